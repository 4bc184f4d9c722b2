// How a kernel reports to the host.
#pragma once

namespace ckv {

// Two words of host-mapped memory and a counter of this GPU's.  *bad becomes 1 on bad news, and *done (if not null; the word behind
// *bad, the two eight-byte aligned) at the kernel's end, which the host sees some microseconds before a stream synchronise
// returns.  `count` is zero between launches and used by one launch at a time.
struct Report {
    int* bad = nullptr;
    int* done = nullptr;
    unsigned* count = nullptr;
};

#ifdef __CUDACC__
__device__ __forceinline__ unsigned count_block(unsigned* count, unsigned add)
{
    unsigned before;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(before) : "l"(count), "r"(add) : "memory");
    return before;
}
__device__ __forceinline__ void tell_host(const Report& r, bool bad)
{
    *reinterpret_cast<volatile unsigned long long*>(r.bad) = (1ull << 32) | (bad ? 1u : 0u);
}
#endif

#if defined(__CUDACC__) || defined(CKV_REPORT_ON_HOST)
// The end of a kernel that reports, reached by all threads of the n_blocks blocks that take part (at most 65535, block (0, 0)
// among them); `bad` of any thread.
// Every access of theirs to this GPU's memory lies before *done: whoever has seen *done, on any stream, finds what the kernel
// wrote there and may overwrite what it read.  (Not what it writes to memory elsewhere, the host's or a peer's: that takes
// a release of system scope, 1.7 us, or a stream synchronise.)
// The blocks' news travel in the counter's upper half, and the host hears of them in one word with *done: no order
// between two words in its memory is needed (an append 15.1 us with two fences of system scope and an atomic in the kernel's
// last block, 10.2 so; 9.8 if its stores are not waited for, but then a call on another stream may meet them on their way).  Block (0, 0) takes off what the others add, so the last addition itself
// leaves the counter at zero, whichever block's it is, and who has seen *done may give the counter to another launch.
__device__ __forceinline__ void report_done(const Report& r, bool bad, unsigned n_blocks)
{
    if (!r.done) {
        if (bad) *reinterpret_cast<volatile int*>(r.bad) = 1;
        return;
    }
    bad = __syncthreads_or(bad);
    if (threadIdx.x != 0) return;
    if (n_blocks > 1) {
        const unsigned add = ((blockIdx.x | blockIdx.y) == 0 ? 1u - n_blocks : 1u) + (bad ? 0x10000u : 0u);
        const unsigned now = count_block(r.count, add) + add;
        if (now & 0xffffu) return;
        bad = now != 0;
        if (bad) {
            *r.count = 0;
            __threadfence();
        }
    } else {
        __threadfence();
    }
    tell_host(r, bad);
}
#endif

}  // namespace ckv
