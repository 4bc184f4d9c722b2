// Prefill router (Sec. 4.3): which global-pool entry a history position selects,
//     I[i][g] = argmin { j : M_ij maximal },   M = X W_g^T + b_g,
// for n positions with d_in-wide inputs X (bf16), per group g a weight matrix W_g stored entry-major
// ([n_entries][d_in] bf16: an entry's weights are contiguous, like a pool row) and an optional fp32 bias.
// The score matrix M (n x n_entries) is never written: every warp keeps the running best (value, entry) of its
// rows in registers while the entries stream through shared memory.
//
// One CTA = 8 warps x 32 positions; the positions' inputs stay in registers as m16n8k16 A fragments.  The group's
// weight rows go through a two-slot shared-memory ring in chunks of 64 entries (cp.async by the whole CTA, rows
// swizzled for ldmatrix), each chunk used by all eight warps.  Products are exact (bf16 x bf16), sums fp32.
#include <cuda_bf16.h>
#include <math_constants.h>

#include "ckv_internal.h"
#include "ptx_helpers.cuh"

namespace ckv {
namespace {

constexpr int kRouteWarps = 8, kRouteChunk = 64;
// 16-position tiles per warp: every weight fragment read from shared memory serves that many MMAs
__host__ __device__ constexpr int route_mt(int) { return 2; }  // (four measured no faster: 334 against 342 TFLOP/s)
__host__ __device__ constexpr int route_rows(int d_in) { return kRouteWarps * 16 * route_mt(d_in); }  // positions per CTA

// 16-byte chunk c of ring row r sits at chunk c ^ swz(r): the eight rows of an ldmatrix block (consecutive
// entries) fall into eight different bank groups
template <int DIN>
__device__ __forceinline__ int swz(int r)
{
    return DIN == 32 ? ((r >> 1) & 3) : (r & 7);
}

template <int DIN>
__global__ void __launch_bounds__(kRouteWarps * 32)
    route_kernel(const uint16_t* __restrict__ x, const uint16_t* __restrict__ W, const float* __restrict__ bias, int n,
                 int m, int G, int32_t* __restrict__ out)
{
    constexpr int KS = DIN / 16, MT = route_mt(DIN), ROWB = DIN * 2, CPR = ROWB / 16, CH = kRouteChunk;
    constexpr int SLOT_B = CH * ROWB;
    extern __shared__ __align__(128) unsigned char rsm[];
    float* bias_s = reinterpret_cast<float*>(rsm + 2 * SLOT_B);  // [2][CH]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gl = lane >> 2, t = lane & 3;
    const int grp = blockIdx.y;
    const int64_t row0 = (int64_t)blockIdx.x * route_rows(DIN) + warp * (16 * MT);
    const uint16_t* Wg = W + (int64_t)grp * m * DIN;
    const float* bg = bias ? bias + (int64_t)grp * m : nullptr;

    uint32_t qa[MT][KS][4];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
        const int64_t r_lo = row0 + 16 * mt + gl, r_hi = r_lo + 8;
        const uint16_t* p_lo = x + r_lo * DIN;
        const uint16_t* p_hi = x + r_hi * DIN;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
            const int c = 16 * ks + 2 * t;
            qa[mt][ks][0] = r_lo < n ? __ldg(reinterpret_cast<const uint32_t*>(p_lo + c)) : 0u;
            qa[mt][ks][1] = r_hi < n ? __ldg(reinterpret_cast<const uint32_t*>(p_hi + c)) : 0u;
            qa[mt][ks][2] = r_lo < n ? __ldg(reinterpret_cast<const uint32_t*>(p_lo + c + 8)) : 0u;
            qa[mt][ks][3] = r_hi < n ? __ldg(reinterpret_cast<const uint32_t*>(p_hi + c + 8)) : 0u;
        }
    }
    float bv[MT][2];
    int bi[MT][2];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
        bv[mt][0] = bv[mt][1] = -CUDART_INF_F;
        bi[mt][0] = bi[mt][1] = 0;
    }

    const uint32_t ring = smem_u32(rsm);
    auto stage = [&](int c) {  // entries 64 c .. 64 c + 63 into slot c & 1 (past the last entry: the last row, bias -inf)
        const int slot = c & 1, j0 = c * CH;
        for (int q = tid; q < CH * CPR; q += kRouteWarps * 32) {
            const int r = q / CPR, cc = q - r * CPR;
            const int j = min(j0 + r, m - 1);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ring + slot * SLOT_B + r * ROWB +
                                                                          ((cc ^ swz<DIN>(r)) << 4)),
                         "l"(Wg + (int64_t)j * DIN + cc * 8)
                         : "memory");
        }
        if (tid < CH) {
            const int j = j0 + tid;
            bias_s[slot * CH + tid] = j < m ? (bg ? __ldg(bg + j) : 0.f) : -CUDART_INF_F;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // ldmatrix row addresses of this lane: matrix lane >> 3 = 16-byte chunk within a k-step pair, row lane & 7
    const int lr = lane & 7, lm = lane >> 3;
    uint32_t offB[KS / 2];
#pragma unroll
    for (int kp = 0; kp < KS / 2; ++kp) offB[kp] = lr * ROWB + ((((4 * kp + lm) ^ swz<DIN>(lr)) & (CPR - 1)) << 4);

    const int nch = (m + CH - 1) / CH;
    stage(0);
    for (int c = 0; c < nch; ++c) {
        if (c + 1 < nch) {
            stage(c + 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const uint32_t wt = ring + (c & 1) * SLOT_B;
        const float* bs = bias_s + (c & 1) * CH;
#pragma unroll 2
        for (int nt = 0; nt < CH / 8; ++nt) {
            uint32_t b[KS][2];
#pragma unroll
            for (int kp = 0; kp < KS / 2; ++kp)
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                             : "=r"(b[2 * kp][0]), "=r"(b[2 * kp][1]), "=r"(b[2 * kp + 1][0]), "=r"(b[2 * kp + 1][1])
                             : "r"(wt + nt * (8 * ROWB) + offB[kp])
                             : "memory");
            const int j = c * CH + 8 * nt + 2 * t;  // entries of this lane's two accumulator columns
            const float b0 = bs[8 * nt + 2 * t], b1 = bs[8 * nt + 2 * t + 1];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int ks = 0; ks < KS; ++ks) mma_bf16(acc, qa[mt][ks], b[ks][0], b[ks][1]);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float v0 = acc[2 * h] + b0, v1 = acc[2 * h + 1] + b1;
                    // entries arrive in increasing order: a strict comparison keeps the lowest entry among equals;
                    // a new best gets rare quickly, so one test of the pair's maximum guards the update
                    if (fmaxf(v0, v1) > bv[mt][h]) {
                        const bool first = v0 >= v1;
                        bv[mt][h] = first ? v0 : v1;
                        bi[mt][h] = first ? j : j + 1;
                    }
                }
            }
        }
        __syncthreads();  // everyone is done with this slot before the chunk after next is staged into it
    }
    // the four lanes of a row hold disjoint entries: best of them, lowest entry among equals
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float v = bv[mt][h];
            int i = bi[mt][h];
#pragma unroll
            for (int o = 1; o <= 2; o <<= 1) {
                const float v2 = __shfl_xor_sync(0xffffffffu, v, o);
                const int i2 = __shfl_xor_sync(0xffffffffu, i, o);
                if (v2 > v || (v2 == v && i2 < i)) {
                    v = v2;
                    i = i2;
                }
            }
            const int64_t r = row0 + 16 * mt + gl + 8 * h;
            if (t == 0 && r < n) out[r * G + grp] = i;
        }
}

template <int DIN>
cudaError_t launch_route_t(const void* x, const void* W, const float* bias, int n, int m, int G, int32_t* out,
                           cudaStream_t s)
{
    const size_t smem = 2 * (size_t)kRouteChunk * DIN * 2 + 2 * kRouteChunk * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(route_kernel<DIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((n + route_rows(DIN) - 1) / route_rows(DIN)), (unsigned)G);
    route_kernel<DIN><<<grid, kRouteWarps * 32, smem, s>>>((const uint16_t*)x, (const uint16_t*)W, bias, n, m, G, out);
    return cudaGetLastError();
}

// Few positions: 32 per block, and its eight warps (of up to eight blocks of a cluster) share the entries, each a run of
// consecutive tiles of eight.  Entry rows go from L2 into the B fragments by 16-byte loads, no shared memory: lane (g, t)
// holds pieces t, t + 4, ... of entry g's row, so that the feature order of the dot product is permuted, in both operands
// alike.  The next four tiles are requested before the four at hand are worked on.  What bounds it is latency, a launch and
// the report to the host included (the tcgen05 kernel has TMEM, barriers, tensor maps and a pipeline to set up first), and
// with more positions the weights, which every block of 32 reads from L2 for itself.
constexpr int kFewRows = 32, kFewWarps = 8, kFewMaxSplit = 8, kFewBatch = 4;
constexpr int kFewBlocks = 2 * 148;  // see route_few

__device__ unsigned few_count[kRouteSlots];  // finished blocks of the launch that holds the slot, zero between launches

template <int DIN>
__global__ void __launch_bounds__(kFewWarps * 32, DIN == 128 ? 1 : 2)
    route_few_kernel(const uint16_t* __restrict__ x, const uint16_t* __restrict__ W, const float* __restrict__ bias, int n,
                     int m, int G, int32_t* __restrict__ out, int* flags, int slot, int n_split)
{
    constexpr int PIECES = DIN / 32, MT = kFewRows / 16, B = kFewBatch;
    __shared__ float2 found[kFewWarps][kFewRows];  // (score, entry) of a warp; row 0: of the block
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int grp = blockIdx.y, split = (int)(blockIdx.x % (uint32_t)n_split);
    const int64_t row0 = (int64_t)(blockIdx.x / (uint32_t)n_split) * kFewRows;
    const uint16_t* Wg = W + (int64_t)grp * m * DIN;
    const float* bg = bias ? bias + (int64_t)grp * m : nullptr;
    const int tiles = (m + 7) / 8, parts = kFewWarps * n_split, part = split * kFewWarps + warp;
    const int first = (int)((int64_t)tiles * part / parts), end = (int)((int64_t)tiles * (part + 1) / parts);

    uint4 w[B][PIECES];
    float b0[B], b1[B];
    auto fetch = [&](int tile) {  // tiles `tile` .. + B - 1 (past the last entry: the last row, bias -inf)
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const int j = min(8 * (tile + i) + g, m - 1), c = 8 * (tile + i) + 2 * t;
#pragma unroll
            for (int q = 0; q < PIECES; ++q) w[i][q] = __ldg(reinterpret_cast<const uint4*>(Wg + (int64_t)j * DIN) + t + 4 * q);
            b0[i] = c < m ? (bg ? __ldg(bg + c) : 0.f) : -CUDART_INF_F;
            b1[i] = c + 1 < m ? (bg ? __ldg(bg + c + 1) : 0.f) : -CUDART_INF_F;
        }
    };
    if (first < end) fetch(first);
    uint4 xa[MT][2][PIECES];  // rows g and g + 8 of each tile of sixteen positions
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t r = row0 + 16 * mt + 8 * h + g;
#pragma unroll
            for (int q = 0; q < PIECES; ++q)
                xa[mt][h][q] = r < n ? __ldg(reinterpret_cast<const uint4*>(x + r * DIN) + t + 4 * q) : make_uint4(0, 0, 0, 0);
        }
    float bv[MT][2];
    int bi[MT][2];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
        bv[mt][0] = bv[mt][1] = -CUDART_INF_F;
        bi[mt][0] = bi[mt][1] = 0;
    }
    for (int tile = first; tile < end; tile += B) {
        uint4 cw[B][PIECES];
        float c0[B], c1[B];
#pragma unroll
        for (int i = 0; i < B; ++i) {
#pragma unroll
            for (int q = 0; q < PIECES; ++q) cw[i][q] = w[i][q];
            c0[i] = b0[i];
            c1[i] = b1[i];
        }
        if (tile + B < end) fetch(tile + B);
#pragma unroll
        for (int i = 0; i < B; ++i) {
            if (tile + i >= end) break;
            const int j = 8 * (tile + i) + 2 * t;  // entries of this lane's two accumulator columns
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int q = 0; q < PIECES; ++q) {
                    const uint4 lo = xa[mt][0][q], hi = xa[mt][1][q];
                    const uint32_t a0[4] = {lo.x, hi.x, lo.y, hi.y}, a1[4] = {lo.z, hi.z, lo.w, hi.w};
                    mma_bf16(acc, a0, cw[i][q].x, cw[i][q].y);
                    mma_bf16(acc, a1, cw[i][q].z, cw[i][q].w);
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    // entries come in increasing order: a strict comparison keeps the lowest among equals, and a score that
                    // is not a number is never taken
                    const float v0 = acc[2 * h] + c0[i], v1 = acc[2 * h + 1] + c1[i];
                    if (v0 > bv[mt][h]) {
                        bv[mt][h] = v0;
                        bi[mt][h] = j;
                    }
                    if (v1 > bv[mt][h]) {
                        bv[mt][h] = v1;
                        bi[mt][h] = j + 1;
                    }
                }
            }
        }
    }
    // the lanes of a row, the warps of the block and the blocks of the cluster hold disjoint entries: the best of them, the
    // lowest entry among equals
    auto better = [](float v2, int i2, float v, int i) { return v2 > v || (v2 == v && i2 < i); };
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float v = bv[mt][h];
            int i = bi[mt][h];
#pragma unroll
            for (int o = 1; o <= 2; o <<= 1) {
                const float v2 = __shfl_xor_sync(0xffffffffu, v, o);
                const int i2 = __shfl_xor_sync(0xffffffffu, i, o);
                if (better(v2, i2, v, i)) {
                    v = v2;
                    i = i2;
                }
            }
            if (t == 0) found[warp][16 * mt + 8 * h + g] = make_float2(v, __int_as_float(i));
        }
    __syncthreads();
    float v = 0.f;
    int i = 0;
    if (warp == 0) {
        v = found[0][lane].x;
        i = __float_as_int(found[0][lane].y);
#pragma unroll
        for (int k = 1; k < kFewWarps; ++k) {
            const float2 f = found[k][lane];
            if (better(f.x, __float_as_int(f.y), v, i)) {
                v = f.x;
                i = __float_as_int(f.y);
            }
        }
        found[0][lane] = make_float2(v, __int_as_float(i));
    }
    if (n_split > 1) {
        asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (split == 0 && warp == 0) {
            for (int r = 1; r < n_split; ++r) {
                uint32_t remote;
                float v2, i2;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(&found[0][lane])), "r"(r));
                asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v2), "=f"(i2) : "r"(remote) : "memory");
                if (better(v2, __float_as_int(i2), v, i)) {
                    v = v2;
                    i = __float_as_int(i2);
                }
            }
        }
        asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    if (warp == 0 && split == 0 && row0 + lane < n) out[(row0 + lane) * G + grp] = i;
    if (slot >= 0 && split == 0) report_done(Report{flags, flags + 1, &few_count[slot]}, false, gridDim.x / (unsigned)n_split * gridDim.y);
}

template <int DIN>
cudaError_t launch_route_few_t(const void* x, const void* W, const float* bias, int n, int m, int G, int32_t* out, int* flags,
                               int* slot, cudaStream_t s)
{
    const int64_t blocks = (int64_t)((n + kFewRows - 1) / kFewRows) * G;
    const int tiles = (m + 7) / 8;
    // a cluster's blocks share the entries as long as there are SMs for them and each warp keeps two batches
    const int resident = DIN == 128 ? 148 : kFewBlocks;
    int split = 1;
    while (split < kFewMaxSplit && blocks * split * 2 <= resident && tiles >= 2 * split * kFewWarps * 2 * kFewBatch) split *= 2;
    const dim3 grid((unsigned)((n + kFewRows - 1) / kFewRows * split), (unsigned)G);
    if (blocks * split > resident) *slot = -1;
    return launch_kernel(Launch{s, nullptr, nullptr}, route_few_kernel<DIN>, grid, kFewWarps * 32, 0, split, (const uint16_t*)x,
                         (const uint16_t*)W, bias, n, m, G, out, flags, *slot, split);
}

// User-specific low-dimensional projection of the prefill (Sec. 4.2): y[i][g][c] = x_i . W[g][c] + b[g][c],
// d_out <= 16 outputs per group.  Memory-bound: one thread per output element, the weights in shared memory
// (rows padded by 16 bytes against bank conflicts), 16-byte loads of the input row, fp32 sums, bf16 result.
__global__ void __launch_bounds__(256) project_kernel(const uint16_t* __restrict__ x, const uint16_t* __restrict__ W,
                                                      const float* __restrict__ bias, int64_t total, int d_in, int gd,
                                                      uint16_t* __restrict__ out)
{
    extern __shared__ __align__(16) unsigned char psm[];
    const int wrow = d_in * 2 + 16;  // bytes per padded weight row
    for (int q = threadIdx.x; q < gd * (d_in / 8); q += blockDim.x) {
        const int r = q / (d_in / 8), c = q - r * (d_in / 8);
        *reinterpret_cast<uint4*>(psm + r * wrow + c * 16) = __ldg(reinterpret_cast<const uint4*>(W + (int64_t)r * d_in) + c);
    }
    __syncthreads();
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / gd;
        const int r = (int)(e - i * gd);  // (group, output) row of W
        const uint4* xr = reinterpret_cast<const uint4*>(x + i * d_in);
        const unsigned char* wr = psm + r * wrow;
        float acc = bias ? __ldg(bias + r) : 0.f;
        for (int c = 0; c < d_in / 8; ++c) {
            const uint4 a = __ldg(xr + c), b = *reinterpret_cast<const uint4*>(wr + c * 16);
            const uint32_t aw[4] = {a.x, a.y, a.z, a.w}, bw[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                acc = fmaf(__uint_as_float(aw[k] << 16), __uint_as_float(bw[k] << 16), acc);
                acc = fmaf(__uint_as_float(aw[k] & 0xffff0000u), __uint_as_float(bw[k] & 0xffff0000u), acc);
            }
        }
        out[e] = __bfloat16_as_ushort(__float2bfloat16_rn(acc));
    }
}

}  // namespace

bool route_supported(int d_in) { return d_in == 32 || d_in == 64 || d_in == 128; }

cudaError_t launch_route(int d_in, const void* x, const void* W, const float* bias, int n, int n_entries, int G,
                         int32_t* out, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    switch (d_in) {
        case 32: return launch_route_t<32>(x, W, bias, n, n_entries, G, out, s);
        case 64: return launch_route_t<64>(x, W, bias, n, n_entries, G, out, s);
        default: return launch_route_t<128>(x, W, bias, n, n_entries, G, out, s);
    }
}

// Up to 1.1e9 products: 500 positions x 16384 entries x 2 groups (d_in 64, 1.05e9) 37 us against 42 with the tcgen05 kernel,
// 1000 x 4096 x 4 27 / 32, 2000 x 4096 x 4 (d_in 32) 29 / 34; at 1.3e9 33 / 32 and 39 / 34, at 2.1e9 40 / 42 and 47 / 40 (a call
// and a wait for the stream, before the report; without that wait the line lies in the same place).  And up to 296 blocks of 32
// positions and a group, two for each SM: a small pool leaves most warps of a block without a tile, and every further round of
// blocks costs 1.5 to 3.5 us, where the tcgen05 kernel has 384 positions to a block.  64 entries, 4 groups (d_in 32): 2000
// positions (252 blocks) 11.8 us against 13.7, 3000 (376) 14.9 / 13.5, 10000 20.5 / 14.1, 100000 89 / 41; 1024 entries, 2 groups
// (d_in 64): 2000 15.9 / 17.5, 5000 (314) 23.7 / 18.4; 32 entries, 4 groups (d_in 128, one block per SM): 2000 16.0 / 18.2, 3000
// 18.5 / 18.3, 5000 22.2 / 18.5.
bool route_few(int d_in, const void* x, const void* W, int n, int n_entries, int G)
{
    if (((uintptr_t)x | (uintptr_t)W) & 15) return false;  // rows are read sixteen bytes at a time
    return (double)n * n_entries * G * d_in <= 1.1e9 && ((int64_t)n + kFewRows - 1) / kFewRows * G <= kFewBlocks;
}

cudaError_t launch_route_few(int d_in, const void* x, const void* W, const float* bias, int n, int n_entries, int G,
                             int32_t* out, int* flags, int* slot, cudaStream_t s)
{
    switch (d_in) {
        case 32: return launch_route_few_t<32>(x, W, bias, n, n_entries, G, out, flags, slot, s);
        case 64: return launch_route_few_t<64>(x, W, bias, n, n_entries, G, out, flags, slot, s);
        default: return launch_route_few_t<128>(x, W, bias, n, n_entries, G, out, flags, slot, s);
    }
}

bool project_supported(int d_in, int d_out, int n_groups)
{
    return d_in >= 8 && d_in <= 256 && d_in % 8 == 0 && d_out >= 1 && d_out <= 16 &&
           (size_t)n_groups * d_out * (d_in * 2 + 16) <= 96 * 1024;
}

cudaError_t launch_project(int d_in, int d_out, int G, const void* x, const void* W, const float* bias, int64_t n,
                           void* out, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    const int gd = G * d_out;
    const size_t smem = (size_t)gd * (d_in * 2 + 16);
    cudaError_t e = cudaFuncSetAttribute(project_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int64_t total = n * gd;
    int64_t blocks = (total + 255) / 256;
    if (blocks > 148 * 16) blocks = 148 * 16;
    project_kernel<<<(unsigned)blocks, 256, smem, s>>>((const uint16_t*)x, (const uint16_t*)W, bias, total, d_in, gd,
                                                       (uint16_t*)out);
    return cudaGetLastError();
}

}  // namespace ckv
