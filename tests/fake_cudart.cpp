// A CUDA runtime without a GPU: the library's object files linked with this instead of libcudart run their whole host side
// on the CPU.  Device memory is host memory, copies happen at once, kernels do not run; every call is counted by name and a
// call can be made to fail.
#include <cuda_runtime.h>

#include <atomic>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#define API extern "C" __attribute__((visibility("default")))

namespace {
std::mutex mu;
std::map<std::string, long> counts, fail_at;        // calls so far; the call that fails (counted from the reset)
std::map<const char*, size_t> device_blocks, host_blocks;
thread_local bool has_context = false;                // as made by the calls that need one, and by cudaSetDevice
long launched[6];                                    // of the last cudaLaunchKernelExC: grid, threads, shared memory, cluster

cudaError_t called(const char* name)
{
    if (!std::strcmp(name, "cudaSetDevice") || !std::strcmp(name, "cudaMalloc") || !std::strncmp(name, "cudaLaunch", 10) ||
        !std::strncmp(name, "cudaMem", 7) || !std::strncmp(name, "cudaStream", 10))
        has_context = true;
    std::lock_guard<std::mutex> lock(mu);
    const long n = ++counts[name];
    auto f = fail_at.find(name);
    return f != fail_at.end() && f->second == n ? cudaErrorMemoryAllocation : cudaSuccess;
}
#define CALLED() do { const cudaError_t e_ = called(__func__); if (e_ != cudaSuccess) return e_; } while (0)

cudaError_t take(void** p, size_t bytes, bool device)
{
    *p = std::aligned_alloc(512, (bytes + 511) / 512 * 512 + 512);
    std::lock_guard<std::mutex> lock(mu);
    (device ? device_blocks : host_blocks)[(const char*)*p] = bytes;
    return cudaSuccess;
}
cudaError_t give(void* p, std::map<const char*, size_t>& blocks)
{
    std::lock_guard<std::mutex> lock(mu);
    blocks.erase((const char*)p);
    std::free(p);
    return cudaSuccess;
}
bool holds(const std::map<const char*, size_t>& blocks, const char* p)
{
    auto it = blocks.upper_bound(p);
    return it != blocks.begin() && p < std::prev(it)->first + std::prev(it)->second;
}
int encode(...) { return has_context ? 0 : 201; }      // cuTensorMapEncodeTiled: CUDA_ERROR_INVALID_CONTEXT
}  // namespace

API long fake_count(const char* name)
{
    std::lock_guard<std::mutex> lock(mu);
    return counts[name];
}
API void fake_reset()
{
    std::lock_guard<std::mutex> lock(mu);
    counts.clear();
    fail_at.clear();
}
API void fake_fail(const char* name, long nth)
{
    std::lock_guard<std::mutex> lock(mu);
    fail_at[name] = counts[name] + nth;
}
API void fake_device_reset()  // what the runtime has allocated is gone
{
    std::lock_guard<std::mutex> lock(mu);
    device_blocks.clear();
    host_blocks.clear();
}
API const long* fake_launched() { return launched; }

// ---- the runtime calls the library makes
API cudaError_t cudaMalloc(void** p, size_t n) { CALLED(); return take(p, n, true); }
API cudaError_t cudaFree(void* p) { CALLED(); return give(p, device_blocks); }
API cudaError_t cudaMallocHost(void** p, size_t n) { CALLED(); return take(p, n, false); }
API cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { CALLED(); return take(p, n, false); }
API cudaError_t cudaFreeHost(void* p) { CALLED(); return give(p, host_blocks); }
API cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { CALLED(); std::memcpy(d, s, n); return cudaSuccess; }
API cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { CALLED(); std::memcpy(d, s, n); return cudaSuccess; }
API cudaError_t cudaMemset(void* d, int v, size_t n) { CALLED(); std::memset(d, v, n); return cudaSuccess; }
API cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p)
{
    CALLED();
    std::memset(a, 0, sizeof *a);
    std::lock_guard<std::mutex> lock(mu);
    a->type = holds(device_blocks, (const char*)p) ? cudaMemoryTypeDevice
              : holds(host_blocks, (const char*)p) ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered;
    return cudaSuccess;
}
API cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
API cudaError_t cudaGetDevice(int* d) { CALLED(); *d = 0; return cudaSuccess; }
API cudaError_t cudaSetDevice(int) { CALLED(); return cudaSuccess; }
API cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int)
{
    CALLED();
    *v = a == cudaDevAttrMultiProcessorCount ? 148 : a == cudaDevAttrMaxPersistingL2CacheSize || a == cudaDevAttrMaxAccessPolicyWindowSize ? 64 << 20 : 0;
    return cudaSuccess;
}
API cudaError_t cudaDeviceGetLimit(size_t* v, cudaLimit) { *v = 0; return cudaSuccess; }
API cudaError_t cudaDeviceSetLimit(cudaLimit, size_t) { return cudaSuccess; }
API cudaError_t cudaCtxResetPersistingL2Cache() { return cudaSuccess; }
API cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { CALLED(); return cudaSuccess; }
API cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)(uintptr_t)16; return cudaSuccess; }
API cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
API cudaError_t cudaStreamSynchronize(cudaStream_t) { CALLED(); return cudaSuccess; }
API cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
API cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)(uintptr_t)16; return cudaSuccess; }
API cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)(uintptr_t)16; return cudaSuccess; }
API cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
API cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
API cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
API cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0; return cudaSuccess; }
API cudaError_t cudaGetLastError() { return cudaSuccess; }
API const char* cudaGetErrorName(cudaError_t) { return "fake"; }
API const char* cudaGetErrorString(cudaError_t) { return "fake"; }
API cudaError_t cudaGetSymbolAddress(void** p, const void*) { static char block[8 << 20]; *p = block; return cudaSuccess; }
API cudaError_t cudaGetDriverEntryPoint(const char*, void** fn, unsigned long long, cudaDriverEntryPointQueryResult* q)
{
    *fn = (void*)&encode;
    if (q) *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
API cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { CALLED(); return cudaSuccess; }
API cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void*, void**)
{
    CALLED();
    std::lock_guard<std::mutex> lock(mu);
    const long now[6] = {c->gridDim.x, c->gridDim.y, c->gridDim.z, c->blockDim.x, (long)c->dynamicSmemBytes, 1};
    std::memcpy(launched, now, sizeof now);
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) launched[5] = c->attrs[i].val.clusterDim.x;
    return cudaSuccess;
}
API unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
API cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st)
{
    *g = *b = dim3(1);
    *s = 0;
    *(void**)st = nullptr;
    return cudaSuccess;
}
API void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
API void __cudaRegisterFatBinaryEnd(void**) {}
API void __cudaUnregisterFatBinary(void**) {}
API void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
API void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}

// What planning a request list cannot do without, for a test to measure a call against: n look-ups through the public call, a
// 40-byte request and a 16-byte item each, and their copies on the way to the device.
API int fake_plan_floor(int (*user_length)(void*, long, long*), void* ctx, int n, const long* users, const int* q_off)
{
    struct Req { long base; int v[8]; };
    struct Item { int v[4]; };
    static std::vector<char> host, device;
    static std::vector<long> users_kept;
    static std::vector<int> q_off_kept;
    host.resize((sizeof(Req) + sizeof(Item)) * n);
    device.resize(host.size());
    std::vector<Req> reqs(n);
    for (int k = 0; k < n; ++k) {
        long L = 0;
        if (int st = user_length(ctx, users[k], &L)) return st;
        reqs[k] = Req{k, {(int)L, (int)L, q_off[k], q_off[k + 1] - q_off[k], -1, 1}};
    }
    std::vector<Item> items;
    items.reserve(n);
    for (int k = 0; k < n; ++k) items.push_back(Item{{k, 0, reqs[k].v[0], -1}});
    std::vector<unsigned> order(n);
    for (int k = 0; k < n; ++k) order[k] = k;
    std::memcpy(host.data(), reqs.data(), sizeof(Req) * n);
    Item* to = (Item*)(host.data() + sizeof(Req) * n);
    for (int k = 0; k < n; ++k) to[k] = items[order[k]];
    std::memcpy(device.data(), host.data(), host.size());
    users_kept.assign(users, users + n);
    q_off_kept.assign(q_off, q_off + n + 1);
    return 0;
}
