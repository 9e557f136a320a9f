// A CUDA runtime without a device, for tests of the host code on the CPU: "device" memory
// is host memory, copies and fills run at once, kernels do nothing.  Every operation on a
// stream counts as pending until that stream or the device is synchronised, so that a
// free that is not ordered after the work before it can be told (fake_unordered_frees).
// Loaded with global symbols ahead of the library under test; what it does not define
// comes from the real runtime.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <set>
#include <string>
#include <vector>

namespace {

struct Block {
    size_t bytes;
    bool pooled;
};
struct Launch {
    std::string name;
    dim3 grid, block;
    size_t smem;
};
std::mutex mu;
std::map<char*, Block> live;
std::set<cudaStream_t> pending;   // streams with work since their last synchronisation
std::map<const void*, std::string> names;
std::vector<Launch> launches;
size_t capacity = ~size_t(0), live_bytes = 0;
size_t kept = 0;                  // freed pool memory not given back yet
size_t kept_pending = 0;          // the part of it whose free a stream has not passed yet
long long fail_in = -1;
int unordered = 0, capturing = 0;
cudaError_t last = cudaSuccess;
dim3 cfg_grid, cfg_block;
size_t cfg_smem;
cudaStream_t cfg_stream;

cudaError_t set(cudaError_t e) {
    if (e != cudaSuccess) last = e;
    return e;
}
cudaError_t alloc(void** p, size_t bytes, bool pooled) {
    if (fail_in == 0) return set(cudaErrorMemoryAllocation);
    if (fail_in > 0) --fail_in;
    // pool memory serves the next pool allocation first
    const size_t reuse = pooled ? (bytes < kept - kept_pending ? bytes : kept - kept_pending) : 0;
    if (live_bytes + kept - reuse + bytes > capacity) return set(cudaErrorMemoryAllocation);
    char* q = static_cast<char*>(malloc(bytes ? bytes : 1));
    kept -= reuse;
    live[q] = {bytes, pooled};
    live_bytes += bytes;
    *p = q;
    return cudaSuccess;
}
void drop(void* p) {
    auto it = live.find(static_cast<char*>(p));
    if (it == live.end()) abort();   // freed twice, or never allocated
    live_bytes -= it->second.bytes;
    if (it->second.pooled) kept += it->second.bytes, kept_pending += it->second.bytes;
    free(it->first);
    live.erase(it);
}

}  // namespace

extern "C" {

// ---- what a test sets and reads
void fake_set_capturing(int on) { capturing = on; }
void fake_set_capacity(size_t bytes) { capacity = bytes; }
void fake_fail_alloc(long long after) { fail_in = after; }   // all after `after` more fail (-1: none)
int fake_unordered_frees() { return unordered; }
size_t fake_live_bytes() { return live_bytes; }
size_t fake_kept_bytes() { return kept; }
int fake_pending() { return (int)pending.size(); }
int fake_launches() { return (int)launches.size(); }
void fake_clear_launches() { launches.clear(); }
const char* fake_launch(int i, unsigned* dims, size_t* smem) {
    const Launch& l = launches[i];
    const unsigned d[6] = {l.grid.x, l.grid.y, l.grid.z, l.block.x, l.block.y, l.block.z};
    memcpy(dims, d, sizeof d);
    *smem = l.smem;
    return l.name.c_str();
}

// ---- memory
cudaError_t cudaMalloc(void** p, size_t n) {
    std::lock_guard<std::mutex> g(mu);
    return alloc(p, n, false);
}
cudaError_t cudaFree(void* p) {   // waits for the device
    std::lock_guard<std::mutex> g(mu);
    if (!p) return cudaSuccess;
    if (capturing) return set(cudaErrorStreamCaptureUnsupported);
    pending.clear();
    drop(p);
    return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) {
    std::lock_guard<std::mutex> g(mu);
    return alloc(p, n, true);
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t s) {
    std::lock_guard<std::mutex> g(mu);
    for (cudaStream_t t : pending) unordered += t != s;
    drop(p);
    return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t* pool, const cudaMemPoolProps*) {
    *pool = reinterpret_cast<cudaMemPool_t>(&kept);
    return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) {
    std::lock_guard<std::mutex> g(mu);
    kept = kept_pending;   // only frees that a synchronisation has passed
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    std::lock_guard<std::mutex> g(mu);
    memset(a, 0, sizeof *a);
    auto it = live.upper_bound(static_cast<char*>(const_cast<void*>(p)));
    const bool in = it != live.begin() && (--it, static_cast<const char*>(p) < it->first + it->second.bytes);
    a->type = in ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
    a->devicePointer = in ? const_cast<void*>(p) : nullptr;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* src, size_t n, cudaMemcpyKind, cudaStream_t s) {
    std::lock_guard<std::mutex> g(mu);
    memmove(d, src, n);
    pending.insert(s);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t s) {
    std::lock_guard<std::mutex> g(mu);
    memset(d, v, n);
    pending.insert(s);
    return cudaSuccess;
}

// ---- devices, streams, events
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int d) { return d == 0 ? cudaSuccess : set(cudaErrorInvalidDevice); }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 1, cudaSuccess; }
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
cudaError_t cudaDeviceSynchronize() {
    std::lock_guard<std::mutex> g(mu);
    if (capturing) return set(cudaErrorStreamCaptureUnsupported);
    pending.clear();
    kept_pending = 0;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    std::lock_guard<std::mutex> g(mu);
    pending.erase(s);
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) {
    *c = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    static char ids[1024];
    static int n = 0;
    *s = reinterpret_cast<cudaStream_t>(&ids[n++ % 1024]);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = reinterpret_cast<cudaEvent_t>(&last), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.f, cudaSuccess; }

// ---- kernels: recorded, not run
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
void** __cudaRegisterFatBinary(void*) {
    static void* handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) {
    names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t s) {
    cfg_grid = grid, cfg_block = block, cfg_smem = smem, cfg_stream = s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
    *grid = cfg_grid, *block = cfg_block, *smem = cfg_smem, *static_cast<cudaStream_t*>(s) = cfg_stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void**, size_t smem, cudaStream_t s) {
    std::lock_guard<std::mutex> g(mu);
    launches.push_back({names[reinterpret_cast<const void*>(k)], grid, block, smem});
    pending.insert(s);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
    return __cudaLaunchKernel(reinterpret_cast<cudaKernel_t>(const_cast<void*>(f)), c->gridDim, c->blockDim, args,
                              c->dynamicSmemBytes, c->stream);
}

}  // extern "C"
