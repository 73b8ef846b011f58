// A stand-in for the CUDA runtime, linked under the library's host code so
// that its routes, workspaces and error returns can be checked without a GPU:
// memory is host memory, kernels are logged instead of run, and a test can
// make a call fail (see host_library.py).
#include <cuda_runtime_api.h>
#include <sys/mman.h>

#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

namespace {

struct Kernel {
    std::string name;
    size_t limit = 44 * 1024;   // dynamic shared memory a launch may ask for (48 KB less what a kernel has of its own)
};
struct Launch {
    std::string name;
    size_t smem;
    unsigned grid, cluster;
};

std::mutex mu;
std::map<const void *, Kernel> kernels;
std::vector<Launch> launches;
std::map<void *, size_t> blocks;
std::map<std::string, long long> knobs = {
    {"clusters", 8},         // clusters that can be resident
    {"refuse_clusters", 0},  // launches of a cluster fail
    {"no_blocks", 0},        // no CTA can be resident
    {"capturing", 0},        // streams are being captured
    {"sms", 152}};
long long frees = 0;
cudaError_t last = cudaSuccess;
struct Config {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
};
thread_local std::vector<Config> pushed;

cudaError_t done(cudaError_t e)
{
    if (e != cudaSuccess) last = e;
    return e;
}

cudaError_t launch(const void *f, dim3 grid, size_t smem, unsigned cluster)
{
    std::lock_guard<std::mutex> lock(mu);
    auto it = kernels.find(f);
    if (it == kernels.end()) return done(cudaErrorInvalidDeviceFunction);
    if (smem > it->second.limit) return done(cudaErrorInvalidValue);
    if (cluster > 1 && knobs["refuse_clusters"]) return done(cudaErrorLaunchOutOfResources);
    launches.push_back({it->second.name, smem, grid.x, cluster});
    return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- what a test reads and sets
void fake_set(const char *knob, long long v) { std::lock_guard<std::mutex> lock(mu); knobs[knob] = v; }
void fake_clear() { std::lock_guard<std::mutex> lock(mu); launches.clear(); }
int fake_launches() { return (int)launches.size(); }
const char *fake_launch_name(int k) { return launches[k].name.c_str(); }
long long fake_frees() { return frees; }
long long fake_held()
{
    long long b = 0;
    for (auto &m : blocks) b += (long long)m.second;
    return b;
}
// the limit of every kernel whose name holds `part`: the smallest of them
long long fake_limit(const char *part)
{
    long long v = -1;
    for (auto &k : kernels)
        if (k.second.name.find(part) != std::string::npos && (v < 0 || (long long)k.second.limit < v))
            v = (long long)k.second.limit;
    return v;
}

// ---- registration and launches
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *)
{
    std::lock_guard<std::mutex> lock(mu);
    kernels[host].name = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st *stream)
{
    pushed.push_back({grid, block, smem, stream});
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream)
{
    const Config c = pushed.back();
    pushed.pop_back();
    *grid = c.grid;
    *block = c.block;
    *smem = c.smem;
    *static_cast<cudaStream_t *>(stream) = c.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f)
{
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void **, size_t smem, cudaStream_t)
{
    return launch((const void *)k, grid, smem, 1);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **)
{
    unsigned cluster = 1;
    for (unsigned k = 0; k < c->numAttrs; ++k)
        if (c->attrs[k].id == cudaLaunchAttributeClusterDimension) cluster = c->attrs[k].val.clusterDim.x;
    return launch(f, c->gridDim, c->dynamicSmemBytes, cluster);
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v)
{
    std::lock_guard<std::mutex> lock(mu);
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
        if (v > 227 * 1024) return done(cudaErrorInvalidValue);
        kernels[f].limit = (size_t)v;
    }
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int, size_t smem, unsigned)
{
    std::lock_guard<std::mutex> lock(mu);
    *n = 0;
    if (smem > kernels[f].limit) return done(cudaErrorInvalidValue);
    *n = knobs["no_blocks"] ? 0 : smem ? (int)(227 * 1024 / smem) : 8;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *)
{
    *n = (int)knobs["clusters"];
    return cudaSuccess;
}

// ---- memory
cudaError_t cudaMalloc(void **p, size_t bytes)
{
    std::lock_guard<std::mutex> lock(mu);
    if (bytes == 0) bytes = 1;
    *p = mmap(nullptr, bytes, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (*p == MAP_FAILED) return done(cudaErrorMemoryAllocation);
    blocks[*p] = bytes;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    std::lock_guard<std::mutex> lock(mu);
    if (!p) return cudaSuccess;
    ++frees;
    munmap(p, blocks[p]);
    blocks.erase(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t bytes, unsigned)
{
    *p = calloc(1, bytes);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *s) { *p = const_cast<void *>(s); return cudaSuccess; }

// ---- device, streams, events, graphs
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int)
{
    *v = a == cudaDevAttrMultiProcessorCount          ? (int)knobs["sms"]
         : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 227 * 1024
                                                        : 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s)
{
    *s = knobs["capturing"] ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)malloc(8); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)malloc(8); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return done(cudaErrorNotSupported); }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { *g = nullptr; return done(cudaErrorNotSupported); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *, cudaGraph_t, unsigned long long) { return done(cudaErrorNotSupported); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return done(cudaErrorNotSupported); }

}  // extern "C"
