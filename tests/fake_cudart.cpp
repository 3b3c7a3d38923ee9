// fake_cudart.cpp - stand-in for the CUDA runtime under the library's host code, for
// tests of what that code calls and in which order (no GPU).  Device memory is host
// memory, copies run at once, kernels do not run.  Every call that a test may ask
// about is a line of the log:
//   kernel S NAME | copy S | set S      work on stream S (0: the default stream)
//   wait S                              the host waits for stream S (device: "wait all")
//   resolve NAME [VALUE]                an attribute of a kernel is set or its occupancy asked for
//   alloc BYTES | begin | end           device allocation; stream capture
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

namespace {
std::mutex mu;
std::string text;
std::map<const void *, std::string> kernels;
std::map<char *, size_t> blocks;          // live device allocations
std::map<void *, int> streams;
int fail_in = 0;                          // > 0: that many allocations from now, one fails
int clusters = 8;                         // what the occupancy query of clusters answers

void add(const std::string &s)
{
    std::lock_guard<std::mutex> g(mu);
    text += s;
    text += '\n';
}
std::string sid(cudaStream_t s)
{
    if (!s || s == cudaStreamLegacy) return "0";
    std::lock_guard<std::mutex> g(mu);
    return std::to_string(streams.emplace(s, (int)streams.size() + 1).first->second);
}
std::string name(const void *f)
{
    std::lock_guard<std::mutex> g(mu);
    auto it = kernels.find(f);
    return it == kernels.end() ? "?" : it->second;
}
template <typename T> cudaError_t take(T **p, size_t n, const char *what)
{
    std::lock_guard<std::mutex> g(mu);
    *p = nullptr;
    if (fail_in > 0 && --fail_in == 0) return cudaErrorMemoryAllocation;
    char *b = static_cast<char *>(aligned_alloc(256, (n + 255) / 256 * 256 + 256));
    memset(b, 0, n);
    blocks[b] = n;
    if (*what) text += std::string(what) + " " + std::to_string(n) + "\n";
    *p = reinterpret_cast<T *>(b);
    return cudaSuccess;
}
void drop(void *p)
{
    std::lock_guard<std::mutex> g(mu);
    blocks.erase(static_cast<char *>(p));
    free(p);
}
cudaError_t move(void *d, const void *s, size_t n)
{
    if (n && (!d || !s)) return cudaErrorInvalidValue;
    memmove(d, s, n);
    return cudaSuccess;
}
struct Config {
    dim3 grid, block;
    size_t smem;
    cudaStream_t st;
};
thread_local Config cfg;
void *handle() { return calloc(1, 16); }
}  // namespace

extern "C" {
const char *fake_log() { return text.c_str(); }
void fake_reset()
{
    text.clear();
    fail_in = 0;
    clusters = 8;
}
void fake_fail_alloc(int k) { fail_in = k; }
void fake_clusters(int n) { clusters = n; }
size_t fake_live_bytes()
{
    size_t n = 0;
    for (auto &b : blocks) n += b.second;
    return n;
}

void **__cudaRegisterFatBinary(void *) { return static_cast<void **>(handle()); }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *dev, int, uint3 *, uint3 *, dim3 *, dim3 *, int *)
{
    std::lock_guard<std::mutex> g(mu);
    kernels[host] = dev;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t st)
{
    cfg = {grid, block, smem, st};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *st)
{
    *grid = cfg.grid;
    *block = cfg.block;
    *smem = cfg.smem;
    *static_cast<cudaStream_t *>(st) = cfg.st;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(void **k, const void *f)
{
    *k = const_cast<void *>(f);
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(void *k, dim3, dim3, void **, size_t, cudaStream_t st)
{
    add("kernel " + sid(st) + " " + name(k));
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **)
{
    add("kernel " + sid(c->stream) + " " + name(f));
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute, int v)
{
    add("resolve " + name(f) + " " + std::to_string(v));
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned)
{
    *n = 2;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *f, const cudaLaunchConfig_t *)
{
    add("resolve " + name(f));
    *n = clusters;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int)
{
    *v = 152;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d)
{
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaDeviceSynchronize()
{
    add("wait all");
    return cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t n) { return take(p, n, "alloc"); }
cudaError_t cudaMallocHost(void **p, size_t n) { return take(p, n, ""); }
cudaError_t cudaFree(void *p)
{
    drop(p);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) { return cudaFree(p); }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind)
{
    add("copy 0");
    return move(d, s, n);
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t st)
{
    add("copy " + sid(st));
    return move(d, s, n);
}
cudaError_t cudaMemset(void *d, int v, size_t n)
{
    add("set 0");
    memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t st)
{
    add("set " + sid(st));
    memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned)
{
    *s = static_cast<cudaStream_t>(handle());
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s)
{
    add("wait " + sid(s));
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode)
{
    add("begin");
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g)
{
    add("end");
    *g = static_cast<cudaGraph_t>(handle());
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long)
{
    *e = static_cast<cudaGraphExec_t>(handle());
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t st)
{
    add("kernel " + sid(st) + " graph");
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e)
{
    *e = static_cast<cudaEvent_t>(handle());
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t)
{
    *ms = 1.0f;
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *)
{
    a->type = cudaMemoryTypeUnregistered;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *)
{
    static char *b = static_cast<char *>(calloc(1, 4 << 20));
    *p = b;
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q)
{
    *f = nullptr;
    if (q) *q = cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *)
{
    *p = static_cast<cudaMemPool_t>(handle());
    return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t, cudaStream_t) { return take(p, n, ""); }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return cudaFree(p); }
}
