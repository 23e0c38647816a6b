// A stand-in for the CUDA runtime calls that libdugks.so makes, for tests of its
// host code on a machine without a GPU: "device" memory is host memory, copies and
// memsets take effect at once, kernels are not run, and every call that orders work
// on a stream is written to a log.  Linked with the library's own object files.
#include <cuda_runtime.h>
#include <sys/mman.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {
struct Rec { std::string op; unsigned long long dst, bytes, stream; };
std::vector<Rec> g_log;
std::map<const void *, std::string> g_names;
std::map<unsigned char *, size_t> g_dev, g_pinned;
int g_capturing = 0;
int *g_late = nullptr;   // a cooperative launch writes 1 here
long g_coop = 0, g_handles = 0x1000;
void add(const char *op, const void *dst = nullptr, size_t bytes = 0, cudaStream_t st = nullptr)
{
    g_log.push_back({op, (unsigned long long)dst, bytes, (unsigned long long)st});
}
bool in(const std::map<unsigned char *, size_t> &m, const void *p)
{
    auto it = m.upper_bound((unsigned char *)p);
    if (it == m.begin()) return false;
    --it;
    return (unsigned char *)p < it->first + it->second;
}
struct Cfg { dim3 g, b; size_t smem; void *st; } g_cfg;
const char *kind_name(cudaMemcpyKind k) { return k == cudaMemcpyHostToDevice ? "h2d" : k == cudaMemcpyDeviceToHost ? "d2h" : "d2d"; }
cudaError_t copy(const char *op, void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t st)
{
    add((std::string(op) + " " + kind_name(k)).c_str(), d, n, st);
    if (k == cudaMemcpyDeviceToHost && in(g_dev, d)) return cudaErrorInvalidValue;
    std::memmove(d, s, n);
    return cudaSuccess;
}
}  // namespace

extern "C" {
// --- the tests' side
void rec_clear() { g_log.clear(); g_coop = 0; }
long rec_count() { return (long)g_log.size(); }
const char *rec_op(long i) { return g_log[i].op.c_str(); }
unsigned long long rec_dst(long i) { return g_log[i].dst; }
unsigned long long rec_bytes(long i) { return g_log[i].bytes; }
unsigned long long rec_stream(long i) { return g_log[i].stream; }
void rec_set_capturing(int on) { g_capturing = on; }
void rec_set_late(unsigned long long p) { g_late = (int *)p; }
long rec_coop_launches() { return g_coop; }
// device memory that the host cannot reach
unsigned long long rec_unreachable(size_t n)
{
    void *p = mmap(nullptr, n, PROT_NONE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
    g_dev[(unsigned char *)p] = n;
    return (unsigned long long)p;
}

// --- the runtime's side
static cudaError_t alloc(void **p, size_t n, std::map<unsigned char *, size_t> &m)
{
    *p = std::calloc(n ? n : 1, 1);
    m[(unsigned char *)*p] = n ? n : 1;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t n) { add("malloc", nullptr, n); return alloc(p, n, g_dev); }
cudaError_t cudaFree(void *p) { g_dev.erase((unsigned char *)p); std::free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return alloc(p, n, g_pinned); }
cudaError_t cudaFreeHost(void *p) { g_pinned.erase((unsigned char *)p); std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind k) { return copy("copy", d, s, n, k, nullptr); }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t st) { return copy("copy", d, s, n, k, st); }
cudaError_t cudaMemset(void *d, int v, size_t n) { add("memset", d, n); std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t st) { add("memset", d, n, st); std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t st) { add("sync", nullptr, 0, st); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *st, unsigned) { *st = (cudaStream_t)(g_handles += 16); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t st, cudaStreamCaptureMode) { add("begin capture", nullptr, 0, st); return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t st, cudaGraph_t *g) { add("end capture", nullptr, 0, st); *g = (cudaGraph_t)(g_handles += 16); return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s)
{
    *s = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) { *x = (cudaGraphExec_t)(g_handles += 16); return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t st) { add("graph", nullptr, 0, st); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)(g_handles += 16); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t st) { add("event", nullptr, 0, st); return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { add("event sync"); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) { *n = 2; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) { *n = 2; return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p)
{
    std::memset(a, 0, sizeof(*a));
    a->type = in(g_dev, p) ? cudaMemoryTypeDevice : in(g_pinned, p) ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered;
    if (a->type != cudaMemoryTypeUnregistered) a->devicePointer = const_cast<void *>(p);
    return cudaSuccess;
}
cudaError_t cudaLaunchCooperativeKernel(const void *f, dim3, dim3, void **, size_t, cudaStream_t st)
{
    add(("cooperative " + g_names[f]).c_str(), nullptr, 0, st);
    g_coop++;
    if (g_late) *g_late = 1;
    return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, void *st) { g_cfg = {g, b, smem, st}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *st)
{
    *g = g_cfg.g;
    *b = g_cfg.b;
    *smem = g_cfg.smem;
    *(void **)st = g_cfg.st;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t, cudaStream_t st)
{
    add(("kernel " + g_names[(const void *)k]).c_str(), nullptr, 0, st);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void *f, dim3, dim3, void **, size_t, cudaStream_t st)
{
    add(("kernel " + g_names[f]).c_str(), nullptr, 0, st);
    return cudaSuccess;
}
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, void *, void *, void *, void *, int *) { g_names[host] = name; }
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
cudaError_t cudaGetSymbolAddress(void **p, const void *) { *p = nullptr; return cudaErrorInvalidValue; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
}
