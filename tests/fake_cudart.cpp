// A stand-in for the CUDA runtime, preloaded into a child process: it launches
// nothing and records which kernels the library asked for, so that routes, error
// handling and memory use of the host code can be tested without a GPU.  Device
// memory is address space that nothing backs, up to a settable size; stream
// handles at and above FAKE_CAPTURING count as being captured, where calls that
// synchronise or allocate fail, as they do in the runtime.
#include <cuda_runtime_api.h>
#include <sys/mman.h>

#include <cstdint>
#include <cstring>
#include <map>
#include <string>

namespace {
constexpr uintptr_t FAKE_CAPTURING = 0x100000;
std::map<const void *, std::string> names;   // kernel entry -> name
std::map<void *, size_t> blocks;
std::string events;
size_t room = (size_t)280 << 30, peak = 0, used = 0;
int regs = 72, has_pools = 1;
bool captured = false;    // some stream is being captured, in the mode that watches all threads
cudaStreamCaptureMode mode = cudaStreamCaptureModeGlobal;   // this thread's
cudaError_t last = cudaSuccess;

cudaError_t err(cudaError_t e)
{
    if (e != cudaSuccess) last = e;
    return e;
}
void note(const std::string &s) { events += s + "\n"; }
bool capturing(cudaStream_t s) { return (uintptr_t)s >= FAKE_CAPTURING; }
cudaError_t take(void **p, size_t n)
{
    if (n > room - used) return err(cudaErrorMemoryAllocation);
    void *m = mmap(nullptr, n ? n : 1, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (m == MAP_FAILED) return err(cudaErrorMemoryAllocation);
    blocks[m] = n;
    used += n;
    if (used > peak) peak = used;
    *p = m;
    return cudaSuccess;
}
cudaError_t give(void *p)
{
    if (!p) return cudaSuccess;
    auto it = blocks.find(p);
    if (it == blocks.end()) return err(cudaErrorInvalidValue);
    munmap(p, it->second ? it->second : 1);
    used -= it->second;
    blocks.erase(it);
    return cudaSuccess;
}
cudaError_t launched(const void *f, dim3 g, cudaStream_t s)
{
    std::string n = names.count(f) ? names[f] : "?";
    size_t i = n.find("k_");   // the mangled name from the kernel's own name on
    note("launch " + n.substr(i == std::string::npos ? 0 : i) + " grid " + std::to_string(g.x) + " stream " +
         std::to_string((uintptr_t)s));
    return cudaSuccess;
}
struct Call { dim3 g, b; size_t sm; cudaStream_t s; } call;
}  // namespace

extern "C" {
// ---- for the test ----
void fake_room(size_t n) { room = n; }
size_t fake_used() { return used; }
size_t fake_peak(int reset) { size_t p = peak; if (reset) peak = used; return p; }
void fake_regs(int n) { regs = n; }
void fake_pools(int on) { has_pools = on; }
void fake_capture(int on) { captured = on; }
const char *fake_events() { static std::string out; out.swap(events); events.clear(); return out.c_str(); }

// ---- registration and launches ----
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *)
{
    names[host] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sm, cudaStream_t s) { call = {g, b, sm, s}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *sm, void *s)
{
    *g = call.g; *b = call.b; *sm = call.sm; *(cudaStream_t *)s = call.s;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(const void **k, const void *f) { *k = f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(const void *k, dim3 g, dim3, void **, size_t, cudaStream_t s) { return launched(k, g, s); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) { return launched(f, c->gridDim, c->stream); }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *)
{
    memset(a, 0, sizeof *a);
    a->numRegs = regs;
    return cudaSuccess;
}

// ---- device ----
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int)
{
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMemoryPoolsSupported ? has_pools : 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return captured ? err(cudaErrorStreamCaptureUnsupported) : cudaSuccess; }
cudaError_t cudaGetLastError() { cudaError_t e = last; last = cudaSuccess; return e; }

// ---- memory ----
cudaError_t cudaMalloc(void **p, size_t n) { return captured ? err(cudaErrorStreamCaptureUnsupported) : take(p, n); }
cudaError_t cudaFree(void *p) { return give(p); }
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t n, cudaStream_t) { note("memset " + std::to_string(n)); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *)
{
    if (captured && mode != cudaStreamCaptureModeRelaxed) return err(cudaErrorStreamCaptureUnsupported);
    *p = (cudaMemPool_t)&blocks;
    return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { note("pool destroyed"); return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t, cudaStream_t s)
{
    if (capturing(s)) note("allocation captured");
    if (captured && mode != cudaStreamCaptureModeRelaxed) return err(cudaErrorStreamCaptureUnsupported);
    return take(p, n);
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return give(p); }

// ---- streams ----
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus *st)
{
    *st = capturing(s) ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *m)
{
    const cudaStreamCaptureMode was = mode;
    mode = *m;
    *m = was;
    return cudaSuccess;
}
}
