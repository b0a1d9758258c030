// A CUDA runtime that runs nothing, for tests of the library's host code on a machine without a GPU: the calls the library makes
// are checked for what the real runtime checks (a stream's and an event's device, a kernel's shared-memory limit), copies are
// done on the spot, launches are noted in a log.  "Device" memory is host memory.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {

struct Thing { int device; int at; };             // a stream, or an event and how many launches came before it
struct Range { size_t bytes; int kind, device; };

thread_local int t_device = 0;
thread_local cudaError_t t_last = cudaSuccess;
std::string g_log;
int g_launches = 0;
std::map<std::string, unsigned> g_grid;           // blocks of a kernel's last launch
std::map<std::string, int> g_fail;                // calls of this name left until one fails
std::map<const void *, std::string> g_name;       // kernels
std::map<const void *, int> g_smem;               // their dynamic shared-memory limits
std::map<const char *, Range> g_memory;
int g_registers = 168;                            // what every kernel says it was built with
void (*g_on_attribute)() = nullptr;               // called once, inside the next cudaFuncSetAttribute, after it took effect

cudaError_t done(cudaError_t e) {
    if (e != cudaSuccess) t_last = e;
    return e;
}
// notes the call; an error if one was asked for
cudaError_t enter(const char *name, const std::string &what = "") {
    g_log += std::string(name) + (what.empty() ? "" : " " + what) + "\n";
    const auto f = g_fail.find(name);
    if (f != g_fail.end() && f->second-- == 0) {
        g_fail.erase(f);
        return done(cudaErrorUnknown);
    }
    return cudaSuccess;
}
int device_of(const void *stream) { return stream ? static_cast<const Thing *>(stream)->device : t_device; }
std::string on(const void *stream) { return stream ? "side" : "main"; }       // the tests pass stream 0 themselves
cudaError_t launch(const void *f, size_t smem, const void *stream) {
    const cudaError_t e = enter("launch", g_name[f] + " " + on(stream));
    if (e != cudaSuccess) return e;
    const auto limit = g_smem.find(f);
    ++g_launches;
    if (smem > (size_t)(limit == g_smem.end() ? 48 * 1024 : limit->second) || device_of(stream) != t_device) return done(cudaErrorInvalidValue);
    return cudaSuccess;
}

}  // namespace

extern "C" {

const char *rt_log() { return g_log.c_str(); }
void rt_reset() {
    g_log.clear();
    g_fail.clear();
    g_on_attribute = nullptr;
    g_registers = 168;
    t_last = cudaSuccess;
}
void rt_fail(const char *name, int after) { g_fail[name] = after; }
void rt_on_attribute(void (*f)()) { g_on_attribute = f; }
void rt_memory(const void *p_, size_t bytes, int kind, int device) {
    const char *p = static_cast<const char *>(p_);
    for (auto r = g_memory.begin(); r != g_memory.end();)       // what lay there before is gone
        r = r->first < p + bytes && p < r->first + r->second.bytes ? g_memory.erase(r) : std::next(r);
    g_memory[p] = Range{bytes, kind, device};
}

cudaError_t cudaGetDevice(int *d) { *d = t_device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { t_device = d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = t_last; t_last = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t) { return "an error of the host runtime"; }
cudaError_t cudaMalloc(void **p, size_t n) {
    enter("malloc", std::to_string(n));
    *p = aligned_alloc(256, (n + 255) / 256 * 256);
    rt_memory(*p, n, cudaMemoryTypeDevice, t_device);
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { *p = aligned_alloc(256, (n + 255) / 256 * 256); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemset(void *p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t s) {
    const cudaError_t e = enter("memset", on(s));
    if (e == cudaSuccess) memset(p, v, n);
    return e;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t st) {
    const cudaError_t e = enter("memcpy", on(st));
    if (e == cudaSuccess) memcpy(d, s, n);
    return e;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
    memset(a, 0, sizeof *a);
    const char *c = static_cast<const char *>(p);
    auto r = g_memory.upper_bound(c);
    if (r != g_memory.begin() && c < (--r)->first + r->second.bytes) {
        a->type = static_cast<cudaMemoryType>(r->second.kind);
        a->device = r->second.device;
    }
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = reinterpret_cast<cudaStream_t>(new Thing{t_device, 0}); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { delete reinterpret_cast<Thing *>(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return enter("synchronize", on(s)); }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = reinterpret_cast<cudaEvent_t>(new Thing{t_device, 0}); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete reinterpret_cast<Thing *>(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    const cudaError_t r = enter("record", on(s));
    if (r != cudaSuccess) return r;
    reinterpret_cast<Thing *>(e)->at = g_launches;
    return device_of(s) == reinterpret_cast<Thing *>(e)->device ? cudaSuccess : done(cudaErrorInvalidResourceHandle);
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t, unsigned) { return enter("wait", on(s)); }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b) {       // in launches
    *ms = (float)(reinterpret_cast<Thing *>(b)->at - reinterpret_cast<Thing *>(a)->at);
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute, int v) {
    g_smem[f] = v;
    if (auto call = g_on_attribute) {
        g_on_attribute = nullptr;
        call();
    }
    return cudaSuccess;
}
void rt_registers(int n) { g_registers = n; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) {
    memset(a, 0, sizeof *a);
    a->numRegs = g_registers;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) { *n = 2; return cudaSuccess; }
unsigned rt_blocks(const char *name) { return g_grid[name]; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) {
    g_grid[g_name[f]] = c->gridDim.x * c->gridDim.y * c->gridDim.z;
    return launch(f, c->dynamicSmemBytes, c->stream);
}
cudaError_t cudaLaunchKernel(const void *f, dim3, dim3, void **, size_t smem, cudaStream_t s) { return launch(f, smem, s); }
cudaError_t cudaGetSymbolAddress(void **p, const void *) {
    static std::vector<char> all(1 << 20);
    *p = all.data();
    return cudaSuccess;
}
static CUresult encode(...) { return CUDA_SUCCESS; }
static CUresult pointer_attributes(unsigned n, CUpointer_attribute *what, void **to, CUdeviceptr p) {
    const char *c = reinterpret_cast<const char *>(p);
    auto r = g_memory.upper_bound(c);
    const bool known = r != g_memory.begin() && c < (--r)->first + r->second.bytes;
    for (unsigned i = 0; i < n; ++i) switch (what[i]) {
        case CU_POINTER_ATTRIBUTE_MEMORY_TYPE: *static_cast<unsigned *>(to[i]) = known ? r->second.kind : 0; break;
        case CU_POINTER_ATTRIBUTE_IS_MANAGED: *static_cast<unsigned *>(to[i]) = 0; break;
        case CU_POINTER_ATTRIBUTE_DEVICE_POINTER: *static_cast<CUdeviceptr *>(to[i]) = known ? p : 0; break;
        case CU_POINTER_ATTRIBUTE_RANGE_START_ADDR: *static_cast<CUdeviceptr *>(to[i]) = known ? reinterpret_cast<CUdeviceptr>(r->first) : 0; break;
        case CU_POINTER_ATTRIBUTE_RANGE_SIZE: *static_cast<size_t *>(to[i]) = known ? r->second.bytes : 0; break;
        default: return CUDA_ERROR_INVALID_VALUE;
    }
    return CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPoint(const char *name, void **p, unsigned long long, cudaDriverEntryPointQueryResult *q) {
    *p = strcmp(name, "cuPointerGetAttributes") ? reinterpret_cast<void *>(encode) : reinterpret_cast<void *>(pointer_attributes);
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
// what the compiler's registration code calls
void **__cudaRegisterFatBinary(void *) { static void *handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {
    const char *k = strstr(name, "k_");              // the kernel's own name out of the mangled one (small letters and underscores)
    const std::string s = k ? std::string(k, strspn(k, "abcdefghijklmnopqrstuvwxyz_")) : name;
    g_name[host] = s;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void *) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }

}  // extern "C"
