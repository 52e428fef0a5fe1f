// A stand-in for the CUDA runtime, linked with the library's own objects so that
// its host code runs without a GPU: kernels do nothing, copies and launches are
// recorded with their streams.  Device memory is address space that faults when
// the CPU touches it; its contents live in a shadow that copies are sent to.
#include <cuda_runtime_api.h>
#include <cudaTypedefs.h>
#include <sys/mman.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {

struct Region {
    size_t bytes;
    int device;
    char *shadow;
};
std::map<char *, Region> regions;  // device memory, by base address
// (kernels and variables register before this file's globals are made)
std::map<const void *, std::string> &names()
{
    static auto *m = new std::map<const void *, std::string>;
    return *m;
}
std::map<const void *, size_t> &vars()
{
    static auto *m = new std::map<const void *, size_t>;
    return *m;
}
std::map<const void *, void *> var_at;
int cc[2] = {10, 3};

char *device_alloc(int device, size_t bytes)
{
    void *p = mmap(nullptr, bytes, PROT_NONE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (p == MAP_FAILED)
        return nullptr;
    regions[(char *)p] = Region{bytes, device, (char *)std::calloc(1, bytes)};
    return (char *)p;
}
const Region *find(const void *p, char **base)
{
    auto it = regions.upper_bound((char *)p);
    if (it == regions.begin())
        return nullptr;
    --it;
    if ((char *)p >= it->first + it->second.bytes)
        return nullptr;
    *base = it->first;
    return &it->second;
}
char *at(const void *p)  // where the CPU finds p's contents
{
    char *base;
    const Region *r = find(p, &base);
    return r ? r->shadow + ((char *)p - base) : (char *)p;
}

}  // namespace

struct Record {
    char what[128];          // "copy", "set", "sync", or a kernel's name
    unsigned long long dst, src, bytes, stream;
    int async, grid;
    unsigned long long arg[16];  // a launch: the first words at its first argument (and what follows it)
};
static std::vector<Record> records;
static Record &record(const char *what, const void *dst, const void *src, size_t bytes, const void *stream, int async)
{
    Record r{};
    std::snprintf(r.what, sizeof r.what, "%s", what);
    r.dst = (unsigned long long)dst;
    r.src = (unsigned long long)src;
    r.bytes = bytes;
    r.stream = (unsigned long long)stream;
    r.async = async;
    records.push_back(r);
    return records.back();
}

extern "C" {

int fake_count() { return (int)records.size(); }
const Record *fake_record(int i) { return &records[i]; }
void fake_clear() { records.clear(); }
void *fake_alloc(int device, size_t bytes) { return device_alloc(device, bytes); }
void *fake_shadow(void *p) { return at(p); }
void fake_capability(int major, int minor) { cc[0] = major, cc[1] = minor; }

// ---- memory
cudaError_t cudaMalloc(void **p, size_t n) { return (*p = device_alloc(0, n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void *p)
{
    auto it = regions.find((char *)p);
    if (it != regions.end()) {
        std::free(it->second.shadow);
        munmap(p, it->second.bytes);
        regions.erase(it);
    }
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return (*p = std::calloc(1, n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaMallocHost(void **p, size_t n) { return cudaHostAlloc(p, n, 0); }
cudaError_t cudaFreeHost(void *p)
{
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p)
{
    char *base;
    const Region *r = find(p, &base);
    std::memset(a, 0, sizeof *a);
    a->type = r ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
    a->device = r ? r->device : -2;
    return cudaSuccess;
}
static cudaError_t copy(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind kind, void *st,
                        int async)
{
    char *base;
    const bool dd = find(d, &base), sd = find(s, &base);  // the kind, where one is given, fits the pointers
    if (kind != cudaMemcpyDefault && kind != (sd ? (dd ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost)
                                                 : (dd ? cudaMemcpyHostToDevice : cudaMemcpyHostToHost)))
        return cudaErrorInvalidValue;
    for (size_t r = 0; r < h; ++r)
        std::memcpy(at((char *)d + r * dp), at((const char *)s + r * sp), w);
    record("copy", d, s, w * h, st, async);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind k) { return copy(d, n, s, n, n, 1, k, nullptr, 0); }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t st)
{
    return copy(d, n, s, n, n, 1, k, st, 1);
}
cudaError_t cudaMemcpy2D(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind k)
{
    return copy(d, dp, s, sp, w, h, k, nullptr, 0);
}
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind k,
                              cudaStream_t st)
{
    return copy(d, dp, s, sp, w, h, k, st, 1);
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t st)
{
    std::memset(at(d), v, n);
    record("set", d, nullptr, n, st, 1);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n)
{
    cudaMemsetAsync(d, v, n, nullptr);
    records.back().async = 0;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *sym)
{
    if (!var_at[sym])
        var_at[sym] = device_alloc(0, vars()[sym]);
    *p = var_at[sym];
    return cudaSuccess;
}

// ---- streams, events, graphs
static long handles = 0;
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned)
{
    *s = (cudaStream_t)(0x10000 + 16 * ++handles);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s)
{
    record("sync", nullptr, nullptr, 0, s, 0);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e)
{
    *e = (cudaEvent_t)(0x10000 + 16 * ++handles);
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t)
{
    *ms = 0.0f;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g)
{
    *g = nullptr;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *g, cudaGraph_t, unsigned long long)
{
    *g = (cudaGraphExec_t)(0x10000 + 16 * ++handles);
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }

// ---- the device: 152 SMs, one CTA pair per two of them
cudaError_t cudaGetDevice(int *d)
{
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceCount(int *n)
{
    *n = 2;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int)
{
    *v = a == cudaDevAttrMultiProcessorCount          ? 152
         : a == cudaDevAttrComputeCapabilityMajor ? cc[0]
         : a == cudaDevAttrComputeCapabilityMinor ? cc[1]
                                                  : 0;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *)
{
    *n = 76;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "an error of the stand-in runtime"; }
static CUresult CUDAAPI encode(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                               const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                               CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill)
{
    return CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q)
{
    *fn = (void *)encode;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}

// ---- kernels
struct Config {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
};
static Config pushed;
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t stream)
{
    pushed = Config{grid, block, smem, stream};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream)
{
    *grid = pushed.grid;
    *block = pushed.block;
    *smem = pushed.smem;
    *(cudaStream_t *)stream = pushed.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fn)
{
    *k = (cudaKernel_t)fn;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void **args, size_t, cudaStream_t stream)
{
    Record &r = record(names()[(const void *)k].c_str(), nullptr, nullptr, 0, stream, 1);
    r.grid = (int)(grid.x * grid.y * grid.z);
    if ((unsigned long long)args[0] % 8 == 0)
        std::memcpy(r.arg, args[0], sizeof r.arg);
    return cudaSuccess;
}
void **__cudaRegisterFatBinary(void *) { return (void **)&pushed; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *host, char *, const char *, int, size_t size, int, int) { vars()[host] = size; }
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *)
{
    names()[host] = name;
}
}
