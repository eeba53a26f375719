// A CUDA runtime that runs nothing: it records the kernels that the library launches and how.  Linked with the library's own
// object files in the place of libcudart, so that a test without a GPU sees what the host code does -- on several devices,
// on streams that capture, after a launch that failed, without memory.
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <stdlib.h>

#include <map>
#include <new>
#include <string>
#include <vector>

namespace {

struct Launch {
    std::string kernel;
    void* stream;
    int overlap;  // launched with programmatic stream serialization
};

std::map<const void*, std::string>& kernels()
{
    static std::map<const void*, std::string> m;
    return m;
}

std::vector<Launch> g_launches;
std::map<void*, int> g_capturing;
int g_device = 0;
bool g_fail_launch = false, g_fail_alloc = false;
cudaError_t g_last = cudaSuccess;
cudaLaunchConfig_t g_pushed;

cudaError_t error(cudaError_t e) { return e == cudaSuccess ? e : g_last = e; }

cudaError_t launch(const void* f, cudaStream_t stream, int overlap)
{
    if (g_fail_launch) {
        g_fail_launch = false;
        return error(cudaErrorLaunchFailure);
    }
    const bool fail = g_fail_alloc;
    g_fail_alloc = false;  // (what is recorded here is not the library's)
    g_launches.push_back({kernels()[f], stream, overlap});
    g_fail_alloc = fail;
    return cudaSuccess;
}

CUresult encode(...) { return CUDA_SUCCESS; }

}  // namespace

// ---- what a test sets and reads
extern "C" {
void fake_device(int d) { g_device = d; }
void fake_capturing(void* stream, int on) { g_capturing[stream] = on; }
void fake_fail_launch() { g_fail_launch = true; }
void fake_fail_alloc(int on) { g_fail_alloc = on; }
int fake_launches() { return static_cast<int>(g_launches.size()); }
const char* fake_kernel(int i) { return g_launches[i].kernel.c_str(); }
int fake_overlap(int i) { return g_launches[i].overlap; }
void fake_clear() { g_launches.clear(); }
}

void* operator new(size_t n)
{
    void* p = g_fail_alloc ? nullptr : malloc(n);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void* p) noexcept { free(p); }
void operator delete(void* p, size_t) noexcept { free(p); }

// ---- the runtime
extern "C" {

void** __cudaRegisterFatBinary(void*)
{
    static void* handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*)
{
    kernels()[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t stream)
{
    g_pushed.gridDim = grid;
    g_pushed.blockDim = block;
    g_pushed.dynamicSmemBytes = smem;
    g_pushed.stream = stream;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream)
{
    *grid = g_pushed.gridDim;
    *block = g_pushed.blockDim;
    *smem = g_pushed.dynamicSmemBytes;
    *static_cast<cudaStream_t*>(stream) = g_pushed.stream;
    return cudaSuccess;
}

cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void**, size_t, cudaStream_t stream) { return launch(f, stream, 0); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* cfg, const void* f, void**)
{
    int overlap = 0;
    for (unsigned i = 0; i < cfg->numAttrs; ++i)
        if (cfg->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization)
            overlap = cfg->attrs[i].val.programmaticStreamSerializationAllowed;
    return launch(f, cfg->stream, overlap);
}

cudaError_t cudaGetLastError()
{
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
cudaError_t cudaGetDevice(int* d)
{
    *d = g_device;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int)
{
    *v = 148;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* cfg)
{
    *n = 144 / static_cast<int>(cfg->attrs[0].val.clusterDim.x);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol)
{
    *p = const_cast<void*>(symbol);
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPoint(const char*, void** fn, unsigned long long, cudaDriverEntryPointQueryResult* q)
{
    *fn = reinterpret_cast<void*>(encode);
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}

cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* status)
{
    *status = g_capturing[s] ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
}
