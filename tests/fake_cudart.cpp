// A stand-in for the CUDA runtime that the host paths of the library are tested on without
// a GPU: device memory is host memory, streams, events and graphs are tokens, and a launch
// is written down (kernel, grid, current device) instead of run. The test controls say how
// many SMs the devices have and which launches fail. Linked with the library's own objects
// in place of the real runtime (fake_gpu.py).
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {

struct Launch {
    std::string kernel;
    unsigned grid;
    int device;
    size_t smem;
};

int g_device = 0;
int g_sms = 152;
cudaError_t g_last = cudaSuccess;
std::vector<Launch> g_launches;
std::string g_fail_kernel;  // launches whose kernel's name holds this fail ...
int g_fail_skip = 0;        // ... after this many of them went through,
int g_fail_times = 0;       // ... this often, with this error
cudaError_t g_fail_code = cudaSuccess;

std::map<const void *, std::string> &kernels() {
    static std::map<const void *, std::string> m;
    return m;
}

std::map<const void *, void *> &variables() {
    static std::map<const void *, void *> m;
    return m;
}

struct Config {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
};
std::vector<Config> g_config;

// The runtime keeps the error of a call that failed until cudaGetLastError asks for it.
cudaError_t note(cudaError_t e) {
    if (e != cudaSuccess) g_last = e;
    return e;
}

cudaError_t launch(const void *fun, dim3 grid, size_t smem) {
    const std::string name = kernels().count(fun) ? kernels()[fun] : "?";
    if (g_fail_times > 0 && name.find(g_fail_kernel) != std::string::npos) {
        if (g_fail_skip > 0) {
            --g_fail_skip;
        } else {
            --g_fail_times;
            return note(g_fail_code);
        }
    }
    g_launches.push_back({name, grid.x, g_device, smem});
    return cudaSuccess;
}

template <class T>
cudaError_t token(T *out) {
    static char t[8];
    *out = reinterpret_cast<T>(t);
    return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- test controls
void fake_reset(int sms) {
    g_launches.clear();
    g_fail_times = 0;
    g_device = 0;
    g_sms = sms;
    g_last = cudaSuccess;
}
void fake_fail(const char *kernel, int skip, int times, int code) {
    g_fail_kernel = kernel;
    g_fail_skip = skip;
    g_fail_times = times;
    g_fail_code = cudaError_t(code);
}
void fake_set_device(int dev) { g_device = dev; }
int fake_device() { return g_device; }
int fake_launches() { return int(g_launches.size()); }
const char *fake_launch_kernel(int i) { return g_launches[size_t(i)].kernel.c_str(); }
int fake_launch_device(int i) { return g_launches[size_t(i)].device; }
int fake_launch_grid(int i) { return int(g_launches[size_t(i)].grid); }
int fake_launch_smem(int i) { return int(g_launches[size_t(i)].smem); }

// ---- registration and launches
void **__cudaRegisterFatBinary(void *) {
    static void *handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *fun, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {
    kernels()[fun] = name;
}
void __cudaRegisterVar(void **, char *var, char *, const char *, int, size_t size, int, int) {
    variables()[var] = std::calloc(1, size);
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st *stream) {
    g_config.push_back({grid, block, smem, stream});
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream) {
    const Config c = g_config.back();
    g_config.pop_back();
    *grid = c.grid;
    *block = c.block;
    *smem = c.smem;
    *static_cast<cudaStream_t *>(stream) = c.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fun) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void *>(fun));
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void **, size_t smem, cudaStream_t) {
    return launch(k, grid, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *fun, void **) {
    return launch(fun, c->gridDim, c->dynamicSmemBytes);
}

// ---- errors and devices
cudaError_t cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "stand-in error"; }
cudaError_t cudaGetDeviceCount(int *n) {
    *n = 3;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) {
    *d = g_device;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
    if (d < 0 || d > 2) return note(cudaErrorInvalidDevice);
    g_device = d;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) {
    std::memset(p, 0, sizeof(*p));
    p->major = 10;
    p->minor = 3;
    p->multiProcessorCount = g_sms;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? g_sms : a == cudaDevAttrClockRate ? 2000000 : 0;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *var) {
    *p = variables().count(var) ? variables()[var] : nullptr;
    return note(*p ? cudaSuccess : cudaErrorInvalidSymbol);
}

// ---- memory
cudaError_t cudaMalloc(void **p, size_t n) {
    *p = std::aligned_alloc(256, (n + 255) / 256 * 256);
    if (!*p) return note(cudaErrorMemoryAllocation);
    std::memset(*p, 0, n);
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void *p) { return cudaFree(p); }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) {
    return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemset(void *d, int v, size_t n) {
    std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }

// ---- streams, events, graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return token(s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { return token(g); }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return token(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return token(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.f;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) { return token(x); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

}  // extern "C"
