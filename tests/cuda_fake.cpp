// cuda_fake.cpp -- the CUDA runtime calls of the library's host code, for tests without a GPU:
// linked with the library's object files in place of the CUDA runtime (tests/test_host_calls.py).
//
// Device memory is host memory.  Work of a stream takes effect when it is enqueued, except that a
// cudaMemcpy from pageable memory to the device (legacy stream) only stages its data, as the CUDA
// runtime may: the data arrive at the next call that waits for that stream or for the device.  A
// kernel launched on another stream before that is recorded: nothing orders it after the copy.
// Kernels compute nothing, but for those that tell the host the row classes, which give the
// classes set by fake_classes.
#include <cuda_runtime_api.h>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {

struct Stream { bool blocking; };
struct Pending { void *dst; std::vector<unsigned char> data; };
struct Classes { int small = 0, mid = 0, large = 0, hubs = 0, dmax = 0, degree = 0, distinct = 0; } classes;

std::map<const void *, std::string> kernels;
std::map<std::string, int> launched;
std::map<void *, size_t> blocks;
std::vector<Pending> pending;
std::string unordered;                     // kernels launched beside a pending copy
int64_t live = 0, fail_in = -1;            // bytes allocated; allocations until one fails
struct Config { dim3 grid, block; size_t smem; cudaStream_t s; };
std::vector<Config> configs;
cudaError_t last = cudaSuccess;

void arrive() {
    for (auto &p : pending) std::memcpy(p.dst, p.data.data(), p.data.size());
    pending.clear();
}
bool legacy(cudaStream_t s) { return !s || reinterpret_cast<Stream *>(s)->blocking; }

cudaError_t allocate(void **p, size_t bytes) {
    if (fail_in >= 0 && fail_in-- == 0) return cudaErrorMemoryAllocation;
    *p = std::calloc(bytes ? bytes : 1, 1);
    blocks[*p] = bytes;
    live += (int64_t)bytes;
    return cudaSuccess;
}
cudaError_t release(void *p) {
    if (!p) return cudaSuccess;
    auto it = blocks.find(p);
    if (it == blocks.end()) return cudaErrorInvalidValue;
    live -= (int64_t)it->second;
    blocks.erase(it);
    std::free(p);
    return cudaSuccess;
}

template <class T> T arg(void **args, int i) { return *static_cast<T *>(args[i]); }

cudaError_t run(const void *fn, void **args, cudaStream_t s) {
    const std::string &name = kernels[fn];
    ++launched[name];
    if (legacy(s)) arrive();
    else if (!pending.empty()) unordered += name + "\n";
    auto is = [&](const char *k) { return name.find(k) != std::string::npos; };
    if (is("classify_count_kernel")) {
        int *hdr = arg<int *>(args, 3);
        int32_t *hubs = arg<int32_t *>(args, 4);
        const int v[7] = {classes.dmax, 64, classes.hubs, 0, classes.small, classes.mid, classes.large};
        std::memcpy(hdr, v, sizeof(v));
        for (int i = 0; i < classes.hubs; ++i) hubs[i] = i;
    } else if (is("hub_bounds_kernel")) {
        const int64_t nh = arg<int64_t>(args, 2);
        int64_t *b = arg<int64_t *>(args, 6);
        for (int64_t i = 0; i < nh; ++i) {
            b[3 * i] = i * classes.degree;
            b[3 * i + 1] = (i + 1) * classes.degree;
            b[3 * i + 2] = arg<int32_t>(args, 3);
        }
    } else if (is("hub_distinct_kernel")) {
        int32_t *lf = arg<int32_t *>(args, 9);
        for (int i = 0; i < classes.hubs; ++i) lf[i] = classes.distinct;
    }
    return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- what the tests set and read --------------------------------------------------------
void *fake_stream(void) { return new Stream{false}; }
void fake_classes(int small, int mid, int large, int hubs, int dmax, int degree, int distinct) {
    classes = Classes{small, mid, large, hubs, dmax, degree, distinct};
}
void fake_fail_allocation(int64_t n) { fail_in = n; }     // the n-th from now (0: the next); -1: none
const char *fake_unordered(void) { return unordered.c_str(); }
int64_t fake_live_bytes(void) { return live; }
int fake_launches(const char *name) {
    int c = 0;
    for (auto &k : launched)
        if (k.first.find(name) != std::string::npos) c += k.second;
    return c;
}

// ---- registration and launches ------------------------------------------------------------
void **__cudaRegisterFatBinary(void *) {
    static void *handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {
    kernels[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st *s) {
    configs.push_back(Config{grid, block, smem, s});
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *s) {
    const Config c = configs.back();
    configs.pop_back();
    *grid = c.grid;
    *block = c.block;
    *smem = c.smem;
    *static_cast<cudaStream_t *>(s) = c.s;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fn) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void *>(fn));
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **args, size_t, cudaStream_t s) { return run(k, args, s); }
cudaError_t cudaLaunchKernel(const void *fn, dim3, dim3, void **args, size_t, cudaStream_t s) { return run(fn, args, s); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *fn, void **args) { return run(fn, args, c->stream); }
cudaError_t cudaLaunchCooperativeKernel(const void *fn, dim3, dim3, void **args, size_t, cudaStream_t s) { return run(fn, args, s); }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
    *n = 1;
    return cudaSuccess;
}

// ---- device ---------------------------------------------------------------------------------
cudaError_t cudaGetDevice(int *d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) {
    *v = 4;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetStreamPriorityRange(int *lo, int *hi) {
    *lo = 0;
    *hi = -1;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize(void) {
    arrive();
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
const char *cudaGetErrorString(cudaError_t) { return "error of the stand-in runtime"; }

// ---- memory ---------------------------------------------------------------------------------
cudaError_t cudaMalloc(void **p, size_t bytes) { return allocate(p, bytes); }
cudaError_t cudaFree(void *p) { return release(p); }
cudaError_t cudaMallocHost(void **p, size_t bytes) {
    *p = std::calloc(bytes ? bytes : 1, 1);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t *pool, const cudaMemPoolProps *) {
    *pool = reinterpret_cast<cudaMemPool_t>(new int);
    return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t bytes, cudaMemPool_t, cudaStream_t) { return allocate(p, bytes); }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return release(p); }
cudaError_t cudaGetSymbolAddress(void **, const void *) { return cudaErrorInvalidValue; }
cudaError_t cudaMemcpy(void *dst, const void *src, size_t bytes, cudaMemcpyKind kind) {
    if (kind == cudaMemcpyHostToDevice) {
        const unsigned char *p = static_cast<const unsigned char *>(src);
        pending.push_back(Pending{dst, std::vector<unsigned char>(p, p + bytes)});
    } else {
        arrive();
        std::memcpy(dst, src, bytes);
    }
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t bytes, cudaMemcpyKind, cudaStream_t s) {
    if (legacy(s)) arrive();
    std::memmove(dst, src, bytes);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t bytes, cudaStream_t s) {
    if (legacy(s)) arrive();
    std::memset(p, v, bytes);
    return cudaSuccess;
}

// ---- streams, events, graphs ----------------------------------------------------------------
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned flags) {
    *s = reinterpret_cast<cudaStream_t>(new Stream{!(flags & cudaStreamNonBlocking)});
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned flags, int) { return cudaStreamCreateWithFlags(s, flags); }
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    delete reinterpret_cast<Stream *>(s);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    if (legacy(s)) arrive();
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
    *g = nullptr;
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) {
    *e = reinterpret_cast<cudaEvent_t>(new int);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    delete reinterpret_cast<int *>(e);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.0f;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) {
    *x = nullptr;
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

}  // extern "C"
