// See fake_cuda.h. Linked with the library's objects in place of the CUDA runtime.
#include "fake_cuda.h"

#include <sys/mman.h>

#include <cstdlib>
#include <cstring>
#include <mutex>

namespace fake {

Runtime& runtime() {
    static Runtime* r = new Runtime();
    return *r;
}

namespace {

constexpr size_t kDefaultShared = 48 * 1024;

std::mutex mu;
std::map<char*, size_t> blocks;
cudaError_t last = cudaSuccess;
uintptr_t names = 0x1000;

struct Config {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
};
thread_local Config config;

cudaError_t answer(cudaError_t e) {
    if (e != cudaSuccess) last = e;
    return e;
}

cudaError_t launch(const void* kernel, size_t smem, cudaStream_t s, bool cooperative) {
    Runtime& R = runtime();
    {
        std::lock_guard<std::mutex> lk(mu);
        const auto a = R.allowed.find({R.device, kernel});
        if (smem > (a == R.allowed.end() ? kDefaultShared : a->second)) {
            ++R.refused;
            return answer(cudaErrorInvalidValue);
        }
        R.calls.push_back({cooperative ? "cooperative" : "launch", kernel, s, nullptr});
    }
    return R.on_launch ? answer(R.on_launch(kernel, cooperative)) : cudaSuccess;
}

template <class T>
cudaError_t name(T* p) {
    std::lock_guard<std::mutex> lk(mu);
    *p = reinterpret_cast<T>(names += 16);
    return cudaSuccess;
}

}  // namespace

}  // namespace fake

using namespace fake;

extern "C" {

void** __cudaRegisterFatBinary(void*) {
    static void* handle = nullptr;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}

unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st* s) {
    config = {grid, block, smem, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
    *grid = config.grid;
    *block = config.block;
    *smem = config.smem;
    *static_cast<cudaStream_t*>(s) = config.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fun) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(fun));
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t smem, cudaStream_t s) {
    return launch(k, smem, s, false);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* cfg, const void* fun, void**) {
    return launch(fun, cfg->dynamicSmemBytes, cfg->stream, false);
}
cudaError_t cudaLaunchCooperativeKernel(const void* fun, dim3, dim3, void**, size_t smem, cudaStream_t s) {
    return launch(fun, smem, s, true);
}
cudaError_t cudaFuncSetAttribute(const void* fun, cudaFuncAttribute a, int value) {
    Runtime& R = runtime();
    if (R.attribute_error != cudaSuccess) return answer(R.attribute_error);
    std::lock_guard<std::mutex> lk(mu);
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) R.allowed[{R.device, fun}] = static_cast<size_t>(value);
    return cudaSuccess;
}

cudaError_t cudaGetDevice(int* d) {
    *d = runtime().device;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
    runtime().device = d;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t* p, int) { return name(p); }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaDeviceSetLimit(cudaLimit, size_t) { return cudaSuccess; }
cudaError_t cudaCtxResetPersistingL2Cache() { return cudaSuccess; }
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t) { return "an error of the test's runtime"; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
    *p = nullptr;
    return answer(cudaErrorInvalidSymbol);
}

cudaError_t cudaMallocAsync(void** p, size_t bytes, cudaStream_t) {
    std::lock_guard<std::mutex> lk(mu);
    Runtime& R = runtime();
    *p = nullptr;
    if (bytes > R.limit || R.live > R.limit - bytes) return answer(cudaErrorMemoryAllocation);
    void* m = mmap(nullptr, bytes ? bytes : 1, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (m == MAP_FAILED) return answer(cudaErrorMemoryAllocation);
    blocks[static_cast<char*>(m)] = bytes;
    R.live += bytes;
    if (R.live > R.peak) R.peak = R.live;
    *p = m;
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {
    std::lock_guard<std::mutex> lk(mu);
    const auto b = blocks.find(static_cast<char*>(p));
    if (b == blocks.end()) return answer(cudaErrorInvalidValue);
    runtime().live -= b->second;
    munmap(p, b->second ? b->second : 1);
    blocks.erase(b);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t bytes, unsigned) {
    *p = std::calloc(1, bytes);
    return *p ? cudaSuccess : answer(cudaErrorMemoryAllocation);
}
cudaError_t cudaFreeHost(void* p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* to, const void* from, size_t bytes, cudaMemcpyKind, cudaStream_t) {
    std::memcpy(to, from, bytes);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* to, const void* from, size_t bytes, cudaMemcpyKind) {
    std::memcpy(to, from, bytes);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t bytes, cudaStream_t) {
    std::memset(p, v, bytes);
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    std::lock_guard<std::mutex> lk(mu);
    std::memset(a, 0, sizeof(*a));
    a->type = cudaMemoryTypeUnregistered;
    auto b = blocks.upper_bound(static_cast<char*>(const_cast<void*>(p)));
    if (b != blocks.begin() && static_cast<const char*>(p) < (--b)->first + b->second) {
        a->type = cudaMemoryTypeDevice;
        a->device = runtime().device;
    }
    return cudaSuccess;
}

cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return name(s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSetAttribute(cudaStream_t, cudaLaunchAttributeID, const cudaLaunchAttributeValue*) {
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    std::lock_guard<std::mutex> lk(mu);
    runtime().calls.push_back({"wait", nullptr, s, e});
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return name(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return name(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 0.f;
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    std::lock_guard<std::mutex> lk(mu);
    runtime().calls.push_back({"record", nullptr, s, e});
    return cudaSuccess;
}

cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
    *n = 1;
    return cudaSuccess;
}

cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) { return name(g); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle* h, cudaGraph_t, unsigned, unsigned) {
    *h = 1;
    return cudaSuccess;
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                             cudaGraphNodeParams* p) {
    static cudaGraph_t body = reinterpret_cast<cudaGraph_t>(uintptr_t{0x100});
    if (p->type == cudaGraphNodeTypeConditional) p->conditional.phGraph_out = &body;
    return name(n);
}
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*,
                                          size_t, cudaStreamCaptureMode) {
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { return name(e); }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return launch(nullptr, 0, nullptr, false); }

}  // extern "C"
