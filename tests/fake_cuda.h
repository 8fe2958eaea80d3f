// A CUDA runtime without a GPU, for tests of the library's host code: memory is
// host memory with a limit, streams and events are names, kernels do not run (a
// test may stand in for them), and every call that matters is written down.
#pragma once

#include <cuda_runtime.h>

#include <functional>
#include <map>
#include <string>
#include <utility>
#include <vector>

namespace fake {

struct Call {
    std::string what;            // "launch", "cooperative", "record", "wait"
    const void* kernel;
    cudaStream_t stream;
    cudaEvent_t event;
};

struct Runtime {
    int device = 0;              // the current one, of every thread
    size_t live = 0, peak = 0, limit = ~size_t{0};               // device memory in bytes
    std::vector<Call> calls;
    std::map<std::pair<int, const void*>, size_t> allowed;       // dynamic shared memory, per device and kernel
    int refused = 0;             // launches that asked for more than that
    cudaError_t attribute_error = cudaSuccess;                   // what cudaFuncSetAttribute answers
    std::function<cudaError_t(const void* kernel, bool cooperative)> on_launch;
};

Runtime& runtime();

}  // namespace fake
