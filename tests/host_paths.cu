// Scenarios of the library's host code on the runtime of fake_cuda.h, one per
// run, named on the command line. Prints what failed and returns 1, or returns 0.
#include <cstdio>
#include <cstring>
#include <functional>
#include <map>
#include <string>
#include <vector>

#include "bisim.h"
#include "common.cuh"
#include "fake_cuda.h"
#include "rounds.cuh"

using namespace bisim;

namespace {

int failures = 0;

void expect(bool ok, const char* what) {
    if (ok) return;
    std::printf("failed: %s\n", what);
    ++failures;
}

// A sort of more than 2^20 pairs asks for more shared memory than a kernel has
// by default, on each device that sorts. Where it is not allowed the sort says so.
void sort_on_two_devices() {
    const int64_t m = (int64_t{1} << 20) + 1;
    std::vector<int64_t> tmp(radix_temp_words(m));
    int which = 0;
    const auto sort = [&] {
        return radix_sort_pairs(nullptr, nullptr, nullptr, nullptr, m, 16, tmp.data(), nullptr, "radix", &which);
    };
    for (int device : {0, 1, 0, 1}) {
        fake::runtime().device = device;
        expect(sort() == cudaSuccess, "the sort failed");
        expect(fake::runtime().refused == 0, "a pass asked for shared memory that was not allowed on its device");
    }
    fake::runtime().device = 2;
    fake::runtime().attribute_error = cudaErrorInvalidValue;
    expect(sort() == cudaErrorInvalidValue, "shared memory that could not be had went unnoticed");
}

}  // namespace

int main(int argc, char** argv) {
    const std::map<std::string, std::function<void()>> scenarios = {
        {"sort_on_two_devices", sort_on_two_devices},
    };
    const auto s = scenarios.find(argc > 1 ? argv[1] : "");
    if (s == scenarios.end()) {
        std::printf("no such scenario\n");
        return 2;
    }
    s->second();
    return failures ? 1 : 0;
}
