// Scenarios of the library's host code on the runtime of fake_cuda.h, one per
// run, named on the command line. Prints what failed and returns 1, or returns 0.
#include <cstdio>
#include <cstring>
#include <functional>
#include <map>
#include <string>
#include <type_traits>
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

// So do the kernels of the wide rows, in the rounds and in the incremental levels.
void wide_rows_on_two_devices() {
    bisim_ctx c;
    c.n = 1000;
    c.m = 100000;
    c.opt.hash_bits = 64;
    c.opt.mid_max_degree = kMidMaxN;
    c.dense_ready = true;
    c.nslots = 2048;
    for (int q = 0; q <= kDClasses; ++q) c.dbegin[q] = 10 * q;
    Buckets B{};
    for (int q = 0; q <= kNumClasses; ++q) B.begin[q] = 10 * q;
    void* state = nullptr;
    cudaMallocAsync(&state, 4096, nullptr);
    c.dstate = static_cast<DevState*>(state);
    c.hstate = static_cast<DevState*>(pinned_take());
    cudaMallocAsync(&state, sizeof(Slot) * c.nslots, nullptr);
    c.table = static_cast<Slot*>(state);
    for (int device : {0, 1}) {
        fake::runtime().device = c.device = device;
        int64_t blocks = 0;
        expect(dense_round(&c, nullptr, &blocks) == BISIM_OK, "a round failed");
        expect(signature_launch(&c, B, nullptr, nullptr, nullptr, 10, nullptr, nullptr) == BISIM_OK, "signatures failed");
        expect(fake::runtime().refused == 0, "a kernel asked for shared memory that was not allowed on its device");
    }
}

// A context of `n` vertices with short rows, laid out as far as the round loop's host code looks.
bisim_ctx& looping_context(int32_t n) {
    bisim_ctx& c = *new bisim_ctx();
    c.n = n;
    c.m = n;
    c.opt.hash_bits = 64;
    c.dense_ready = true;
    c.nslots = 2048;
    for (int q = 1; q <= kDClasses; ++q) c.dbegin[q] = n;
    return c;
}

// Two loops on the per-thread default stream may come from two threads, for which
// the one handle names two streams: the second waits for the first all the same.
void loops_on_one_handle() {
    bisim_ctx* c[2] = {&looping_context(1 << 20), &looping_context(1 << 20)};
    const auto& calls = fake::runtime().calls;
    cudaEvent_t last = nullptr;
    for (int i = 0; i < 2; ++i) {
        fake::runtime().on_launch = [&](const void*, bool) {
            static_cast<LoopState*>(c[i]->hloop)->stop = kStopDone;
            return cudaSuccess;
        };
        LoopState init{}, out{};
        expect(round_loop(c[i], cudaStreamPerThread, true, init, nullptr, &out) == BISIM_OK, "a loop failed");
        size_t at = calls.size();
        while (at > 0 && calls[at - 1].what != "cooperative") --at;
        expect(at > 0, "the loop was not a cooperative launch");
        if (at == 0) return;
        if (i == 1) expect(at > 1 && calls[at - 2].what == "wait" && calls[at - 2].event == last, "the second loop did not wait for the first");
        expect(at < calls.size() && calls[at].what == "record", "no event follows the loop");
        if (at < calls.size()) last = calls[at].event;
    }
}

// A loop that is refused its SMs, or gives up at a barrier, leaves the rounds to
// the captured graph, from P_0 again.
void rounds_without_the_loop() {
    bisim_ctx& c = looping_context(1 << 20);
    const auto device_array = [](auto** p, size_t count) {
        void* q = nullptr;
        cudaMallocAsync(&q, count * sizeof(**p), nullptr);
        *p = static_cast<std::remove_reference_t<decltype(*p)>>(q);
    };
    device_array(&c.P0, c.n);
    device_array(&c.P[0], c.n);
    device_array(&c.P[1], c.n);
    device_array(&c.djoined, c.n);
    device_array(&c.dstate, 1);
    device_array(&c.table, c.nslots);
    c.hstate = static_cast<DevState*>(pinned_take());
    for (int i = 0; i < c.n; ++i) c.P0[i] = 7;
    c.last_blocks = 5;
    for (const bool refuse : {true, false}) {
        int graphs = 0;
        c.P[0][1] = 0;                          // as if the loop had got some way
        fake::runtime().on_launch = [&](const void* kernel, bool cooperative) {
            if (cooperative) return refuse ? cudaErrorCooperativeLaunchTooLarge : cudaSuccess;
            if (kernel == nullptr) {            // the graph
                ++graphs;
                LoopState* L = static_cast<LoopState*>(c.dloop);
                expect(L->prev_blocks == 5 && L->limit == 3 && c.P[0][1] == 7, "the graph did not start from P_0");
                L->stop = kStopDone;
                L->executed = L->rounds = 3;
                L->blocks = 11;
            }
            return cudaSuccess;
        };
        int32_t rounds = 0, executed = 0;
        int64_t blocks = 0;
        expect(dense_rounds_all(&c, 3, 0, nullptr, &rounds, &executed, &blocks, true) == BISIM_OK, "the rounds failed");
        expect(graphs == 1 && rounds == 3 && executed == 3 && blocks == 11, "the graph's result is not the call's");
    }
}

// An init that does not fit with P_0 beside the build fits with P_0 after it.
void init_at_the_memory_limit() {
    const int32_t n = 200000, graphs = 2;
    const int64_t m = 1000000;
    int32_t* a[4];                              // sources, targets, labels; vertex labels
    for (int32_t*& p : a) {
        void* q = nullptr;
        cudaMallocAsync(&q, sizeof(int32_t) * m, nullptr);
        p = static_cast<int32_t*>(q);
    }
    const std::vector<int64_t> vo = {0, n / 2, n}, eo = {0, m / 2, m};
    void* rp = nullptr;
    cudaMallocAsync(&rp, sizeof(int64_t) * (n + 1), nullptr);
    bisim_options o;
    bisim_default_options(&o);
    const std::map<std::string, std::function<bisim_status(bisim_ctx**)>> inits = {
        {"edge list", [&](bisim_ctx** c) { return summarize_init_coo(c, n, m, a[0], a[1], a[2], a[3], nullptr, &o, nullptr); }},
        {"CSR", [&](bisim_ctx** c) { return summarize_init(c, n, m, static_cast<int64_t*>(rp), a[1], a[2], a[3], nullptr, &o, nullptr); }},
        {"batch", [&](bisim_ctx** c) { return summarize_init_batched(c, graphs, vo.data(), eo.data(), a[0], a[1], a[2], a[3], &o, nullptr); }},
    };
    fake::Runtime& R = fake::runtime();
    const size_t before = R.live;
    for (const int direction : {BISIM_DIR_FORWARD, BISIM_DIR_BOTH}) {
        o.direction = direction;
        for (const auto& [what, init] : inits) {
            if (what == "CSR" && direction == BISIM_DIR_FORWARD) continue;      // nothing is staged: no peak to avoid
            bisim_ctx* c = nullptr;
            R.limit = ~size_t{0};
            R.peak = before;
            expect(init(&c) == BISIM_OK, what.c_str());
            summarize_destroy(c);
            R.limit = R.peak - 1;
            expect(init(&c) == BISIM_OK, (what + ", a byte below the peak").c_str());
            summarize_destroy(c);
            R.limit = before + 1000;
            expect(init(&c) != BISIM_OK && c == nullptr, (what + ", next to no memory").c_str());
            expect(R.live == before, (what + ": memory is left behind").c_str());
        }
    }
}

}  // namespace

int main(int argc, char** argv) {
    const std::map<std::string, std::function<void()>> scenarios = {
        {"sort_on_two_devices", sort_on_two_devices},
        {"wide_rows_on_two_devices", wide_rows_on_two_devices},
        {"loops_on_one_handle", loops_on_one_handle},
        {"rounds_without_the_loop", rounds_without_the_loop},
        {"init_at_the_memory_limit", init_at_the_memory_limit},
    };
    const auto s = scenarios.find(argc > 1 ? argv[1] : "");
    if (s == scenarios.end()) {
        std::printf("no such scenario\n");
        return 2;
    }
    s->second();
    return failures ? 1 : 0;
}
