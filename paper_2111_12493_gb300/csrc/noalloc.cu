// bisim_refine_round_noalloc: one refinement round that allocates nothing.
//
// Some callers cannot allocate device memory at all: code running as a plugin
// inside another runtime that owns the whole device heap (a database engine's
// user-defined function, a custom operator of an inference server), or a
// latency-critical service loop that reserves every buffer up front because an
// allocation call may synchronise the device or fail under fragmentation. They
// pass their inputs and outputs; this entry point keeps all of its scratch in
// one fixed array compiled into the library (sized by kNoAlloc* below), which
// every GPU that loads the library holds until the process exits.
//
// A call is two kernels and one read-back: the first checks the CSR, computes every vertex's set and puts it
// into the table, the second confirms every vertex against its slot's smallest
// one. (With a check of its own and its read-back first, a warp a row and sets
// compared a CTA a pair, a call on 10k vertices and 50k edges took 84 us; it takes
// 42, 10 and 5 of them in the two kernels, the rest in launches and the read-back.)
// Both kernels wait for chains of dependent loads, row offsets to edges to blocks
// to the table, so all that is done for speed is to keep a chain short: the vertices
// spread over every SM, a row's loads in flight together, a table so sparse that
// the first probe mostly ends.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "common.cuh"
#include "prof.cuh"

namespace bisim {

namespace {

constexpr int64_t kNoAllocMaxVertices = 65536;
constexpr int64_t kNoAllocMaxEdges = 1 << 20;
constexpr int64_t kNoAllocMaxDegree = kMidMaxN;
constexpr int64_t kNoAllocSlots = 2 * kNoAllocMaxVertices;   // >= 2n, a power of two

constexpr size_t align256(size_t b) { return (b + 255) & ~size_t(255); }
constexpr size_t kOffState = 0;
constexpr size_t kOffTable = kOffState + align256(sizeof(DevState) * (kEpochCycle + 1));   // one status word per epoch
constexpr size_t kOffVal = kOffTable + align256(sizeof(Slot) * kNoAllocSlots);
constexpr size_t kOffHash = kOffVal + align256(sizeof(unsigned long long) * kNoAllocMaxEdges);
constexpr size_t kOffSlot = kOffHash + align256(sizeof(unsigned long long) * kNoAllocMaxVertices);
constexpr size_t kOffCnt = kOffSlot + align256(sizeof(uint32_t) * kNoAllocMaxVertices);
constexpr size_t kOffU0 = kOffCnt + align256(sizeof(int32_t) * kNoAllocMaxVertices);
constexpr size_t kOffU1 = kOffU0 + align256(sizeof(int32_t) * kNoAllocMaxVertices);
constexpr size_t kNoAllocBytes = kOffU1 + align256(sizeof(int32_t) * kNoAllocMaxVertices);   // about 10.5 MB

constexpr unsigned kErrLongRow = 8u;               // an out-degree above the limit (DevState::error)

// The fixed scratch. In host code this name is only a stand-in for the
// symbol; its device address comes from cudaGetSymbolAddress below.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

// Rows of at most LANE edges are one lane's, of at most kWarpRow a warp's (its set
// has 2 * kWarpRow slots of shared memory), longer ones a CTA's. Two forms of each
// kernel: for a mean row of at most kLongMean edges LANE = 32 in CTAs of at most 512
// threads (each lane's row has a column of shared memory), above it LANE = 8 in CTAs
// of 1024, since it takes the warps of a full SM to hide a row's chain of loads
// (20k rows of 50 edges: 115 against 69 us).
constexpr int kWarpRow = 256;
constexpr int kLongMean = 24;
constexpr int kMaxThreads = 1024;
// Words of shared memory a warp has: its set, or its lanes' columns of LANE values.
template <int LANE>
constexpr int kWarpWords = LANE * 32 > 2 * kWarpRow ? LANE * 32 : 2 * kWarpRow;
constexpr size_t kRoundSmem = sizeof(unsigned long long) * 2 * kNoAllocMaxDegree;
static_assert(sizeof(unsigned long long) * (512 / 32) * kWarpWords<32> <= kRoundSmem, "512 threads");
static_assert(sizeof(unsigned long long) * (kMaxThreads / 32) * kWarpWords<8> <= kRoundSmem, "1024 threads");

struct RoundView {
    const int64_t* rp;
    const int32_t* col;
    const int32_t* lab;
    const int32_t* in;
    int32_t* out;
    int32_t n;
    int64_t m;
    TableRef t;
    unsigned long long* val;       // a row's distinct pair values, from the row's offset on
    unsigned long long* hash;      // by vertex: signature hash, |S|, table slot
    int32_t* cnt;
    uint32_t* slot;
    DevState* st;
};

__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }

// Pair value of edge e; a target out of range is reported and read as vertex 0.
__device__ __forceinline__ uint64_t value_at(const RoundView& V, int32_t target, int32_t label, bool* bad) {
    const bool ok = target >= 0 && target < V.n;
    if (!ok) *bad = true;
    return pair_value(label, V.in[ok ? target : 0]);
}

__device__ __forceinline__ void put_row(const RoundView& V, int32_t v, int32_t own, unsigned count, uint64_t sum) {
    const uint64_t h = sig_hash(own, count, sum);
    V.cnt[v] = static_cast<int32_t>(count);
    V.hash[v] = h;
    V.slot[v] = table_insert(V.t, h, v, &V.st->error);
}

// A lane's row of up to 32 edges, eight at a time: the loads of eight edges are in
// flight together, and their values are compared with each other and with the
// distinct values before them, which lie in the lane's column of shared memory. No
// comparison ends early, so none waits for the one before it; and one loop serves
// every length: straight-line code for 32 values in registers is 30 KB of
// instructions that a call of a few microseconds has to wait for.
__device__ __forceinline__ void lane_row(const RoundView& V, int32_t v, int64_t b, int d, int32_t own,
                                         unsigned long long* mine, bool* bad) {
    uint64_t sum = 0;
    int u = 0;
    int32_t c[8], l[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        c[j] = j < d ? V.col[b + j] : 0;
        l[j] = j < d ? V.lab[b + j] : 0;
    }
    for (int j0 = 0; j0 < d; j0 += 8) {
        uint64_t x[8];
        bool fresh[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = j0 + j < d ? value_at(V, c[j], l[j], bad) : 0ull;
#pragma unroll
        for (int j = 0; j < 8; ++j) {                  // the next eight arrive meanwhile
            c[j] = j0 + 8 + j < d ? V.col[b + j0 + 8 + j] : 0;
            l[j] = j0 + 8 + j < d ? V.lab[b + j0 + 8 + j] : 0;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            fresh[j] = j0 + j < d;
#pragma unroll
            for (int q = 0; q < j; ++q) fresh[j] = fresh[j] & (x[q] != x[j]);
        }
#pragma unroll 4
        for (int q = 0; q < u; ++q) {
            const uint64_t y = mine[32 * q];
#pragma unroll
            for (int j = 0; j < 8; ++j) fresh[j] = fresh[j] & (y != x[j]);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (!fresh[j]) continue;
            if (j0 + 8 < d) mine[32 * u] = x[j];
            V.val[b + u] = x[j];
            sum += x[j];
            ++u;
        }
    }
    put_row(V, v, own, static_cast<unsigned>(u), sum);
}

// A longer row by a group of `size` threads (a warp, or the CTA): every thread
// takes each size-th edge and puts its value into the group's set; values new to
// the set go to the row's list in any order. `out` and `zero` are the group's
// words of shared memory (0 at the start). Returns the warp's part of the sum.
__device__ __forceinline__ uint64_t group_row(const RoundView& V, int64_t b, int d, int at, int size,
                                              unsigned long long* set, uint32_t mask, unsigned* out, unsigned* zero,
                                              bool* bad) {
    uint64_t sum = 0;
    for (int j0 = 0; j0 < d; j0 += size) {
        const int j = j0 + at;
        uint64_t x = 0;
        if (j < d) x = value_at(V, V.col[b + j], V.lab[b + j], bad);
        const bool fresh = j < d && smem_set_insert(set, mask, zero, x);
        const unsigned who = __ballot_sync(0xffffffffu, fresh);
        unsigned to = 0;
        if (lane_id() == 0 && who) to = atomicAdd(out, static_cast<unsigned>(__popc(who)));
        to = __shfl_sync(0xffffffffu, to, 0);
        if (fresh) {
            V.val[b + to + __popc(who & ((1u << lane_id()) - 1u))] = x;
            sum += x;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    return sum;
}

__device__ __forceinline__ uint32_t set_size(int d) {
    uint32_t size = 64;
    while (size < 2u * static_cast<uint32_t>(d)) size <<= 1;
    return size;
}

struct RoundShared {
    int32_t list[kMaxThreads];       // vertices left to the whole CTA
    int32_t other[kMaxThreads];
    unsigned listed;
    unsigned out[kMaxThreads / 32], zero[kMaxThreads / 32];
    unsigned long long sum[kMaxThreads / 32];
    unsigned blocks;
};

// The items are dealt to the CTAs in units of 1 << shift consecutive ones, the CTAs
// turned from round to round so that no period of the ids lands on one of them: a
// CTA's t-th item. Its warps take turns at the units too (my_item). With consecutive
// items a CTA's and a warp's, wide rows that lie side by side (ids by degree) were one
// CTA's or one warp's, one after the other: 20 rows of 8000 edges first among 10k
// vertices took 626 us and take 95, 500 of 300 edges 232 and 71. From 96 items a CTA
// on a unit has four, which keep the short rows' loads together: 65k vertices of four
// edges and two labels 49 us one at a time, 43 in fours (and the 20 rows 177).
__device__ __forceinline__ int64_t dealt_item(int64_t t, int shift) {
    const int64_t u = t >> shift;
    return ((u * gridDim.x + (blockIdx.x + u * 61) % gridDim.x) << shift) + (t & ((1 << shift) - 1));
}

__device__ __forceinline__ int my_item(int warp, int warps, int lane, int shift) {
    return ((((lane >> shift) * warps) + warp) << shift) + (lane & ((1 << shift) - 1));
}

int item_shift(int per_cta) { return per_cta >= 96 ? 2 : 0; }

// Pass 1. A CTA takes `per_cta` vertices at a time, one a lane.
template <int LANE, int THREADS>
__global__ void __launch_bounds__(THREADS) k_noalloc_sign(const RoundView V, int per_cta, int shift) {
    extern __shared__ unsigned long long sets[];
    __shared__ RoundShared sh;
    const int warp = static_cast<int>(threadIdx.x >> 5), warps = static_cast<int>(blockDim.x >> 5);
    const int lane = static_cast<int>(lane_id());
    const int mine = my_item(warp, warps, lane, shift);     // of the CTA's items
    if (threadIdx.x == 0) sh.listed = 0u;
    __syncthreads();
    for (int64_t t0 = 0; t0 * gridDim.x < V.n; t0 += per_cta) {
        const int64_t i = dealt_item(t0 + mine, shift);
        const int32_t v = static_cast<int32_t>(i);
        int32_t own = 0;
        int64_t b = 0;
        int d = -1;                                     // no row to do
        bool bad = false;
        if (mine < per_cta && i < V.n) {
            own = V.in[v];
            b = V.rp[v];
            const int64_t e = V.rp[v + 1];
            bad = b < 0 || e < b || e > V.m || (v == 0 && b != 0) || (v == V.n - 1 && e != V.m);
            if (!bad && e - b > kNoAllocMaxDegree) atomicOr(&V.st->error, kErrLongRow);
            else if (!bad) d = static_cast<int>(e - b);
        }
        if (d >= 0 && d <= LANE) lane_row(V, v, b, d, own, sets + warp * kWarpWords<LANE> + lane, &bad);
        __syncwarp();
        for (unsigned todo = __ballot_sync(0xffffffffu, d > LANE && d <= kWarpRow); todo; todo &= todo - 1u) {
            const int from = __ffs(todo) - 1;
            const int64_t rb = __shfl_sync(0xffffffffu, b, from);
            const int rd = __shfl_sync(0xffffffffu, d, from);
            unsigned long long* set = sets + warp * kWarpWords<LANE>;
            const uint32_t size = set_size(rd);
            for (uint32_t j = lane; j < size; j += 32) set[j] = 0ull;
            if (lane == 0) sh.out[warp] = sh.zero[warp] = 0u;
            __syncwarp();
            const uint64_t sum = group_row(V, rb, rd, lane, 32, set, size - 1, &sh.out[warp], &sh.zero[warp], &bad);
            __syncwarp();
            if (lane == from) put_row(V, v, own, sh.out[warp], sum);
            __syncwarp();
        }
        if (d > kWarpRow) sh.list[atomicAdd(&sh.listed, 1u)] = v;
        __syncthreads();
        const unsigned listed = sh.listed;
        for (unsigned k = 0; k < listed; ++k) {
            const int32_t r = sh.list[k];
            const int64_t rb = V.rp[r];
            const int rd = static_cast<int>(V.rp[r + 1] - rb);
            const uint32_t size = set_size(rd);
            for (uint32_t j = threadIdx.x; j < size; j += blockDim.x) sets[j] = 0ull;
            if (threadIdx.x == 0) sh.out[0] = sh.zero[0] = 0u;
            __syncthreads();
            const uint64_t sum = group_row(V, rb, rd, static_cast<int>(threadIdx.x), static_cast<int>(blockDim.x), sets,
                                           size - 1, &sh.out[0], &sh.zero[0], &bad);
            if (lane == 0) sh.sum[warp] = sum;
            __syncthreads();
            if (threadIdx.x == 0) {
                uint64_t total = 0;
                for (int w = 0; w < warps; ++w) total += sh.sum[w];
                put_row(V, r, V.in[r], sh.out[0], total);
            }
            __syncthreads();
        }
        if (bad) atomicOr(&V.st->error, kErrBadInput);
        if (threadIdx.x == 0) sh.listed = 0u;
        __syncthreads();
    }
}

// Whether two rows of c distinct values are the same set.
__device__ __forceinline__ bool lane_same(const unsigned long long* __restrict__ a,
                                          const unsigned long long* __restrict__ b, int c) {
    int found = 0;
    for (int j0 = 0; j0 < c; j0 += 8) {
        uint64_t x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = j0 + j < c ? a[j0 + j] : 0ull;
#pragma unroll 4
        for (int k = 0; k < c; ++k) {
            const uint64_t y = b[k];
#pragma unroll
            for (int j = 0; j < 8; ++j) found += (j0 + j < c && x[j] == y) ? 1 : 0;
        }
    }
    return found == c;
}

// The same for a group of threads; a thread's answer covers its own part of a.
__device__ __forceinline__ bool group_same(const unsigned long long* a, const unsigned long long* b, int c, int at, int size,
                                           unsigned long long* set, uint32_t mask, unsigned* zero, bool cta) {
    for (int j = at; j < c; j += size) smem_set_insert(set, mask, zero, b[j]);
    if (cta) __syncthreads(); else __syncwarp();
    bool same = true;
    for (int j = at; j < c && same; j += size) same = smem_set_contains(set, mask, *zero, a[j]);
    return same;
}

// Pass 2: every vertex (list null), or every listed one, against its slot's
// smallest vertex: the same own block, size and set, or the vertex goes to the
// list of the next collision level. Does nothing when pass 1 refused the input.
template <int LANE, int THREADS>
__global__ void __launch_bounds__(THREADS) k_noalloc_verify(const RoundView V, const int32_t* __restrict__ list,
                                                            int32_t count, int per_cta, int shift,
                                                            int32_t* __restrict__ next) {
    extern __shared__ unsigned long long sets[];
    __shared__ RoundShared sh;
    if (*reinterpret_cast<volatile unsigned*>(&V.st->error) != 0u) return;   // the same for the whole grid: only pass 1 sets it
    const int warp = static_cast<int>(threadIdx.x >> 5);
    const int lane = static_cast<int>(lane_id());
    const int warps = static_cast<int>(blockDim.x >> 5);
    const int mine = my_item(warp, warps, lane, shift);     // of the CTA's items
    if (threadIdx.x == 0) sh.listed = sh.blocks = 0u;
    __syncthreads();
    for (int64_t t0 = 0; t0 * gridDim.x < count; t0 += per_cta) {
        const int64_t i = dealt_item(t0 + mine, shift);
        int32_t v = -1, r = -1;
        int c = -1;                                     // size of the sets to compare
        bool own = false, push = false;
        if (mine < per_cta && i < count) {
            v = list ? list[i] : static_cast<int32_t>(i);
            r = table_rep(V.t.slots, V.slot[v]);
            if (r == v) own = true;
            else if (V.hash[v] != V.hash[r] || V.cnt[v] != V.cnt[r] || V.in[v] != V.in[r]) push = true;
            else c = V.cnt[v];
        }
        bool same = c == 0;
        const int64_t bv = c > 0 ? V.rp[v] : 0, br = c > 0 ? V.rp[r] : 0;
        if (c > 0 && c <= LANE) same = lane_same(V.val + bv, V.val + br, c);
        __syncwarp();
        for (unsigned todo = __ballot_sync(0xffffffffu, c > LANE && c <= kWarpRow); todo; todo &= todo - 1u) {
            const int from = __ffs(todo) - 1;
            const int64_t a = __shfl_sync(0xffffffffu, bv, from), b = __shfl_sync(0xffffffffu, br, from);
            const int rc = __shfl_sync(0xffffffffu, c, from);
            unsigned long long* set = sets + warp * kWarpWords<LANE>;
            const uint32_t size = set_size(rc);
            for (uint32_t j = lane; j < size; j += 32) set[j] = 0ull;
            if (lane == 0) sh.zero[warp] = 0u;
            __syncwarp();
            const bool all = __all_sync(0xffffffffu, group_same(V.val + a, V.val + b, rc, lane, 32, set, size - 1, &sh.zero[warp], false));
            if (lane == from) same = all;
            __syncwarp();
        }
        bool asked = c > kWarpRow;
        if (asked) {
            const unsigned at = atomicAdd(&sh.listed, 1u);
            sh.list[at] = v;
            sh.other[at] = r;
        }
        __syncthreads();
        const unsigned listed = sh.listed;
        for (unsigned k = 0; k < listed; ++k) {
            const int32_t x = sh.list[k];
            const int rc = V.cnt[x];
            const uint32_t size = set_size(rc);
            for (uint32_t j = threadIdx.x; j < size; j += blockDim.x) sets[j] = 0ull;
            if (threadIdx.x == 0) sh.zero[0] = 0u;
            __syncthreads();
            const bool mine = group_same(V.val + V.rp[x], V.val + V.rp[sh.other[k]], rc, static_cast<int>(threadIdx.x),
                                         static_cast<int>(blockDim.x), sets, size - 1, &sh.zero[0], true);
            const bool all = __syncthreads_and(mine) != 0;
            if (x == v && asked) {
                same = all;
                asked = false;
            }
        }
        if (threadIdx.x == 0) sh.listed = 0u;
        if (own || (c >= 0 && same)) V.out[v] = r;
        push = push || (c >= 0 && !same);
        const unsigned bo = __ballot_sync(0xffffffffu, own), bp = __ballot_sync(0xffffffffu, push);
        if (lane == 0 && bo) atomicAdd(&sh.blocks, static_cast<unsigned>(__popc(bo)));
        if (bp) {
            unsigned at = 0;
            if (lane == 0) at = atomicAdd(&V.st->unresolved, static_cast<unsigned>(__popc(bp)));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (push) next[at + __popc(bp & ((1u << lane) - 1u))] = v;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0 && sh.blocks) atomicAdd(&V.st->blocks, static_cast<unsigned long long>(sh.blocks));
}

// A collision level: the listed vertices enter the table with a re-mixed hash.
__global__ void __launch_bounds__(256) k_noalloc_level(const RoundView V, const int32_t* __restrict__ list, int32_t count,
                                                       uint32_t level) {
    const int i = static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x);
    if (i >= count) return;
    const int32_t v = list[i];
    V.slot[v] = table_insert(V.t, level_hash(V.hash[v], level, ~0ull), v, &V.st->error);
}

std::mutex g_setup_mu;
unsigned char* g_scratch_addr[64] = {};

// Device address of the scratch array for the current device, looked up once
// per device.
cudaError_t scratch_address(int device, unsigned char** out) {
    std::lock_guard<std::mutex> lk(g_setup_mu);
    if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
    if (g_scratch_addr[device] == nullptr) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_scratch_addr[device] = static_cast<unsigned char*>(p);
    }
    *out = g_scratch_addr[device];
    return cudaSuccess;
}

// Whether the kernels of `device` may read or write `p` in place: managed
// memory, or device memory of that same device (memory of another GPU would
// need a peer mapping, which this call does not assume).
bool on_device(const void* p, int device) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (a.type == cudaMemoryTypeManaged) return true;
    return a.type == cudaMemoryTypeDevice && a.device == device;
}

// The next epoch of the device's table and status words. All of them are cleared,
// on `s`, when the epochs start over (and before the first call).
std::mutex g_epoch_mu;
uint32_t g_epoch[64] = {};
uint32_t next_epoch(int device, unsigned char* base, cudaStream_t s) {
    std::lock_guard<std::mutex> lk(g_epoch_mu);
    uint32_t& e = g_epoch[device];
    if (e == 0 || e == kEpochCycle) {
        // a failed clearing (reported with the call's launches) is tried again
        e = cudaMemsetAsync(base, 0, kOffTable + sizeof(Slot) * kNoAllocSlots, s) == cudaSuccess ? 0 : kEpochCycle;
        if (e != 0) return 1;
    }
    return ++e;
}

// The kernels' shared memory, allowed once per device.
cudaError_t allow_round_smem(int device) {
    static std::mutex mu;
    static bool done[64] = {};
    std::lock_guard<std::mutex> lk(mu);
    if (done[device]) return cudaSuccess;
    const auto allow = [](auto kernel) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kRoundSmem));
    };
    cudaError_t e;
    if ((e = allow(k_noalloc_sign<32, 512>)) || (e = allow(k_noalloc_sign<8, 1024>)) ||
        (e = allow(k_noalloc_verify<32, 512>)) || (e = allow(k_noalloc_verify<8, 1024>)))
        return e;
    done[device] = true;
    return cudaSuccess;
}

}  // namespace

}  // namespace bisim

using namespace bisim;

extern "C" bisim_status bisim_refine_round_noalloc(int32_t n_vertices, int64_t n_edges, const int64_t* row_ptr,
                                                   const int32_t* col, const int32_t* edge_label,
                                                   const int32_t* block_in, int32_t* block_out,
                                                   int64_t* out_num_blocks, void* stream) {
    const int32_t n = n_vertices;
    const int64_t m = n_edges;
    if (n < 0 || m < 0) return set_error(nullptr, BISIM_EINVAL, "negative vertex or edge count");
    if (n > kNoAllocMaxVertices || m > kNoAllocMaxEdges)
        return set_error(nullptr, BISIM_EINVAL,
                         "graph exceeds the allocation-free limits (65536 vertices, 1048576 edges)");
    if (n == 0) {
        if (out_num_blocks) *out_num_blocks = 0;
        return BISIM_OK;
    }
    if (row_ptr == nullptr || block_in == nullptr || block_out == nullptr ||
        (m > 0 && (col == nullptr || edge_label == nullptr)))
        return set_error(nullptr, BISIM_EINVAL, "a required array is NULL");
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e) return cuda_error(nullptr, e, "cudaGetDevice");
    if (!on_device(row_ptr, device) || !on_device(block_in, device) || !on_device(block_out, device) ||
        (m > 0 && (!on_device(col, device) || !on_device(edge_label, device))))
        return set_error(nullptr, BISIM_EINVAL,
                         "the allocation-free round needs arrays in the current device's memory");
    if (block_in == block_out) return set_error(nullptr, BISIM_EINVAL, "block_in and block_out must differ");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    unsigned char* base = nullptr;
    if ((e = scratch_address(device, &base))) return cuda_error(nullptr, e, "cudaGetSymbolAddress(scratch)");

    if ((e = allow_round_smem(device))) return cuda_error(nullptr, e, "cudaFuncSetAttribute");

    // The array keeps whatever the previous calls left in it: every call (and
    // every collision level) takes an epoch, whose status word is blank and in
    // which every slot of the table is free. The table is the whole one also for
    // few vertices: nothing is cleared for it, and a probe beyond the first slot
    // costs a read of the L2 cache.
    DevState hs;
    std::memset(&hs, 0, sizeof(hs));
    RoundView V{};
    V.rp = row_ptr;
    V.col = col;
    V.lab = edge_label;
    V.in = block_in;
    V.out = block_out;
    V.n = n;
    V.m = m;
    V.t.slots = reinterpret_cast<Slot*>(base + kOffTable);
    V.t.mask = kNoAllocSlots - 1;
    V.t.hmask = ~0ull;
    V.val = reinterpret_cast<unsigned long long*>(base + kOffVal);
    V.hash = reinterpret_cast<unsigned long long*>(base + kOffHash);
    V.cnt = reinterpret_cast<int32_t*>(base + kOffCnt);
    V.slot = reinterpret_cast<uint32_t*>(base + kOffSlot);
    DevState* states = reinterpret_cast<DevState*>(base + kOffState);
    const auto take_epoch = [&] {
        const uint32_t epoch = next_epoch(device, base, s);
        V.t.epoch = static_cast<uint64_t>(epoch) << 32;
        V.st = states + epoch;
    };
    take_epoch();
    int32_t* list[2] = {reinterpret_cast<int32_t*>(base + kOffU0), reinterpret_cast<int32_t*>(base + kOffU1)};
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    const bool long_rows = m > kLongMean * static_cast<int64_t>(n);
    // small CTAs while they are enough, so that a short list still meets every SM
    const unsigned threads = long_rows ? 1024 : n <= sms * 128 ? 128 : 512;
    // the vertices dealt evenly to the SMs, as far as a CTA has lanes for them
    const auto per_cta = [&](int32_t count) {
        const int32_t even = (count + sms - 1) / sms, unit = 1 << item_shift(even);
        return std::min<int32_t>((even + unit - 1) / unit * unit, static_cast<int32_t>(threads));
    };
    const auto grid = [&](int32_t count) { return std::min<unsigned>((count + per_cta(count) - 1) / per_cta(count), sms); };
    const auto verify = [&](const int32_t* from, int32_t count, int32_t* next) {
        if (long_rows) k_noalloc_verify<8, 1024><<<grid(count), threads, kRoundSmem, s>>>(V, from, count, per_cta(count), item_shift(per_cta(count)), next);
        else k_noalloc_verify<32, 512><<<grid(count), threads, kRoundSmem, s>>>(V, from, count, per_cta(count), item_shift(per_cta(count)), next);
    };
    BISIM_SITE(site_sign, "noalloc_sign");
    BISIM_SITE(site_verify, "noalloc_verify");
    {
        Launch L(site_sign, s, n, m, 28.0 * n + 20.0 * m);
        if (long_rows) k_noalloc_sign<8, 1024><<<grid(n), threads, kRoundSmem, s>>>(V, per_cta(n), item_shift(per_cta(n)));
        else k_noalloc_sign<32, 512><<<grid(n), threads, kRoundSmem, s>>>(V, per_cta(n), item_shift(per_cta(n)));
    }
    {
        Launch L(site_verify, s, n, m, 48.0 * n + 16.0 * m);
        verify(nullptr, n, list[0]);
    }
    const auto read_back = [&]() -> cudaError_t {
        // a launch that failed would leave the status word blank
        cudaError_t err = cudaGetLastError();
        if (err == cudaSuccess) err = cudaMemcpyAsync(&hs, V.st, sizeof(DevState), cudaMemcpyDeviceToHost, s);
        return err == cudaSuccess ? cudaStreamSynchronize(s) : err;
    };
    if ((e = read_back())) return cuda_error(nullptr, e, "allocation-free round");
    if (hs.error & kErrBadInput)
        return set_error(nullptr, BISIM_EINVAL, "malformed CSR: row_ptr not a prefix sum of [0, m] or a target out of range");
    if (hs.error & kErrLongRow)
        return set_error(nullptr, BISIM_EINVAL, "an out-degree exceeds the allocation-free limit of 8192");
    int64_t blocks = static_cast<int64_t>(hs.blocks);
    for (uint32_t level = 1; hs.error == 0 && hs.unresolved > 0; ++level) {
        if (level > 1u << 16) return set_error(nullptr, BISIM_ETIMEOUT, "hash collision resolution did not converge");
        const int32_t left = static_cast<int32_t>(hs.unresolved);
        const int32_t* from = list[(level + 1) & 1];
        take_epoch();
        k_noalloc_level<<<(left + 255) / 256, 256, 0, s>>>(V, from, left, level);
        verify(from, left, list[level & 1]);
        if ((e = read_back())) return cuda_error(nullptr, e, "resolve hash collisions");
        blocks += static_cast<int64_t>(hs.blocks);
    }
    if (hs.error) return set_error(nullptr, BISIM_ETIMEOUT, "signature table probe limit reached");
    if (out_num_blocks) *out_num_blocks = blocks;
    return BISIM_OK;
}
