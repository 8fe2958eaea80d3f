// Out-CSR construction, validation and degree bucketing.
#include <algorithm>

#include "common.cuh"
#include "prof.cuh"

namespace bisim {

namespace {

int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }
unsigned grid_for(int64_t n, int threads) {
    return static_cast<unsigned>(std::max<int64_t>(1, cdiv(n, threads)));
}

// Runs of equal keys among a warp's lanes (lane order): a lane heads a run
// when its key differs from the previous lane's. Sources grouped in the edge
// list give a few runs per warp; any order stays correct, with more runs.
__device__ __forceinline__ unsigned run_heads(int32_t key, unsigned lane) {
    const int32_t prev = __shfl_up_sync(0xffffffffu, key, 1);
    return __ballot_sync(0xffffffffu, lane == 0 || prev != key);
}

// Lanes in the run headed by `lane` (a head): up to the next head.
__device__ __forceinline__ int run_length(unsigned heads, unsigned lane) {
    const unsigned after = lane == 31 ? 0u : heads >> (lane + 1);
    return after ? __ffs(after) : 32 - static_cast<int>(lane);
}

// The head of the run that holds `lane`.
__device__ __forceinline__ int run_head(unsigned heads, unsigned lane) {
    const unsigned upto = lane == 31 ? heads : heads & ((2u << lane) - 1u);
    return 31 - __clz(upto);
}

// A flag that other CTAs raise, as this SM's L1 last saw it: a hint that may be
// late. (Past L1 the reads of all warps queue at one sector: 0.55 ms more for
// 100M edges when every edge looked, and 0.09 ms through L1; so the threads
// look at their first two edges and then at every eighth.)
__device__ __forceinline__ bool cached_flag(const unsigned* p) {
    unsigned v;
    asm volatile("ld.global.ca.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v != 0u;
}

// A look at 32 sources in a row at each of up to 4864 places of a long list: whether
// any of them is out of order, before the check below sends its first atomics.
constexpr int64_t kPeekMin = int64_t{1} << 20;
__global__ void __launch_bounds__(256) k_peek_unsorted(const int32_t* __restrict__ src, int64_t m, DevState* st) {
    const int64_t warps = static_cast<int64_t>(gridDim.x) * 8, w = static_cast<int64_t>(blockIdx.x) * 8 + (threadIdx.x >> 5);
    for (int k = 0; k < 4; ++k) {
        const int64_t e = (m - 33) * (4 * w + k) / (4 * warps) + (threadIdx.x & 31u);
        if (__any_sync(0xffffffffu, src[e] > src[e + 1]) && (threadIdx.x & 31u) == 0u) {
            *reinterpret_cast<volatile unsigned*>(&st->unsorted) = 1u;
            return;
        }
    }
}

// Checks every edge (or, with dst null, every source; k_validate_dst then
// checks the targets), and finds out whether the list is sorted by source. For
// a sorted list each source's edges form one run [start, end) of the list:
// the run's first edge records start[v] and adds -start to deg[v], its last
// edge adds end, so deg[v] = end - start (in modular 32-bit arithmetic, exact
// for any degree below 2^32) with two atomics per vertex on distinct
// addresses. For an unsorted list these values are not used (k_count_coo
// counts again), so threads leave the atomics out once the list was found
// unsorted: in a shuffled list every edge ends a run, and a hub's edges
// all go to one address (1.10 ms for 16M shuffled edges of a 1M-vertex
// power-law graph with them; 103 us when the first warps of all had to find out,
// 25 with k_peek_unsorted before. Warps that looked at their own first edges instead
// made a sorted list's check 6% slower). A list that fails the check is not used at all.
// A thread takes four consecutive edges, in 16-byte loads where both arrays allow
// them (`wide`): one edge a thread with 4-byte loads took 0.25 ms for 100M edges.
__global__ void __launch_bounds__(256) k_validate_coo(const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                                                      int64_t m, int32_t n, const uint8_t* __restrict__ alive,
                                                      uint32_t* __restrict__ deg, int64_t* __restrict__ start,
                                                      DevState* st, bool wide) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const int64_t quads = (m + 3) / 4;
    bool unsorted = false;
    unsigned turn = 0;
    for (int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; q < quads; q += stride) {
        const int64_t e0 = 4 * q;
        int32_t s[6], d[4] = {0, 0, 0, 0};                 // s[0] and s[5]: the sources before and after the four
        if (wide && e0 + 4 <= m) {
            const int4 x = __ldcs(reinterpret_cast<const int4*>(src + e0));
            s[1] = x.x;
            s[2] = x.y;
            s[3] = x.z;
            s[4] = x.w;
            if (dst != nullptr) {
                const int4 y = __ldcs(reinterpret_cast<const int4*>(dst + e0));
                d[0] = y.x;
                d[1] = y.y;
                d[2] = y.z;
                d[3] = y.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                s[k + 1] = e0 + k < m ? src[e0 + k] : -1;
                if (dst != nullptr && e0 + k < m) d[k] = dst[e0 + k];
            }
        }
        s[0] = e0 > 0 ? src[e0 - 1] : -1;
        s[5] = e0 + 4 < m ? src[e0 + 4] : -1;
        if (++turn <= 2u || (turn & 7u) == 0u) unsorted = cached_flag(&st->unsorted);
        bool bad = false, back = false;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (e0 + k >= m) break;
            const int32_t v = s[k + 1];
            bool ok = v >= 0 && v < n && d[k] >= 0 && d[k] < n;
            if (ok && alive != nullptr) ok = alive[v] && (dst == nullptr || alive[d[k]]);
            bad = bad || !ok;
            if (!ok || unsorted) continue;
            back = back || s[k] > v;
            if (s[k] != v) {
                start[v] = e0 + k;
                atomicAdd(&deg[v], 0u - static_cast<uint32_t>(e0 + k));
            }
            if (s[k + 2] != v) atomicAdd(&deg[v], static_cast<uint32_t>(e0 + k + 1));
        }
        if (bad) atomicOr(&st->error, kErrBadInput);
        if (back) *reinterpret_cast<volatile unsigned*>(&st->unsorted) = 1u;
    }
}

// The graph of edge e, known to lie in [lo, hi].
__device__ __forceinline__ int32_t graph_of(const int64_t* __restrict__ eoff, int64_t e, int32_t lo, int32_t hi) {
    while (lo < hi) {
        const int32_t mid = lo + (hi - lo + 1) / 2;
        if (eoff[mid] <= e) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// The same for a batched list, whose edges name vertices of their own graph: the
// union's ids are written to B.src and B.dst on the way (deg null: only those, and
// the check). A warp's 128 edges are looked up once: unless a graph ends among
// them, all have the offset of one graph. (A search over all graphs for every
// edge, in a pass before the check: 219 and 77 us for the 37M edges of 512 graphs.)
__global__ void __launch_bounds__(256) k_validate_local(const BatchedList B, const int32_t* __restrict__ src,
                                                        const int32_t* __restrict__ dst, int64_t m,
                                                        uint32_t* __restrict__ deg, int64_t* __restrict__ start, DevState* st,
                                                        bool wide) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const int64_t quads = (m + 3) / 4;
    const int64_t lane = threadIdx.x & 31u;
    bool unsorted = false;
    unsigned turn = 0;
    for (int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; q - lane < quads; q += stride) {
        const int64_t e0 = 4 * q;
        int32_t s[6] = {-1, -1, -1, -1, -1, -1}, d[4] = {0, 0, 0, 0};    // s[0] and s[5]: the sources beside the four
        if (wide && e0 + 4 <= m) {
            const int4 x = __ldcs(reinterpret_cast<const int4*>(src + e0));
            const int4 y = __ldcs(reinterpret_cast<const int4*>(dst + e0));
            s[1] = x.x;
            s[2] = x.y;
            s[3] = x.z;
            s[4] = x.w;
            d[0] = y.x;
            d[1] = y.y;
            d[2] = y.z;
            d[3] = y.w;
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (e0 + k >= m) break;
                s[k + 1] = src[e0 + k];
                d[k] = dst[e0 + k];
            }
        }
        if (e0 > 0 && e0 <= m) s[0] = src[e0 - 1];
        if (e0 + 4 < m) s[5] = src[e0 + 4];
        const int64_t w0 = 4 * (q - lane), w1 = min(w0 + 128, m - 1);    // the warp's edges and the one after
        const int32_t glo = graph_of(B.eoff, max(w0 - 1, int64_t{0}), 0, B.n_graphs - 1);
        const int32_t ghi = B.eoff[glo + 1] > w1 ? glo : graph_of(B.eoff, w1, glo, B.n_graphs - 1);
        int64_t first[6], size[6];
        if (glo == ghi) {
            const int64_t f = B.voff[glo], z = B.voff[glo + 1] - f;
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                first[k] = f;
                size[k] = z;
            }
        } else {
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const int32_t g = graph_of(B.eoff, min(max(e0 + k - 1, int64_t{0}), m - 1), glo, ghi);
                first[k] = B.voff[g];
                size[k] = B.voff[g + 1] - first[k];
            }
        }
        if (++turn <= 2u || (turn & 7u) == 0u) unsorted = cached_flag(&st->unsorted);
        bool bad = false, back = false;
        int32_t v[6], t[4];
#pragma unroll
        for (int k = 0; k < 6; ++k) v[k] = s[k] < 0 ? -1 : static_cast<int32_t>(first[k] + s[k]);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const bool ok = s[k + 1] >= 0 && s[k + 1] < size[k + 1] && d[k] >= 0 && d[k] < size[k + 1];
            t[k] = ok ? static_cast<int32_t>(first[k + 1] + d[k]) : -1;
            if (e0 + k >= m) continue;
            bad = bad || !ok;
            if (!ok || unsorted || deg == nullptr) continue;
            const int32_t x = v[k + 1];
            back = back || v[k] > x;
            if (v[k] != x) {
                start[x] = e0 + k;
                atomicAdd(&deg[x], 0u - static_cast<uint32_t>(e0 + k));
            }
            if (v[k + 2] != x) atomicAdd(&deg[x], static_cast<uint32_t>(e0 + k + 1));
        }
        if (e0 + 4 <= m) {
            *reinterpret_cast<int4*>(B.src + e0) = make_int4(v[1], v[2], v[3], v[4]);
            *reinterpret_cast<int4*>(B.dst + e0) = make_int4(t[0], t[1], t[2], t[3]);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (e0 + k >= m) break;
                B.src[e0 + k] = v[k + 1];
                B.dst[e0 + k] = t[k];
            }
        }
        if (bad) atomicOr(&st->error, kErrBadInput);
        if (back) *reinterpret_cast<volatile unsigned*>(&st->unsorted) = 1u;
    }
}

// The targets' check of a list whose sources k_validate_coo checked alone.
__global__ void __launch_bounds__(256) k_validate_dst(const int32_t* __restrict__ dst, int64_t m, int32_t n,
                                                      const uint8_t* __restrict__ alive, DevState* st) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < m; e += stride) {
        const int32_t d = dst[e];
        if (d < 0 || d >= n || (alive != nullptr && !alive[d])) atomicOr(&st->error, kErrBadInput);
    }
}

__device__ __forceinline__ unsigned long long pack_word(int32_t label, int32_t target) {
    return (static_cast<unsigned long long>(static_cast<uint32_t>(label)) << 32) | static_cast<uint32_t>(target);
}

// Every edge written into its source's packed row of the layout: the row of
// position p is [prp[p], prp[p+1]). A sorted list places edge e at offset
// e - start[v] of its row: no atomics, and the row keeps the list's order.
__global__ void __launch_bounds__(256) k_place_sorted(const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                                                      const int32_t* __restrict__ elab, int64_t m,
                                                      const int32_t* __restrict__ vpos, const int64_t* __restrict__ prp,
                                                      const int64_t* __restrict__ start,
                                                      unsigned long long* __restrict__ pe) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < m; e += stride) {
        const int32_t v = src[e];
        pe[prp[vpos[v]] + (e - start[v])] = pack_word(elab[e], dst[e]);
    }
}

// Unsorted lists: one atomic per edge (per run of equal sources in a warp) counts
// the degrees, and one that returns the edge's place in its row places it. What
// bounds that is the one address of a hub: on a shuffled forward-backward 1M / 16M
// power-law list it took 0.53 ms to count and 1.28 ms to place. So every CTA keeps
// the first sources it meets in a shared-memory table of kHotSources slots, one
// source per slot of its hash. A hub, met within the first few dozen edges, finds
// its slot free; its edges are counted there and sent as one atomic. Any other
// source that finds its slot taken goes straight to memory. (A table that ranks
// all edges of a tile of 2048 was slower on lists without hubs, 0.28 against
// 0.09 ms to count 20M uniform edges.)
constexpr int kTileThreads = 256;
constexpr int kTilePer = 8;
constexpr int kTileEdges = kTileThreads * kTilePer;
constexpr int kHotSources = 1024;

struct HotTable {
    int32_t key[kHotSources];              // source, -1 free
    unsigned cnt[kHotSources];             // its edges since the last flush
    unsigned long long base[kHotSources];  // placement: where the flushed ones start
};

__device__ __forceinline__ void hot_clear(HotTable& t) {
    for (int j = threadIdx.x; j < kHotSources; j += kTileThreads) {
        t.key[j] = -1;
        t.cnt[j] = 0u;
    }
    __syncthreads();
}

// The slot that holds source s, taken by it if free; -1 when another source has it.
__device__ __forceinline__ int hot_slot(HotTable& t, int32_t s) {
    static_assert(kHotSources == 1 << 10, "hash shift");
    const int at = static_cast<int>((static_cast<uint32_t>(s) * 0x9e3779b1u) >> (32 - 10));
    int32_t k = *reinterpret_cast<volatile int32_t*>(&t.key[at]);
    if (k == -1) {
        k = atomicCAS(&t.key[at], -1, s);
        if (k == -1) k = s;
    }
    return k == s ? at : -1;
}

// Out-degrees of an unsorted list.
__global__ void __launch_bounds__(kTileThreads) k_count_coo(const int32_t* __restrict__ src, int64_t m,
                                                            uint32_t* __restrict__ deg) {
    __shared__ HotTable t;
    const unsigned lane = threadIdx.x & 31u;
    hot_clear(t);
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kTileEdges;
    for (int64_t e0 = static_cast<int64_t>(blockIdx.x) * kTileEdges; e0 < m; e0 += stride) {
        int32_t s[kTilePer];
#pragma unroll
        for (int k = 0; k < kTilePer; ++k) {
            const int64_t e = e0 + k * kTileThreads + threadIdx.x;
            s[k] = e < m ? src[e] : -1;
        }
#pragma unroll
        for (int k = 0; k < kTilePer; ++k) {
            const unsigned heads = run_heads(s[k], lane);
            if (s[k] < 0 || !((heads >> lane) & 1u)) continue;
            const unsigned len = static_cast<unsigned>(run_length(heads, lane));
            const int at = hot_slot(t, s[k]);
            if (at >= 0) atomicAdd(&t.cnt[at], len);
            else atomicAdd(&deg[s[k]], len);
        }
    }
    __syncthreads();
    for (int j = threadIdx.x; j < kHotSources; j += kTileThreads)
        if (t.cnt[j]) atomicAdd(&deg[t.key[j]], t.cnt[j]);
}

// Where every vertex's row starts in the packed rows: the cursors of the placement.
__global__ void __launch_bounds__(256) k_row_starts(const int32_t* __restrict__ vpos, int32_t n, int64_t n_live,
                                                    const int64_t* __restrict__ prp,
                                                    unsigned long long* __restrict__ cursor) {
    const int64_t v = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (v >= n) return;
    const int32_t p = vpos[v];
    cursor[v] = p < n_live ? static_cast<unsigned long long>(prp[p]) : 0ull;
}

// Every edge of an unsorted list into its source's row. Signatures are sets,
// so the order of the edges inside a row is never read; it follows the order
// in which the warps and tiles reach the row's cursor.
__global__ void __launch_bounds__(kTileThreads) k_place_coo(const int32_t* __restrict__ src,
                                                            const int32_t* __restrict__ dst,
                                                            const int32_t* __restrict__ elab, int64_t m,
                                                            unsigned long long* __restrict__ cursor,
                                                            unsigned long long* __restrict__ pe) {
    __shared__ HotTable t;
    const unsigned lane = threadIdx.x & 31u;
    hot_clear(t);
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kTileEdges;
    for (int64_t e0 = static_cast<int64_t>(blockIdx.x) * kTileEdges; e0 < m; e0 += stride) {
        int32_t s[kTilePer];
        unsigned long long word[kTilePer], at[kTilePer];
        int hot[kTilePer];
#pragma unroll
        for (int k = 0; k < kTilePer; ++k) {
            const int64_t e = e0 + k * kTileThreads + threadIdx.x;
            s[k] = e < m ? src[e] : -1;
        }
        // the atomics of all of a thread's edges are in flight before any result is used
#pragma unroll
        for (int k = 0; k < kTilePer; ++k) {
            const unsigned heads = run_heads(s[k], lane);
            hot[k] = -1;
            at[k] = 0ull;
            if (s[k] >= 0 && ((heads >> lane) & 1u)) {
                const unsigned len = static_cast<unsigned>(run_length(heads, lane));
                hot[k] = hot_slot(t, s[k]);
                at[k] = hot[k] >= 0 ? atomicAdd(&t.cnt[hot[k]], len) : atomicAdd(&cursor[s[k]], len);
            }
        }
#pragma unroll
        for (int k = 0; k < kTilePer; ++k) {
            const int64_t e = e0 + k * kTileThreads + threadIdx.x;
            word[k] = e < m ? pack_word(elab[e], dst[e]) : 0ull;
        }
        __syncthreads();
        for (int j = threadIdx.x; j < kHotSources; j += kTileThreads) {
            const unsigned c = t.cnt[j];
            if (c) {
                t.base[j] = atomicAdd(&cursor[t.key[j]], static_cast<unsigned long long>(c));
                t.cnt[j] = 0u;
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kTilePer; ++k) {
            const int h = run_head(run_heads(s[k], lane), lane);
            if (hot[k] >= 0) at[k] += t.base[hot[k]];
            const unsigned long long first = __shfl_sync(0xffffffffu, at[k], h);
            if (s[k] >= 0) pe[first + (lane - static_cast<unsigned>(h))] = word[k];
        }
        // the next tile's counts start after every thread passed the first barrier
        // above, and its bases are written after the next one
    }
}

// The check of a CSR, which also makes the context's copy of it (the `to` arrays;
// null: the given ones are the copy). Four edges a thread in 16-byte accesses where
// `wide` says that the given arrays take them: three copies and then a check of one
// edge a thread took 28 and 20 us for 4M edges; this takes 17.
struct CsrCopy {
    int64_t* rp;
    int32_t* col;
    int32_t* elab;
};

__global__ void __launch_bounds__(256) k_validate_csr(const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                                      const int32_t* __restrict__ elab, int32_t n, int64_t m,
                                                      const uint8_t* __restrict__ alive, const CsrCopy to, bool wide,
                                                      unsigned* err) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const int64_t t0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    bool bad = false;
    for (int64_t v = t0; v <= n; v += stride) {
        int64_t a = rp[v];
        bool ok = a >= 0 && a <= m;
        if (v == 0) ok = ok && a == 0;
        if (v == n) ok = ok && a == m;
        if (v < n) {
            int64_t b = rp[v + 1];
            ok = ok && b >= a;
            if (alive != nullptr && !alive[v]) ok = ok && b == a;
        }
        if (to.rp != nullptr) to.rp[v] = a;
        bad = bad || !ok;
    }
    const auto check = [&](int32_t d) { return d >= 0 && d < n && (alive == nullptr || alive[d]); };
    const int64_t quads = wide ? m / 4 : 0;
    for (int64_t q = t0; q < quads; q += stride) {
        const int4 d = reinterpret_cast<const int4*>(col)[q];
        if (to.col != nullptr) {
            reinterpret_cast<int4*>(to.col)[q] = d;
            reinterpret_cast<int4*>(to.elab)[q] = __ldcs(reinterpret_cast<const int4*>(elab) + q);
        }
        bad = bad || !check(d.x) || !check(d.y) || !check(d.z) || !check(d.w);
    }
    for (int64_t e = 4 * quads + t0; e < m; e += stride) {
        const int32_t d = col[e];
        if (to.col != nullptr) {
            to.col[e] = d;
            to.elab[e] = elab[e];
        }
        bad = bad || !check(d);
    }
    if (bad) atomicOr(err, kErrBadInput);
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

void launch_validate_local(bisim_ctx* ctx, const BatchedList& B, const int32_t* src, const int32_t* dst, uint32_t* deg,
                           int64_t* start, cudaStream_t s) {
    const int64_t m = ctx->m;
    if (m <= 0) return;
    BISIM_SITE(site, "batch_globalize");
    Launch L(site, s, 0, m, 16.0 * m);
    k_validate_local<<<grid_for(std::min<int64_t>(cdiv(m, 4), 1 << 22), 256), 256, 0, s>>>(
        B, src, dst, m, deg, start, ctx->dstate, aligned16(src) && aligned16(dst));
}

}  // namespace

bisim_status globalize_edges(bisim_ctx* ctx, const BatchedList& batch, const int32_t* src, const int32_t* dst,
                             cudaStream_t s) {
    cudaMemsetAsync(&ctx->dstate->error, 0, sizeof(unsigned), s);
    launch_validate_local(ctx, batch, src, dst, nullptr, nullptr, s);
    cudaMemcpyAsync(ctx->hstate, ctx->dstate, sizeof(DevState), cudaMemcpyDeviceToHost, s);
    cudaError_t e;
    if ((e = cudaStreamSynchronize(s))) return cuda_error(ctx, e, "globalize batched edges");
    if (ctx->hstate->error & kErrBadInput)
        return set_error(ctx, BISIM_EINVAL, "a graph-local edge endpoint is out of range");
    return BISIM_OK;
}

// COO -> the round layout directly: out-degrees, then the positions of the
// layout (vertices grouped by degree class) and their row offsets, then every
// edge placed into its source's row (k_place_coo). The (label, target) words
// are the layout's packed rows; the vertex-ordered CSR is rebuilt from them
// only if an update or the list-mode path asks for it.
bisim_status build_from_coo(bisim_ctx* ctx, const int32_t* src, const int32_t* dst,
                            const int32_t* elab, cudaStream_t s, const CooArrival* arrival,
                            const BatchedList* batch) {
    const int32_t n = ctx->n;
    const int64_t m = ctx->m;
    const int64_t cap = std::max<int64_t>(m, 1);
    cudaError_t e;
    // scratch: out-degrees, then the runs' first edges (sorted list) or the
    // rows' cursors (unsorted list)
    const size_t nv = static_cast<size_t>(n) + 1;
    const size_t deg_bytes = (sizeof(uint32_t) * nv + 255) & ~size_t(255);
    const size_t bytes = deg_bytes + sizeof(int64_t) * nv;
    char* base = nullptr;
    if ((e = cudaMallocAsync(reinterpret_cast<void**>(&base), bytes, s))) return cuda_error(ctx, e, "alloc CSR scratch");
    uint32_t* deg = reinterpret_cast<uint32_t*>(base);
    int64_t* start = reinterpret_cast<int64_t*>(base + deg_bytes);
    unsigned long long* cursor = reinterpret_cast<unsigned long long*>(start);
    unsigned long long* rows = nullptr;
    if ((e = ctx_alloc(ctx, reinterpret_cast<void**>(&rows), sizeof(unsigned long long) * cap, s))) {
        cudaFreeAsync(base, s);
        return cuda_error(ctx, e, "alloc packed rows");
    }

    cudaMemsetAsync(&ctx->dstate->error, 0, sizeof(unsigned), s);
    cudaMemsetAsync(&ctx->dstate->unsorted, 0, sizeof(unsigned), s);
    cudaMemsetAsync(deg, 0, sizeof(uint32_t) * nv, s);
    BISIM_SITE(site_val, "validate_edges");
    BISIM_SITE(site_cnt, "count_edges");
    BISIM_SITE(site_pack, "csr_place");
    const unsigned grid = grid_for(std::min<int64_t>(m, 1 << 22), 256);
    const unsigned tile_grid = static_cast<unsigned>(std::min<int64_t>(cdiv(m, kTileEdges), 152 * 8));
    const bool wide = aligned16(src) && (arrival || aligned16(dst));
    // arriving arrays: the sources are checked and counted while the targets
    // and labels are still being copied in
    if (arrival != nullptr) cudaStreamWaitEvent(s, arrival->src, 0);
    if (batch == nullptr && m >= kPeekMin) {
        Launch L(site_val, s, 0, 0, 0.0);
        k_peek_unsorted<<<152, 256, 0, s>>>(src, m, ctx->dstate);
    }
    if (batch != nullptr) {
        launch_validate_local(ctx, *batch, src, dst, deg, start, s);
        src = batch->src;
        dst = batch->dst;
    } else if (m > 0)
        Launch(site_val, s, 0, m, arrival ? 4.0 * m : 8.0 * m),
        k_validate_coo<<<grid_for(std::min<int64_t>(cdiv(m, 4), 1 << 22), 256), 256, 0, s>>>(
            src, arrival ? nullptr : dst, m, n, ctx->alive, deg, start, ctx->dstate, wide);
    // the layout of a sorted list follows at once (the degrees of a list that
    // failed the check are never used, whatever they are): one read-back tells
    // both what the check found and where the classes lie
    cudaMemcpyAsync(ctx->hstate, ctx->dstate, sizeof(DevState), cudaMemcpyDeviceToHost, s);
    bisim_status st = dense_layout_positions(ctx, reinterpret_cast<const int32_t*>(deg), s, &ctx->dstate->unsorted);
    if (st == BISIM_OK && ctx->hstate->bad_label) st = edge_view_bad_label(ctx);
    if (st == BISIM_OK && (ctx->hstate->error & kErrBadInput))
        st = set_error(ctx, BISIM_EINVAL, batch ? "a graph-local edge endpoint is out of range"
                                                : "edge endpoint out of range [0, n) or on a dead vertex");
    const bool sorted = ctx->hstate->unsorted == 0;
    if (st == BISIM_OK && !sorted && m > 0) {
        cudaMemsetAsync(deg, 0, sizeof(uint32_t) * nv, s);
        {
            Launch L(site_cnt, s, 0, m, 4.0 * m);
            k_count_coo<<<tile_grid, kTileThreads, 0, s>>>(src, m, deg);
        }
        st = dense_layout_positions(ctx, reinterpret_cast<const int32_t*>(deg), s);
    }
    if (st != BISIM_OK) {
        cudaFreeAsync(base, s);
        return st;
    }
    if (arrival != nullptr && m > 0) {
        cudaStreamWaitEvent(s, arrival->dst, 0);
        {
            Launch L(site_val, s, 0, m, 4.0 * m);
            k_validate_dst<<<grid, 256, 0, s>>>(dst, m, n, ctx->alive, ctx->dstate);
        }
        cudaStreamWaitEvent(s, arrival->lab, 0);
        if (arrival->arrived != nullptr) {
            // the host link is free again: let the next upload start
            if ((e = cudaEventSynchronize(arrival->lab))) {
                cudaFreeAsync(base, s);
                return cuda_error(ctx, e, "edge labels copy");
            }
            arrival->arrived(arrival->arrived_arg);
        }
    }
    if (m > 0) {
        // read src, dst, label, the source's position and row offset; write the packed word
        Launch L(site_pack, s, 0, m, 24.0 * m);
        if (sorted) {
            k_place_sorted<<<grid, 256, 0, s>>>(src, dst, elab, m, ctx->dvpos, ctx->dprp, start, rows);
        } else {
            k_row_starts<<<grid_for(n, 256), 256, 0, s>>>(ctx->dvpos, n, ctx->dbegin[kDClasses], ctx->dprp, cursor);
            k_place_coo<<<tile_grid, kTileThreads, 0, s>>>(src, dst, elab, m, cursor, rows);
        }
    }
    ctx_free(ctx, ctx->dpe, sizeof(unsigned long long) * ctx->dpe_cap, s);
    ctx->dpe = rows;
    ctx->dpe_cap = cap;
    cudaFreeAsync(base, s);
    if ((e = cudaGetLastError())) return cuda_error(ctx, e, "build layout");
    if (arrival != nullptr && m > 0) {
        // the targets' check ran after the layout was made: read it now
        cudaMemcpyAsync(ctx->hstate, ctx->dstate, sizeof(DevState), cudaMemcpyDeviceToHost, s);
        if ((e = cudaStreamSynchronize(s))) return cuda_error(ctx, e, "validate edge targets");
        if (ctx->hstate->error & kErrBadInput)
            return set_error(ctx, BISIM_EINVAL, "edge endpoint out of range [0, n) or on a dead vertex");
    }
    return dense_layout_hubs(ctx, false, s);
}

bisim_status build_from_csr(bisim_ctx* ctx, const int64_t* row_ptr, const int32_t* col,
                            const int32_t* elab, cudaStream_t s, unsigned* later) {
    const int32_t n = ctx->n;
    const int64_t m = ctx->m;
    cudaError_t e;
    if ((e = ctx_alloc(ctx, reinterpret_cast<void**>(&ctx->row_ptr), sizeof(int64_t) * (n + 1), s))) return cuda_error(ctx, e, "alloc row_ptr");
    if ((e = ctx_alloc(ctx, reinterpret_cast<void**>(&ctx->col), sizeof(int32_t) * std::max<int64_t>(m, 1), s))) return cuda_error(ctx, e, "alloc col");
    if ((e = ctx_alloc(ctx, reinterpret_cast<void**>(&ctx->elab), sizeof(int32_t) * std::max<int64_t>(m, 1), s))) return cuda_error(ctx, e, "alloc elab");
    CsrCopy to{ctx->row_ptr, ctx->col, ctx->elab};
    if (!device_accessible(row_ptr) || (m > 0 && (!device_accessible(col) || !device_accessible(elab)))) {
        cudaMemcpyAsync(ctx->row_ptr, row_ptr, sizeof(int64_t) * (n + 1), cudaMemcpyDefault, s);
        if (m > 0) {
            cudaMemcpyAsync(ctx->col, col, sizeof(int32_t) * m, cudaMemcpyDefault, s);
            cudaMemcpyAsync(ctx->elab, elab, sizeof(int32_t) * m, cudaMemcpyDefault, s);
        }
        row_ptr = ctx->row_ptr;
        col = ctx->col;
        elab = ctx->elab;
        to = CsrCopy{nullptr, nullptr, nullptr};
    }
    cudaMemsetAsync(&ctx->dstate->error, 0, sizeof(unsigned), s);
    BISIM_SITE(site_vcsr, "validate_csr");
    const unsigned grid = static_cast<unsigned>(std::min<int64_t>(cdiv(std::max<int64_t>(cdiv(m, 4), n + 1), 256), 152 * 8));
    Launch(site_vcsr, s, n + 1, m, (to.rp ? 16.0 : 8.0) * (n + 1) + (to.rp ? 16.0 : 4.0) * m),
    k_validate_csr<<<grid, 256, 0, s>>>(row_ptr, col, elab, n, m, ctx->alive, to, aligned16(col) && aligned16(elab),
                                        &ctx->dstate->error);
    if (later != nullptr) {
        cudaMemcpyAsync(later, &ctx->dstate->error, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
        return BISIM_OK;
    }
    cudaMemcpyAsync(ctx->hstate, ctx->dstate, sizeof(DevState), cudaMemcpyDeviceToHost, s);
    if ((e = cudaStreamSynchronize(s))) return cuda_error(ctx, e, "validate CSR");
    return csr_checked(ctx, ctx->hstate->error);
}

bisim_status csr_checked(bisim_ctx* ctx, unsigned error) {
    if (error & kErrBadInput)
        return set_error(ctx, BISIM_EINVAL, "malformed CSR: row_ptr not a prefix sum of [0, m], a target out of range, or an edge on a dead vertex");
    return BISIM_OK;
}

}  // namespace bisim
