// The summary graph of the current partition: its vertices' payload (the
// number of vertices each block summarizes) and its edges.
//
// Section 2.6 defines the graph summary SG: one vertex per equivalence class,
// and an edge labelled l from the class of u to the class of w for the edges
// (u, w) of the data graph with label l; parallel edges of one label between
// two classes collapse into one. Section 3.1 names counting the summarized
// vertices as the typical payload, merged by adding counts when vertex
// summaries merge. For the partition P held by a context:
//
//   size(b)  = |{ v : P[v] = b }|                          (b a block id)
//   E_vs     = { (P[u], l, P[w]) : (u, w, l) a live edge }  (a set)
//
// The context's rows are the edges by source, so the edges of a source block are
// a few whole rows: every row is copied to its block's segment as (label, target
// block) keys, each segment is sorted and its repeats dropped where it lies, and
// the segments' keys are emitted in the blocks' order. Segments of up to 32 keys
// are sorted in a warp's registers (several at once), up to 256 in a warp's
// shared memory, up to 2048 in a CTA's; the keys of longer ones are brought
// together and radix-sorted by target block, label and segment. A backward
// context's rows hold the edges by target: there, and where few edges lie between
// many vertices, the triples of all edges are radix-sorted by target block, label and
// source block.
//
// On a 1M / 10M power-law graph at k = 2 (9.7M summary edges) ten radix passes over
// all edges took 2.0 of 2.26 ms.
#include <algorithm>
#include <cstddef>
#include <vector>

#include "common.cuh"
#include "prof.cuh"

namespace bisim {

namespace {

__host__ __device__ inline int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

unsigned grid_for(int64_t n, int threads) {
    return static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>(cdiv(n, threads), 152 * 32)));
}

int bits_for(int64_t n) {
    int b = 0;
    while ((int64_t{1} << b) < n) ++b;
    return std::max(b, 1);
}

constexpr uint32_t kLabelFlip = 0x80000000u;   // signed labels sort in signed order as unsigned keys

__global__ void k_block_sizes(const int32_t* __restrict__ P, int32_t n, int32_t* __restrict__ sizes) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t v = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; v < n; v += stride) {
        const int32_t b = P[v];
        if (b >= 0) atomicAdd(&sizes[b], 1);
    }
}

// The last vertex v with rp[v] <= e (rp non-decreasing, rp[0] = 0 <= e < rp[n]),
// searched in [lo, hi].
__device__ __forceinline__ int32_t row_of(const int64_t* __restrict__ rp, int64_t e, int32_t lo, int32_t hi) {
    while (lo < hi) {
        const int32_t mid = lo + (hi - lo + 1) / 2;
        if (rp[mid] <= e) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Pass A keys: every edge's target block (key) with (source block, flipped
// label) as the value. Edges with a dead endpoint get the source block n, so
// that they sort after every live triple. Each CTA takes a tile of edges and
// narrows the search for their source rows to the rows the tile spans.
constexpr int kKeyTile = 2048;
// The context's own edges map back to the caller's (direction.cu): backward
// contexts hold every edge reversed; forward-backward contexts hold (u, w, 2l)
// and the in-edge copy (w, u, 2l + 1), which is left out here.
__global__ void __launch_bounds__(256) k_summary_keys(const int64_t* __restrict__ rp, int32_t n,
                                                      const int32_t* __restrict__ col,
                                                      const int32_t* __restrict__ elab, int64_t m,
                                                      const int32_t* __restrict__ P, int32_t dir,
                                                      uint32_t* __restrict__ key, uint64_t* __restrict__ val) {
    __shared__ int32_t span[2];
    const int64_t tiles = cdiv(m, kKeyTile);
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int64_t e0 = t * kKeyTile;
        const int64_t e1 = e0 + kKeyTile < m ? e0 + kKeyTile : m;
        if (threadIdx.x < 2) span[threadIdx.x] = row_of(rp, threadIdx.x == 0 ? e0 : e1 - 1, 0, n - 1);
        __syncthreads();
        const int32_t lo = span[0], hi = span[1];
        for (int64_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
            const int32_t u = row_of(rp, e, lo, hi);
            int32_t sb = P[u], tb = P[col[e]], l = elab[e];
            bool live = sb >= 0 && tb >= 0;
            if (dir == BISIM_DIR_BACKWARD) {
                const int32_t t = sb;
                sb = tb;
                tb = t;
            } else if (dir == BISIM_DIR_BOTH) {
                live = live && (l & 1) == 0;
                l >>= 1;                                   // arithmetic: 2l -> l for negative l too
            }
            key[e] = live ? static_cast<uint32_t>(tb) : 0u;
            val[e] = (static_cast<uint64_t>(live ? static_cast<uint32_t>(sb) : static_cast<uint32_t>(n)) << 32) |
                     (static_cast<uint32_t>(l) ^ kLabelFlip);
        }
        __syncthreads();
    }
}

// After pass A (key = target block, value = source << 32 | label): key = label,
// value = source << 32 | target.
__global__ void k_summary_to_label(const uint32_t* __restrict__ ki, const uint64_t* __restrict__ vi, int64_t m,
                                   uint32_t* __restrict__ ko, uint64_t* __restrict__ vo) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < m; e += stride) {
        const uint64_t v = vi[e];
        ko[e] = static_cast<uint32_t>(v);
        vo[e] = (v & 0xffffffff00000000ull) | ki[e];
    }
}

// After pass B (key = label, value = source << 32 | target): key = source,
// value = label << 32 | target.
__global__ void k_summary_to_source(const uint32_t* __restrict__ ki, const uint64_t* __restrict__ vi, int64_t m,
                                    uint32_t* __restrict__ ko, uint64_t* __restrict__ vo) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < m; e += stride) {
        const uint64_t v = vi[e];
        ko[e] = static_cast<uint32_t>(v >> 32);
        vo[e] = (static_cast<uint64_t>(ki[e]) << 32) | static_cast<uint32_t>(v);
    }
}

// Sorted triples (key = source, value = label << 32 | target): 1 for the first
// of every run of equal live triples.
__global__ void k_summary_heads(const uint32_t* __restrict__ k, const uint64_t* __restrict__ v, int64_t m,
                                int32_t n, int64_t* __restrict__ head) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e <= m; e += stride) {
        if (e == m) {
            head[e] = 0;
            continue;
        }
        const bool live = k[e] < static_cast<uint32_t>(n);
        head[e] = live && (e == 0 || k[e] != k[e - 1] || v[e] != v[e - 1]) ? 1 : 0;
    }
}

__global__ void k_summary_emit(const uint32_t* __restrict__ k, const uint64_t* __restrict__ v, int64_t m,
                               int32_t n, const int64_t* __restrict__ at, int32_t* __restrict__ os,
                               int32_t* __restrict__ ol, int32_t* __restrict__ ot) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < m; e += stride) {
        if (at[e + 1] == at[e]) continue;                    // not the head of a run
        const int64_t i = at[e];
        os[i] = static_cast<int32_t>(k[e]);
        ol[i] = static_cast<int32_t>(static_cast<uint32_t>(v[e] >> 32) ^ kLabelFlip);
        ot[i] = static_cast<int32_t>(static_cast<uint32_t>(v[e]));
    }
}

// ----------------------------------------------------------------------------- segments by source block

constexpr uint64_t kNoKey = ~0ull;             // not a summary edge (no key has all ones: a block id is below 2^31)
constexpr int kSegWarp = 256;                  // longest segment sorted by a warp
constexpr int kSegCta = 2048;                  // ... by a CTA
constexpr int kSegWarps = 8;

struct SegLists {
    int32_t* cta;                              // blocks with a segment of kSegWarp + 1 .. kSegCta keys
    int32_t* big;                              // longer ones
    unsigned long long* count;                 // [0] cta blocks, [1] big blocks, [2] keys of the big ones,
                                               // [3] smallest and [4] largest label (flipped) of all
};

// Adds `x` to at[b] for the lanes with `on`; the lanes that share the first
// one's b add once (a block can hold most vertices). Returns the value before,
// as if the lanes came in order.
__device__ __forceinline__ int64_t add_grouped(bool on, int32_t b, int64_t x, unsigned long long* at) {
    const unsigned lane = threadIdx.x & 31u;
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (m == 0u) return 0;
    const int lead = __ffs(m) - 1;
    const int32_t lb = __shfl_sync(0xffffffffu, b, lead);
    const bool same = on && b == lb;
    int64_t inc = same ? x : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (static_cast<int>(lane) >= o) inc += y;
    }
    const int64_t total = __shfl_sync(0xffffffffu, inc, 31);
    unsigned long long before = 0;
    if (static_cast<int>(lane) == lead) before = atomicAdd(&at[lb], static_cast<unsigned long long>(total));
    else if (on && !same) before = atomicAdd(&at[b], static_cast<unsigned long long>(x));
    const unsigned long long group = __shfl_sync(0xffffffffu, before, lead);
    return static_cast<int64_t>(same ? group + static_cast<unsigned long long>(inc - x) : before);
}

// Keys per block, and where each vertex's row starts within its block's segment.
__global__ void __launch_bounds__(256) k_seg_sizes(const int64_t* __restrict__ rp, int32_t n,
                                                   const int32_t* __restrict__ P, unsigned long long* __restrict__ size,
                                                   int64_t* __restrict__ at) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t v0 = static_cast<int64_t>(blockIdx.x) * blockDim.x; v0 < n; v0 += stride) {
        const int64_t v = v0 + threadIdx.x;
        const int32_t b = v < n ? P[v] : -1;
        const int64_t d = b >= 0 ? rp[v + 1] - rp[v] : 0;
        const int64_t before = add_grouped(d > 0, b, d, size);
        if (v < n) at[v] = before;
    }
}

// Files the blocks whose segment a warp does not sort.
__global__ void __launch_bounds__(256) k_seg_lists(const int64_t* __restrict__ off, int32_t n, SegLists L) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t b = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; b < n; b += stride) {
        const int64_t len = off[b + 1] - off[b];
        if (len <= kSegWarp) continue;
        if (len <= kSegCta) {
            L.cta[atomicAdd(&L.count[0], 1ull)] = static_cast<int32_t>(b);
        } else {
            L.big[atomicAdd(&L.count[1], 1ull)] = static_cast<int32_t>(b);
            atomicAdd(&L.count[2], static_cast<unsigned long long>(len));
        }
    }
}

// Every edge's key into its block's segment. Each CTA takes a tile of edges and
// narrows the search for their source rows to the rows the tile spans. at[v]:
// where v's row starts in the segment of its block.
__global__ void __launch_bounds__(256) k_seg_keys(const int64_t* __restrict__ rp, int32_t n,
                                                  const int32_t* __restrict__ col, const int32_t* __restrict__ elab,
                                                  int64_t m, const int32_t* __restrict__ P, int32_t dir,
                                                  const int64_t* __restrict__ off, const int64_t* __restrict__ at,
                                                  unsigned long long* __restrict__ seg,
                                                  unsigned long long* __restrict__ range) {
    __shared__ int32_t span[2];
    __shared__ unsigned least, most;
    unsigned lo_l = ~0u, hi_l = 0u;
    if (threadIdx.x == 0) {
        least = ~0u;
        most = 0u;
    }
    const int64_t tiles = cdiv(m, kKeyTile);
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int64_t e0 = t * kKeyTile;
        const int64_t e1 = e0 + kKeyTile < m ? e0 + kKeyTile : m;
        if (threadIdx.x < 2) span[threadIdx.x] = row_of(rp, threadIdx.x == 0 ? e0 : e1 - 1, 0, n - 1);
        __syncthreads();
        const int32_t lo = span[0], hi = span[1];
        for (int64_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
            const int32_t u = row_of(rp, e, lo, hi);
            const int32_t sb = P[u];
            if (sb < 0) continue;                            // a dead vertex's row is in no segment
            const int32_t tb = P[col[e]];
            int32_t l = elab[e];
            bool live = tb >= 0;
            if (dir == BISIM_DIR_BOTH) {
                live = live && (l & 1) == 0;
                l >>= 1;                                     // arithmetic: 2l -> l for negative l too
            }
            const uint32_t fl = static_cast<uint32_t>(l) ^ kLabelFlip;
            if (live) {
                lo_l = min(lo_l, fl);
                hi_l = max(hi_l, fl);
            }
            seg[off[sb] + at[u] + (e - rp[u])] =
                live ? (static_cast<uint64_t>(fl) << 32) | static_cast<uint32_t>(tb) : kNoKey;
        }
        __syncthreads();
    }
    // the labels' range, for the radix passes of the big segments
    lo_l = __reduce_min_sync(0xffffffffu, lo_l);
    hi_l = __reduce_max_sync(0xffffffffu, hi_l);
    __syncthreads();
    if ((threadIdx.x & 31u) == 0) {
        atomicMin(&least, lo_l);
        atomicMax(&most, hi_l);
    }
    __syncthreads();
    if (threadIdx.x == 0 && least <= most) {
        if (least < *reinterpret_cast<volatile unsigned long long*>(&range[0])) atomicMin(&range[0], static_cast<unsigned long long>(least));
        if (most > *reinterpret_cast<volatile unsigned long long*>(&range[1])) atomicMax(&range[1], static_cast<unsigned long long>(most));
    }
}

// Compare-exchange of a bitonic network of `size` keys (a power of two) in
// shared memory by `threads` threads; `sync` separates the steps.
template <class Sync>
__device__ __forceinline__ void bitonic_sort(unsigned long long* c, int size, int t, int threads, const Sync& sync) {
    for (int k = 2; k <= size; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int q = t; q < size / 2; q += threads) {
                const int i = 2 * q - (q & (j - 1));         // the lower index of the q-th pair at distance j
                const unsigned long long a = c[i], b = c[i + j];
                if ((a > b) == ((i & k) == 0)) {
                    c[i] = b;
                    c[i + j] = a;
                }
            }
            sync();
        }
    }
}

// Segments of at most kSegWarp keys: a warp per 32 consecutive blocks. Whole
// segments are packed into the 32 lanes, as many as fit, and sorted together by
// (segment, key) in registers; a segment of 33 keys and more takes the warp's
// shared memory. The distinct keys go back to the segment's start, their number
// to uniq[b].
__global__ void __launch_bounds__(kSegWarps * 32) k_seg_sort_warp(const int64_t* __restrict__ off, int32_t n,
                                                                 unsigned long long* __restrict__ seg,
                                                                 int64_t* __restrict__ uniq) {
    __shared__ unsigned long long buf_all[kSegWarps][kSegWarp];
    const unsigned lane = threadIdx.x & 31u;
    unsigned long long* buf = buf_all[threadIdx.x >> 5];
    const int64_t warps = static_cast<int64_t>(gridDim.x) * kSegWarps;
    for (int64_t b0 = (static_cast<int64_t>(blockIdx.x) * kSegWarps + (threadIdx.x >> 5)) * 32; b0 < n; b0 += warps * 32) {
        const int64_t b = b0 + lane;
        const int64_t o = b < n ? off[b] : 0;
        const int64_t len64 = b < n ? off[b + 1] - o : 0;
        if (b < n && len64 == 0) uniq[b] = 0;
        const int len = len64 <= 32 ? static_cast<int>(len64) : 0;
        int incl = len;
#pragma unroll
        for (int q = 1; q < 32; q <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, q);
            if (static_cast<int>(lane) >= q) incl += y;
        }
        const int excl = incl - len;
        int cur = 0;                                         // first block not done yet
        while (cur < 32) {
            const int done = __shfl_sync(0xffffffffu, excl, cur);
            const unsigned fit = __ballot_sync(0xffffffffu, static_cast<int>(lane) >= cur && incl - done <= 32);
            const int end = cur + __popc(fit);               // incl ascends: the lanes from cur on that fit
            const bool mine = static_cast<int>(lane) >= cur && static_cast<int>(lane) < end && len > 0;
            const unsigned starts = __reduce_or_sync(0xffffffffu, mine ? 1u << (excl - done) : 0u);
            const unsigned owners = __ballot_sync(0xffffffffu, mine);
            const int total = __shfl_sync(0xffffffffu, incl, end - 1) - done;
            cur = end;
            if (total == 0) continue;
            // lane t holds key t - start of the r-th packed segment, the one of lane j
            const unsigned upto = starts & (lane == 31 ? ~0u : (2u << lane) - 1u);
            int r = __popc(upto) - 1;
            const int start = 31 - __clz(upto);              // bit 0 is always set
            const int j = static_cast<int>(__fns(owners, 0, r + 1));
            const int64_t so = __shfl_sync(0xffffffffu, o, j);
            const bool in = static_cast<int>(lane) < total;
            unsigned long long key = in ? seg[so + static_cast<int>(lane) - start] : kNoKey;
            int own = in ? r : 32;
#pragma unroll
            for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
                for (int d = k >> 1; d > 0; d >>= 1) {
                    const unsigned long long pk = __shfl_xor_sync(0xffffffffu, key, d);
                    const int po = __shfl_xor_sync(0xffffffffu, own, d);
                    const bool low = (lane & d) == 0, up = (lane & k) == 0;
                    const bool less = po < own || (po == own && pk < key);       // the partner's is smaller
                    const bool more = po > own || (po == own && pk > key);
                    if (low == up ? less : more) {
                        key = pk;
                        own = po;
                    }
                }
            }
            // a segment's keys are back in its own lanes, in order
            const unsigned long long before = __shfl_up_sync(0xffffffffu, key, 1);
            const bool keep = in && key != kNoKey && (static_cast<int>(lane) == start || before != key);
            const unsigned kept = __ballot_sync(0xffffffffu, keep);
            const unsigned from = kept & ~((1u << start) - 1u);          // from the segment's first lane on
            if (keep) seg[so + __popc(from & ((1u << lane) - 1u))] = key;
            if (mine) {
                const int s0 = excl - done;
                const unsigned lanes = (len == 32 ? ~0u : ((1u << len) - 1u)) << s0;
                uniq[b] = __popc(kept & lanes);
            }
        }
        for (unsigned todo = __ballot_sync(0xffffffffu, len64 > 32 && len64 <= kSegWarp); todo; todo &= todo - 1u) {
            const int q = __ffs(todo) - 1;
            const int64_t so = __shfl_sync(0xffffffffu, o, q);
            const int sl = static_cast<int>(__shfl_sync(0xffffffffu, len64, q));
            const int size = sl <= 64 ? 64 : sl <= 128 ? 128 : 256;
            for (int i = lane; i < size; i += 32) buf[i] = i < sl ? seg[so + i] : kNoKey;
            __syncwarp();
            bitonic_sort(buf, size, static_cast<int>(lane), 32, [] { __syncwarp(); });
            int at = 0;
            for (int i0 = 0; i0 < sl; i0 += 32) {
                const int i = i0 + static_cast<int>(lane);
                const unsigned long long key = i < sl ? buf[i] : kNoKey;
                const bool keep = key != kNoKey && (i == 0 || buf[i - 1] != key);
                const unsigned kept = __ballot_sync(0xffffffffu, keep);
                if (keep) seg[so + at + __popc(kept & ((1u << lane) - 1u))] = key;
                at += __popc(kept);
            }
            if (lane == 0) uniq[b0 + q] = at;
            __syncwarp();                                    // buf is filled again
        }
    }
}

// Segments of kSegWarp + 1 to kSegCta keys: a CTA each.
__global__ void __launch_bounds__(256) k_seg_sort_cta(const int64_t* __restrict__ off, const SegLists L,
                                                      unsigned long long* __restrict__ seg, int64_t* __restrict__ uniq) {
    __shared__ unsigned long long c[kSegCta];
    __shared__ unsigned wsum[8];
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const unsigned long long count = *reinterpret_cast<const volatile unsigned long long*>(&L.count[0]);
    for (unsigned long long s = blockIdx.x; s < count; s += gridDim.x) {
        const int32_t b = L.cta[s];
        const int64_t so = off[b];
        const int len = static_cast<int>(off[b + 1] - so);
        int size = 2 * kSegWarp;
        while (size < len) size <<= 1;
        for (int i = threadIdx.x; i < size; i += 256) c[i] = i < len ? seg[so + i] : kNoKey;
        __syncthreads();
        bitonic_sort(c, size, static_cast<int>(threadIdx.x), 256, [] { __syncthreads(); });
        int at = 0;
        for (int i0 = 0; i0 < len; i0 += 256) {
            const int i = i0 + static_cast<int>(threadIdx.x);
            const unsigned long long key = i < len ? c[i] : kNoKey;
            const bool keep = key != kNoKey && (i == 0 || c[i - 1] != key);
            const unsigned kept = __ballot_sync(0xffffffffu, keep);
            if (lane == 0) wsum[warp] = static_cast<unsigned>(__popc(kept));
            __syncthreads();
            int mine = at, all = 0;
            for (unsigned w = 0; w < 8; ++w) {
                if (w < warp) mine += static_cast<int>(wsum[w]);
                all += static_cast<int>(wsum[w]);
            }
            if (keep) seg[so + mine + __popc(kept & ((1u << lane) - 1u))] = key;
            at += all;
            __syncthreads();
        }
        if (threadIdx.x == 0) uniq[b] = at;
    }
}

// The big segments' keys brought together in the order of the segments' numbers
// (first: the exclusive sum of their lengths). With `tbits` > 0 as one word,
// segment << (tbits + lbits) | (label - lo) << tbits | target, whose low half is
// the key; else key = target block, val = segment << 32 | label.
__global__ void __launch_bounds__(256) k_big_gather(const int64_t* __restrict__ off, const SegLists L, int32_t big,
                                                    const int64_t* __restrict__ first, int64_t m,
                                                    const unsigned long long* __restrict__ seg, int tbits, int lbits,
                                                    uint32_t lo, uint32_t hi, uint32_t* __restrict__ key,
                                                    uint64_t* __restrict__ val) {
    __shared__ int32_t span[2];
    const int64_t tiles = cdiv(m, kKeyTile);
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int64_t e0 = t * kKeyTile;
        const int64_t e1 = e0 + kKeyTile < m ? e0 + kKeyTile : m;
        if (threadIdx.x < 2) span[threadIdx.x] = row_of(first, threadIdx.x == 0 ? e0 : e1 - 1, 0, big - 1);
        __syncthreads();
        const int32_t slo = span[0], shi = span[1];
        for (int64_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
            const int32_t s = row_of(first, e, slo, shi);
            const unsigned long long k = seg[off[L.big[s]] + (e - first[s])];
            const uint32_t l = static_cast<uint32_t>(k >> 32), tb = static_cast<uint32_t>(k);
            uint64_t v = (static_cast<uint64_t>(s) << 32) | l;
            if (tbits > 0) {
                // what is no edge has all ones for its target, which no target has
                v = (((static_cast<uint64_t>(s) << lbits) | (min(l, hi) - lo)) << tbits) |
                    (tb & static_cast<uint32_t>((uint64_t{1} << tbits) - 1));
            }
            key[e] = tbits > 0 ? static_cast<uint32_t>(v) : tb;
            val[e] = v;
        }
        __syncthreads();
    }
}

// The words' high halves as the next keys.
__global__ void k_big_high(const uint64_t* __restrict__ v, int64_t m, uint32_t* __restrict__ key) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < m; e += stride)
        key[e] = static_cast<uint32_t>(v[e] >> 32);
}

// The words taken apart: key = segment, val = label << 32 | target (all ones: no edge).
__global__ void k_big_split(uint32_t* __restrict__ key, uint64_t* __restrict__ val, int64_t m, int tbits, int lbits,
                            uint32_t lo) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const uint64_t tmask = (uint64_t{1} << tbits) - 1;
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < m; e += stride) {
        const uint64_t v = val[e];
        const uint32_t l = static_cast<uint32_t>(v >> tbits) & static_cast<uint32_t>((uint64_t{1} << lbits) - 1);
        const uint32_t t = (v & tmask) == tmask ? ~0u : static_cast<uint32_t>(v & tmask);
        key[e] = static_cast<uint32_t>(v >> (tbits + lbits));
        val[e] = (static_cast<uint64_t>(l + lo) << 32) | t;
    }
}

// After the sort by target block: key = label above the smallest one, val =
// segment << 32 | target. An edge that is none keeps its place among the rest
// (its target word is all ones).
__global__ void k_big_to_label(const uint32_t* __restrict__ ki, const uint64_t* __restrict__ vi, int64_t m, uint32_t lo,
                               uint32_t hi, uint32_t* __restrict__ ko, uint64_t* __restrict__ vo) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < m; e += stride) {
        const uint64_t v = vi[e];
        ko[e] = min(static_cast<uint32_t>(v), hi) - lo;
        vo[e] = (v & 0xffffffff00000000ull) | ki[e];
    }
}

// After the sort by label: key = segment, val = label << 32 | target.
__global__ void k_big_to_segment(const uint32_t* __restrict__ ki, const uint64_t* __restrict__ vi, int64_t m, uint32_t lo,
                                 uint32_t* __restrict__ ko, uint64_t* __restrict__ vo) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < m; e += stride) {
        const uint64_t v = vi[e];
        ko[e] = static_cast<uint32_t>(v >> 32);
        vo[e] = (static_cast<uint64_t>(ki[e] + lo) << 32) | static_cast<uint32_t>(v);
    }
}

// Sorted big keys: 1 for the first of every run of equal ones of a segment.
__global__ void k_big_heads(const uint32_t* __restrict__ k, const uint64_t* __restrict__ v, int64_t m,
                            int64_t* __restrict__ head) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e <= m; e += stride) {
        if (e == m) {
            head[e] = 0;
            continue;
        }
        const bool live = static_cast<uint32_t>(v[e]) != ~0u;
        head[e] = live && (e == 0 || k[e] != k[e - 1] || v[e] != v[e - 1]) ? 1 : 0;
    }
}

// The distinct keys back to their segments' starts. Segments come in the order
// of their numbers, each at the exclusive sum of the lengths before it.
__global__ void k_big_scatter(const uint32_t* __restrict__ k, const uint64_t* __restrict__ v, int64_t m,
                              const int64_t* __restrict__ rank, const int64_t* __restrict__ first,
                              const int64_t* __restrict__ off, const SegLists L, unsigned long long* __restrict__ seg,
                              int64_t* __restrict__ uniq) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const int64_t t0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    for (int64_t e = t0; e < m; e += stride) {
        if (rank[e + 1] == rank[e]) continue;                // not the head of a run
        const uint32_t s = k[e];
        seg[off[L.big[s]] + (rank[e] - rank[first[s]])] = v[e];
    }
    const int64_t big = static_cast<int64_t>(L.count[1]);
    for (int64_t s = t0; s < big; s += stride) uniq[L.big[s]] = rank[first[s + 1]] - rank[first[s]];
}

// Lengths of the big segments (for the exclusive sum that gives `first`).
__global__ void k_big_lengths(const int64_t* __restrict__ off, const SegLists L, int64_t* __restrict__ len) {
    const int64_t big = static_cast<int64_t>(L.count[1]);
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t s = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; s <= big; s += stride)
        len[s] = s < big ? off[L.big[s] + 1] - off[L.big[s]] : 0;
}

// Summary edge i (below `take`) is key i - at[b] of the block b whose keys are
// emitted from at[b] on. Tiles narrow the search for b as for the source rows.
__global__ void __launch_bounds__(256) k_seg_emit(const int64_t* __restrict__ at, int32_t n, int64_t take,
                                                  const int64_t* __restrict__ off,
                                                  const unsigned long long* __restrict__ seg, int32_t* __restrict__ os,
                                                  int32_t* __restrict__ ol, int32_t* __restrict__ ot) {
    __shared__ int32_t span[2];
    const int64_t tiles = cdiv(take, kKeyTile);
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int64_t i0 = t * kKeyTile;
        const int64_t i1 = i0 + kKeyTile < take ? i0 + kKeyTile : take;
        if (threadIdx.x < 2) span[threadIdx.x] = row_of(at, threadIdx.x == 0 ? i0 : i1 - 1, 0, n - 1);
        __syncthreads();
        const int32_t lo = span[0], hi = span[1];
        for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
            const int32_t b = row_of(at, i, lo, hi);
            const unsigned long long k = seg[off[b] + (i - at[b])];
            os[i] = b;
            ol[i] = static_cast<int32_t>(static_cast<uint32_t>(k >> 32) ^ kLabelFlip);
            ot[i] = static_cast<int32_t>(static_cast<uint32_t>(k));
        }
        __syncthreads();
    }
}

// The segments take a dozen passes over all blocks, the radix sorts ten over all
// edges: many vertices with few edges between them are better sorted. us by segments
// and by radix, vertices and edges in millions: 1 and 0.5 280 / 457; 3 and 0.3 457 /
// 430; 3 and 1.5 564 / 617; 10 and 0.5 794 / 490; 10 and 5 1,328 / 1,059; 10 and 10
// 1,515 / 1,803; 30 and 3 1,749 / 880; 30 and 15 3,500 / 2,680.
bool fewer_edges_than_passes_over_blocks(int64_t n, int64_t m) { return 10 * m < 7 * (n - 1250000); }

// A backward context, or few edges for its vertices: the triples of all edges sorted
// by target block, label and source block. *out_base (freed by the caller) holds the compacted triples
// os, ol, ot.
bisim_status summary_by_radix(bisim_ctx* ctx, cudaStream_t s, char** out_base, const int32_t** out_os,
                              const int32_t** out_ol, const int32_t** out_ot, int64_t* out_count) {
    cudaError_t e;
    const int32_t n = ctx->n;
    const int64_t m = ctx->m;
    // scratch: keys and values twice (radix ping-pong), run heads and their offsets, the radix temp,
    // the compacted triples
    const size_t tmp_words = std::max(radix_temp_words(m), scan_temp_words(m + 1));
    // every piece starts on a 256-byte boundary: the allocation is the sum of the rounded sizes
    auto r256 = [](size_t b) { return (b + 255) & ~size_t(255); };
    const size_t mm = static_cast<size_t>(m);
    const size_t bytes = 2 * r256(sizeof(uint32_t) * mm) + 2 * r256(sizeof(uint64_t) * mm) +
                         2 * r256(sizeof(int64_t) * (mm + 1)) + r256(sizeof(int64_t) * tmp_words) +
                         3 * r256(sizeof(int32_t) * mm);
    char* base = nullptr;
    if ((e = cudaMallocAsync(reinterpret_cast<void**>(&base), bytes, s))) return cuda_error(ctx, e, "alloc summary scratch");
    char* cur = base;
    auto carve = [&](size_t b) { char* p = cur; cur += r256(b); return p; };
    uint32_t* k0 = reinterpret_cast<uint32_t*>(carve(sizeof(uint32_t) * m));
    uint32_t* k1 = reinterpret_cast<uint32_t*>(carve(sizeof(uint32_t) * m));
    uint64_t* v0 = reinterpret_cast<uint64_t*>(carve(sizeof(uint64_t) * m));
    uint64_t* v1 = reinterpret_cast<uint64_t*>(carve(sizeof(uint64_t) * m));
    int64_t* head = reinterpret_cast<int64_t*>(carve(sizeof(int64_t) * (m + 1)));
    int64_t* at = reinterpret_cast<int64_t*>(carve(sizeof(int64_t) * (m + 1)));
    int64_t* tmp = reinterpret_cast<int64_t*>(carve(sizeof(int64_t) * tmp_words));
    int32_t* os = reinterpret_cast<int32_t*>(carve(sizeof(int32_t) * m));
    int32_t* ol = reinterpret_cast<int32_t*>(carve(sizeof(int32_t) * m));
    int32_t* ot = reinterpret_cast<int32_t*>(carve(sizeof(int32_t) * m));
    const int32_t* P = ctx->P[ctx->cur];
    BISIM_SITE(site, "summary_edges");
    int64_t count = 0;
    {
        Launch L(site, s, n, m, 48.0 * m);
        k_summary_keys<<<grid_for(cdiv(m, kKeyTile) * 256, 256), 256, 0, s>>>(ctx->row_ptr, n, ctx->col, ctx->elab, m,
                                                                                P, ctx->opt.direction, k0, v0);
    }
    const auto fail = [&](cudaError_t err, const char* what) {
        cudaFreeAsync(base, s);
        return cuda_error(ctx, err, what);
    };
    // pass A: by target block (stable), the result in (k0, v0) or (k1, v1)
    int w = 0;
    if ((e = radix_sort_pairs(k0, v0, k1, v1, m, bits_for(n), tmp, s, "summary_radix", &w))) return fail(e, "summary sort");
    uint32_t* ka = w ? k1 : k0;
    uint64_t* va = w ? v1 : v0;
    uint32_t* kb = w ? k0 : k1;
    uint64_t* vb = w ? v0 : v1;
    k_summary_to_label<<<grid_for(m, 256), 256, 0, s>>>(ka, va, m, kb, vb);
    // pass B: by label
    if ((e = radix_sort_pairs(kb, vb, ka, va, m, 32, tmp, s, "summary_radix", &w))) return fail(e, "summary sort");
    uint32_t* kc = w ? ka : kb;
    uint64_t* vc = w ? va : vb;
    uint32_t* kd = w ? kb : ka;
    uint64_t* vd = w ? vb : va;
    k_summary_to_source<<<grid_for(m, 256), 256, 0, s>>>(kc, vc, m, kd, vd);
    // pass C: by source block (dead-endpoint edges carry n and sort last)
    if ((e = radix_sort_pairs(kd, vd, kc, vc, m, bits_for(static_cast<int64_t>(n) + 1), tmp, s, "summary_radix", &w)))
        return fail(e, "summary sort");
    const uint32_t* kf = w ? kc : kd;
    const uint64_t* vf = w ? vc : vd;
    {
        Launch L(site, s, 0, m, 36.0 * m);
        k_summary_heads<<<grid_for(m + 1, 256), 256, 0, s>>>(kf, vf, m, n, head);
        exclusive_scan_i64(head, at, m + 1, tmp, s);
        k_summary_emit<<<grid_for(m, 256), 256, 0, s>>>(kf, vf, m, n, at, os, ol, ot);
    }
    cudaMemcpyAsync(&count, at + m, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
    if ((e = cudaStreamSynchronize(s))) return fail(e, "summary edges");
    if (cur - base != static_cast<ptrdiff_t>(bytes) || count < 0 || count > m) {
        cudaFreeAsync(base, s);
        return set_error(ctx, BISIM_ECUDA, "summary edges: inconsistent scratch layout or count");
    }
    *out_base = base;
    *out_os = os;
    *out_ol = ol;
    *out_ot = ot;
    *out_count = count;
    return BISIM_OK;
}

// Any other context: keys by source block in *out_seg (from off[b] on), of which
// the first at[b + 1] - at[b] of a block are its summary edges. *out_base (freed
// by the caller) holds it all.
bisim_status summary_by_segment(bisim_ctx* ctx, cudaStream_t s, char** out_base, const unsigned long long** out_seg,
                                const int64_t** out_off, const int64_t** out_at, int64_t* out_count) {
    cudaError_t e;
    const int32_t n = ctx->n;
    const int64_t m = ctx->m;
    const size_t nn = static_cast<size_t>(n) + 1, mm = static_cast<size_t>(m);
    const size_t n_cta = std::min(nn, mm / (kSegWarp + 1) + 1), n_big = std::min(nn, mm / (kSegCta + 1) + 1);
    auto r256 = [](size_t b) { return (b + 255) & ~size_t(255); };
    const size_t bytes = r256(8 * mm) + 4 * r256(8 * nn) + r256(4 * n_cta) + r256(4 * n_big) + r256(8 * 5) + r256(8 * scan_temp_words(n + 1));
    char* base = nullptr;
    if ((e = cudaMallocAsync(reinterpret_cast<void**>(&base), bytes, s))) return cuda_error(ctx, e, "alloc summary scratch");
    char* cur = base;
    auto carve = [&](size_t b) { char* p = cur; cur += r256(b); return p; };
    unsigned long long* seg = reinterpret_cast<unsigned long long*>(carve(8 * mm));
    int64_t* size = reinterpret_cast<int64_t*>(carve(8 * nn));         // keys per block, later the distinct ones
    int64_t* off = reinterpret_cast<int64_t*>(carve(8 * nn));
    int64_t* row = reinterpret_cast<int64_t*>(carve(8 * nn));
    int64_t* at = reinterpret_cast<int64_t*>(carve(8 * nn));
    SegLists L;
    L.cta = reinterpret_cast<int32_t*>(carve(4 * n_cta));
    L.big = reinterpret_cast<int32_t*>(carve(4 * n_big));
    L.count = reinterpret_cast<unsigned long long*>(carve(8 * 5));
    int64_t* tmp = reinterpret_cast<int64_t*>(carve(8 * scan_temp_words(n + 1)));
    const int32_t* P = ctx->P[ctx->cur];
    BISIM_SITE(site, "summary_edges");
    Branch warps, ctas;
    auto fail = [&](cudaError_t err, const char* what) {
        branch_join(ctx->device, &warps, s);
        branch_join(ctx->device, &ctas, s);
        cudaFreeAsync(base, s);
        return cuda_error(ctx, err, what);
    };
    cudaMemsetAsync(size, 0, 8 * nn, s);
    cudaMemsetAsync(L.count, 0, 8 * 5, s);
    cudaMemsetAsync(L.count + 3, 0xff, 8, s);
    {
        Launch Lk(site, s, n, 0, 28.0 * n);
        k_seg_sizes<<<grid_for(n, 256), 256, 0, s>>>(ctx->row_ptr, n, P, reinterpret_cast<unsigned long long*>(size), row);
    }
    exclusive_scan_i64(size, off, n + 1, tmp, s);
    {
        Launch Lk(site, s, n, 0, 8.0 * n);
        k_seg_lists<<<grid_for(n, 256), 256, 0, s>>>(off, n, L);
    }
    {
        Launch Lk(site, s, n, m, 20.0 * m);
        k_seg_keys<<<grid_for(cdiv(m, kKeyTile) * 256, 256), 256, 0, s>>>(ctx->row_ptr, n, ctx->col, ctx->elab, m, P,
                                                                         ctx->opt.direction, off, row, seg, L.count + 3);
    }
    int64_t* uniq = size;
    cudaMemsetAsync(uniq + n, 0, 8, s);
    // the three kinds of segments are sorted beside each other: the long ones' passes
    // on `s`, started by the host as soon as it knows how many there are, and the
    // others, which run from shared memory, on branches (1M / 10M: 131 and 119 us of
    // kernels beside 400)
    if (!prof_enabled()) {
        warps = branch_fork(ctx->device, s);
        ctas = branch_fork(ctx->device, s);
    }
    const cudaStream_t ws = warps.s ? warps.s : s, ts = ctas.s ? ctas.s : s;
    unsigned long long h[5] = {};
    {
        Launch Lk(site, ws, n, m, 16.0 * m);
        k_seg_sort_warp<<<grid_for(cdiv(n, 32 * kSegWarps) * 256, 256), kSegWarps * 32, 0, ws>>>(off, n, seg, uniq);
    }
    {
        Launch Lk(site, ts, 0, 0, 0.0);
        k_seg_sort_cta<<<static_cast<unsigned>(std::min<size_t>(n_cta, 152 * 8)), 256, 0, ts>>>(off, L, seg, uniq);
    }
    cudaMemcpyAsync(h, L.count, sizeof(h), cudaMemcpyDeviceToHost, s);
    if ((e = cudaStreamSynchronize(s))) return fail(e, "summary segments");
    const int64_t big = static_cast<int64_t>(h[1]), bm = static_cast<int64_t>(h[2]);
    if (big > 0) {
        const size_t tw = std::max({radix_temp_words(bm), scan_temp_words(bm + 1), scan_temp_words(big + 1)});
        const size_t bytes2 = 2 * r256(4 * bm) + 2 * r256(8 * (bm + 1)) + 2 * r256(8 * (big + 1)) + r256(8 * tw);
        char* more = nullptr;
        if ((e = cudaMallocAsync(reinterpret_cast<void**>(&more), bytes2, s))) return fail(e, "alloc summary sort");
        char* q = more;
        auto carve2 = [&](size_t b) { char* p = q; q += r256(b); return p; };
        uint32_t* ka = reinterpret_cast<uint32_t*>(carve2(4 * bm));
        uint32_t* kb = reinterpret_cast<uint32_t*>(carve2(4 * bm));
        uint64_t* va = reinterpret_cast<uint64_t*>(carve2(8 * (bm + 1)));
        uint64_t* vb = reinterpret_cast<uint64_t*>(carve2(8 * (bm + 1)));
        int64_t* len = reinterpret_cast<int64_t*>(carve2(8 * (big + 1)));
        int64_t* first = reinterpret_cast<int64_t*>(carve2(8 * (big + 1)));
        int64_t* btmp = reinterpret_cast<int64_t*>(carve2(8 * tw));
        const uint32_t lo = h[3] > h[4] ? 0u : static_cast<uint32_t>(h[3]), hi = h[3] > h[4] ? 0u : static_cast<uint32_t>(h[4]);
        Launch Lk(site, s, big, bm, 40.0 * bm);
        const int tbits = bits_for(static_cast<int64_t>(n) + 1);       // all ones: above every target
        const int lbits = bits_for(static_cast<int64_t>(hi - lo) + 1), sbits = bits_for(big);
        const bool one = tbits + lbits + sbits <= 64;                  // a triple fits in one word
        k_big_lengths<<<grid_for(big + 1, 256), 256, 0, s>>>(off, L, len);
        exclusive_scan_i64(len, first, big + 1, btmp, s);
        k_big_gather<<<grid_for(cdiv(bm, kKeyTile) * 256, 256), 256, 0, s>>>(off, L, static_cast<int32_t>(big), first, bm, seg,
                                                                           one ? tbits : 0, lbits, lo, hi, ka, va);
        // the result of each sort in (ka, va), the other pair free; after a sort that
        // failed nothing is looked up by its keys any more
        auto turn = [&] {
            std::swap(ka, kb);
            std::swap(va, vb);
        };
        auto sort = [&](int bits) {
            int w = 0;
            e = radix_sort_pairs(ka, va, kb, vb, bm, bits, btmp, s, "summary_radix", &w);
            if (w) turn();
            return e == cudaSuccess;
        };
        if (one) {
            if (sort(std::min(32, tbits + lbits + sbits))) {
                if (tbits + lbits + sbits > 32) {
                    k_big_high<<<grid_for(bm, 256), 256, 0, s>>>(va, bm, ka);
                    sort(tbits + lbits + sbits - 32);
                }
                k_big_split<<<grid_for(bm, 256), 256, 0, s>>>(ka, va, bm, tbits, lbits, lo);
            }
        } else if (sort(tbits)) {
            k_big_to_label<<<grid_for(bm, 256), 256, 0, s>>>(ka, va, bm, lo, hi, kb, vb);
            turn();
            if (sort(lbits)) {
                k_big_to_segment<<<grid_for(bm, 256), 256, 0, s>>>(ka, va, bm, lo, kb, vb);
                turn();
                sort(sbits);
            }
        }
        if (e) {
            cudaFreeAsync(more, s);
            return fail(e, "summary sort");
        }
        int64_t* rank = reinterpret_cast<int64_t*>(vb);
        k_big_heads<<<grid_for(bm + 1, 256), 256, 0, s>>>(ka, va, bm, rank);
        exclusive_scan_i64(rank, rank, bm + 1, btmp, s);
        k_big_scatter<<<grid_for(bm, 256), 256, 0, s>>>(ka, va, bm, rank, first, off, L, seg, uniq);
        cudaFreeAsync(more, s);
    }
    branch_join(ctx->device, &warps, s);
    branch_join(ctx->device, &ctas, s);
    exclusive_scan_i64(uniq, at, n + 1, tmp, s);
    int64_t count = 0;
    cudaMemcpyAsync(&count, at + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
    if ((e = cudaStreamSynchronize(s))) return fail(e, "summary edges");
    if (cur - base != static_cast<ptrdiff_t>(bytes) || count < 0 || count > m) {
        cudaFreeAsync(base, s);
        return set_error(ctx, BISIM_ECUDA, "summary edges: inconsistent scratch layout or count");
    }
    *out_base = base;
    *out_seg = seg;
    *out_off = off;
    *out_at = at;
    *out_count = count;
    return BISIM_OK;
}

}  // namespace

}  // namespace bisim

using namespace bisim;

extern "C" {

bisim_status get_block_sizes(bisim_ctx* ctx, int32_t* sizes, void* stream) {
    if (ctx == nullptr) return set_error(nullptr, BISIM_EINVAL, "ctx is NULL");
    ctx->last_stream = stream;
    if (ctx->n == 0) return BISIM_OK;
    if (sizes == nullptr) return set_error(ctx, BISIM_EINVAL, "output is NULL");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaError_t e;
    int32_t* d = nullptr;
    if ((e = cudaMallocAsync(reinterpret_cast<void**>(&d), sizeof(int32_t) * ctx->n, s)))
        return cuda_error(ctx, e, "alloc block sizes");
    cudaMemsetAsync(d, 0, sizeof(int32_t) * ctx->n, s);
    BISIM_SITE(site, "block_sizes");
    {
        Launch L(site, s, ctx->n, 0, 8.0 * ctx->n);
        k_block_sizes<<<grid_for(ctx->n, 256), 256, 0, s>>>(ctx->P[ctx->cur], ctx->n, d);
    }
    e = cudaMemcpyAsync(sizes, d, sizeof(int32_t) * ctx->n, cudaMemcpyDefault, s);
    cudaFreeAsync(d, s);
    if (e || (e = cudaStreamSynchronize(s))) return cuda_error(ctx, e, "block sizes");
    return BISIM_OK;
}

bisim_status get_summary_edges(bisim_ctx* ctx, int32_t* src_block, int32_t* label, int32_t* dst_block,
                               int64_t capacity, int64_t* out_count, void* stream) {
    if (ctx == nullptr) return set_error(nullptr, BISIM_EINVAL, "ctx is NULL");
    ctx->last_stream = stream;
    if (out_count == nullptr || capacity < 0) return set_error(ctx, BISIM_EINVAL, "invalid count or capacity");
    if (capacity > 0 && (src_block == nullptr || label == nullptr || dst_block == nullptr))
        return set_error(ctx, BISIM_EINVAL, "an output array is NULL");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaError_t e;
    bisim_status st;
    *out_count = 0;
    if ((st = ensure_vertex_csr(ctx, s)) != BISIM_OK) return st;
    const int32_t n = ctx->n;
    const int64_t m = ctx->m;
    if (n == 0 || m == 0) return BISIM_OK;
    const bool by_radix = ctx->opt.direction == BISIM_DIR_BACKWARD || fewer_edges_than_passes_over_blocks(n, m);
    char* base = nullptr;
    const int32_t *os = nullptr, *ol = nullptr, *ot = nullptr;
    const unsigned long long* seg = nullptr;
    const int64_t *off = nullptr, *at = nullptr;
    int64_t count = 0;
    st = by_radix ? summary_by_radix(ctx, s, &base, &os, &ol, &ot, &count)
                  : summary_by_segment(ctx, s, &base, &seg, &off, &at, &count);
    if (st != BISIM_OK) return st;
    const int64_t take = std::min(capacity, count);
    char* stage = nullptr;
    if (!by_radix && take > 0) {
        // straight into the caller's arrays where a kernel may write them
        int32_t* o[3] = {src_block, label, dst_block};
        const bool direct = device_accessible(src_block) && device_accessible(label) && device_accessible(dst_block);
        if (!direct) {
            const size_t one = (sizeof(int32_t) * take + 255) & ~size_t(255);
            if ((e = cudaMallocAsync(reinterpret_cast<void**>(&stage), 3 * one, s))) {
                cudaFreeAsync(base, s);
                return cuda_error(ctx, e, "alloc summary output");
            }
            for (int i = 0; i < 3; ++i) o[i] = reinterpret_cast<int32_t*>(stage + i * one);
            os = o[0];
            ol = o[1];
            ot = o[2];
        }
        BISIM_SITE(site, "summary_edges");
        Launch L(site, s, 0, take, 24.0 * take);
        k_seg_emit<<<grid_for(cdiv(take, kKeyTile) * 256, 256), 256, 0, s>>>(at, n, take, off, seg, o[0], o[1], o[2]);
    }
    if (take > 0 && os != nullptr) {
        cudaMemcpyAsync(src_block, os, sizeof(int32_t) * take, cudaMemcpyDefault, s);
        cudaMemcpyAsync(label, ol, sizeof(int32_t) * take, cudaMemcpyDefault, s);
        cudaMemcpyAsync(dst_block, ot, sizeof(int32_t) * take, cudaMemcpyDefault, s);
    }
    if (stage) cudaFreeAsync(stage, s);
    cudaFreeAsync(base, s);
    if ((e = cudaStreamSynchronize(s))) return cuda_error(ctx, e, "copy summary edges");
    *out_count = count;
    return BISIM_OK;
}

}  // extern "C"
