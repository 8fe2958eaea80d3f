// The round loop as one cooperative kernel, for lists whose rows have at most
// 256 edges (the thread and warp classes of the dense layout).
//
// What it replaces is a loop of about a dozen kernels a round. Each of those is
// near empty once the list is short (a late round of a power-law graph) or the
// graph is small, and a round then costs its launches: 77 us on 300k vertices in
// paths, 60 us on 10k vertices. Here a round is two or three phases with a grid
// barrier after each, one CTA per SM (on small graphs one cluster, or one CTA):
//   A  the entries of the list that are not alone in their block compute their
//      signatures
//   B  every entry is confirmed by an exact comparison, inside the thread for rows of
//      at most eight edges (the pairs with longer rows are shared out to the CTA's
//      warps afterwards), against the smallest vertex of its slot of the signature
//      table, which phase A filled; in a round that is likely to keep most blocks
//      (see keeps_blocks) against the smallest vertex of its present block, and those
//      that differ from it enter the table instead
//   C  (only then, and only them) and are confirmed against their slots
//
// The list is cut among the CTAs at the start and each keeps its part to the end
// (dealt in units of up to 32 entries, rotated from row to row so that no period
// of the graph lands on one CTA), so that no list position is handed out by an
// atomic and no entry waits for one: thousands of warps on one address are what
// bounded the phases with a shared list. A barrier carries the CTAs' counts, so
// every CTA knows the totals and takes the same decision: another round, done, or
// back to the host at a hash collision (with the state the host-driven levels
// expect).
//
// The two partition buffers alternate as input and output; a vertex that leaves
// the list writes its final block into the other one, so both agree on every
// vertex that is not listed.
#include <algorithm>
#include <climits>
#include <cstring>
#include <mutex>

#include "common.cuh"
#include "prof.cuh"
#include "rounds.cuh"

namespace bisim {

namespace {

constexpr int kLoopThreads = 1024;        // at most; 512 for short lists
constexpr int kLoopWarps = kLoopThreads / 32;
constexpr int kLoopGroups = 4;            // degree <= 8, <= 16, <= 32, <= 256: classes 0-4, 5, 6, 7-9
constexpr int kHotSlots = 64;
constexpr int kSeenSlots = 1024;
constexpr int kLoopWarpSet = 512;         // slots of a warp's set: twice the longest row
constexpr unsigned kSpinLimit = 1u << 22; // polls of a barrier before the kernel gives up (seconds): the rounds
                                          // then run again without it
constexpr int kUnits = 4;                 // work units a warp takes between two flushes of the CTA
constexpr int kStage = kUnits * 32;
constexpr uint8_t kCold = 255;

// Values of an entry's `own` flag.
constexpr uint8_t kMember = 0;            // not its block's smallest vertex
constexpr uint8_t kOwner = 1;             // the smallest vertex; joined says whether others are in the block
constexpr uint8_t kOwnerLeft = 3;         // ... and some left since: joined may be out of date
constexpr uint8_t kOwnerAsks = 5;         // ... and this round those that stay set it anew

int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

// What one barrier carries: the CTAs' listed (high half) and owned entries
// added up, the number of CTAs that raise each of three flags (8 bits each), and
// above those the CTAs' moved entries.
struct __align__(16) BarrierSum {
    unsigned long long counts;
    unsigned long long flags;
};

// What a launch leaves behind is cleared by the next one, which uses the other copy.
struct LoopCopy {
    BarrierSum sum[3];                          // of barrier k: sum[k % 3]
    unsigned arrived;                           // barrier arrivals since the launch
    unsigned gcount[kLoopGroups];               // list entries per group, when the list goes back to the host
    unsigned gcursor[kLoopGroups];
    unsigned unresolved;
    unsigned error;
};

struct LoopCtl {
    LoopCopy copy[2];
    unsigned abort;                       // a barrier gave up
};

struct LoopView {
    const int32_t* vert;
    const int32_t* vpos;
    const int64_t* prp;
    const unsigned long long* pe;
    const int32_t* P0;
    int32_t* P[2];
    SigRec* sig;
    uint32_t* slot;
    uint8_t* joined;
    uint8_t* own;
    int32_t* act[2];
    int64_t* aoff;
    unsigned long long* ccount;
    const int32_t* gid;
    const int64_t* rbase;
    const uint32_t* rmask;
    TableRef t;                           // epoch: set per round
    uint64_t nslots;
    uint32_t epoch;                       // the table's last epoch (kEpochCycle: blank it first)
    int32_t* unresolved;
    int32_t* wide;                        // entries that confirm_wide compares, at their CTA's places
    int32_t* split;                       // entries that left their block's smallest vertex this round, the same
    DevState* st;
    LoopCtl* ctl;
    LoopState* L;
    LoopState* host;                      // pinned: where the host reads the result
    int64_t gb[kLoopGroups + 1];          // first position of each group
    int64_t n_live;
    int32_t n;
    int32_t copy;                         // which LoopCopy this launch uses
    int32_t cluster;                      // the grid is one cluster
    unsigned polls;                       // kSpinLimit, or what a test sets
    int32_t start;                        // 1: from P_0 with every live position listed; 0: from act[0] / aoff and *L
    LoopState init;                       // start: the loop state to begin with
};

struct Shared {
    unsigned long long hot_key[kHotSlots];
    unsigned hot_min[kHotSlots];
    uint32_t hot_slot[kHotSlots];
    int32_t stage_pos[kLoopWarps][kStage];    // the warp's short rows that stay listed
    uint8_t stage_hot[kLoopWarps][kStage];    // their hot slot, or kCold (already in the table)
    unsigned wcnt[kLoopWarps];
    unsigned wbase[kLoopWarps];
    unsigned zero[kLoopWarps];
    int32_t seen[kSeenSlots];                 // positions whose joined flag this CTA has set this round
    unsigned next_cnt[kLoopGroups];           // entries of the next list so far
    unsigned owned;                           // entries that are their block's id
    unsigned wide;                            // entries on the wide list
    unsigned split;                           // and on the split list
    unsigned moved;                           // members that are in another block now
    unsigned error;                           // kErr* bits
    unsigned flags;                           // barrier result: kAny* of all CTAs
    unsigned total[3];                        // barrier result: listed, owned, moved
    int ok;
};

__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }

// Pair value of a packed word. Arrays that one phase writes and a later one
// reads (partitions, signatures, flags, slots, lists) are read with plain loads:
// every barrier's acquire makes the SM's L1 forget them, and within a phase L1
// serves what all vertices of a large block read.
__device__ __forceinline__ uint64_t word_value(unsigned long long w, const int32_t* P) {
    return pair_value(static_cast<int32_t>(w >> 32), P[static_cast<uint32_t>(w)]);
}

// Sum and number of the distinct values among the lanes that have one (every lane gets both).
__device__ __forceinline__ void distinct_of_warp(uint64_t val, bool has, uint64_t* sum, unsigned* cnt) {
    const unsigned m = __ballot_sync(0xffffffffu, has);
    bool first = false;
    if (has) first = __ffs(__match_any_sync(m, val)) - 1 == static_cast<int>(lane_id());
    uint64_t s = first ? val : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    *sum = s;
    *cnt = static_cast<unsigned>(__popc(__ballot_sync(0xffffffffu, first)));
}

// ----------------------------------------------------------------------------- barrier

constexpr unsigned kAnySplit = 1u, kAnyUnresolved = 2u, kAnyError = 4u;

__device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void add_release(unsigned* p, unsigned v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Grid barrier number `k` (from 1) of this launch; false when it gave up. One
// counter and one poller per CTA: 2.9k cycles for 152 CTAs with stores in
// flight, against 7k to 9k when every CTA reads a word of every other, 4.2k with
// one CTA collecting and 3.1k of the runtime's grid sync. A grid that is one
// cluster uses the cluster's barrier.
__device__ bool arrive_and_wait(const LoopView& V, unsigned k, Shared& sh) {
    LoopCopy* c = &V.ctl->copy[V.copy];
    if (V.cluster) {
        asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
        return true;
    }
    if (gridDim.x == 1) {
        __syncthreads();
        return true;
    }
    if (threadIdx.x == 0) {
        sh.ok = 1;
        add_release(&c->arrived, 1u);
        const unsigned target = gridDim.x * k;
        unsigned spin = 0;
        while (load_acquire(&c->arrived) < target) {
            if (++spin > V.polls || ((spin & 255u) == 0u && load_acquire(&V.ctl->abort) != 0u)) {
                atomicExch(&V.ctl->abort, 1u);
                sh.ok = 0;
                break;
            }
        }
    }
    __syncthreads();
    return sh.ok != 0;
}

__device__ bool grid_barrier(const LoopView& V, unsigned k, Shared& sh) {
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0) V.ctl->copy[V.copy].sum[(k + 1) % 3] = BarrierSum{0ull, 0ull};
    return arrive_and_wait(V, k, sh);
}

// The same with the sums of all CTAs' counts and the union of their flags, in
// sh.total and sh.flags. Three sums rotate: that of barrier k + 1 is cleared
// before anyone leaves barrier k, and was last read before anyone reached k - 1.
__device__ bool grid_barrier(const LoopView& V, unsigned k, unsigned flags, unsigned listed, unsigned owned,
                             unsigned moved, Shared& sh) {
    LoopCopy* c = &V.ctl->copy[V.copy];
    __syncthreads();
    if (threadIdx.x == 0) {
        if (blockIdx.x == 0) c->sum[(k + 1) % 3] = BarrierSum{0ull, 0ull};
        atomicAdd(&c->sum[k % 3].counts, (static_cast<unsigned long long>(listed) << 32) | owned);
        const unsigned long long raised = (flags & kAnySplit ? 1ull : 0ull) | (flags & kAnyUnresolved ? 1ull << 8 : 0ull) |
                                          (flags & kAnyError ? 1ull << 16 : 0ull) | static_cast<unsigned long long>(moved) << 24;
        if (raised) atomicAdd(&c->sum[k % 3].flags, raised);
    }
    const bool fine = arrive_and_wait(V, k, sh);
    if (threadIdx.x == 0) {
        const ulonglong2 t = __ldcg(reinterpret_cast<const ulonglong2*>(&c->sum[k % 3]));
        sh.total[0] = static_cast<unsigned>(t.x >> 32);
        sh.total[1] = static_cast<unsigned>(t.x);
        sh.total[2] = static_cast<unsigned>(t.y >> 24);
        sh.flags = (t.y & 0xffull ? kAnySplit : 0u) | (t.y & 0xff00ull ? kAnyUnresolved : 0u) |
                   (t.y & 0xff0000ull ? kAnyError : 0u);
    }
    __syncthreads();
    return fine;
}

// ----------------------------------------------------------------------------- list

// The CTA's part of the list. Group g was dealt at the start in units of
// 1 << shift[g] entries, a row of one unit per CTA at a time; entry j of this
// CTA's part sits where its j-th dealt entry sat, in `buf` (null: the list is
// every position in order) from base[g] on.
struct List {
    const int32_t* buf;
    int64_t base[kLoopGroups];
    unsigned cnt[kLoopGroups];            // entries of this CTA
    unsigned shift[kLoopGroups];
};

__device__ __forceinline__ int64_t dealt(const List& l, int g, unsigned j) {
    const unsigned row = j >> l.shift[g];
    const unsigned turn = (blockIdx.x + row * 61u) % gridDim.x;
    return ((static_cast<int64_t>(row) * gridDim.x + turn) << l.shift[g]) + (j & ((1u << l.shift[g]) - 1u));
}

// How many of `count` entries are dealt to this CTA.
__device__ __forceinline__ unsigned dealt_count(int64_t count, unsigned shift) {
    const int64_t units = (count + (1 << shift) - 1) >> shift;
    if (units == 0) return 0u;
    const int64_t rows = (units + gridDim.x - 1) / gridDim.x;
    const unsigned turn = (blockIdx.x + static_cast<unsigned>(rows - 1) * 61u) % gridDim.x;
    const int64_t u = (rows - 1) * gridDim.x + turn;               // this CTA's unit of the last row
    const int64_t last = u >= units ? 0 : min(static_cast<int64_t>(1) << shift, count - (u << shift));
    return static_cast<unsigned>(((rows - 1) << shift) + last);
}

__device__ __forceinline__ int32_t list_at(const List& l, int g, unsigned j) {
    const int64_t at = l.base[g] + dealt(l, g, j);
    return l.buf ? l.buf[at] : static_cast<int32_t>(at);
}

__device__ __forceinline__ unsigned list_size(const List& l) { return l.cnt[0] + l.cnt[1] + l.cnt[2] + l.cnt[3]; }

// Entry i of the CTA's groups in turn: its group, and i becomes its number in it.
__device__ __forceinline__ int group_of(const List& l, unsigned* i) {
    int g = 0;
#pragma unroll
    for (int q = 0; q < kLoopGroups - 1; ++q) {
        if (g == q && *i >= l.cnt[q]) {
            *i -= l.cnt[q];
            g = q + 1;
        }
    }
    return g;
}

__device__ __forceinline__ int32_t entry_of(const List& l, unsigned i) {
    const int g = group_of(l, &i);
    return list_at(l, g, i);
}

// A place among all positions that is this CTA's alone, one for each of its entries.
__device__ __forceinline__ int64_t place_of(const LoopView& V, const List& l, unsigned i) {
    const int g = group_of(l, &i);
    return V.gb[g] + dealt(l, g, i);
}

// ----------------------------------------------------------------------------- table

// Table insert of the lanes with `on`. Lanes of one hash (and region) enter as
// one, by their smallest vertex: every vertex of a popular signature would
// queue at one slot otherwise. Two rounds of comparing with one lane's hash
// find the popular ones at a fraction of a full match. Returns the lane that
// inserts for this one and the lanes it stands for.
__device__ __forceinline__ int combine(bool on, uint64_t h, int64_t base, int32_t v, unsigned* members) {
    int rep = static_cast<int>(lane_id());
    *members = 1u;
    unsigned todo = __ballot_sync(0xffffffffu, on);
#pragma unroll
    for (int it = 0; it < 2; ++it) {
        if (todo == 0u) break;                                     // the same for the whole warp
        const int lead = __ffs(todo) - 1;
        const uint64_t lh = __shfl_sync(0xffffffffu, h, lead);
        const int64_t lb = __shfl_sync(0xffffffffu, base, lead);
        const bool same = ((todo >> lane_id()) & 1u) && lh == h && lb == base;
        const unsigned grp = __ballot_sync(0xffffffffu, same);
        const unsigned lowest = __reduce_min_sync(0xffffffffu, same ? static_cast<unsigned>(v) : ~0u);
        const unsigned who = __ballot_sync(0xffffffffu, same && static_cast<unsigned>(v) == lowest);
        if (same) {
            rep = __ffs(who) - 1;
            *members = static_cast<unsigned>(__popc(grp));
        }
        todo &= ~grp;
    }
    return rep;
}

// Table insert of the warp's lanes with `on`; returns the lane's slot.
__device__ __forceinline__ uint32_t insert_warp(const TableRef& tt, bool on, uint64_t h, int64_t base, uint64_t mask,
                                                int32_t v, unsigned* err) {
    unsigned members;
    const int rep = combine(on, h, base, v, &members);
    uint32_t sl = ~0u;
    if (on && rep == static_cast<int>(lane_id())) sl = table_insert_in(tt, h, v, static_cast<uint64_t>(base), mask, err);
    return __shfl_sync(0xffffffffu, sl, rep);
}

__device__ __forceinline__ void table_span(const LoopView& V, int32_t v, int64_t* base, uint64_t* mask) {
    *base = 0;
    *mask = V.t.mask;
    if (V.gid) {
        const int32_t g = __ldg(V.gid + v);
        *base = __ldg(V.rbase + g);
        *mask = __ldg(V.rmask + g);
    }
}

__device__ __forceinline__ void put_sig(const LoopView& V, int64_t pos, uint64_t hash, unsigned cnt, int32_t own) {
    SigRec r;
    r.hash = hash;
    r.cnt = static_cast<int32_t>(cnt);
    r.own = own;
    V.sig[pos] = r;
}

// ----------------------------------------------------------------------------- phase A

// What a round is: `first` of the launch, when every entry stays and the list is
// kept as it is, and whether every entry enters the table.
struct Round {
    bool first, insert;
    const int32_t* Pin;
    int32_t* Pout;
    int32_t* next;                        // buffer of the next list
    TableRef t;
};

// Does the entry stay on the list? Not when its vertex is alone in its block.
// An owner whose block lost members asks those that stay, once.
template <bool KEEPS>
__device__ __forceinline__ bool stays_listed(const LoopView& V, const Round& R, int32_t pos) {
    if (R.first) return true;
    const uint8_t o = V.own[pos];
    if (o == kMember) return true;
    if (KEEPS && o == kOwnerLeft) {
        V.own[pos] = kOwnerAsks;
        V.joined[pos] = 0;
        return true;
    }
    if (!V.joined[pos]) return false;
    if (KEEPS && o == kOwnerAsks) V.own[pos] = kOwner;
    return true;
}

// A unit of up to 32 short rows (group 0): a thread per vertex. The entries that
// stay listed are staged in shared memory; the CTA's flush appends them to its
// next list.
template <bool KEEPS>
__device__ __forceinline__ void unit_threads(const LoopView& V, const Round& R, const List& l, unsigned j0, Shared& sh,
                                             int warp, int* staged) {
    const unsigned j = j0 + lane_id();
    const bool in = j < l.cnt[0];
    bool stay = false;
    int32_t pos = 0, v = 0, own = 0;
    int64_t e0 = 0;
    int d = 0;
    if (in) {
        pos = list_at(l, 0, j);
        v = __ldg(V.vert + pos);
        e0 = __ldg(V.prp + pos);
        d = static_cast<int>(__ldg(V.prp + pos + 1) - e0);
        stay = stays_listed<KEEPS>(V, R, pos);
        own = R.Pin[v];
    }
    // the list is grouped by degree, so the warp's longest row is mostly short:
    // what lies beyond it is skipped by the warp as a whole
    const int widest = static_cast<int>(__reduce_max_sync(0xffffffffu, stay ? static_cast<unsigned>(d) : 0u));
    uint64_t h = 0, mask = 0;
    int64_t base = 0;
    if (in && !stay) R.Pout[v] = own;
    if (stay) {
        uint64_t x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) x[q] = q < d ? __ldcs(V.pe + e0 + q) : 0ull;
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (q < widest) x[q] = q < d ? word_value(x[q], R.Pin) : 0ull;
        uint64_t sum = 0;
        unsigned u = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            if (q >= widest) break;
            bool fresh = q < d;
#pragma unroll
            for (int p = 0; p < q; ++p) fresh = fresh && x[p] != x[q];
            if (fresh) {
                sum += x[q];
                ++u;
            }
        }
        const uint64_t hash = sig_hash(own, u, sum);
        put_sig(V, pos, hash, u, own);
        h = hash & R.t.hmask;
    }
    unsigned hot = kCold;
    if (!KEEPS || R.insert) {                                      // the same for the whole grid
        if (stay) {
            V.joined[pos] = 0;
            table_span(V, v, &base, &mask);
        }
        unsigned members;
        const int rep = combine(stay, h, base, v, &members);
        const bool doer = stay && rep == static_cast<int>(lane_id());
        if (doer && members >= 4u && V.gid == nullptr && h != 0ull) {
            // popular in the warp: combine over the CTA too, at the flush
            const unsigned at = static_cast<unsigned>(h ^ (h >> 29)) & (kHotSlots - 1);
            const unsigned long long prev = atomicCAS(&sh.hot_key[at], 0ull, static_cast<unsigned long long>(h));
            if (prev == 0ull || prev == h) {
                atomicMin(&sh.hot_min[at], static_cast<unsigned>(v));
                hot = at;
            }
        }
        uint32_t sl = ~0u;
        if (doer && hot == kCold) sl = table_insert_in(R.t, h, v, static_cast<uint64_t>(base), mask, &sh.error);
        sl = __shfl_sync(0xffffffffu, sl, rep);
        hot = __shfl_sync(0xffffffffu, hot, rep);
        if (stay && hot == kCold) V.slot[pos] = sl;
    }
    const unsigned stays = __ballot_sync(0xffffffffu, stay);
    if (stay) {
        const int at = *staged + __popc(stays & ((1u << lane_id()) - 1u));
        sh.stage_pos[warp][at] = pos;
        sh.stage_hot[warp][at] = static_cast<uint8_t>(hot);
    }
    *staged += __popc(stays);
}

// A unit of up to `per` rows of group g (9 to 256 edges): a warp per row, several
// rows of at most 32 edges at a time to keep their loads in flight together.
// Lane q keeps the result of row q, and the lanes finish all of them together.
template <bool KEEPS>
__device__ __forceinline__ void unit_warps(const LoopView& V, const Round& R, const List& l, int g, unsigned j0,
                                           unsigned per, Shared& sh, int warp, unsigned long long* sets) {
    const unsigned lane = lane_id();
    const unsigned cnt_g = g == 3 ? l.cnt[3] : g == 2 ? l.cnt[2] : l.cnt[1];
    bool stay = false;
    int32_t pos = 0, v = 0, own = 0;
    int64_t e0 = 0;
    int d = 0;
    if (lane < per && j0 + lane < cnt_g) {
        pos = g == 3 ? list_at(l, 3, j0 + lane) : g == 2 ? list_at(l, 2, j0 + lane) : list_at(l, 1, j0 + lane);
        v = __ldg(V.vert + pos);
        e0 = __ldg(V.prp + pos);
        d = static_cast<int>(__ldg(V.prp + pos + 1) - e0);
        stay = stays_listed<KEEPS>(V, R, pos);
        own = R.Pin[v];
        if (!stay) R.Pout[v] = own;
    }
    const unsigned stays = __ballot_sync(0xffffffffu, stay);
    uint64_t sum = 0;
    unsigned cnt = 0;
    if (g < 3) {
        constexpr int kAtOnce = 4;
        for (unsigned todo = stays; todo;) {
            int q[kAtOnce];
            uint64_t w[kAtOnce];
            bool has[kAtOnce];
#pragma unroll
            for (int k = 0; k < kAtOnce; ++k) {
                q[k] = todo ? __ffs(todo) - 1 : -1;
                if (todo) todo &= todo - 1u;
                const int src = q[k] < 0 ? 0 : q[k];
                const int64_t e = __shfl_sync(0xffffffffu, e0, src);
                const int dd = __shfl_sync(0xffffffffu, d, src);
                has[k] = q[k] >= 0 && static_cast<int>(lane) < dd;
                w[k] = has[k] ? __ldcs(V.pe + e + lane) : 0ull;
            }
#pragma unroll
            for (int k = 0; k < kAtOnce; ++k)
                if (has[k]) w[k] = word_value(w[k], R.Pin);
#pragma unroll
            for (int k = 0; k < kAtOnce; ++k) {
                if (q[k] < 0) break;                               // the same for the whole warp
                uint64_t s;
                unsigned c;
                distinct_of_warp(w[k], has[k], &s, &c);
                if (static_cast<int>(lane) == q[k]) {
                    sum = s;
                    cnt = c;
                }
            }
        }
    } else {
        unsigned long long* tab = sets + warp * kLoopWarpSet;
        for (unsigned todo = stays; todo; todo &= todo - 1u) {
            const int q = __ffs(todo) - 1;
            const int64_t e = __shfl_sync(0xffffffffu, e0, q);
            const int dd = __shfl_sync(0xffffffffu, d, q);
            uint64_t mv[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int j = k * 32 + static_cast<int>(lane);
                mv[k] = j < dd ? __ldcs(V.pe + e + j) : 0ull;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (k * 32 + static_cast<int>(lane) < dd) mv[k] = word_value(mv[k], R.Pin);
            uint32_t size = 64;
            while (size < 2u * static_cast<uint32_t>(dd)) size <<= 1;
            for (uint32_t j = lane; j < size; j += 32) tab[j] = 0ull;
            if (lane == 0) sh.zero[warp] = 0u;
            __syncwarp();
            uint64_t s = 0;
            unsigned c = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (k * 32 >= dd) break;                           // the same for the whole warp
                const int j = k * 32 + static_cast<int>(lane);
                const bool fresh = j < dd && smem_set_insert(tab, size - 1, &sh.zero[warp], mv[k]);
                c += static_cast<unsigned>(__popc(__ballot_sync(0xffffffffu, fresh)));
                if (fresh) s += mv[k];
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (static_cast<int>(lane) == q) {
                sum = s;
                cnt = c;
            }
            __syncwarp();                                          // the set is cleared for the next row
        }
    }
    uint64_t h = 0, mask = 0;
    int64_t base = 0;
    if (stay) {
        const uint64_t hash = sig_hash(own, cnt, sum);
        put_sig(V, pos, hash, cnt, own);
        h = hash & R.t.hmask;
    }
    if (!KEEPS || R.insert) {
        if (stay) {
            V.joined[pos] = 0;
            table_span(V, v, &base, &mask);
        }
        const uint32_t sl = insert_warp(R.t, stay, h, base, mask, v, &sh.error);
        if (stay) V.slot[pos] = sl;
    }
    if (!R.first && stays) {
        unsigned at = 0;
        if (lane == 0) at = atomicAdd(&sh.next_cnt[g], static_cast<unsigned>(__popc(stays)));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(stays & ((1u << lane) - 1u));
        if (stay) {
            const int64_t to = g == 3 ? V.gb[3] + dealt(l, 3, at) : g == 2 ? V.gb[2] + dealt(l, 2, at) : V.gb[1] + dealt(l, 1, at);
            R.next[to] = pos;
        }
    }
}

// Phase A over the CTA's part of the list. It is cut into units, one warp's
// work: 32 short rows, or up to 32 longer ones (fewer when there are not enough
// to go round). After every kUnits units the CTA enters its hot signatures, one
// insert each, and appends its staged rows to its next list.
template <bool KEEPS>
__device__ void phase_a(const LoopView& V, const Round& R, const List& l, Shared& sh, unsigned long long* sets) {
    const int warp = static_cast<int>(threadIdx.x >> 5);
    const unsigned lane = lane_id();
    const unsigned warps = blockDim.x / 32;
    const unsigned per3 = max(1u, min(32u, l.cnt[3] / warps)), per2 = max(1u, min(32u, l.cnt[2] / warps)),
                   per1 = max(1u, min(32u, l.cnt[1] / warps));
    const unsigned end3 = (l.cnt[3] + per3 - 1) / per3, end2 = end3 + (l.cnt[2] + per2 - 1) / per2,
                   end1 = end2 + (l.cnt[1] + per1 - 1) / per1, units = end1 + (l.cnt[0] + 31) / 32;
    for (unsigned u0 = 0; u0 < units; u0 += warps * kUnits) {
        int staged = 0;
        for (int k = 0; k < kUnits; ++k) {
            const unsigned u = u0 + k * warps + warp;
            if (u >= units) break;                                 // the same for the whole warp
            if (u >= end1) unit_threads<KEEPS>(V, R, l, (u - end1) * 32, sh, warp, &staged);
            else if (u < end3) unit_warps<KEEPS>(V, R, l, 3, u * per3, per3, sh, warp, sets);
            else if (u < end2) unit_warps<KEEPS>(V, R, l, 2, (u - end3) * per2, per2, sh, warp, sets);
            else unit_warps<KEEPS>(V, R, l, 1, (u - end2) * per1, per1, sh, warp, sets);
        }
        if (lane == 0) sh.wcnt[warp] = static_cast<unsigned>(staged);
        __syncthreads();
        if (threadIdx.x < kHotSlots) {
            const unsigned long long key = sh.hot_key[threadIdx.x];
            if (key) {
                sh.hot_slot[threadIdx.x] = table_insert(R.t, key, static_cast<int32_t>(sh.hot_min[threadIdx.x]), &sh.error);
                sh.hot_key[threadIdx.x] = 0ull;
                sh.hot_min[threadIdx.x] = ~0u;
            }
        } else if (warp == 2) {
            const unsigned c = lane < warps ? sh.wcnt[lane] : 0u;
            unsigned inc = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= static_cast<unsigned>(o)) inc += y;
            }
            const unsigned before = sh.next_cnt[0];
            if (lane < warps) sh.wbase[lane] = before + inc - c;
            __syncwarp();
            if (lane == 31) sh.next_cnt[0] = before + inc;
        }
        __syncthreads();
        for (int i = static_cast<int>(lane); i < staged; i += 32) {
            const int32_t pos = sh.stage_pos[warp][i];
            const unsigned hot = sh.stage_hot[warp][i];
            if (hot != kCold) V.slot[pos] = sh.hot_slot[hot];
            if (!R.first) R.next[V.gb[0] + dealt(l, 0, sh.wbase[warp] + i)] = pos;
        }
        if (u0 + warps * kUnits < units) __syncthreads();          // hot_slot and wcnt are written again
    }
}

// ----------------------------------------------------------------------------- phases B and C

// One entry and the representative it is to be confirmed against.
struct Pair {
    int32_t pos, v, r, rpos;              // rpos < 0: nothing to confirm
};

__device__ __forceinline__ int4 record(const LoopView& V, int32_t pos) {
    return *reinterpret_cast<const int4*>(V.sig + pos);            // hash low, hash high, |S|, own block
}

// The representative's joined flag, set once per CTA as far as a small filter
// in shared memory remembers: the stores of a large block's vertices would queue
// at one sector, and so would reads past L1 to see whether it is set (1M chains:
// 35k cycles a round for this phase, against 100k and 60k). Threads that race in
// the filter only store again.
__device__ __forceinline__ void mark_joined(const LoopView& V, int32_t rpos, Shared& sh) {
    volatile int32_t* seen = &sh.seen[rpos & (kSeenSlots - 1)];
    if (*seen == rpos) return;
    *seen = rpos;
    V.joined[rpos] = 1;
}

// The entry joins the representative's block (with `mark` the representative is
// told), or (with `push`) goes on the unresolved list. For the whole warp.
__device__ __forceinline__ void settle(const LoopView& V, const Round& R, const Pair& p, bool join, bool mark, bool push,
                                       Shared& sh) {
    if (join) {
        R.Pout[p.v] = p.r;
        if (mark) mark_joined(V, p.rpos, sh);
    }
    const unsigned m = __ballot_sync(0xffffffffu, push);
    if (m) {
        unsigned at = 0;
        if (lane_id() == 0) at = atomicAdd(&V.ctl->copy[V.copy].unresolved, static_cast<unsigned>(__popc(m)));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (push) V.unresolved[at + __popc(m & ((1u << lane_id()) - 1u))] = p.pos;
    }
}

// Confirms the lanes' pairs exactly: with `test`, the records a and c have equal own
// blocks and sizes. Pairs with a row too long for that go on the wide list
// (confirm_wide).
__device__ __forceinline__ void confirm(const LoopView& V, const Round& R, const List& l, const Pair& p, bool test,
                                        bool mark, bool push, const int4& a, const int4& c, Shared& sh) {
    bool join = false, wide = false;
    int64_t ev = 0, er = 0;
    int dv = 0, dr = 0;
    if (test && a.z <= 1) {                                        // the full hash decides (a bijection of the pair)
        join = a.x == c.x && a.y == c.y;
        push = !join;
    } else if (test) {
        ev = __ldg(V.prp + p.pos);
        dv = static_cast<int>(__ldg(V.prp + p.pos + 1) - ev);
        er = __ldg(V.prp + p.rpos);
        dr = static_cast<int>(__ldg(V.prp + p.rpos + 1) - er);
        if (dv <= 8 && dr <= 8) {
            // S_v inside S_r with equal sizes means equal sets
            uint64_t x[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = j < dr ? __ldg(V.pe + er + j) : 0ull;
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = j < dr ? word_value(x[j], R.Pin) : 0ull;
            bool all = true;
#pragma unroll 1
            for (int j0 = 0; j0 < dv && all; j0 += 4) {            // four of v's values at a time in flight
                uint64_t y[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) y[j] = j0 + j < dv ? __ldg(V.pe + ev + j0 + j) : 0ull;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (j0 + j < dv) y[j] = word_value(y[j], R.Pin);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    bool found = j0 + j >= dv;
#pragma unroll
                    for (int q = 0; q < 8; ++q) found = found || (q < dr && x[q] == y[j]);
                    all = all && found;
                }
            }
            join = all;
            push = !all;
        } else {
            wide = true;
        }
    }
    settle(V, R, p, join, mark, push, sh);
    const unsigned m = __ballot_sync(0xffffffffu, wide);
    if (m) {
        unsigned at = 0;
        if (lane_id() == 0) at = atomicAdd(&sh.wide, static_cast<unsigned>(__popc(m)));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane_id()) - 1u));
        if (wide) V.wide[place_of(V, l, at)] = p.pos;
    }
}

// Adds the threads' counts to the CTA's.
__device__ __forceinline__ void add_owned(unsigned owned, Shared& sh) {
    owned = __reduce_add_sync(0xffffffffu, owned);
    if (lane_id() == 0 && owned) atomicAdd(&sh.owned, owned);
}

// Confirms the CTA's entries pos_of(i), i < total, against their table slots'
// smallest vertices. (Two entries a thread at once: no faster.)
template <bool KEEPS, class F>
__device__ __forceinline__ void verify_slots(const LoopView& V, const Round& R, const List& l, unsigned total,
                                             const F& pos_of, Shared& sh) {
    const unsigned lane = lane_id();
    unsigned owned = 0, moved = 0;
    for (unsigned b = threadIdx.x - lane; b < total; b += blockDim.x) {
        Pair p{-1, -1, -1, -1};
        bool test = false, push = false;
        int4 a{}, c{};
        if (b + lane < total) {
            p.pos = pos_of(b + lane);
            const uint32_t sv = V.slot[p.pos];
            p.v = __ldg(V.vert + p.pos);
            p.r = sv == ~0u ? -1 : table_rep(V.t.slots, sv);
            if (p.r < 0 || p.r >= V.n) {                           // failed insert
                atomicOr(&sh.error, kErrTableFull);
                R.Pout[p.v] = -1;
            } else if (p.r == p.v) {
                R.Pout[p.v] = p.v;
                V.own[p.pos] = kOwner;
                ++owned;
            } else {
                p.rpos = __ldg(V.vpos + p.r);
                a = record(V, p.pos);
                c = record(V, p.rpos);
                V.own[p.pos] = kMember;
                test = a.z == c.z && a.w == c.w;
                push = !test;
                if (KEEPS && a.w != p.r) ++moved;
            }
        }
        confirm(V, R, l, p, test, true, push, a, c, sh);
    }
    add_owned(owned, sh);
    if (KEEPS) {
        moved = __reduce_add_sync(0xffffffffu, moved);
        if (lane == 0 && moved) atomicAdd(&sh.moved, moved);
    }
}

// Phase B of a round that is likely to keep its blocks: every entry against the
// smallest vertex b of its present block. b stays in the part of its block that keeps
// the block's id, whatever happens to the others, so a vertex with b's signature needs
// neither the table nor a flag; those that leave b go on the split list, and b asks next
// round whether it is alone now (see stays_listed).
__device__ __forceinline__ void keep_or_split(const LoopView& V, const Round& R, const List& l, Shared& sh) {
    const unsigned total = list_size(l);
    const unsigned lane = lane_id();
    unsigned owned = 0;
    for (unsigned b = threadIdx.x - lane; b < total; b += blockDim.x) {
        Pair p{-1, -1, -1, -1};
        bool test = false, leave = false, asks = false;
        int4 a{}, c{};
        if (b + lane < total) {
            p.pos = entry_of(l, b + lane);
            p.v = __ldg(V.vert + p.pos);
            a = record(V, p.pos);
            p.r = a.w;
            if (p.r == p.v) {
                R.Pout[p.v] = p.v;
                ++owned;
            } else {
                p.rpos = __ldg(V.vpos + p.r);
                c = record(V, p.rpos);
                asks = V.own[p.rpos] == kOwnerAsks;
                test = a.x == c.x && a.y == c.y && a.z == c.z;
                leave = !test;
            }
        }
        confirm(V, R, l, p, test, asks, false, a, c, sh);
        const unsigned leaves = __ballot_sync(0xffffffffu, leave);
        if (leaves) {
            unsigned at = 0;
            if (lane == 0) at = atomicAdd(&sh.split, static_cast<unsigned>(__popc(leaves)));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(leaves & ((1u << lane) - 1u));
            if (leave) {
                V.split[place_of(V, l, at)] = p.pos;
                if (__ldcg(V.own + p.rpos) != kOwnerLeft) V.own[p.rpos] = kOwnerLeft;
            }
        }
    }
    add_owned(owned, sh);
}

// The entries of the split list enter the table, equal signatures of a warp as one.
__device__ __forceinline__ void insert_split(const LoopView& V, const Round& R, const List& l, Shared& sh) {
    const unsigned split = sh.split, lane = lane_id();
    for (unsigned b = threadIdx.x - lane; b < split; b += blockDim.x) {
        const bool on = b + lane < split;
        int32_t pos = 0, v = 0;
        uint64_t h = 0, mask = 0;
        int64_t base = 0;
        if (on) {
            pos = V.split[place_of(V, l, b + lane)];
            v = __ldg(V.vert + pos);
            h = V.sig[pos].hash & R.t.hmask;
            table_span(V, v, &base, &mask);
        }
        const uint32_t sl = insert_warp(R.t, on, h, base, mask, v, &sh.error);
        if (on) V.slot[pos] = sl;
    }
}

// Pairs with a row of more than eight edges, cut evenly among the CTA's warps: rows
// of up to 32 edges eight lanes a pair, longer ones through a set in shared memory.
// (Each compared by the warp that met it, against 32 shuffles of the other row at a
// time, a CTA's few wide pairs were one warp's: 1,000 vertices of 250 edges with equal
// sets took 678 us a round, 98 in the kernels of the single classes.) `keep`: against
// the present block's smallest vertex, as keep_or_split, else the table slot's.
__device__ void confirm_wide(const LoopView& V, const Round& R, const List& l, bool keep, Shared& sh,
                             unsigned long long* sets) {
    const unsigned count = sh.wide, lane = lane_id(), warp = threadIdx.x >> 5, warps = blockDim.x / 32;
    const unsigned per = max(4u, min(32u, (count + warps - 1) / warps));
    const auto value = [&](unsigned long long w) { return word_value(w, R.Pin); };
    for (unsigned b = warp * per; b < count; b += warps * per) {
        const bool in = lane < per && b + lane < count;
        Pair p{-1, -1, -1, -1};
        int64_t ev = 0, er = 0;
        int dv = 0, dr = 0;
        if (in) {
            p.pos = V.wide[place_of(V, l, b + lane)];
            p.v = __ldg(V.vert + p.pos);
            p.r = keep ? record(V, p.pos).w : table_rep(V.t.slots, V.slot[p.pos]);
            p.rpos = __ldg(V.vpos + p.r);
            ev = __ldg(V.prp + p.pos);
            dv = static_cast<int>(__ldg(V.prp + p.pos + 1) - ev);
            er = __ldg(V.prp + p.rpos);
            dr = static_cast<int>(__ldg(V.prp + p.rpos + 1) - er);
        }
        const bool by_eights = in && dv <= 32 && dr <= 32;
        bool same = rows_inside(by_eights, ev, dv, er, dr, V.pe, value);
        unsigned long long* tab = sets + warp * kLoopWarpSet;
        for (unsigned todo = __ballot_sync(0xffffffffu, in && !by_eights); todo; todo &= todo - 1u) {
            const int q = __ffs(todo) - 1;
            const int64_t qev = __shfl_sync(0xffffffffu, ev, q), qer = __shfl_sync(0xffffffffu, er, q);
            const int qdv = __shfl_sync(0xffffffffu, dv, q), qdr = __shfl_sync(0xffffffffu, dr, q);
            uint32_t size = 64;
            while (size < 2u * static_cast<uint32_t>(qdr)) size <<= 1;
            for (uint32_t j = lane; j < size; j += 32) tab[j] = 0ull;
            if (lane == 0) sh.zero[warp] = 0u;
            __syncwarp();
            bool miss = false;
#pragma unroll 1
            for (int pass = 0; pass < 2; ++pass) {                 // r's row into the set, then v's against it
                const int64_t e = pass ? qev : qer;
                const int d = pass ? qdv : qdr;
                uint64_t x[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int j = k * 32 + static_cast<int>(lane);
                    x[k] = j < d ? __ldg(V.pe + e + j) : 0ull;
                }
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (k * 32 + static_cast<int>(lane) < d) x[k] = value(x[k]);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    if (k * 32 + static_cast<int>(lane) >= d) break;
                    if (pass == 0) smem_set_insert(tab, size - 1, &sh.zero[warp], x[k]);
                    else miss = miss || !smem_set_contains(tab, size - 1, sh.zero[warp], x[k]);
                }
                __syncwarp();
            }
            miss = __any_sync(0xffffffffu, miss);
            if (static_cast<int>(lane) == q) same = !miss;
        }
        const bool mark = !keep || (in && V.own[p.rpos] == kOwnerAsks);
        settle(V, R, p, in && same, mark, in && !same, sh);
    }
}

// ----------------------------------------------------------------------------- the loop

// The list and the state of a round that ended in a hash collision (or an
// error) as the host-driven levels expect them: P_i in P[0], P_{i+1} as far as
// it is known in P[1], the list in act[0] / aoff, the counts in the status word.
template <bool KEEPS>
__device__ bool hand_back(const LoopView& V, const List& l, const Round& R, int out, unsigned long long blocks,
                          unsigned listed, unsigned* bar, Shared& sh) {
    LoopCopy* c = &V.ctl->copy[V.copy];
    if (threadIdx.x < kLoopGroups && l.cnt[threadIdx.x]) atomicAdd(&c->gcount[threadIdx.x], l.cnt[threadIdx.x]);
    if (threadIdx.x == 0 && sh.error) atomicOr(&c->error, sh.error);
    for (unsigned i = threadIdx.x; i < list_size(l); i += blockDim.x) {
        const int32_t pos = entry_of(l, i);
        const int32_t v = __ldg(V.vert + pos);
        if (V.start && R.first) {
            V.P[0][v] = V.P0[v];
        } else if (out == 0) {
            const int32_t x = V.P[0][v];
            V.P[0][v] = V.P[1][v];
            V.P[1][v] = x;
        }
        if (KEEPS && V.own[pos] > kOwner) {                        // whether it is alone is not known: listed on
            V.own[pos] = kOwner;
            V.joined[pos] = 1;
        }
    }
    if (!grid_barrier(V, ++*bar, sh)) return false;
    int64_t first[kLoopGroups + 1] = {0, 0, 0, 0, 0};
    for (int g = 0; g < kLoopGroups; ++g) first[g + 1] = first[g] + __ldcg(&c->gcount[g]);
    const bool in_place = R.first && !V.start;
    if (!in_place) {
        // flat into the buffer the list is not in, then (if that is act[1]) over to act[0]
        int32_t* flat = l.buf == V.act[1] ? V.act[0] : V.act[1];
        if (threadIdx.x < kLoopGroups) sh.wcnt[threadIdx.x] = atomicAdd(&c->gcursor[threadIdx.x], l.cnt[threadIdx.x]);
        __syncthreads();
        for (int g = 0; g < kLoopGroups; ++g)
            for (unsigned j = threadIdx.x; j < l.cnt[g]; j += blockDim.x) flat[first[g] + sh.wcnt[g] + j] = list_at(l, g, j);
        if (!grid_barrier(V, ++*bar, sh)) return false;
        if (flat != V.act[0])
            for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < listed;
                 i += static_cast<int64_t>(gridDim.x) * blockDim.x)
                V.act[0][i] = flat[i];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (!in_place) {
            // the groups as classes: 0 (0 to 4), 5, 6, 7 (7 to 9)
            V.aoff[0] = 0;
            for (int q = 1; q <= kDClasses; ++q) V.aoff[q] = q <= 5 ? first[1] : q == 6 ? first[2] : q == 7 ? first[3] : first[4];
            for (int q = 0; q < kDClasses; ++q) V.ccount[q] = 0ull;
        }
        DevState z{};
        z.blocks = blocks;
        z.unresolved = __ldcg(&c->unresolved);
        z.error = __ldcg(&c->error);
        z.listed = listed;
        *V.st = z;
    }
    return true;
}

// Whether the next round is likely to keep most blocks. Then comparing with them saves
// an insert at a random or a popular slot per entry; what has to pay for it is the third
// phase, and the entries that leave, one by one. Two signs of it, from the last round:
// few new blocks, and blocks of at most kKeepSize listed entries on average (entries
// cannot leave small blocks without new ones in proportion); or few entries in another
// block than before on a long list (13 us for the phase and 5 ns for an entry that
// leaves, against 50 ps an insert). us to the fixpoint with no such round, with any
// round that made few new blocks, with these two: power law 1.4M / 4M 613 / 561 / 562,
// 4M / 16M 1,220 / 1,147 / 1,158, with a label filter 500k / 1.5M 494 / 413 / 423 and 3M /
// 9M 1,267 / 1,130 / 1,137; beside a wide row, paths of 300k vertices with 3,000 more edges
// 330 / 503 / 332, two edges a vertex with two labels, 200k, 246 / 400 / 248, 600 rounds
// of paths on 300k 13,270 / 15,920 / 13,740.
constexpr int64_t kKeepSize = 32;
constexpr int64_t kKeepListed = 210000;
constexpr int64_t kKeepMoved = 200;
__device__ __forceinline__ bool keeps_blocks(int64_t grown, int64_t moved, int64_t owned, int64_t listed) {
    return (grown * 32 < listed && listed <= owned * kKeepSize) || kKeepListed + kKeepMoved * (moved + grown) < listed;
}

// KEEPS: with rounds that keep_or_split begins. The rest of the kernel is 2% to 3%
// slower with them in it, so loops from P_0 on have them only where many vertices have
// no edges and stay in large blocks: a fourth of them, on a list long enough (chains
// with two extra edges a vertex behind a label filter, 56% without edges, 500k 431 to
// 380 us, 3M 1,579 to 1,482; unfiltered ones 186 to 190 and 697 to 717, uniform graphs of
// mean five 178 to 182 and 713 to 730).
template <bool KEEPS>
__global__ void __launch_bounds__(kLoopThreads, 1) k_round_loop(const LoopView V) {
    extern __shared__ unsigned long long sets[];           // a set per warp, when warp-class rows exist
    __shared__ Shared sh;
    LoopState S = V.init;
    if (!V.start) S = *V.L;
    if (blockIdx.x == 0) {                                 // the next launch's copy starts out zero
        unsigned* z = reinterpret_cast<unsigned*>(&V.ctl->copy[V.copy ^ 1]);
        for (unsigned i = threadIdx.x; i < sizeof(LoopCopy) / sizeof(unsigned); i += blockDim.x) z[i] = 0u;
    }
    List l;
    l.buf = V.start ? nullptr : V.act[0];
    const unsigned warps = gridDim.x * (blockDim.x / 32);
#pragma unroll
    for (int g = 0; g < kLoopGroups; ++g) {
        constexpr int c0[kLoopGroups + 1] = {0, 5, 6, 7, 10};
        l.base[g] = V.start ? V.gb[g] : V.aoff[c0[g]];
        const int64_t count = V.start ? V.gb[g + 1] - V.gb[g] : V.aoff[c0[g + 1]] - V.aoff[c0[g]];
        unsigned shift = 5;
        while (g > 0 && shift > 0 && (count >> shift) < warps) --shift;
        l.shift[g] = shift;
        l.cnt[g] = dealt_count(count, shift);
    }
    if (!V.start && S.stop == kStopNo && V.aoff[kDClasses] != V.aoff[kDMid0]) S.stop = kStopWideRows;
    if (threadIdx.x < kHotSlots) {
        sh.hot_key[threadIdx.x] = 0ull;
        sh.hot_min[threadIdx.x] = ~0u;
    }
    if (threadIdx.x == 0) sh.error = 0u;
    uint32_t ep = V.epoch;
    unsigned bar = 0;
    int nbuf = V.start ? 0 : 1;                            // the list buffer the next list goes to
    int out = 1;
    bool fine = true, keep = false;
    Round R;
    R.Pin = V.start ? V.P0 : V.P[0];
    R.t = V.t;
    for (R.first = true; S.stop == kStopNo; R.first = false) {
        if (ep == kEpochCycle) {                           // every epoch is used up: blank the table
            uint4* w = reinterpret_cast<uint4*>(V.t.slots);
            const uint64_t st = static_cast<uint64_t>(gridDim.x) * blockDim.x;
            for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < V.nslots / 2; i += st)
                w[i] = make_uint4(0u, 0u, 0u, 0u);
            ep = 0;
            if (!(fine = grid_barrier(V, ++bar, sh))) break;
        }
        ++ep;
        R.t.epoch = static_cast<uint64_t>(ep) << 32;
        R.Pout = V.P[out];
        R.next = V.act[nbuf];
        R.insert = !KEEPS || !keep;
        for (int i = threadIdx.x; i < kSeenSlots; i += blockDim.x) sh.seen[i] = -1;
        if (threadIdx.x < kLoopGroups) sh.next_cnt[threadIdx.x] = 0u;
        if (threadIdx.x == 0) sh.owned = sh.wide = sh.split = sh.moved = 0u;
        __syncthreads();
        phase_a<KEEPS>(V, R, l, sh, sets);
        if (!(fine = grid_barrier(V, ++bar, sh))) break;
        if (!R.first) {
            l.buf = R.next;
#pragma unroll
            for (int g = 0; g < kLoopGroups; ++g) {
                l.base[g] = V.gb[g];
                l.cnt[g] = sh.next_cnt[g];
            }
            nbuf ^= 1;
        }
        if (KEEPS && keep) keep_or_split(V, R, l, sh);
        else verify_slots<KEEPS>(V, R, l, list_size(l), [&](unsigned i) { return entry_of(l, i); }, sh);
        __syncthreads();
        for (bool against_block = KEEPS && keep;; against_block = false) {
            if (sh.wide) confirm_wide(V, R, l, KEEPS && against_block, sh, sets);
            if (KEEPS && against_block && sh.split) insert_split(V, R, l, sh);
            __syncthreads();
            // unresolved entries are rare: every CTA looks at the counter
            const unsigned flags = (sh.split ? kAnySplit : 0u) | (sh.error ? kAnyError : 0u) |
                                   (__ldcg(&V.ctl->copy[V.copy].unresolved) ? kAnyUnresolved : 0u);
            if (!(fine = grid_barrier(V, ++bar, flags, list_size(l), sh.owned, sh.moved + sh.split, sh))) break;
            if (!KEEPS || !against_block || !(sh.flags & kAnySplit)) break;
            if (threadIdx.x == 0) sh.wide = 0u;
            __syncthreads();
            verify_slots<false>(V, R, l, sh.split, [&](unsigned i) { return V.split[place_of(V, l, i)]; }, sh);
            __syncthreads();
        }
        if (!fine) break;
        const unsigned listed = sh.total[0];
        const unsigned long long blocks = static_cast<unsigned long long>(V.n_live - listed) + sh.total[1];
        if (KEEPS) keep = keeps_blocks(static_cast<int64_t>(blocks - S.prev_blocks), sh.total[2], sh.total[1], listed);
        loop_advance(S, blocks, sh.flags & kAnyUnresolved, sh.flags & kAnyError);
        if (S.stop == kStopDone) {
            if (out != 0)                                  // the result belongs in P[0]
                for (unsigned i = threadIdx.x; i < list_size(l); i += blockDim.x) {
                    const int32_t v = __ldg(V.vert + entry_of(l, i));
                    V.P[0][v] = V.P[1][v];
                }
        } else if (S.stop != kStopNo) {
            if (!(fine = hand_back<KEEPS>(V, l, R, out, blocks, listed, &bar, sh))) break;
        }
        R.Pin = R.Pout;
        out ^= 1;
        __syncthreads();                                   // the counts are cleared for the next round
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && fine) {
        S.epoch = static_cast<int32_t>(ep);
        *V.L = S;
        *V.host = S;
        __threadfence_system();
    }
}

// Cooperative launches of this process follow one another on a device, whatever
// their streams: each waits for the event recorded after the one before, so that
// two of them never share the SMs half resident. That includes launches on equal
// handles: the per-thread default stream is another stream in every thread.
struct CoopLane {
    std::mutex mu;
    cudaEvent_t done[64] = {};
};

CoopLane& coop_lane() {
    static CoopLane* lane = new CoopLane();
    return *lane;
}

cudaError_t launch_in_lane(int device, const void* kernel, unsigned grid, unsigned threads, void** args, size_t smem,
                           cudaStream_t s) {
    if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
    CoopLane& lane = coop_lane();
    std::lock_guard<std::mutex> lk(lane.mu);
    cudaError_t e;
    if (lane.done[device] == nullptr) {
        if ((e = cudaEventCreateWithFlags(&lane.done[device], cudaEventDisableTiming))) return e;
    } else if ((e = cudaStreamWaitEvent(s, lane.done[device], 0))) {
        return e;
    }
    if ((e = cudaLaunchCooperativeKernel(kernel, dim3(grid), dim3(threads), args, smem, s))) return e;
    return cudaEventRecord(lane.done[device], s);
}

cudaLaunchConfig_t cluster_config(unsigned grid, unsigned threads, size_t smem) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    return cfg;
}

cudaLaunchAttribute cluster_attribute(unsigned size) {
    cudaLaunchAttribute a{};
    a.id = cudaLaunchAttributeClusterDimension;
    a.val.clusterDim.x = size;
    a.val.clusterDim.y = 1;
    a.val.clusterDim.z = 1;
    return a;
}

// The largest cluster of full SMs the device takes (16 where a GPC has them, else 8).
template <bool KEEPS>
int largest_cluster(int device, size_t smem) {
    static std::mutex mu;
    static int known[64][2] = {};
    if (device < 0 || device >= 64) return 1;
    std::lock_guard<std::mutex> lk(mu);
    int& k = known[device][smem ? 1 : 0];
    if (k == 0) {
        cudaFuncSetAttribute(k_round_loop<KEEPS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(sizeof(unsigned long long) * kLoopWarps * kLoopWarpSet));
        cudaFuncSetAttribute(k_round_loop<KEEPS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        for (k = 16; k > 1; k >>= 1) {
            cudaLaunchConfig_t cfg = cluster_config(static_cast<unsigned>(k), kLoopThreads, smem);
            cudaLaunchAttribute attr = cluster_attribute(static_cast<unsigned>(k));
            cfg.attrs = &attr;
            cfg.numAttrs = 1;
            int fit = 0;
            if (cudaOccupancyMaxActiveClusters(&fit, k_round_loop<KEEPS>, &cfg) == cudaSuccess && fit > 0) break;
            cudaGetLastError();
        }
    }
    return k;
}

}  // namespace

bool round_loop_usable(const bisim_ctx* ctx) {
    return ctx->dense_ready && ctx->n > 0 && !prof_enabled() && !(ctx->opt.flags & (BISIM_FLAG_EAGER | BISIM_FLAG_L2_PIN));
}

bool round_loop_covers(const bisim_ctx* ctx) {
    return ctx->dbegin[kDClasses] == ctx->dbegin[kDMid0];
}

bisim_status round_loop_state(bisim_ctx* ctx, cudaStream_t s) {
    static_assert(sizeof(LoopState) <= 256, "pinned blocks hold 256 bytes");
    cudaError_t e;
    if (ctx->dloop == nullptr) {
        const size_t ls = (sizeof(LoopState) + 255) & ~size_t(255);
        if ((e = ctx_alloc(ctx, &ctx->dloop, ls + sizeof(LoopCtl), s))) return cuda_error(ctx, e, "alloc loop state");
        cudaMemsetAsync(ctx->dloop, 0, ls + sizeof(LoopCtl), s);
    }
    if (ctx->hloop == nullptr && (ctx->hloop = pinned_take()) == nullptr)
        return set_error(ctx, BISIM_ENOMEM, "pinned loop state mirror");
    return BISIM_OK;
}

bisim_status round_loop(bisim_ctx* ctx, cudaStream_t s, bool start, const LoopState& init, unsigned long long* ccount,
                        LoopState* out) {
    bisim_status st = round_loop_state(ctx, s);
    if (st != BISIM_OK) return st;
    const size_t ls = (sizeof(LoopState) + 255) & ~size_t(255);
    LoopState* h = static_cast<LoopState*>(ctx->hloop);
    LoopView V{};
    V.vert = ctx->dvert;
    V.vpos = ctx->dvpos;
    V.prp = ctx->dprp;
    V.pe = ctx->dpe;
    V.P0 = ctx->P0;
    V.P[0] = ctx->P[0];
    V.P[1] = ctx->P[1];
    V.sig = ctx->dsig;
    V.slot = ctx->dslot;
    V.joined = ctx->djoined;
    V.own = ctx->downs;
    V.act[0] = ctx->dact;
    V.act[1] = ctx->dact2;
    V.aoff = ctx->daoff;
    V.ccount = ccount;
    const bool regions = ctx->rtable != nullptr;
    V.gid = regions ? ctx->gid : nullptr;
    V.rbase = ctx->rbase;
    V.rmask = ctx->rmask;
    V.t.slots = regions ? ctx->rtable : ctx->table;
    V.nslots = regions ? ctx->n_rslots : ctx->nslots;
    V.t.mask = V.nslots - 1;
    const int hb = ctx->opt.hash_bits;
    V.t.hmask = hb >= 64 ? ~0ull : ((1ull << hb) - 1ull);
    V.epoch = regions || ctx->epoch32 == 0 ? kEpochCycle : (ctx->epoch32 - 1) % kEpochCycle + 1;
    V.unresolved = ctx->ulist[0];
    V.wide = ctx->ulist[1];
    V.split = ctx->dlist;
    V.st = ctx->dstate;
    V.L = static_cast<LoopState*>(ctx->dloop);
    V.ctl = reinterpret_cast<LoopCtl*>(static_cast<char*>(ctx->dloop) + ls);
    V.host = h;
    const int64_t* db = ctx->dbegin;
    const int64_t gb[kLoopGroups + 1] = {db[0], db[5], db[6], db[7], db[10]};
    for (int g = 0; g <= kLoopGroups; ++g) V.gb[g] = gb[g];
    V.n_live = db[kDClasses];
    V.n = ctx->n;
    V.copy = ctx->loop_copy;
    ctx->loop_copy ^= 1;
    V.start = start ? 1 : 0;
    V.polls = ctx->loop_polls ? ctx->loop_polls : kSpinLimit;
    V.init = init;
    std::memset(h, 0, sizeof(*h));
    h->stop = kStopLost;                                   // overwritten by the kernel
    const size_t smem = db[kDMid0] > db[kDWarp0] ? sizeof(unsigned long long) * kLoopWarps * kLoopWarpSet : 0;
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
    cudaError_t e;
    // a warp per unit of phase A as far as the SMs go, in CTAs of 512 threads while
    // that is enough of them (16 warps an SM issue their work sooner: 15k against
    // 30k cycles a round on 10k vertices), of 1024 above; a grid of up to one
    // cluster is one
    const int64_t units = cdiv(gb[1], 32) + gb[4] - gb[1];
    const unsigned threads = units <= static_cast<int64_t>(sms) * 16 ? 512 : kLoopThreads;
    const int64_t want = std::max<int64_t>(1, std::min<int64_t>(sms, cdiv(units, threads / 32)));
    const bool keeps = !start || (V.n_live > kKeepListed && 4 * (db[1] - db[0]) >= V.n_live);
    const int cl = keeps ? largest_cluster<true>(ctx->device, smem) : largest_cluster<false>(ctx->device, smem);   // also sets the kernel's attributes, so always asked
    const bool cluster = want > 1 && want <= cl;
    const unsigned grid = static_cast<unsigned>(want);
    V.cluster = cluster ? 1 : 0;
    void* args[] = {&V};
    const void* kernel = keeps ? reinterpret_cast<const void*>(k_round_loop<true>) : reinterpret_cast<const void*>(k_round_loop<false>);
    if (grid == 1 || cluster) {
        cudaLaunchConfig_t cfg = cluster_config(grid, threads, smem);
        cudaLaunchAttribute attr = cluster_attribute(grid);
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        cfg.stream = s;
        e = cudaLaunchKernelExC(&cfg, kernel, args);
    } else {
        e = launch_in_lane(ctx->device, kernel, grid, threads, args, smem, s);
    }
    // refused (too few SMs for a grid that has to be resident as a whole): no result either
    if (e) cudaGetLastError();
    else prof_add_launches(1);
    if ((e = cudaStreamSynchronize(s))) return cuda_error(ctx, e, "round loop");
    *out = *h;
    if (out->stop == kStopLost) {
        cudaMemsetAsync(V.ctl, 0, sizeof(LoopCtl), s);     // both copies of the counters
        ctx->epoch32 = kEpochCycle;                        // the next epoch starts with a blank table
        return BISIM_OK;
    }
    if (!regions) ctx->epoch32 = static_cast<uint32_t>(out->epoch) + kEpochCycle;
    return BISIM_OK;
}

}  // namespace bisim

extern "C" void bisim_loop_polls(bisim_ctx* ctx, uint32_t polls) {
    if (ctx != nullptr) ctx->loop_polls = polls;
}
