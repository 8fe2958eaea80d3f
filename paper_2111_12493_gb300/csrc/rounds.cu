// The round loop as one cooperative kernel, for lists whose rows have at most
// 256 edges (the thread and warp classes of the dense layout).
//
// What it replaces is a loop of about a dozen kernels a round. Each of those is
// near empty once the list is short (a late round of a power-law graph) or the
// graph is small, and a round then costs its launches: 77 us on 300k vertices in
// paths, 60 us on 10k vertices. Here a round is two phases with a grid barrier
// after each, one CTA of 1024 threads per SM (fewer on small graphs, and no
// barrier but the CTA's own when one CTA holds them all):
//   A  of the previous round's list, the entries that are not alone in their
//      block go on the new list; each computes its signature and enters the table
//   B  every entry of the new list is confirmed against its slot's smallest
//      vertex by an exact comparison, inside the thread for rows of at most
//      eight edges, in the warp for longer ones
// The two partition buffers alternate as input and output; a vertex that leaves
// the list writes its final block into the other one, so both agree on every
// vertex that is not listed. After B all CTAs read the same counts and take the
// same decision: another round, done, or back to the host at a hash collision
// (with the state the host-driven levels expect).
#include <algorithm>
#include <climits>
#include <cstring>
#include <mutex>

#include "common.cuh"
#include "prof.cuh"
#include "rounds.cuh"

namespace bisim {

namespace {

constexpr int kLoopThreads = 1024;
constexpr int kLoopWarps = kLoopThreads / 32;
constexpr int kLoopGroups = 4;            // degree <= 8, <= 16, <= 32, <= 256: classes 0-4, 5, 6, 7-9
constexpr int kHotSlots = 64;
constexpr int kLoopWarpSet = 512;         // slots of a warp's set: twice the longest row
constexpr unsigned kSpinLimit = 1u << 22; // polls of a barrier before the kernel gives up (seconds)

int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

// Counters of one round; three of them rotate, so that one can be cleared
// while the others are read.
struct RoundSet {
    unsigned long long blocks;            // listed vertices that are their block's id
    unsigned cnt[kLoopGroups];            // entries of the round's list per group
    unsigned unresolved;
    unsigned error;
};

struct LoopCtl {
    RoundSet set[3];
    unsigned arrived;                     // barrier arrivals since the launch
    unsigned left;                        // CTAs that returned
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
    DevState* st;
    LoopCtl* ctl;
    LoopState* L;
    LoopState* host;                      // pinned: where the host reads the result
    int64_t gb[kLoopGroups + 1];          // first position of each group
    int64_t n_live;
    int32_t n;
    int32_t start;                        // 1: from P_0 with every live position listed; 0: from act[0] / aoff and *L
    LoopState init;                       // start: the loop state to begin with
};

__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }

__device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Pair value of a packed word over the labelling P, which other CTAs write
// between barriers: read through L2.
__device__ __forceinline__ uint64_t word_value(unsigned long long w, const int32_t* P) {
    return pair_value(static_cast<int32_t>(w >> 32), __ldcg(P + static_cast<uint32_t>(w)));
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

struct Shared {
    unsigned long long hot_key[2][kHotSlots];
    unsigned hot_min[2][kHotSlots];
    uint32_t hot_slot[kHotSlots];
    unsigned wcnt[kLoopWarps];
    unsigned wbase[kLoopWarps];
    unsigned long long wsum[kLoopWarps];
    unsigned zero[kLoopWarps];
    int ok;
};

// Grid barrier number `k` (from 1) of this launch; false when it gave up.
__device__ bool grid_barrier(LoopCtl* c, unsigned k, Shared& sh) {
    __syncthreads();
    if (gridDim.x == 1) return true;
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&c->arrived, 1u);
        const unsigned target = gridDim.x * k;
        unsigned spin = 0;
        bool ok = true;
        while (load_acquire(&c->arrived) < target) {
            if (++spin > kSpinLimit || load_acquire(&c->abort) != 0u) {
                atomicExch(&c->abort, 1u);
                ok = false;
                break;
            }
        }
        __threadfence();
        sh.ok = ok ? 1 : 0;
    }
    __syncthreads();
    return sh.ok != 0;
}

// The current list: group g's entries are base[g][0 .. cnt[g]), or (identity)
// the positions from first[g] on.
struct List {
    const int32_t* base[kLoopGroups];
    int64_t cnt[kLoopGroups];
    bool identity;
};

__device__ __forceinline__ int32_t list_at(const LoopView& V, const List& l, int g, int64_t i) {
    return l.identity ? static_cast<int32_t>(V.gb[g] + i) : __ldcg(l.base[g] + i);
}

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

// Does position `pos` go on the next list? Not when its vertex was its block's
// id last round and no other joined it.
__device__ __forceinline__ bool not_alone(const LoopView& V, int32_t pos) {
    return !(__ldcg(V.own + pos) && !__ldcg(V.joined + pos));
}

// Phase A, group 0: a thread per vertex.
__device__ void phase_a_threads(const LoopView& V, const TableRef& tt, const List& l, bool first, const int32_t* Pin,
                                int32_t* Pout, int32_t* next, RoundSet* rs, Shared& sh, int* parity) {
    const int64_t count = l.cnt[0];
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kLoopThreads;
    const int warp = static_cast<int>(threadIdx.x >> 5);
    for (int64_t b = static_cast<int64_t>(blockIdx.x) * kLoopThreads; b < count; b += stride, *parity ^= 1) {
        const int par = *parity;
        const int64_t i = b + threadIdx.x;
        bool stay = false;
        int32_t pos = 0, v = 0;
        uint64_t h = 0, mask = 0;
        int64_t base = 0;
        if (i < count) {
            pos = list_at(V, l, 0, i);
            stay = first || not_alone(V, pos);
            v = __ldg(V.vert + pos);
            const int32_t own = __ldcg(Pin + v);
            if (!stay) {
                Pout[v] = own;
            } else {
                const int64_t e0 = __ldg(V.prp + pos);
                const int d = static_cast<int>(__ldg(V.prp + pos + 1) - e0);
                uint64_t x[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) x[j] = j < d ? __ldcs(V.pe + e0 + j) : 0ull;
#pragma unroll
                for (int j = 0; j < 8; ++j) x[j] = j < d ? word_value(x[j], Pin) : 0ull;
                uint64_t sum = 0;
                unsigned u = 0;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    bool fresh = j < d;
#pragma unroll
                    for (int q = 0; q < j; ++q) fresh = fresh && x[q] != x[j];
                    if (fresh) {
                        sum += x[j];
                        ++u;
                    }
                }
                const uint64_t hash = sig_hash(own, u, sum);
                put_sig(V, pos, hash, u, own);
                V.joined[pos] = 0;
                h = hash & tt.hmask;
                table_span(V, v, &base, &mask);
            }
        }
        unsigned members;
        const int rep = combine(stay, h, base, v, &members);
        const bool doer = stay && rep == static_cast<int>(lane_id());
        int hot = -1;
        if (doer && members >= 4u && V.gid == nullptr && h != 0ull) {
            // popular in the warp: combine over the CTA too
            const int at = static_cast<int>((h ^ (h >> 29)) & (kHotSlots - 1));
            const unsigned long long prev = atomicCAS(&sh.hot_key[par][at], 0ull, static_cast<unsigned long long>(h));
            if (prev == 0ull || prev == h) {
                atomicMin(&sh.hot_min[par][at], static_cast<unsigned>(v));
                hot = at;
            }
        }
        uint32_t sl = ~0u;
        if (doer && hot < 0) sl = table_insert_in(tt, h, v, static_cast<uint64_t>(base), mask, &rs->error);
        const unsigned stays = __ballot_sync(0xffffffffu, stay);
        if (lane_id() == 0) sh.wcnt[warp] = static_cast<unsigned>(__popc(stays));
        __syncthreads();
        if (threadIdx.x < kHotSlots) {
            const unsigned long long key = sh.hot_key[par][threadIdx.x];
            if (key)
                sh.hot_slot[threadIdx.x] = table_insert(tt, key, static_cast<int32_t>(sh.hot_min[par][threadIdx.x]),
                                                        &rs->error);
            sh.hot_key[par ^ 1][threadIdx.x] = 0ull;
            sh.hot_min[par ^ 1][threadIdx.x] = ~0u;
        } else if (warp == 2 && !first) {
            const unsigned c = sh.wcnt[lane_id()];
            unsigned inc = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane_id() >= static_cast<unsigned>(o)) inc += y;
            }
            unsigned at = 0;
            if (lane_id() == 31 && inc) at = atomicAdd(&rs->cnt[0], inc);
            at = __shfl_sync(0xffffffffu, at, 31);
            sh.wbase[lane_id()] = at + inc - c;
        }
        __syncthreads();
        if (hot >= 0) sl = sh.hot_slot[hot];
        sl = __shfl_sync(0xffffffffu, sl, rep);
        if (stay) {
            V.slot[pos] = sl;
            if (!first) next[V.gb[0] + sh.wbase[warp] + __popc(stays & ((1u << lane_id()) - 1u))] = pos;
        }
    }
}

// Phase A, groups 1 to 3: a warp takes up to 32 entries, one at a time with
// all lanes (several at a time for rows of at most 32 edges, to keep their
// loads in flight together); lane q keeps the result of entry q, and the lanes
// finish all of them together. Few entries are spread over all warps.
__device__ void phase_a_warps(const LoopView& V, const TableRef& tt, const List& l, int g, bool first,
                              const int32_t* Pin, int32_t* Pout, int32_t* next, RoundSet* rs, Shared& sh,
                              unsigned long long* sets) {
    const int64_t count = l.cnt[g];
    const int warp = static_cast<int>(threadIdx.x >> 5);
    const unsigned lane = lane_id();
    const int64_t warps = static_cast<int64_t>(gridDim.x) * kLoopWarps;
    const int64_t per = min(static_cast<int64_t>(32), (count + warps - 1) / warps);
    const int64_t gw = static_cast<int64_t>(warp) * gridDim.x + blockIdx.x;      // neighbours on different SMs
    for (int64_t b = gw * per; b < count; b += warps * per) {
        bool stay = false;
        int32_t pos = 0, v = 0, own = 0;
        int64_t e0 = 0;
        int d = 0;
        if (lane < per && b + lane < count) {
            pos = list_at(V, l, g, b + lane);
            stay = first || not_alone(V, pos);
            v = __ldg(V.vert + pos);
            own = __ldcg(Pin + v);
            if (!stay) {
                Pout[v] = own;
            } else {
                e0 = __ldg(V.prp + pos);
                d = static_cast<int>(__ldg(V.prp + pos + 1) - e0);
            }
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
                    if (has[k]) w[k] = word_value(w[k], Pin);
#pragma unroll
                for (int k = 0; k < kAtOnce; ++k) {
                    if (q[k] < 0) break;                           // the same for the whole warp
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
                    if (k * 32 + static_cast<int>(lane) < dd) mv[k] = word_value(mv[k], Pin);
                uint32_t size = 64;
                while (size < 2u * static_cast<uint32_t>(dd)) size <<= 1;
                for (uint32_t j = lane; j < size; j += 32) tab[j] = 0ull;
                if (lane == 0) sh.zero[warp] = 0u;
                __syncwarp();
                uint64_t s = 0;
                unsigned c = 0;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    if (k * 32 >= dd) break;                       // the same for the whole warp
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
                __syncwarp();                                      // the set is cleared for the next row
            }
        }
        uint64_t h = 0, mask = 0;
        int64_t base = 0;
        if (stay) {
            const uint64_t hash = sig_hash(own, cnt, sum);
            put_sig(V, pos, hash, cnt, own);
            V.joined[pos] = 0;
            h = hash & tt.hmask;
            table_span(V, v, &base, &mask);
        }
        unsigned members;
        const int rep = combine(stay, h, base, v, &members);
        uint32_t sl = ~0u;
        if (stay && rep == static_cast<int>(lane))
            sl = table_insert_in(tt, h, v, static_cast<uint64_t>(base), mask, &rs->error);
        sl = __shfl_sync(0xffffffffu, sl, rep);
        unsigned at = 0;
        if (!first && stays) {
            if (lane == 0) at = atomicAdd(&rs->cnt[g], static_cast<unsigned>(__popc(stays)));
            at = __shfl_sync(0xffffffffu, at, 0);
        }
        if (stay) {
            V.slot[pos] = sl;
            if (!first) next[V.gb[g] + at + __popc(stays & ((1u << lane) - 1u))] = pos;
        }
    }
}

// Is every pair value of row [ea, ea + da) among those of row [eb, eb + db)?
// All lanes of the warp take part; at most 256 entries each.
__device__ bool row_inside(const LoopView& V, const int32_t* P, int64_t ea, int da, int64_t eb, int db) {
    const int lane = static_cast<int>(lane_id());
    bool miss = false;
    for (int a0 = 0; a0 < da && !miss; a0 += 32) {
        const bool ha = a0 + lane < da;
        const uint64_t a = ha ? word_value(__ldg(V.pe + ea + a0 + lane), P) : 0ull;
        bool found = !ha;
        for (int b0 = 0; b0 < db; b0 += 32) {
            const uint64_t b = b0 + lane < db ? word_value(__ldg(V.pe + eb + b0 + lane), P) : 0ull;
            const int lim = min(32, db - b0);
            for (int k = 0; k < lim; ++k) {
                const uint64_t bk = __shfl_sync(0xffffffffu, b, k);    // every lane takes part in every shuffle
                found = found || bk == a;
            }
        }
        miss = __any_sync(0xffffffffu, !found);
    }
    return !miss;
}

// Phase B: every listed entry against its slot's representative.
__device__ void phase_b(const LoopView& V, const List& l, const int32_t* Pin, int32_t* Pout, RoundSet* rs,
                        Shared& sh) {
    const int64_t c01 = l.cnt[0] + l.cnt[1], c012 = c01 + l.cnt[2], total = c012 + l.cnt[3];
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kLoopThreads;
    const unsigned lane = lane_id();
    unsigned long long owned = 0;
    for (int64_t b = static_cast<int64_t>(blockIdx.x) * kLoopThreads + (threadIdx.x & ~31u); b < total; b += stride) {
        const int64_t i = b + lane;
        int32_t pos = -1, v = -1, r = -1, rpos = -1;
        bool join = false, push = false, wide = false;
        int64_t ev = 0, er = 0;
        int dv = 0, dr = 0;
        if (i < total) {
            pos = i < l.cnt[0]  ? list_at(V, l, 0, i)
                  : i < c01     ? list_at(V, l, 1, i - l.cnt[0])
                  : i < c012    ? list_at(V, l, 2, i - c01)
                                : list_at(V, l, 3, i - c012);
            v = __ldg(V.vert + pos);
            const uint32_t sv = __ldcg(V.slot + pos);
            r = sv == ~0u ? -1 : static_cast<int32_t>(static_cast<uint32_t>(__ldcg(&V.t.slots[sv].w)));
            if (r < 0 || r >= V.n) {                               // failed insert
                atomicOr(&rs->error, kErrTableFull);
                Pout[v] = -1;
            } else if (r == v) {
                Pout[v] = v;
                V.own[pos] = 1;
                ++owned;
            } else {
                rpos = __ldg(V.vpos + r);
                V.own[pos] = 0;
                const int4 a = __ldcg(reinterpret_cast<const int4*>(V.sig + pos));
                const int4 c = __ldcg(reinterpret_cast<const int4*>(V.sig + rpos));
                if (a.z != c.z || a.w != c.w) {                    // |S| or own block differ
                    push = true;
                } else if (a.z <= 1) {                             // the full hash decides (a bijection of the pair)
                    join = a.x == c.x && a.y == c.y;
                    push = !join;
                } else {
                    ev = __ldg(V.prp + pos);
                    dv = static_cast<int>(__ldg(V.prp + pos + 1) - ev);
                    er = __ldg(V.prp + rpos);
                    dr = static_cast<int>(__ldg(V.prp + rpos + 1) - er);
                    if (dv <= 8 && dr <= 8) {
                        // S_v inside S_r with equal sizes means equal sets
                        uint64_t x[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) x[j] = j < dr ? __ldg(V.pe + er + j) : 0ull;
#pragma unroll
                        for (int j = 0; j < 8; ++j) x[j] = j < dr ? word_value(x[j], Pin) : 0ull;
                        bool all = true;
                        for (int j = 0; j < dv; ++j) {
                            const uint64_t y = word_value(__ldg(V.pe + ev + j), Pin);
                            bool found = false;
#pragma unroll
                            for (int q = 0; q < 8; ++q) found = found || (q < dr && x[q] == y);
                            all = all && found;
                        }
                        join = all;
                        push = !all;
                    } else {
                        wide = true;
                    }
                }
            }
        }
        for (unsigned todo = __ballot_sync(0xffffffffu, wide); todo; todo &= todo - 1u) {
            const int q = __ffs(todo) - 1;
            const bool same = row_inside(V, Pin, __shfl_sync(0xffffffffu, ev, q), __shfl_sync(0xffffffffu, dv, q),
                                         __shfl_sync(0xffffffffu, er, q), __shfl_sync(0xffffffffu, dr, q));
            if (static_cast<int>(lane) == q) {
                join = same;
                push = !same;
            }
        }
        if (join) {
            Pout[v] = r;
            if (!__ldcg(V.joined + rpos)) V.joined[rpos] = 1;
        }
        const unsigned p = __ballot_sync(0xffffffffu, push);
        if (p) {
            unsigned at = 0;
            if (lane == 0) at = atomicAdd(&rs->unresolved, static_cast<unsigned>(__popc(p)));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (push) V.unresolved[at + __popc(p & ((1u << lane) - 1u))] = pos;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) owned += __shfl_xor_sync(0xffffffffu, owned, o);
    if (lane == 0) sh.wsum[threadIdx.x >> 5] = owned;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long s = 0;
        for (int w = 0; w < kLoopWarps; ++w) s += sh.wsum[w];
        if (s) atomicAdd(&rs->blocks, s);
    }
}

// Every listed position through f(pos).
template <class F>
__device__ __forceinline__ void for_listed(const LoopView& V, const List& l, const F& f) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * kLoopThreads;
    const int64_t t = static_cast<int64_t>(blockIdx.x) * kLoopThreads + threadIdx.x;
    int64_t before = 0;
    for (int g = 0; g < kLoopGroups; before += l.cnt[g], ++g)
        for (int64_t i = t; i < l.cnt[g]; i += stride) f(list_at(V, l, g, i), before + i);
}

__global__ void __launch_bounds__(kLoopThreads, 1) k_round_loop(const LoopView V) {
    extern __shared__ unsigned long long sets[];           // kLoopWarps * kLoopWarpSet when warp-class rows exist
    __shared__ Shared sh;
    LoopCtl* ctl = V.ctl;
    LoopState S = V.init;
    if (!V.start) S = *V.L;
    List l;
    l.identity = V.start != 0;
    if (V.start) {
        for (int g = 0; g < kLoopGroups; ++g) {
            l.base[g] = nullptr;
            l.cnt[g] = V.gb[g + 1] - V.gb[g];
        }
    } else {
        constexpr int c0[kLoopGroups + 1] = {0, 5, 6, 7, 10};
        for (int g = 0; g < kLoopGroups; ++g) {
            l.base[g] = V.act[0] + V.aoff[c0[g]];
            l.cnt[g] = V.aoff[c0[g + 1]] - V.aoff[c0[g]];
        }
        if (S.stop == 0 && V.aoff[16] != V.aoff[10]) S.stop = kStopWideRows;   // rows above 256 edges are listed
    }
    if (threadIdx.x < kHotSlots) {
        for (int p = 0; p < 2; ++p) {
            sh.hot_key[p][threadIdx.x] = 0ull;
            sh.hot_min[p][threadIdx.x] = ~0u;
        }
    }
    __syncthreads();
    uint32_t ep = V.epoch;
    unsigned bar = 0;
    int parity = 0, nbuf = V.start ? 0 : 1;                // the list buffer the next list goes to
    bool fine = true;
    const int32_t* Pin = V.start ? V.P0 : V.P[0];
    int out = 1;
    for (int round = 0; S.stop == 0; ++round) {
        const bool first = round == 0;
        RoundSet* rs = &ctl->set[round % 3];
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            RoundSet z{};
            ctl->set[(round + 1) % 3] = z;
        }
        if (ep == kEpochCycle) {                           // every epoch is used up: blank the table
            uint4* w = reinterpret_cast<uint4*>(V.t.slots);
            const uint64_t st = static_cast<uint64_t>(gridDim.x) * kLoopThreads;
            for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * kLoopThreads + threadIdx.x; i < V.nslots / 2; i += st)
                w[i] = make_uint4(0u, 0u, 0u, 0u);
            ep = 0;
            if (!(fine = grid_barrier(ctl, ++bar, sh))) break;
        }
        ++ep;
        TableRef tt = V.t;
        tt.epoch = static_cast<uint64_t>(ep) << 32;
        int32_t* Pout = V.P[out];
        int32_t* next = V.act[nbuf];
        for (int g = 1; g < kLoopGroups; ++g)
            if (l.cnt[g] > 0) phase_a_warps(V, tt, l, g, first, Pin, Pout, next, rs, sh, sets);
        phase_a_threads(V, tt, l, first, Pin, Pout, next, rs, sh, &parity);
        if (!(fine = grid_barrier(ctl, ++bar, sh))) break;
        if (!first) {
            l.identity = false;
            for (int g = 0; g < kLoopGroups; ++g) {
                l.base[g] = next + V.gb[g];
                l.cnt[g] = __ldcg(&rs->cnt[g]);
            }
            nbuf ^= 1;
        }
        phase_b(V, l, Pin, Pout, rs, sh);
        if (!(fine = grid_barrier(ctl, ++bar, sh))) break;
        const int64_t listed = l.cnt[0] + l.cnt[1] + l.cnt[2] + l.cnt[3];
        const unsigned long long blocks = static_cast<unsigned long long>(V.n_live - listed) + __ldcg(&rs->blocks);
        loop_advance(S, blocks, __ldcg(&rs->unresolved), __ldcg(&rs->error));
        if (S.stop == kStopDone) {
            if (out != 0)                                  // the result belongs in P[0]
                for_listed(V, l, [&](int32_t pos, int64_t) {
                    const int32_t v = __ldg(V.vert + pos);
                    V.P[0][v] = __ldcg(V.P[1] + v);
                });
        } else if (S.stop != 0) {
            // back to the host within this round: P_i in P[0], P_{i+1} as far as it is
            // known in P[1], the list in act[0] / aoff, the counts in the status word
            int32_t* flat = V.act[1];
            const bool in_place = first && !V.start;
            if (!in_place) {
                // a list in act[1]'s own regions first moves to act[0]'s
                if (!l.identity && l.base[0] == V.act[1] + V.gb[0]) {
                    for (int g = 0; g < kLoopGroups; ++g) {
                        const int64_t st = static_cast<int64_t>(gridDim.x) * kLoopThreads;
                        for (int64_t i = static_cast<int64_t>(blockIdx.x) * kLoopThreads + threadIdx.x; i < l.cnt[g]; i += st)
                            V.act[0][V.gb[g] + i] = __ldcg(l.base[g] + i);
                        l.base[g] = V.act[0] + V.gb[g];
                    }
                    if (!(fine = grid_barrier(ctl, ++bar, sh))) break;
                }
                for_listed(V, l, [&](int32_t pos, int64_t i) { flat[i] = pos; });
            }
            if (V.start && first) {
                for_listed(V, l, [&](int32_t pos, int64_t) {
                    const int32_t v = __ldg(V.vert + pos);
                    V.P[0][v] = __ldg(V.P0 + v);
                });
            } else if (out == 0) {
                for_listed(V, l, [&](int32_t pos, int64_t) {
                    const int32_t v = __ldg(V.vert + pos);
                    const int32_t a = __ldcg(V.P[0] + v), c = __ldcg(V.P[1] + v);
                    V.P[0][v] = c;
                    V.P[1][v] = a;
                });
            }
            if (!(fine = grid_barrier(ctl, ++bar, sh))) break;
            if (!in_place)
                for (int64_t i = static_cast<int64_t>(blockIdx.x) * kLoopThreads + threadIdx.x; i < listed;
                     i += static_cast<int64_t>(gridDim.x) * kLoopThreads)
                    V.act[0][i] = __ldcg(flat + i);
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                if (!in_place) {
                    // the groups as classes: 0 (0 to 4), 5, 6, 7 (7 to 9)
                    const int64_t o[4] = {l.cnt[0], l.cnt[0] + l.cnt[1], l.cnt[0] + l.cnt[1] + l.cnt[2], listed};
                    V.aoff[0] = 0;
                    for (int c = 1; c <= kDClasses; ++c) V.aoff[c] = c <= 5 ? o[0] : c == 6 ? o[1] : c == 7 ? o[2] : o[3];
                    for (int c = 0; c < kDClasses; ++c) V.ccount[c] = 0ull;
                }
                DevState z{};
                z.blocks = blocks;
                z.unresolved = __ldcg(&rs->unresolved);
                z.error = __ldcg(&rs->error);
                z.listed = static_cast<unsigned>(listed);
                *V.st = z;
            }
        }
        Pin = Pout;
        out ^= 1;
    }
    // the last CTA to leave writes the result and clears the counters for the next launch
    __syncthreads();
    if (threadIdx.x == 0 && fine) {
        __threadfence();
        const unsigned left = atomicAdd(&ctl->left, 1u);
        if (left == gridDim.x - 1) {
            RoundSet z{};
            for (int k = 0; k < 3; ++k) ctl->set[k] = z;
            ctl->arrived = 0u;
            ctl->left = 0u;
            S.epoch = static_cast<int32_t>(ep);
            *V.L = S;
            *V.host = S;
            __threadfence_system();
        }
    }
}

// Cooperative launches of this process follow one another on a device, whatever
// their streams: each waits for the event recorded after the one before, so that
// two of them never share the SMs half resident.
struct CoopLane {
    std::mutex mu;
    cudaEvent_t done[64] = {};
    cudaStream_t last[64] = {};
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
    } else if (lane.last[device] != s) {
        if ((e = cudaStreamWaitEvent(s, lane.done[device], 0))) return e;
    }
    if ((e = cudaLaunchCooperativeKernel(kernel, dim3(grid), dim3(threads), args, smem, s))) return e;
    lane.last[device] = s;
    return cudaEventRecord(lane.done[device], s);
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
    V.st = ctx->dstate;
    V.L = static_cast<LoopState*>(ctx->dloop);
    V.ctl = reinterpret_cast<LoopCtl*>(static_cast<char*>(ctx->dloop) + ls);
    V.host = h;
    const int64_t* db = ctx->dbegin;
    const int64_t gb[kLoopGroups + 1] = {db[0], db[5], db[6], db[7], db[10]};
    for (int g = 0; g <= kLoopGroups; ++g) V.gb[g] = gb[g];
    V.n_live = db[kDClasses];
    V.n = ctx->n;
    V.start = start ? 1 : 0;
    V.init = init;
    std::memset(h, 0, sizeof(*h));
    h->stop = kStopLost;                                   // overwritten by the kernel
    const size_t smem = db[kDMid0] > db[kDWarp0] ? sizeof(unsigned long long) * kLoopWarps * kLoopWarpSet : 0;
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
    cudaError_t e;
    static std::once_flag once;
    std::call_once(once, [] {
        cudaFuncSetAttribute(k_round_loop, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(sizeof(unsigned long long) * kLoopWarps * kLoopWarpSet));
    });
    // a thread per vertex of the short rows, a warp for every four longer ones;
    // fewer CTAs make a cheaper barrier
    const int64_t need = std::max(cdiv(gb[1], kLoopThreads), cdiv(gb[4] - gb[1], 4 * kLoopWarps));
    const unsigned grid = static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>(sms, need)));
    void* args[] = {&V};
    if ((e = launch_in_lane(ctx->device, reinterpret_cast<const void*>(k_round_loop), grid, kLoopThreads, args, smem, s)))
        return cuda_error(ctx, e, "launch round loop");
    prof_add_launches(1);
    if ((e = cudaStreamSynchronize(s))) return cuda_error(ctx, e, "round loop");
    *out = *h;
    if (out->stop == kStopLost) {
        cudaMemsetAsync(V.ctl, 0, sizeof(LoopCtl), s);
        cudaStreamSynchronize(s);
        ctx->epoch32 = kEpochCycle;
        return set_error(ctx, BISIM_ETIMEOUT, "round loop: a grid barrier ran out of polls");
    }
    if (!regions) ctx->epoch32 = static_cast<uint32_t>(out->epoch) + kEpochCycle;
    return BISIM_OK;
}

}  // namespace bisim
