// The device-side round loop: its state, shared by the cooperative kernel
// (rounds.cu) and the captured graph (dense.cu).
#pragma once

#include "common.cuh"

namespace bisim {

// Why a loop of rounds ended on the device.
enum : int32_t {
    kStopNo = 0,
    kStopDone = 1,
    kStopCollision = 2,     // the last round's hash collisions are left to the host
    kStopError = 3,         // error bits in the status word
    kStopWideRows = 4,      // cooperative kernel: rows above 256 edges are listed; nothing was done
    kStopLost = 5,          // cooperative kernel: it could not run, or gave up at a barrier
};

// State of a run of rounds (device memory, and its pinned mirror).
struct LoopState {
    unsigned long long prev_blocks;   // block count of the partition the next round refines
    unsigned long long blocks;        // block count after the last round
    int32_t executed;                 // rounds run
    int32_t limit;                    // rounds allowed
    int32_t fixpoint;                 // 1: stop as soon as a round keeps the block count
    int32_t rounds;                   // the result r (k, or the fixpoint round)
    int32_t stop;                     // kStop*
    int32_t epoch;                    // cooperative kernel: the table epoch of its last round
};

// The state after a round that ended with `blocks` blocks and the given
// unresolved positions and error bits.
__host__ __device__ inline void loop_advance(LoopState& L, unsigned long long blocks, unsigned unresolved,
                                             unsigned error) {
    L.executed += 1;
    if (error != 0u) {
        L.stop = kStopError;
    } else if (unresolved != 0u) {
        L.stop = kStopCollision;
    } else if (blocks == L.prev_blocks) {     // P_{i+1} refines P_i with as many blocks: the fixpoint
        L.stop = kStopDone;
        L.rounds = L.fixpoint ? L.executed - 1 : L.limit;
    } else if (L.executed >= L.limit) {
        L.stop = kStopDone;
        L.rounds = L.limit;
    }
    if (L.stop < kStopCollision) L.prev_blocks = blocks;
    L.blocks = blocks;
}

// For the lanes with `on`: is every pair value of the row [ev, ev + dv) of the packed
// rows among those of [er, er + dr)? Rows of at most 32 edges; the whole warp takes
// part. Four pairs at a time, eight lanes a pair, four values of each row a lane.
// `value`: the pair value of a packed word.
template <class Value>
__device__ __forceinline__ bool rows_inside(bool on, int64_t ev, int dv, int64_t er, int dr,
                                            const unsigned long long* __restrict__ pe, const Value& value) {
    const unsigned lane = threadIdx.x & 31u;
    const int sub = static_cast<int>(lane & 7u);
    bool inside = false;
    unsigned todo = __ballot_sync(0xffffffffu, on);
    while (todo) {
        unsigned mine = todo;                                        // from the (lane / 8)-th pair that is left on
        for (unsigned k = 0; k < lane / 8; ++k) mine &= mine - 1u;
        const int q = mine ? __ffs(mine) - 1 : 0;
        const int64_t qev = __shfl_sync(0xffffffffu, ev, q), qer = __shfl_sync(0xffffffffu, er, q);
        const int gdv = __shfl_sync(0xffffffffu, dv, q), gdr = __shfl_sync(0xffffffffu, dr, q);
        const int qdv = mine ? gdv : 0, qdr = mine ? gdr : 0;
        uint64_t va[4], vb[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            va[j] = sub + 8 * j < qdv ? pe[qev + sub + 8 * j] : 0ull;
            vb[j] = sub + 8 * j < qdr ? pe[qer + sub + 8 * j] : 0ull;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (sub + 8 * j < qdv) va[j] = value(va[j]);
            if (sub + 8 * j < qdr) vb[j] = value(vb[j]);
        }
        unsigned found = 0u;                                         // which of the lane's four are among r's
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (__all_sync(0xffffffffu, qdr <= 8 * i)) break;
            for (int k = 0; k < 8; ++k) {
                const uint64_t b = __shfl_sync(0xffffffffu, vb[i], k, 8);   // every lane takes part
                const bool is = 8 * i + k < qdr;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (is && va[j] == b) found |= 1u << j;
            }
        }
        bool miss = false;
#pragma unroll
        for (int j = 0; j < 4; ++j) miss = miss || (sub + 8 * j < qdv && !((found >> j) & 1u));
        const unsigned missed = __ballot_sync(0xffffffffu, miss);
        for (int g = 0; g < 4 && todo; ++g, todo &= todo - 1u)       // the same for the whole warp
            if (static_cast<int>(lane) == __ffs(todo) - 1) inside = ((missed >> (8 * g)) & 0xffu) == 0u;
    }
    return inside;
}

// Whether runs of rounds may go through the cooperative kernel at all.
bool round_loop_usable(const bisim_ctx* ctx);
// Whether it covers the whole graph (no live vertex above 256 edges).
bool round_loop_covers(const bisim_ctx* ctx);
// Allocates the loop state and its mirror.
bisim_status round_loop_state(bisim_ctx* ctx, cudaStream_t s);
// Runs the loop: from P_0 with every live vertex listed (start; `init` is the
// state to begin with), or from the current list and the loop state in device
// memory. The result is in P[0] unless out->stop is kStopCollision or
// kStopError: then the last round stands as the host-driven levels expect it.
// kStopLost: the partition and the list are left anyhow, and the rounds have to
// start from P_0 again without the loop.
// `ccount`: the list's per-class survivor counters. Synchronises s.
bisim_status round_loop(bisim_ctx* ctx, cudaStream_t s, bool start, const LoopState& init, unsigned long long* ccount,
                        LoopState* out);

}  // namespace bisim

// Sets the polls after which the context's loop gives up at a barrier (0: the
// usual number, a few seconds), so that tests see what follows. Not part of the
// public interface.
extern "C" void bisim_loop_polls(bisim_ctx* ctx, uint32_t polls);
