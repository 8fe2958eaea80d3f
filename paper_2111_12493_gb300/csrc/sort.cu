// Device-wide exclusive scan and stable LSD radix sort (key u32, value u64).
//
// The radix sort is the classic three-phase scheme per 8-bit digit: per-tile
// digit histograms, one exclusive scan over the (digit, tile) counts, and a
// stable scatter in which every warp ranks its own items with match masks and
// the tile is put in digit order in shared memory before it is written.
#include <algorithm>
#include <string>

#include "common.cuh"
#include "prof.cuh"

namespace bisim {

namespace {

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;   // 4096

constexpr int kRadixThreads = 256;
// Items a thread: tiles of 4096 pairs, or of 1024 below kRadixShort pairs, where
// tiles of 4096 leave most SMs without one.
constexpr int kRadixItems = 16;
constexpr int kRadixShortItems = 4;
constexpr int64_t kRadixShort = int64_t{1} << 20;
constexpr int kRadixBins = 256;
constexpr int kRadixWarps = kRadixThreads / 32;

__device__ __forceinline__ int64_t warp_inclusive_scan(int64_t x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// Scans one tile of kScanTile values; writes the exclusive prefix within the
// tile and the tile total to block_sums[blockIdx.x].
__global__ void __launch_bounds__(kScanThreads) k_scan_tile(const int64_t* __restrict__ in,
                                                            int64_t* __restrict__ out, int64_t n,
                                                            int64_t* __restrict__ block_sums) {
    __shared__ int64_t warp_tot[kScanThreads / 32];
    const int64_t base = static_cast<int64_t>(blockIdx.x) * kScanTile +
                         static_cast<int64_t>(threadIdx.x) * kScanItems;
    int64_t v[kScanItems];
    int64_t run = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        int64_t idx = base + i;
        v[i] = idx < n ? in[idx] : 0;
        run += v[i];
    }
    int64_t inc = warp_inclusive_scan(run);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        int64_t t = warp_tot[lane];
        int64_t ti = warp_inclusive_scan(t);
        warp_tot[lane] = ti - t;   // exclusive per warp
    }
    __syncthreads();
    int64_t excl = warp_tot[warp] + inc - run;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        int64_t idx = base + i;
        if (idx < n) out[idx] = excl;
        excl += v[i];
    }
    if (threadIdx.x == kScanThreads - 1) block_sums[blockIdx.x] = excl;
}

__global__ void k_scan_add(int64_t* __restrict__ out, int64_t n, const int64_t* __restrict__ offs) {
    int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < n) out[i] += offs[i / kScanTile];
}

template <int ITEMS>
__global__ void __launch_bounds__(kRadixThreads) k_radix_hist(const uint32_t* __restrict__ keys,
                                                               int64_t m, int shift,
                                                               int64_t* __restrict__ counts,
                                                               int64_t ntiles) {
    __shared__ unsigned hist[kRadixBins];
    hist[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = static_cast<int64_t>(blockIdx.x) * kRadixThreads * ITEMS;
#pragma unroll 4
    for (int r = 0; r < ITEMS; ++r) {
        int64_t idx = base + static_cast<int64_t>(r) * kRadixThreads + threadIdx.x;
        if (idx < m) atomicAdd(&hist[(keys[idx] >> shift) & 0xffu], 1u);
    }
    __syncthreads();
    counts[static_cast<int64_t>(threadIdx.x) * ntiles + blockIdx.x] = hist[threadIdx.x];
}

// Stable scatter. Warp w of a tile takes its w-th run of 32 * ITEMS items in
// order; an item's rank is the warp's earlier items of its digit (counted in the
// warp's own row of shared memory, so the ranking needs no CTA barrier) plus
// those of the warps before it. The tile then goes through shared memory in
// digit order, so that a warp writes runs of one digit's items. (Ranking by
// rounds of 256 items with three CTA barriers each and scattered writes: 37
// against 20 us for a pass over 2.9M pairs.)
template <int ITEMS>
struct RadixShared {
    unsigned wcnt[kRadixWarps][kRadixBins];      // per warp: items of a digit, later those before the warp's
    unsigned first[kRadixBins];                  // the digit's first item in the tile's order
    int64_t base[kRadixBins];                    // where the digit's items go, less `first`
    unsigned wsum[kRadixWarps];
    uint64_t val[kRadixThreads * ITEMS];
    uint32_t key[kRadixThreads * ITEMS];
};

template <int ITEMS>
__global__ void __launch_bounds__(kRadixThreads, 3) k_radix_scatter(
    const uint32_t* __restrict__ kin, const uint64_t* __restrict__ vin, uint32_t* __restrict__ kout,
    uint64_t* __restrict__ vout, int64_t m, int shift, const int64_t* __restrict__ offs,
    int64_t ntiles) {
    extern __shared__ __align__(16) unsigned char raw[];
    RadixShared<ITEMS>& sh = *reinterpret_cast<RadixShared<ITEMS>*>(raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t tbase = static_cast<int64_t>(blockIdx.x) * kRadixThreads * ITEMS;
    const int64_t wbase = tbase + static_cast<int64_t>(warp) * 32 * ITEMS;
    uint32_t k[ITEMS];
    uint64_t v[ITEMS];
    unsigned rank[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int64_t idx = wbase + r * 32 + lane;
        k[r] = idx < m ? kin[idx] : 0u;
        v[r] = idx < m ? vin[idx] : 0ull;
    }
    for (int d = lane; d < kRadixBins; d += 32) sh.wcnt[warp][d] = 0u;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const bool valid = wbase + r * 32 + lane < m;
        const unsigned d = valid ? (k[r] >> shift) & 0xffu : static_cast<unsigned>(kRadixBins);
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const unsigned before = valid ? sh.wcnt[warp][d] : 0u;
        rank[r] = before + static_cast<unsigned>(__popc(peers & lt));
        __syncwarp();
        if (valid && lane == __ffs(peers) - 1) sh.wcnt[warp][d] = before + static_cast<unsigned>(__popc(peers));
        __syncwarp();
    }
    __syncthreads();
    // thread d: its digit's items before each warp, and where the digit starts in the tile
    unsigned total = 0;
#pragma unroll
    for (int w = 0; w < kRadixWarps; ++w) {
        const unsigned c = sh.wcnt[w][tid];
        sh.wcnt[w][tid] = total;
        total += c;
    }
    unsigned inc = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) sh.wsum[warp] = inc;
    __syncthreads();
    unsigned at = inc - total;
    for (int w = 0; w < warp; ++w) at += sh.wsum[w];
    sh.first[tid] = at;
    sh.base[tid] = offs[static_cast<int64_t>(tid) * ntiles + blockIdx.x] - static_cast<int64_t>(at);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        if (wbase + r * 32 + lane >= m) continue;
        const unsigned d = (k[r] >> shift) & 0xffu;
        const unsigned to = sh.first[d] + sh.wcnt[warp][d] + rank[r];
        sh.key[to] = k[r];
        sh.val[to] = v[r];
    }
    __syncthreads();
    const int count = static_cast<int>(m - tbase < kRadixThreads * ITEMS ? m - tbase : kRadixThreads * ITEMS);
    for (int i = tid; i < count; i += kRadixThreads) {
        const uint32_t key = sh.key[i];
        const int64_t to = sh.base[(key >> shift) & 0xffu] + i;
        kout[to] = key;
        vout[to] = sh.val[i];
    }
}

template <int ITEMS>
cudaError_t radix_pass(const uint32_t* ki, const uint64_t* vi, uint32_t* ko, uint64_t* vo, int64_t m, int shift, int64_t ntiles,
                int64_t* counts, int64_t* offs, int64_t* stmp, int site_h, int site_s, cudaStream_t s) {
    cudaError_t e = allow_smem(reinterpret_cast<const void*>(k_radix_scatter<ITEMS>), sizeof(RadixShared<ITEMS>));
    if (e) return e;
    {
        Launch L(site_h, s, 0, m, 4.0 * m);
        k_radix_hist<ITEMS><<<static_cast<unsigned>(ntiles), kRadixThreads, 0, s>>>(ki, m, shift, counts, ntiles);
    }
    exclusive_scan_i64(counts, offs, ntiles * kRadixBins, stmp, s);
    Launch L(site_s, s, 0, m, 24.0 * m);
    k_radix_scatter<ITEMS><<<static_cast<unsigned>(ntiles), kRadixThreads, sizeof(RadixShared<ITEMS>), s>>>(
        ki, vi, ko, vo, m, shift, offs, ntiles);
    return cudaGetLastError();
}

int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

// Inputs of at most kSmallSortMax pairs (update batches, small frontiers): one
// CTA runs all radix passes over (key, input index) in shared memory, in one
// launch instead of three per 8-bit digit. Ranking is that of the scatter above.
// (A bitonic network of the same size is bound by its own instructions on the one
// SM it runs on: 19 us a sort of 2k.)
constexpr int kSmallSortMax = 4096;
constexpr int kSmallSortThreads = 512;
constexpr int kSmallSortWarps = kSmallSortThreads / 32;

template <int ITEMS>
__global__ void __launch_bounds__(kSmallSortThreads) k_small_sort(const uint32_t* __restrict__ k0,
                                                                  const uint64_t* __restrict__ v0,
                                                                  uint32_t* __restrict__ k1, uint64_t* __restrict__ v1,
                                                                  int m, int bits) {
    __shared__ unsigned wcnt[kSmallSortWarps][kRadixBins];
    __shared__ unsigned first[kRadixBins];
    __shared__ unsigned wsum[kRadixBins / 32];
    __shared__ uint32_t skey[kSmallSortThreads * ITEMS];
    __shared__ uint16_t sidx[kSmallSortThreads * ITEMS];
    const int tid = static_cast<int>(threadIdx.x), warp = tid >> 5, lane = tid & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int wbase = warp * 32 * ITEMS + lane;
    uint32_t k[ITEMS];
    unsigned idx[ITEMS], rank[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        idx[r] = static_cast<unsigned>(wbase + r * 32);
        k[r] = idx[r] < static_cast<unsigned>(m) ? k0[idx[r]] : 0u;
    }
    for (int shift = 0; shift < bits; shift += 8) {
        const unsigned mask = bits - shift >= 8 ? 0xffu : (1u << (bits - shift)) - 1u;
        for (int d = lane; d < kRadixBins; d += 32) wcnt[warp][d] = 0u;
        __syncwarp();
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            const bool valid = wbase + r * 32 < m;
            const unsigned d = valid ? (k[r] >> shift) & mask : static_cast<unsigned>(kRadixBins);
            const unsigned peers = __match_any_sync(0xffffffffu, d);
            const unsigned before = valid ? wcnt[warp][d] : 0u;
            rank[r] = before + static_cast<unsigned>(__popc(peers & lt));
            __syncwarp();
            if (valid && lane == __ffs(peers) - 1) wcnt[warp][d] = before + static_cast<unsigned>(__popc(peers));
            __syncwarp();
        }
        __syncthreads();
        unsigned total = 0, inc = 0;
        if (tid < kRadixBins) {
#pragma unroll
            for (int w = 0; w < kSmallSortWarps; ++w) {
                const unsigned c = wcnt[w][tid];
                wcnt[w][tid] = total;
                total += c;
            }
            inc = total;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            if (lane == 31) wsum[warp] = inc;
        }
        __syncthreads();
        if (tid < kRadixBins) {
            unsigned at = inc - total;
            for (int w = 0; w < warp; ++w) at += wsum[w];
            first[tid] = at;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            if (wbase + r * 32 >= m) continue;
            const unsigned d = (k[r] >> shift) & mask;
            const unsigned to = first[d] + wcnt[warp][d] + rank[r];
            skey[to] = k[r];
            sidx[to] = static_cast<uint16_t>(idx[r]);
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            if (wbase + r * 32 >= m) continue;
            k[r] = skey[wbase + r * 32];
            idx[r] = sidx[wbase + r * 32];
        }
    }
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int i = wbase + r * 32;
        if (i >= m) continue;
        k1[i] = k[r];
        v1[i] = v0[idx[r]];
    }
}

}  // namespace

size_t scan_temp_words(int64_t n) {
    size_t words = 0;
    while (n > 1) {
        int64_t nb = cdiv(n, kScanTile);
        words += static_cast<size_t>(2 * nb);   // block sums and their scan
        n = nb;
    }
    return words + 2;
}

void exclusive_scan_i64(const int64_t* in, int64_t* out, int64_t n, int64_t* tmp, cudaStream_t s) {
    if (n <= 0) return;
    int64_t nb = cdiv(n, kScanTile);
    int64_t* sums = tmp;
    int64_t* sums_scan = tmp + nb;
    BISIM_SITE(site, "scan");
    {
        Launch L(site, s, 0, 0, 16.0 * n);
        k_scan_tile<<<static_cast<unsigned>(nb), kScanThreads, 0, s>>>(in, out, n, sums);
    }
    if (nb > 1) {
        exclusive_scan_i64(sums, sums_scan, nb, tmp + 2 * nb, s);
        Launch L(site, s, 0, 0, 16.0 * n);
        k_scan_add<<<static_cast<unsigned>(cdiv(n, 256)), 256, 0, s>>>(out, n, sums_scan);
    }
}

int64_t radix_tiles(int64_t m) {
    return cdiv(m > 0 ? m : 1, kRadixThreads * (m <= kRadixShort ? kRadixShortItems : kRadixItems));
}

size_t radix_temp_words(int64_t m) {
    // a caller may sort fewer pairs than it sized the scratch for, in smaller tiles
    const int64_t ntiles = std::max(radix_tiles(m), radix_tiles(std::min(m, kRadixShort)));
    int64_t nc = ntiles * kRadixBins;
    return static_cast<size_t>(2 * nc) + scan_temp_words(nc);
}

cudaError_t radix_sort_pairs(uint32_t* k0, uint64_t* v0, uint32_t* k1, uint64_t* v1, int64_t m, int bits,
                             int64_t* tmp, cudaStream_t s, const char* site_name, int* which) {
    *which = 0;
    if (m <= 0 || bits <= 0) return cudaSuccess;
    if (m <= kSmallSortMax) {
        BISIM_SITE(site_small, "small_sort");
        Launch L(site_small, s, 0, m, 24.0 * m);
        const int mi = static_cast<int>(m);
        if (m <= 2 * kSmallSortThreads) k_small_sort<2><<<1, kSmallSortThreads, 0, s>>>(k0, v0, k1, v1, mi, bits);
        else k_small_sort<8><<<1, kSmallSortThreads, 0, s>>>(k0, v0, k1, v1, mi, bits);
        *which = 1;
        return cudaGetLastError();
    }
    const int64_t ntiles = radix_tiles(m);
    const int64_t nc = ntiles * kRadixBins;
    int64_t* counts = tmp;
    int64_t* offs = tmp + nc;
    int64_t* stmp = tmp + 2 * nc;
    for (int shift = 0; shift < bits; shift += 8) {
        const uint32_t* ki = *which ? k1 : k0;
        const uint64_t* vi = *which ? v1 : v0;
        uint32_t* ko = *which ? k0 : k1;
        uint64_t* vo = *which ? v0 : v1;
        // the site's passes are timed apart from other callers' (the CSR build's
        // full-size passes are the ones the benchmark's roofline names)
        const std::string name = site_name;
        const int site_h = prof_site((name + "_hist").c_str());
        const int site_s = prof_site((name + "_scatter").c_str());
        const cudaError_t e =
            m <= kRadixShort ? radix_pass<kRadixShortItems>(ki, vi, ko, vo, m, shift, ntiles, counts, offs, stmp, site_h, site_s, s)
                             : radix_pass<kRadixItems>(ki, vi, ko, vo, m, shift, ntiles, counts, offs, stmp, site_h, site_s, s);
        if (e) return e;
        *which ^= 1;
    }
    return cudaSuccess;
}

}  // namespace bisim
