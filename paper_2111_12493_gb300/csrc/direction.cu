// Direction and label parameterizations (Section 2.4.2 and Section 2.5):
// forward bisimulation compares the out-edges of two vertices, backward
// bisimulation their in-edges, and the forward-backward variant both; a label
// filter restricts the edges taken into account to a set of labels.
//
// The refinement kernels always compare out-edges of the graph they are given,
// so each variant becomes an edge list that the unchanged path refines:
//   forward     the edges as given
//   backward    every edge (u, w, l) reversed to (w, u, l)
//   both        every edge twice: (u, w, 2l) for the out-edge of u and
//               (w, u, 2l + 1) for the in-edge of w, so a pair's label keeps
//               its direction and no out-pair can equal an in-pair (labels
//               must lie in [-2^30, 2^30) for this to be injective)
//   filter      edges whose label is not listed are left out
// Update batches go through the same mapping (an edge operation becomes one
// or two operations on the internal edge list, in order), and the summary
// graph reports edges in the caller's direction and labels.
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "prof.cuh"

namespace bisim {

namespace {

constexpr int32_t kBothLabelMin = -(1 << 30);
constexpr int32_t kBothLabelMax = (1 << 30) - 1;

unsigned grid_for(int64_t n, int threads) {
    return static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>((n + threads - 1) / threads, 152 * 32)));
}

__device__ __forceinline__ bool listed(const int32_t* __restrict__ f, int32_t nf, int32_t l) {
    if (nf == 0) return true;
    int32_t lo = 0, hi = nf - 1;
    while (lo < hi) {
        const int32_t mid = (lo + hi) >> 1;
        if (f[mid] < l) lo = mid + 1; else hi = mid;
    }
    return f[lo] == l;
}

// Internal edges per input edge (0, 1 or 2); cnt[m] = 0 closes the scan.
__global__ void k_view_count(const int32_t* __restrict__ lab, int64_t m, const int32_t* __restrict__ filt, int32_t nf,
                             int32_t dir, int64_t* __restrict__ cnt, unsigned* err) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e <= m; e += stride) {
        if (e == m) {
            cnt[e] = 0;
            continue;
        }
        const int32_t l = lab[e];
        const bool keep = listed(filt, nf, l);
        if (keep && dir == BISIM_DIR_BOTH && (l < kBothLabelMin || l > kBothLabelMax)) atomicOr(err, kErrBadInput);
        cnt[e] = keep ? (dir == BISIM_DIR_BOTH ? 2 : 1) : 0;
    }
}

__global__ void k_view_emit(const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                            const int32_t* __restrict__ lab, int64_t m, const int64_t* __restrict__ pos, int32_t dir,
                            int32_t* __restrict__ os, int32_t* __restrict__ od, int32_t* __restrict__ ol) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t e = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < m; e += stride) {
        const int64_t p = pos[e];
        if (pos[e + 1] == p) continue;
        const int32_t u = src[e], w = dst[e], l = lab[e];
        if (dir == BISIM_DIR_FORWARD) {
            os[p] = u; od[p] = w; ol[p] = l;
        } else if (dir == BISIM_DIR_BACKWARD) {
            os[p] = w; od[p] = u; ol[p] = l;
        } else {
            os[p] = u; od[p] = w; ol[p] = 2 * l;
            os[p + 1] = w; od[p + 1] = u; ol[p + 1] = 2 * l + 1;
        }
    }
}

// Both directions of every edge, unfiltered: edge e becomes entries 2e and 2e + 1, so
// nothing is counted and nothing read back (counts, their scan and an emission that
// looks places up: 168 us for 8M edges, against 50). A label out of range is left to
// the build's read-back. Two edges a thread, 16-byte stores; 8-byte loads where the
// arrays take them (`wide`).
__global__ void __launch_bounds__(256) k_view_both(const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                                                   const int32_t* __restrict__ lab, int64_t m, bool wide,
                                                   int32_t* __restrict__ os, int32_t* __restrict__ od,
                                                   int32_t* __restrict__ ol, DevState* st) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    bool bad = false;
    for (int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; 2 * q < m; q += stride) {
        const int64_t e = 2 * q;
        const bool two = e + 1 < m;
        int2 u, w, l;
        if (wide && two) {
            u = __ldcs(reinterpret_cast<const int2*>(src + e));
            w = __ldcs(reinterpret_cast<const int2*>(dst + e));
            l = __ldcs(reinterpret_cast<const int2*>(lab + e));
        } else {
            u = make_int2(src[e], two ? src[e + 1] : 0);
            w = make_int2(dst[e], two ? dst[e + 1] : 0);
            l = make_int2(lab[e], two ? lab[e + 1] : 0);
        }
        bad = bad || l.x < kBothLabelMin || l.x > kBothLabelMax || l.y < kBothLabelMin || l.y > kBothLabelMax;
        const int32_t l0 = static_cast<int32_t>(2u * static_cast<uint32_t>(l.x)), l1 = static_cast<int32_t>(2u * static_cast<uint32_t>(l.y));
        if (two) {
            reinterpret_cast<int4*>(os)[q] = make_int4(u.x, w.x, u.y, w.y);
            reinterpret_cast<int4*>(od)[q] = make_int4(w.x, u.x, w.y, u.y);
            reinterpret_cast<int4*>(ol)[q] = make_int4(l0, l0 + 1, l1, l1 + 1);
        } else {
            reinterpret_cast<int2*>(os)[e] = make_int2(u.x, w.x);
            reinterpret_cast<int2*>(od)[e] = make_int2(w.x, u.x);
            reinterpret_cast<int2*>(ol)[e] = make_int2(l0, l0 + 1);
        }
    }
    if (bad) atomicOr(&st->bad_label, 1u);
}

// Per-graph offsets of the view's edges (pos null: two of every edge).
__global__ void k_view_offsets(const int64_t* __restrict__ pos, const int64_t* __restrict__ eoff, int32_t G,
                               int64_t* __restrict__ out) {
    const int64_t g = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (g <= G) out[g] = pos ? pos[eoff[g]] : 2 * eoff[g];
}

// Internal operations per operation: edge operations as edges above, vertex
// operations (and unknown kinds, which the batch check rejects) once.
__global__ void k_ops_count(const bisim_op* __restrict__ ops, int64_t n, const int32_t* __restrict__ filt, int32_t nf,
                            int32_t dir, int64_t* __restrict__ cnt, unsigned* err) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i <= n; i += stride) {
        if (i == n) {
            cnt[i] = 0;
            continue;
        }
        const bisim_op o = ops[i];
        int64_t c = 1;
        if (o.kind == BISIM_OP_EDGE_ADD || o.kind == BISIM_OP_EDGE_DEL) {
            const bool keep = listed(filt, nf, o.label);
            if (keep && dir == BISIM_DIR_BOTH && (o.label < kBothLabelMin || o.label > kBothLabelMax))
                atomicOr(err, kErrBadInput);
            c = keep ? (dir == BISIM_DIR_BOTH ? 2 : 1) : 0;
        }
        cnt[i] = c;
    }
}

__global__ void k_ops_emit(const bisim_op* __restrict__ ops, int64_t n, const int64_t* __restrict__ pos, int32_t dir,
                           bisim_op* __restrict__ out) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) {
        const int64_t p = pos[i];
        if (pos[i + 1] == p) continue;
        bisim_op o = ops[i];
        if (o.kind != BISIM_OP_EDGE_ADD && o.kind != BISIM_OP_EDGE_DEL) {
            out[p] = o;
        } else if (dir == BISIM_DIR_FORWARD) {
            out[p] = o;
        } else if (dir == BISIM_DIR_BACKWARD) {
            out[p] = bisim_op{o.kind, o.dst, o.src, o.label};
        } else {
            out[p] = bisim_op{o.kind, o.src, o.dst, 2 * o.label};
            out[p + 1] = bisim_op{o.kind, o.dst, o.src, 2 * o.label + 1};
        }
    }
}

// One warp per vertex writes the vertex into its row's entries; rows outside
// [0, m] or running backwards only raise the error flag.
__global__ void k_csr_sources(const int64_t* __restrict__ rp, int32_t n, int64_t m, int32_t* __restrict__ src,
                              unsigned* err) {
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
    const unsigned lane = threadIdx.x & 31u;
    for (int64_t v = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); v <= n; v += warps) {
        const int64_t a = rp[v];
        if (v == n) {
            if (lane == 0 && a != m) atomicOr(err, kErrBadInput);
            continue;
        }
        const int64_t b = rp[v + 1];
        if (a < 0 || b < a || b > m || (v == 0 && a != 0)) {
            if (lane == 0) atomicOr(err, kErrBadInput);
            continue;
        }
        for (int64_t e = a + lane; e < b; e += 32) src[e] = static_cast<int32_t>(v);
    }
}

}  // namespace

bisim_status csr_sources(bisim_ctx* ctx, const int64_t* row_ptr, int32_t n, int64_t m, int32_t* src, cudaStream_t s) {
    cudaMemsetAsync(&ctx->dstate->error, 0, sizeof(unsigned), s);
    BISIM_SITE(site, "csr_sources");
    {
        Launch L(site, s, n, m, 8.0 * n + 4.0 * m);
        k_csr_sources<<<grid_for(static_cast<int64_t>(n + 1) * 32, 256), 256, 0, s>>>(row_ptr, n, m, src,
                                                                                     &ctx->dstate->error);
    }
    unsigned err = 0;
    cudaError_t e;
    cudaMemcpyAsync(&err, &ctx->dstate->error, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
    if ((e = cudaStreamSynchronize(s))) return cuda_error(ctx, e, "CSR sources");
    if (err & kErrBadInput) return set_error(ctx, BISIM_EINVAL, "row_ptr is not a prefix sum of [0, m]");
    return BISIM_OK;
}

bool edge_view_identity(const bisim_ctx* ctx) {
    return ctx->opt.direction == BISIM_DIR_FORWARD && ctx->nfilter == 0;
}

bool edge_view_reversal(const bisim_ctx* ctx) {
    return ctx->opt.direction == BISIM_DIR_BACKWARD && ctx->nfilter == 0;
}

bisim_status edge_view_setup(bisim_ctx* ctx, const bisim_options* opt, cudaStream_t s) {
    ctx->opt.label_filter = nullptr;                // caller memory: never kept
    if (opt == nullptr || opt->n_label_filter <= 0) return BISIM_OK;
    if (opt->label_filter == nullptr) return set_error(ctx, BISIM_EINVAL, "label_filter is NULL");
    std::vector<int32_t> f(static_cast<size_t>(opt->n_label_filter));
    cudaError_t e;
    if ((e = cudaMemcpyAsync(f.data(), opt->label_filter, sizeof(int32_t) * f.size(), cudaMemcpyDefault, s)) ||
        (e = cudaStreamSynchronize(s)))
        return cuda_error(ctx, e, "read label filter");
    std::sort(f.begin(), f.end());
    f.erase(std::unique(f.begin(), f.end()), f.end());
    if ((e = ctx_alloc(ctx, reinterpret_cast<void**>(&ctx->dfilter), sizeof(int32_t) * f.size(), s)))
        return cuda_error(ctx, e, "alloc label filter");
    ctx->nfilter = static_cast<int32_t>(f.size());
    if ((e = cudaMemcpyAsync(ctx->dfilter, f.data(), sizeof(int32_t) * f.size(), cudaMemcpyHostToDevice, s)) ||
        (e = cudaStreamSynchronize(s)))
        return cuda_error(ctx, e, "upload label filter");
    return BISIM_OK;
}

bisim_status edge_view_bad_label(bisim_ctx* ctx) {
    return set_error(ctx, BISIM_EINVAL, "the forward-backward direction needs edge labels in [-2^30, 2^30)");
}

bisim_status edge_view_coo(bisim_ctx* ctx, const int32_t* src, const int32_t* dst, const int32_t* lab, int64_t m,
                           const int64_t* eoff, int32_t G, cudaStream_t s, EdgeView* out) {
    *out = EdgeView{};
    cudaError_t e;
    const int32_t dir = ctx->opt.direction;
    BISIM_SITE(site, "edge_view");
    const auto alloc = [&](int64_t total) -> cudaError_t {
        const size_t eb = sizeof(int32_t) * static_cast<size_t>(std::max<int64_t>(total, 1));
        cudaError_t err = cudaMallocAsync(reinterpret_cast<void**>(&out->src), eb, s);
        if (err == cudaSuccess) err = cudaMallocAsync(reinterpret_cast<void**>(&out->dst), eb, s);
        if (err == cudaSuccess) err = cudaMallocAsync(reinterpret_cast<void**>(&out->lab), eb, s);
        if (err == cudaSuccess && eoff) err = cudaMallocAsync(reinterpret_cast<void**>(&out->eoff), sizeof(int64_t) * (G + 1), s);
        return err;
    };
    if (dir == BISIM_DIR_BOTH && ctx->nfilter == 0) {
        if ((e = alloc(2 * m))) {
            edge_view_free(out, s);
            return cuda_error(ctx, e, "alloc edge view");
        }
        const auto even = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 7u) == 0; };
        {
            Launch L(site, s, 0, m, 36.0 * m);
            k_view_both<<<grid_for((m + 1) / 2, 256), 256, 0, s>>>(src, dst, lab, m, even(src) && even(dst) && even(lab),
                                                                  out->src, out->dst, out->lab, ctx->dstate);
        }
        if (eoff) k_view_offsets<<<(G + 256) / 256, 256, 0, s>>>(nullptr, eoff, G, out->eoff);
        out->m = 2 * m;
        if ((e = cudaGetLastError())) return cuda_error(ctx, e, "edge view");
        return BISIM_OK;
    }
    const size_t scan_words = scan_temp_words(m + 1);
    int64_t* pos = nullptr;
    if ((e = cudaMallocAsync(reinterpret_cast<void**>(&pos), sizeof(int64_t) * (2 * (m + 1) + scan_words), s)))
        return cuda_error(ctx, e, "alloc edge view");
    int64_t* cnt = pos + (m + 1);
    int64_t* tmp = cnt + (m + 1);
    cudaMemsetAsync(&ctx->dstate->error, 0, sizeof(unsigned), s);
    {
        Launch L(site, s, 0, m, 24.0 * m);
        k_view_count<<<grid_for(m + 1, 256), 256, 0, s>>>(lab, m, ctx->dfilter, ctx->nfilter, dir, cnt,
                                                          &ctx->dstate->error);
    }
    exclusive_scan_i64(cnt, pos, m + 1, tmp, s);
    int64_t total = 0;
    unsigned err = 0;
    cudaMemcpyAsync(&total, pos + m, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
    cudaMemcpyAsync(&err, &ctx->dstate->error, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
    if ((e = cudaStreamSynchronize(s))) {
        cudaFreeAsync(pos, s);
        return cuda_error(ctx, e, "count edge view");
    }
    if (err & kErrBadInput) {
        cudaFreeAsync(pos, s);
        return edge_view_bad_label(ctx);
    }
    if ((e = alloc(total))) {
        cudaFreeAsync(pos, s);
        edge_view_free(out, s);
        return cuda_error(ctx, e, "alloc edge view");
    }
    {
        Launch L(site, s, 0, m, 24.0 * m + 12.0 * total);
        k_view_emit<<<grid_for(m, 256), 256, 0, s>>>(src, dst, lab, m, pos, dir, out->src, out->dst, out->lab);
        if (eoff) k_view_offsets<<<(G + 256) / 256, 256, 0, s>>>(pos, eoff, G, out->eoff);
    }
    out->m = total;
    cudaFreeAsync(pos, s);
    if ((e = cudaGetLastError())) return cuda_error(ctx, e, "edge view");
    return BISIM_OK;
}

void edge_view_free(EdgeView* v, cudaStream_t s) {
    if (v->src) cudaFreeAsync(v->src, s);
    if (v->dst) cudaFreeAsync(v->dst, s);
    if (v->lab) cudaFreeAsync(v->lab, s);
    if (v->eoff) cudaFreeAsync(v->eoff, s);
    *v = EdgeView{};
}

bisim_status edge_view_ops(bisim_ctx* ctx, const bisim_op* ops, int64_t n, cudaStream_t s, bisim_op** out,
                           int64_t* out_n) {
    *out = nullptr;
    *out_n = 0;
    cudaError_t e;
    const size_t scan_words = scan_temp_words(n + 1);
    int64_t* pos = nullptr;
    if ((e = cudaMallocAsync(reinterpret_cast<void**>(&pos), sizeof(int64_t) * (2 * (n + 1) + scan_words), s)))
        return cuda_error(ctx, e, "alloc op view");
    int64_t* cnt = pos + (n + 1);
    int64_t* tmp = cnt + (n + 1);
    const int32_t dir = ctx->opt.direction;
    cudaMemsetAsync(&ctx->dstate->error, 0, sizeof(unsigned), s);
    k_ops_count<<<grid_for(n + 1, 256), 256, 0, s>>>(ops, n, ctx->dfilter, ctx->nfilter, dir, cnt, &ctx->dstate->error);
    exclusive_scan_i64(cnt, pos, n + 1, tmp, s);
    int64_t total = 0;
    unsigned err = 0;
    cudaMemcpyAsync(&total, pos + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
    cudaMemcpyAsync(&err, &ctx->dstate->error, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
    if ((e = cudaStreamSynchronize(s))) {
        cudaFreeAsync(pos, s);
        return cuda_error(ctx, e, "count op view");
    }
    if (err & kErrBadInput) {
        cudaFreeAsync(pos, s);
        return edge_view_bad_label(ctx);
    }
    if ((e = cudaMallocAsync(reinterpret_cast<void**>(out), sizeof(bisim_op) * std::max<int64_t>(total, 1), s))) {
        cudaFreeAsync(pos, s);
        return cuda_error(ctx, e, "alloc op view");
    }
    k_ops_emit<<<grid_for(n, 256), 256, 0, s>>>(ops, n, pos, dir, *out);
    cudaFreeAsync(pos, s);
    if ((e = cudaGetLastError())) return cuda_error(ctx, e, "op view");
    *out_n = total;
    return BISIM_OK;
}

}  // namespace bisim
