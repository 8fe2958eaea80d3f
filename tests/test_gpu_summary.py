"""The summary graph and its count payload (get_summary_edges, get_block_sizes)
against the oracle.

Section 2.6 defines the summary graph (one vertex per block, an l-labelled
edge between the blocks of the endpoints of every l-edge, parallel edges of
one label collapsed); Section 3.1 the count payload (vertices per block).
Both sides compute them from the same partition, which is itself checked
against the oracle, so the triples and counts must match exactly.
"""

import numpy as np
import pytest

import oracle
from paper_2111_12493_gb300 import graphgen
from refcheck import edges_to_arrays, parse_golden

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2111_12493_gb300 import bisim
    return bisim


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _gpu_summary(B, ctx):
    s, l, t = (x.cpu().numpy() for x in B.get_summary_edges(ctx))
    return list(zip(s.tolist(), l.tolist(), t.tolist()))


def _check(B, ctx, src, dst, elabel, P):
    got_P = B.get_partition(ctx).cpu().numpy()
    assert np.array_equal(got_P, P)
    assert _gpu_summary(B, ctx) == oracle.summary_edges(src, dst, elabel, P)
    assert B.get_block_sizes(ctx).cpu().numpy().tolist() == oracle.block_sizes(P).tolist()


def test_summary_of_the_worked_example(B):
    gf = parse_golden("fig3_worked_example.txt")
    s, d, l = edges_to_arrays(gf["edges"])
    vl = np.array(gf["vlabel"]["L"], np.int32)
    ctx = B.summarize_init_coo(gf["n"], _dev(s), _dev(d), _dev(l), _dev(vl))
    B.bisim_iterate(ctx, 2, 0)
    assert _gpu_summary(B, ctx) == gf["summary"][2]
    assert B.get_block_sizes(ctx).cpu().numpy().tolist() == gf["sizes"][2].tolist()
    B.summarize_destroy(ctx)


@pytest.mark.parametrize("k", [0, 1, 2, -1])
def test_uniform_graph_every_k(B, k):
    g = graphgen.uniform_graph(seed=1)
    # signed labels exercise the label order of the output
    lab = (g["elabel"] - 4).astype(np.int32)
    ctx = B.summarize_init_coo(g["n"], _dev(g["src"]), _dev(g["dst"]), _dev(lab), _dev(g["vlabel"]))
    B.bisim_iterate(ctx, k, 10)
    P, _, _ = oracle.refine(g["n"], g["src"], g["dst"], lab, g["vlabel"], k, 10)
    _check(B, ctx, g["src"], g["dst"], lab, P)
    B.summarize_destroy(ctx)


def test_powerlaw_graph_with_hubs_and_dead_vertices(B):
    g = graphgen.powerlaw_graph(n=100_000, m=1_000_000, dmax=50_000, n_elabels=40, n_vlabels=6, seed=31)
    alive = (np.random.default_rng(5).random(g["n"]) > 0.05).astype(np.uint8)
    keep = alive[g["src"]].astype(bool) & alive[g["dst"]].astype(bool)
    src, dst, lab = g["src"][keep], g["dst"][keep], g["elabel"][keep]
    ctx = B.summarize_init_coo(g["n"], _dev(src), _dev(dst), _dev(lab), _dev(g["vlabel"]), alive=_dev(alive))
    for k in (1, -1):
        B.bisim_iterate(ctx, k, 10)
        P, _, _ = oracle.refine(g["n"], src, dst, lab, g["vlabel"], k, 10, alive=alive)
        _check(B, ctx, src, dst, lab, P)
    B.summarize_destroy(ctx)


def test_batched_graphs_report_union_ids(B):
    b = graphgen.batched_graphs(n_graphs=40, nmin=20, nmax=3000, seed=12)
    ctx = B.summarize_init_batched(*(_dev(b[x]) for x in ("vertex_offsets", "edge_offsets", "src_local",
                                                           "dst_local", "elabel", "vlabel")))
    B.bisim_iterate(ctx, 3, 0)
    u = graphgen.batched_union(b)
    P, _, _ = oracle.refine(u["n"], u["src"], u["dst"], u["elabel"], u["vlabel"], 3, graph=u["graph"])
    assert _gpu_summary(B, ctx) == oracle.summary_edges(u["src"], u["dst"], u["elabel"], P)
    assert B.get_block_sizes(ctx).cpu().numpy().tolist() == oracle.block_sizes(P).tolist()
    B.summarize_destroy(ctx)


def test_summary_follows_update_batches(B):
    from test_gpu_updates import random_batch
    rng = np.random.default_rng(9)
    g = graphgen.uniform_graph(n=400, m=1600, n_elabels=3, n_vlabels=3, seed=41)
    state = dict(n=g["n"], alive=np.ones(g["n"], np.uint8), vlabel=g["vlabel"].copy(), src=g["src"],
                 dst=g["dst"], elabel=g["elabel"])
    ctx = B.summarize_init_coo(g["n"], _dev(g["src"]), _dev(g["dst"]), _dev(g["elabel"]), _dev(g["vlabel"]),
                               options=B.default_options(k_incremental=2))
    B.apply_updates(ctx, _dev(np.zeros((0, 4), np.int32)))
    for _ in range(6):
        ops = random_batch(rng, state, int(rng.integers(5, 80)))
        try:
            new_state = oracle.apply_ops(state, ops)
        except oracle.UpdateRejected:
            continue
        B.apply_updates(ctx, _dev(ops))
        state = new_state
        P, _, _ = oracle.refine(state["n"], state["src"], state["dst"], state["elabel"], state["vlabel"], 2,
                                alive=state["alive"])
        _check(B, ctx, state["src"], state["dst"], state["elabel"], P)
    B.summarize_destroy(ctx)


def test_host_outputs_and_capacity(B):
    import ctypes
    import torch
    g = graphgen.uniform_graph(n=2000, m=9000, n_elabels=3, n_vlabels=2, seed=13)
    ctx = B.summarize_init_coo(g["n"], _dev(g["src"]), _dev(g["dst"]), _dev(g["elabel"]), _dev(g["vlabel"]))
    B.bisim_iterate(ctx, 1, 0)
    P, _, _ = oracle.refine(g["n"], g["src"], g["dst"], g["elabel"], g["vlabel"], 1)
    want = oracle.summary_edges(g["src"], g["dst"], g["elabel"], P)
    sizes = torch.empty(g["n"], dtype=torch.int32).pin_memory()
    B.get_block_sizes(ctx, out=sizes)
    assert sizes.numpy().tolist() == oracle.block_sizes(P).tolist()
    # capacity 0 sizes the output; a short capacity writes a prefix; host arrays work
    count = ctypes.c_int64()
    assert B._lib.get_summary_edges(ctx.ptr, None, None, None, 0, ctypes.byref(count), None) == 0
    assert count.value == len(want)
    cap = len(want) // 2
    outs = [torch.empty(cap, dtype=torch.int32).pin_memory() for _ in range(3)]
    assert B._lib.get_summary_edges(ctx.ptr, *[ctypes.c_void_p(o.data_ptr()) for o in outs], cap,
                                    ctypes.byref(count), None) == 0
    assert count.value == len(want)
    assert list(zip(*(o.numpy().tolist() for o in outs))) == want[:cap]
    B.summarize_destroy(ctx)


@pytest.mark.parametrize("direction", ["DIR_FORWARD", "DIR_BOTH", "DIR_BACKWARD"])
@pytest.mark.parametrize("k", [0, 1])
def test_segments_of_every_length(B, direction, k):
    # rows at the edges of the ways a block's edges are sorted (a packed warp, a
    # warp's and a CTA's shared memory, the radix sort), repeated edges among
    # them; at k = 0 whole label classes form segments
    rng = np.random.default_rng(17)
    lengths = [0, 1, 2, 7, 8, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 129, 255, 256, 257, 511, 513, 2047, 2048, 2049, 9000]
    lengths += [int(x) for x in rng.integers(0, 40, 300)] + [5000, 2500]
    n = len(lengths)
    src = np.repeat(np.arange(n), lengths).astype(np.int32)
    dst = rng.integers(0, n, len(src)).astype(np.int32)
    top = 2**30 - 1 if direction == "DIR_BOTH" else 2**31 - 1
    lab = rng.choice(np.array([-top - 1, -3, 0, 1, 2, 700, top], np.int64), len(src)).astype(np.int32)
    vl = (np.arange(n) % 9).astype(np.int32)
    o = rng.permutation(len(src))
    src, dst, lab = src[o], dst[o], lab[o]
    ctx = B.summarize_init_coo(n, _dev(src), _dev(dst), _dev(lab), _dev(vl),
                               options=B.default_options(direction=getattr(B, direction)))
    B.bisim_iterate(ctx, k, 0)
    P = B.get_partition(ctx).cpu().numpy()
    assert _gpu_summary(B, ctx) == oracle.summary_edges(src, dst, lab, P)
    B.summarize_destroy(ctx)


def test_big_segments_whose_triples_exceed_a_word(B):
    # 2^22 + 3 vertices (23 bits) and labels over the whole range (32 bits) with
    # more than 512 long rows (10 bits): target, label and segment are sorted apart
    import torch
    n, rows, length = (1 << 22) + 3, 600, 2100
    rng = np.random.default_rng(23)
    src = np.repeat(rng.choice(n, rows, replace=False), length).astype(np.int32)
    dst = rng.integers(0, n, len(src)).astype(np.int32)
    lab = rng.choice(np.array([-2**31, -5, 0, 2**31 - 1], np.int64), len(src)).astype(np.int32)
    dst[1::2], lab[1::2] = dst[::2], lab[::2]              # every second edge repeats the one before it
    vl = np.arange(n, dtype=np.int32)                      # every vertex a block of its own
    ctx = B.summarize_init_coo(n, _dev(src), _dev(dst), _dev(lab), _dev(vl))
    got = np.stack([x.cpu().numpy() for x in B.get_summary_edges(ctx)])
    want = np.unique(np.stack([src, lab, dst], 1).astype(np.int64), axis=0).T
    assert np.array_equal(got, want)
    B.summarize_destroy(ctx)


@pytest.mark.parametrize("direction", [0, 2])
@pytest.mark.parametrize("m", [68_000, 72_000])
def test_few_edges_between_many_vertices(B, m, direction):
    """On both sides of the line below which the triples are sorted, not the blocks' segments (0.7 edges for every
    vertex above 1.25 million); forward-backward contexts hold every edge twice."""
    rng = np.random.default_rng(m)
    n = 1_350_000
    m //= 2 if direction == 2 else 1
    src, dst = (rng.integers(0, n, m).astype(np.int32) for _ in range(2))
    src[: m // 4] = 5                                       # one long row, and repeated triples
    lab, vl = rng.integers(-3, 3, m).astype(np.int32), rng.integers(0, 3, n).astype(np.int32)
    alive = np.ones(n, np.uint8)
    alive[rng.integers(0, n, 1000)] = 0
    alive[5] = 1
    keep = alive[src].astype(bool) & alive[dst].astype(bool)
    src, dst, lab = src[keep], dst[keep], lab[keep]
    with B.summarize_init_coo(n, _dev(src), _dev(dst), _dev(lab), _dev(vl), alive=_dev(alive),
                              options=B.default_options(direction=direction)) as ctx:
        B.bisim_iterate(ctx, 1)
        P = B.get_partition(ctx).cpu().numpy()
        if direction == 0:
            want, _, _ = oracle.refine(n, src, dst, lab, vl, 1, 0, alive=alive)
            assert np.array_equal(P, want)
        assert _gpu_summary(B, ctx) == oracle.summary_edges(src, dst, lab, P)
