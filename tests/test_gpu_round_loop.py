"""The cooperative round loop at the edges of what it takes: row lengths around
its groups, list lengths around a CTA and the grid, the epoch cycle of the table,
hash collisions that hand a round back to the host, and rows it leaves to the
kernels of the wide classes. Partitions and rounds equal the oracle's."""

import numpy as np
import pytest

import oracle
from test_gpu_parity import B, check  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def rows_graph(n, degree, seed, copies=3, n_labels=2):
    """n vertices of out-degree `degree` - 1, `degree` or `degree` + 1; groups of `copies` vertices share a row (in
    another order, one entry doubled), so that many pairs need the exact comparison."""
    rng = np.random.default_rng(seed)
    src, dst, lab = [], [], []
    for v0 in range(0, n, copies):
        d = max(0, degree + int(rng.integers(-1, 2)))
        t, l = rng.integers(0, n, d), rng.integers(0, n_labels, d)
        for v in range(v0, min(n, v0 + copies)):
            o = rng.permutation(d)
            if d > 1 and v % 2:
                o[0] = o[1]                                # a repeated entry in place of one: another set
            src.append(np.full(d, v)); dst.append(t[o]); lab.append(l[o])
    cat = lambda a: np.concatenate(a).astype(np.int32) if a else np.zeros(0, np.int32)  # noqa: E731
    return dict(n=n, src=cat(src), dst=cat(dst), elabel=cat(lab), vlabel=rng.integers(0, 2, n).astype(np.int32))


def with_hub(g, edges):
    """The graph with a row of `edges` more edges, whose vertex is alone in its block from round 1 on."""
    rng = np.random.default_rng(edges)
    more = dict(src=np.full(edges, 17), dst=rng.integers(0, g["n"], edges), elabel=2 + np.arange(edges))
    return dict(g, **{k: np.concatenate([g[k], more[k]]).astype(np.int32) for k in more})


def path_graph(lengths, marked=()):
    n = int(sum(lengths))
    ends = np.cumsum(lengths) - 1
    v = np.setdiff1d(np.arange(n), ends)
    vl = np.zeros(n, np.int32)
    vl[list(marked)] = 1
    return dict(n=n, src=v.astype(np.int32), dst=(v + 1).astype(np.int32), elabel=np.zeros(len(v), np.int32), vlabel=vl)


@pytest.mark.parametrize("n", [1, 33, 1024, 1025, 6000])
@pytest.mark.parametrize("degree", [1, 8, 16, 32])
def test_row_lengths_of_every_group(B, n, degree):
    check(B, rows_graph(n, degree, seed=n + degree), [1, 2, oracle.FIXPOINT])


@pytest.mark.parametrize("degree", [64, 200, 255])
def test_rows_of_the_warp_classes(B, degree):
    check(B, rows_graph(2100, degree, seed=degree), [2, oracle.FIXPOINT])


@pytest.mark.parametrize("k", [1, 2, 14, 15, 16, 31])
def test_rounds_around_the_epoch_cycle(B, k):
    check(B, path_graph([40] * 30 + [7, 1, 90], marked=(3, 600)), [k])


@pytest.mark.parametrize("bits", [3, 9, 16])
@pytest.mark.parametrize("n,degree", [(300, 3), (3000, 9), (3000, 40)])
def test_collisions_hand_the_round_back(B, bits, n, degree):
    check(B, rows_graph(n, degree, seed=bits), [1, 3, oracle.FIXPOINT], options=B.default_options(hash_bits=bits))


def test_collisions_in_a_late_round(B):
    # few blocks at first, so the narrow hash collides only rounds later
    g = path_graph([60] * 200, marked=(5, 4000, 7001))
    check(B, g, [oracle.FIXPOINT], options=B.default_options(hash_bits=13))


def test_a_popular_signature_over_many_ctas(B):
    # 200k vertices with one signature in round 1 (a hot table slot), dead vertices among them
    n = 200_000
    rng = np.random.default_rng(4)
    alive = np.ones(n, np.uint8)
    alive[rng.integers(100, n, 500)] = 0
    src = np.flatnonzero(alive[:-1] & (np.arange(n - 1) % 7 != 0)).astype(np.int32)
    g = dict(n=n, src=src, dst=rng.integers(0, 100, len(src)).astype(np.int32), elabel=np.zeros(len(src), np.int32),
             vlabel=np.zeros(n, np.int32))
    check(B, g, [1, oracle.FIXPOINT], alive=alive)


@pytest.mark.parametrize("wide", [257, 9000])
def test_wide_rows_that_stay_listed_leave_the_loop(B, wide):
    # twins with equal rows are never alone: a wide pair keeps every round in the kernels of its class
    rng = np.random.default_rng(wide)
    base = path_graph([30] * 500)
    n = base["n"]
    t = rng.integers(0, n, wide)
    src = np.concatenate([base["src"], np.full(wide, 2), np.full(wide, 32)]).astype(np.int32)
    dst = np.concatenate([base["dst"], t, t[::-1]]).astype(np.int32)
    g = dict(base, src=src, dst=dst, elabel=np.zeros(len(src), np.int32))
    check(B, g, [1, 5, oracle.FIXPOINT])


def test_wide_rows_that_become_alone_enter_the_loop(B):
    rng = np.random.default_rng(8)
    base = path_graph([30] * 500)
    n = base["n"]
    src = np.concatenate([base["src"], np.full(700, 2), np.full(10_000, 32)]).astype(np.int32)
    dst = np.concatenate([base["dst"], rng.integers(0, n, 10_700)]).astype(np.int32)
    g = dict(base, src=src, dst=dst, elabel=np.zeros(len(src), np.int32))
    check(B, g, [1, 2, 17, oracle.FIXPOINT])


def test_resident_context_alternates_routes(B):
    # the same context by the loop, host-driven, and again: nothing of one run leaks into the next
    g = path_graph([25] * 300, marked=(11,))
    dev = [__import__("torch").from_numpy(g[k]).cuda() for k in ("src", "dst", "elabel", "vlabel")]
    ctx = B.summarize_init_coo(g["n"], *dev)
    for k in (3, oracle.FIXPOINT, 0, 40, 1, oracle.FIXPOINT):
        rounds, blocks = B.bisim_iterate(ctx, k, 10_000)
        want, wr, _ = oracle.refine(g["n"], g["src"], g["dst"], g["elabel"], g["vlabel"], k, 10_000)
        assert np.array_equal(B.get_partition(ctx).cpu().numpy(), want) and rounds == wr
        assert blocks == len(np.unique(want))
    B.summarize_destroy(ctx)


def test_one_cta_with_a_warp_row_as_the_first_call():
    # in a process of its own: the kernel's attributes are set whatever graph comes first
    import subprocess
    import sys
    code = ("import torch; from paper_2111_12493_gb300 import bisim as B; i = lambda a: torch.tensor(a, dtype=torch.int32).cuda();"
            "c = B.summarize_init_coo(3, i([0] * 40 + [1]), i([k % 3 for k in range(40)] + [2]), i(list(range(40)) + [0]), i([0, 0, 0]));"
            "assert B.bisim_iterate(c, 1)[1] == 3; assert B.get_partition(c).tolist() == [0, 1, 2]")
    subprocess.run([sys.executable, "-c", code], check=True, timeout=300)


@pytest.mark.parametrize("hub", [0, 300])
@pytest.mark.parametrize("degree", [3, 20])
def test_rounds_go_on_without_a_loop_that_gave_up(B, degree, hub):
    """With one poll a barrier the CTAs give up while others are on their way; the rounds then run again from P_0 by
    the captured graph. The next call has the loop back."""
    import torch
    g = rows_graph(60_000, degree, seed=degree)
    if hub:
        g = with_hub(g, hub)
    want, rounds, _ = oracle.refine(g["n"], g["src"], g["dst"], g["elabel"], g["vlabel"], oracle.FIXPOINT, 20)
    t = {k: torch.from_numpy(g[k]).cuda() for k in ("src", "dst", "elabel", "vlabel")}
    with B.summarize_init_coo(g["n"], t["src"], t["dst"], t["elabel"], t["vlabel"]) as ctx:
        launches = []
        for polls in (0, 1, 0):
            B._lib.bisim_loop_polls(ctx.ptr, polls)
            before = B.bisim_launch_count()
            got = B.bisim_iterate(ctx, oracle.FIXPOINT, 20)
            launches.append(B.bisim_launch_count() - before)
            assert got == (rounds, len(np.unique(want)))
            assert np.array_equal(B.get_partition(ctx).cpu().numpy(), want)
        assert launches[1] > launches[0] == launches[2]


@pytest.mark.parametrize("bits", [2, 64])
@pytest.mark.parametrize("n,degree", [(25, 9), (26, 32), (800, 17), (20_000, 24), (20_000, 8)])
def test_pairs_of_the_single_class_kernels(B, n, degree, bits):
    """Equal and (with two bits of hash) unequal rows of 8 to 33 edges, compared eight lanes a pair in the kernels of
    host-driven rounds: lists shorter than a warp's pairs, and longer than all warps'."""
    check(B, rows_graph(n, degree, seed=n + degree), [1, 2],
          options=B.default_options(flags=B.FLAG_EAGER, hash_bits=bits))


@pytest.mark.parametrize("bits", [3, 64])
@pytest.mark.parametrize("hub", [300, 9000])
def test_one_round_of_every_class(B, hub, bits):
    """A single round beside wide rows ends without a list or a loop, also where the fixpoint's cap is 1, where the
    round changes nothing and where it meets collisions; what follows works on its partition."""
    import torch
    options = B.default_options(hash_bits=bits)
    g = with_hub(rows_graph(2000, 5, seed=hub), hub)
    check(B, g, [1], options=options)
    check(B, g, [oracle.FIXPOINT], cap=1, options=options)
    ring = dict(n=1000, src=np.arange(1000, dtype=np.int32), dst=np.roll(np.arange(1000, dtype=np.int32), 1),
                elabel=np.zeros(1000, np.int32), vlabel=np.zeros(1000, np.int32))
    ring["src"], ring["dst"] = np.append(ring["src"], np.full(hub, 17, np.int32)), np.append(ring["dst"], np.arange(hub, dtype=np.int32) % 1000)
    ring["elabel"] = np.zeros(len(ring["src"]), np.int32)
    check(B, ring, [1, oracle.FIXPOINT], cap=1, options=options)
    check(B, ring, [oracle.FIXPOINT], options=options)
    t = {k: torch.from_numpy(g[k]).cuda() for k in ("src", "dst", "elabel", "vlabel")}
    with B.summarize_init_coo(g["n"], t["src"], t["dst"], t["elabel"], t["vlabel"], options=options) as ctx:
        B.bisim_iterate(ctx, 1)
        want, _, _ = oracle.refine(g["n"], g["src"], g["dst"], g["elabel"], g["vlabel"], 1, 0)
        assert np.array_equal(B.get_block_sizes(ctx).cpu().numpy(), np.bincount(want, minlength=g["n"]))
        B.bisim_iterate(ctx, 3)
        want, _, _ = oracle.refine(g["n"], g["src"], g["dst"], g["elabel"], g["vlabel"], 3, 0)
        assert np.array_equal(B.get_partition(ctx).cpu().numpy(), want)


@pytest.mark.parametrize("bits", [2, 64])
@pytest.mark.parametrize("n,degree", [(40, 12), (1000, 33), (1000, 250), (30_000, 30), (9000, 90)])
def test_wide_pairs_are_shared_out(B, n, degree, bits):
    """Long rows of few values (two labels, two blocks): every entry is a pair with a wide row. Few of them to a CTA
    and several to a warp, equal and (with two bits of hash) unequal."""
    rng = np.random.default_rng(degree)
    g = dict(n=n, src=np.repeat(np.arange(n), degree).astype(np.int32),
             dst=rng.integers(0, n, n * degree).astype(np.int32),
             elabel=rng.integers(0, 2, n * degree).astype(np.int32), vlabel=rng.integers(0, 2, n).astype(np.int32))
    rare = rng.integers(0, n, n // 10)                      # rows that miss a pair
    g["elabel"][(rare[:, None] * degree + np.arange(degree)).ravel()] = 0
    check(B, g, [1, 2, oracle.FIXPOINT], options=B.default_options(hash_bits=bits))


def test_wide_pairs_do_not_wait_for_one_warp(B):
    """1,000 rows of 250 edges, all pairs (two labels) against none (many labels): 14 times the time when the warp
    that met a CTA's pairs compared them all."""
    import time

    import torch
    rng = np.random.default_rng(1)
    n, d = 1000, 250
    took = []
    for labels, blocks in ((2, 2), (1000, 200)):
        a = [np.repeat(np.arange(n), d), rng.integers(0, n, n * d), rng.integers(0, labels, n * d), rng.integers(0, blocks, n)]
        with B.summarize_init_coo(n, *(torch.from_numpy(x.astype(np.int32)).cuda() for x in a)) as ctx:
            best = 1.0
            for _ in range(30):
                t = time.perf_counter()
                B.bisim_iterate(ctx, 1)
                best = min(best, time.perf_counter() - t)
        took.append(best)
    assert took[0] < 4 * took[1], took


@pytest.mark.parametrize("n", [400_000, 400_001])
def test_first_round_on_both_sides_of_its_line(B, n):
    """Up to 400,000 rows above eight edges are the loop's from P_0 on; more have their first round in the kernels of
    the single classes."""
    rng = np.random.default_rng(n)
    d = 9
    g = dict(n=n, src=np.repeat(np.arange(n), d).astype(np.int32), dst=rng.integers(0, n, n * d).astype(np.int32),
             elabel=rng.integers(0, 2, n * d).astype(np.int32), vlabel=rng.integers(0, 2, n).astype(np.int32))
    check(B, g, [1, 2])


@pytest.mark.parametrize("bits", [6, 64])
@pytest.mark.parametrize("degree", [3, 14, 60])
@pytest.mark.parametrize("tails", [1, 40])
def test_rounds_that_keep_small_blocks(B, tails, degree, bits):
    """Triplets with equal rows stay blocks of three from the first rounds on, while paths beside them split one
    vertex each off a block for 30 rounds more; a wide row makes the loop start after a round of the single classes,
    where such rounds compare with the blocks first."""
    g = rows_graph(3000, degree, seed=degree + tails)
    n, length = g["n"], 30
    v = np.arange(tails * length)
    v = v[v % length != length - 1] + n
    path = dict(src=v, dst=v + 1, elabel=np.zeros(len(v)))
    g = dict(n=n + tails * length, vlabel=np.append(g["vlabel"], np.zeros(tails * length, np.int32)),
             **{k: np.concatenate([g[k], path[k]]).astype(np.int32) for k in path})
    check(B, with_hub(g, 300), [2, 5, 29, oracle.FIXPOINT], options=B.default_options(hash_bits=bits))


@pytest.mark.parametrize("bits", [10, 64])
def test_rounds_that_keep_large_blocks(B, bits):
    """20 paths of 11,000 vertices: 20 entries of a long list leave the large block in every round; a wide row makes
    the loop start after a round of the single classes, where such rounds compare with the blocks first."""
    g = with_hub(path_graph([11_000] * 20, marked=(7, 30_000)), 300)
    check(B, g, [3, 24], options=B.default_options(hash_bits=bits))
    # from P_0 on beside as many vertices without edges
    g = path_graph([11_000] * 20 + [1] * 80_000, marked=(7, 30_000, 250_000))
    check(B, g, [3, 24], options=B.default_options(hash_bits=bits))
