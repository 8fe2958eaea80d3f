"""The allocation-free round (bisim_refine_round_noalloc).

Some callers cannot allocate device memory: a plugin inside another runtime
that owns the device heap, or a loop that reserves every buffer up front
because an allocation may synchronise the device or fail under fragmentation.
For them the library runs one refinement round with its scratch in a fixed
array compiled into the library. Its output must equal what the regular entry
point (bisim_iterate) computes and what the CPU oracle computes: two calls in
a row, raw vertex labels -> P_1 -> P_2, compared bit for bit. The array keeps
the last call's contents, so calls are also checked after a larger call has
left it dirty, and at the exact size limits. Every rejection must happen
before any kernel touches the caller's arrays.

This file is collected last so that a stop-at-first-failure run has run every
other test before it.
"""

import numpy as np
import pytest

import oracle
from paper_2111_12493_gb300 import graphgen

pytestmark = pytest.mark.gpu

MAX_N = 65536
MAX_M = 1 << 20
MAX_DEG = 8192


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2111_12493_gb300 import bisim
    return bisim


def _csr(g):
    order = np.argsort(g["src"], kind="stable")
    rp = np.zeros(g["n"] + 1, np.int64)
    rp[1:] = np.cumsum(np.bincount(g["src"], minlength=g["n"]))
    return rp, g["dst"][order].astype(np.int32), g["elabel"][order].astype(np.int32)


def _dev(*arrays):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


def _two_rounds(B, g):
    """P_1 and P_2 from the allocation-free round, with their block counts."""
    import torch
    rp, col, lab, vl = _dev(*_csr(g), g["vlabel"])
    p1 = torch.empty(g["n"], dtype=torch.int32, device="cuda")
    p2 = torch.empty(g["n"], dtype=torch.int32, device="cuda")
    b1 = B.bisim_refine_round_noalloc(g["n"], rp, col, lab, vl, p1)
    b2 = B.bisim_refine_round_noalloc(g["n"], rp, col, lab, p1, p2)
    return (p1.cpu().numpy(), b1), (p2.cpu().numpy(), b2)


def _oracle_rounds(g):
    P0 = g["vlabel"]          # any labelling of the label partition: the round only compares ids
    P1 = oracle.refine_round(g["n"], g["src"], g["dst"], g["elabel"], g["vlabel"], P0)
    P2 = oracle.refine_round(g["n"], g["src"], g["dst"], g["elabel"], g["vlabel"], P1)
    return P1, P2


def _check_against_oracle(B, g):
    (p1, b1), (p2, b2) = _two_rounds(B, g)
    w1, w2 = _oracle_rounds(g)
    assert np.array_equal(p1, w1) and b1 == len(np.unique(w1))
    assert np.array_equal(p2, w2) and b2 == len(np.unique(w2))


@pytest.mark.parametrize("seed", [0, 1])
def test_two_noalloc_rounds_match_bisim_iterate_and_the_oracle(B, seed):
    g = graphgen.powerlaw_graph(n=60_000, m=600_000, dmax=6_000, n_elabels=40, n_vlabels=8, seed=100 + seed)
    rp, col, lab, vl = _dev(*_csr(g), g["vlabel"])
    expected = []
    ctx = B.summarize_init(g["n"], rp, col, lab, vl)
    for k in (1, 2):
        _, blocks = B.bisim_iterate(ctx, k, 10)
        expected.append((B.get_partition(ctx).cpu().numpy(), blocks))
    B.summarize_destroy(ctx)
    (p1, b1), (p2, b2) = _two_rounds(B, g)
    assert np.array_equal(p1, expected[0][0]) and b1 == expected[0][1]
    assert np.array_equal(p2, expected[1][0]) and b2 == expected[1][1]
    w1, w2 = _oracle_rounds(g)
    assert np.array_equal(p1, w1) and np.array_equal(p2, w2)


def test_noalloc_at_the_exact_size_limits(B):
    # n = 65536 fills the whole 2n-slot table; m = 2^20 the whole list array
    g = graphgen.powerlaw_graph(n=MAX_N, m=MAX_M, dmax=MAX_DEG, n_elabels=30, n_vlabels=6, seed=140)
    assert g["n"] == MAX_N and len(g["src"]) == MAX_M
    assert np.bincount(g["src"], minlength=g["n"]).max() <= MAX_DEG
    (p1, b1), _ = _two_rounds(B, g)
    rp, col, lab, vl = _dev(*_csr(g), g["vlabel"])
    ctx = B.summarize_init(g["n"], rp, col, lab, vl)
    _, blocks = B.bisim_iterate(ctx, 1, 10)
    assert np.array_equal(p1, B.get_partition(ctx).cpu().numpy()) and b1 == blocks
    B.summarize_destroy(ctx)
    _check_against_oracle(B, g)


def test_noalloc_after_a_larger_call_left_the_array_dirty(B):
    big = graphgen.powerlaw_graph(n=MAX_N, m=500_000, dmax=4_000, n_elabels=20, n_vlabels=5, seed=141)
    small = graphgen.uniform_graph(n=1_000, m=5_000, n_elabels=4, n_vlabels=3, seed=142)
    _check_against_oracle(B, big)
    _check_against_oracle(B, small)
    _check_against_oracle(B, big)


@pytest.mark.parametrize("wide", [False, True])
def test_noalloc_rows_of_every_width(B, wide):
    # rows around the widths at which a lane, a warp and a CTA take over, each twice
    # with its entries repeated and in another order, and once with one entry changed;
    # `wide`: a mean row beyond a lane's, which spreads the vertices over more warps
    rng = np.random.default_rng(150)
    widths = [0, 1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 128, 255, 256, 257, 500, 1024, 4000, 8190, 8192]
    leaves = 200 if wide else 25_000
    src, dst, lab = [], [], []
    n = leaves
    for w in widths:
        t, l = rng.integers(0, leaves, w), rng.integers(0, 50, w)
        if w >= 64:                                   # some of the entries are the same
            t[: w // 3] = t[w // 2]
            l[: w // 3] = l[w // 2]
        for copy in range(3):
            p = rng.permutation(w)
            t2, l2 = t[p].copy(), l[p].copy()
            if copy == 2 and w:
                l2[rng.integers(0, w)] += 50
            src.append(np.full(w, n)); dst.append(t2); lab.append(l2)
            n += 1
    g = dict(n=n, src=np.concatenate(src).astype(np.int32), dst=np.concatenate(dst).astype(np.int32),
             elabel=np.concatenate(lab).astype(np.int32),
             vlabel=np.concatenate([rng.integers(0, 40, leaves), np.zeros(n - leaves)]).astype(np.int32))
    _check_against_oracle(B, g)


def test_noalloc_resolves_colliding_hashes(B):
    # labels of vertices without edges whose hashes share the table's fingerprint (the
    # top 28 bits) and home slot (the low 17): the table merges them, and the
    # confirmation has to take them apart again
    def mix(z):
        z ^= z >> np.uint64(30)
        z *= np.uint64(0xbf58476d1ce4e5b9)
        z ^= z >> np.uint64(27)
        z *= np.uint64(0x94d049bb133111eb)
        z ^= z >> np.uint64(31)
        return z
    h = mix(mix((np.arange(1 << 24, dtype=np.uint64) << np.uint64(32)) ^ np.uint64(0x13198a2e03707344)))
    key = (h >> np.uint64(36) << np.uint64(17)) | (h & np.uint64(MAX_N * 2 - 1))
    order = np.sort(key)
    twice = order[1:][order[1:] == order[:-1]]
    labels = np.flatnonzero(np.isin(key, twice))
    assert len(twice) > 1 and len(labels) >= 2 * len(twice)
    vl = np.tile(labels, 6).astype(np.int32)[np.random.default_rng(7).permutation(6 * len(labels))]
    none = np.zeros(0, np.int32)
    _check_against_oracle(B, dict(n=len(vl), src=none, dst=none, elabel=none, vlabel=vl))


def _rejected(B, *args, match=None):
    with pytest.raises(B.BisimError) as ei:
        B.bisim_refine_round_noalloc(*args)
    assert ei.value.status == 1, ei.value
    if match:
        assert match in ei.value.message, ei.value.message


def test_noalloc_rejects_oversized_graphs(B):
    import torch
    n = MAX_N + 1
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    col = torch.zeros(0, dtype=torch.int32, device="cuda")
    lab = torch.zeros(0, dtype=torch.int32, device="cuda")
    pin = torch.zeros(n, dtype=torch.int32, device="cuda")
    out = torch.empty(n, dtype=torch.int32, device="cuda")
    _rejected(B, n, rp, col, lab, pin, out, match="limit")
    # one edge over the limit
    n = 100
    m = MAX_M + 1
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = m
    col = torch.zeros(m, dtype=torch.int32, device="cuda")
    lab = torch.zeros(m, dtype=torch.int32, device="cuda")
    _rejected(B, n, rp, col, lab, torch.zeros(n, dtype=torch.int32, device="cuda"),
              torch.empty(n, dtype=torch.int32, device="cuda"), match="limit")


def test_noalloc_rejects_malformed_input_and_leaves_the_output_alone(B):
    import torch
    g = graphgen.uniform_graph(n=500, m=3_000, n_elabels=4, n_vlabels=3, seed=143)
    rp, col, lab = _csr(g)
    n = g["n"]
    vl = torch.from_numpy(g["vlabel"]).cuda()
    sentinel = torch.full((n,), 7, dtype=torch.int32, device="cuda")

    def run(rp_, col_, lab_, bin_=vl, bout=sentinel, n_=n):
        _rejected(B, n_, rp_, col_, lab_, bin_, bout)
        assert bool((sentinel == 7).all())

    d_rp, d_col, d_lab = _dev(rp, col, lab)
    # row_ptr not a prefix sum of [0, m]: decreasing, wrong end, wrong start
    bad = rp.copy(); bad[10], bad[11] = bad[11], bad[10] - 1
    run(*_dev(bad), d_col, d_lab)
    bad = rp.copy(); bad[-1] -= 1
    run(*_dev(bad), d_col, d_lab)
    bad = rp.copy(); bad[0] = 1
    run(*_dev(bad), d_col, d_lab)
    # a target out of range, and a negative one
    for v in (n, -1):
        bad = col.copy(); bad[17] = v
        run(d_rp, *_dev(bad), d_lab)
    # block_in and block_out the same array
    same = vl.clone()
    _rejected(B, n, d_rp, d_col, d_lab, same, same, match="differ")
    # host arrays (pinned and pageable)
    run(d_rp, d_col, d_lab, bin_=vl.cpu().pin_memory())
    run(d_rp.cpu(), d_col, d_lab)
    _rejected(B, n, d_rp, d_col, d_lab, vl, torch.empty(n, dtype=torch.int32).pin_memory())
    # one out-degree above the limit
    m = MAX_DEG + 1
    rp2 = np.zeros(11, np.int64)
    rp2[1:] = m
    col2 = np.full(m, 3, np.int32)
    lab2 = np.zeros(m, np.int32)
    out2 = torch.full((10,), 7, dtype=torch.int32, device="cuda")
    _rejected(B, 10, *_dev(rp2, col2, lab2), torch.zeros(10, dtype=torch.int32, device="cuda"), out2,
              match="8192")
    assert bool((out2 == 7).all())


def test_noalloc_rejects_memory_of_another_device(B):
    import torch
    if torch.cuda.device_count() < 2:
        pytest.skip("needs two visible GPUs")
    g = graphgen.uniform_graph(n=200, m=1_000, n_elabels=4, n_vlabels=3, seed=144)
    rp, col, lab = _csr(g)
    with torch.cuda.device(0):
        d_rp, d_col, d_lab = (torch.from_numpy(a).to("cuda:1") for a in (rp, col, lab))
        vl = torch.from_numpy(g["vlabel"]).to("cuda:0")
        out = torch.empty(g["n"], dtype=torch.int32, device="cuda:0")
        _rejected(B, g["n"], d_rp, d_col, d_lab, vl, out, match="current device")


@pytest.mark.parametrize("n,wide,degree", [(153, 4, 300), (10_000, 20, 8000), (19_457, 300, 600), (14_441, 300, 600), (60_000, 800, 1000)])
def test_noalloc_wide_rows_side_by_side(B, n, wide, degree):
    """Rows that take a whole CTA, at the first ids and spread over all: the same partitions as the oracle's, and
    side by side they are not one CTA's work (up to eight times the time of the spread ones, when they were)."""
    import time

    import torch
    rng = np.random.default_rng(n)
    took = []
    for ids in (np.arange(wide), np.sort(rng.choice(n, wide, replace=False))):
        d = np.full(n, 2)
        d[ids] = degree
        m = int(d.sum())
        g = dict(n=n, src=np.repeat(np.arange(n), d).astype(np.int32), dst=rng.integers(0, n, m).astype(np.int32),
                 elabel=rng.integers(0, 3, m).astype(np.int32), vlabel=rng.integers(0, 2, n).astype(np.int32))
        g["dst"][degree * 2:degree * 3] = g["dst"][degree:degree * 2]      # two of the first rows alike
        g["elabel"][degree * 2:degree * 3] = g["elabel"][degree:degree * 2]
        _check_against_oracle(B, g)
        rp, col, lab, vl = _dev(*_csr(g), g["vlabel"])
        out = torch.empty(n, dtype=torch.int32, device="cuda")
        best = 1.0
        for _ in range(30):
            t = time.perf_counter()
            B.bisim_refine_round_noalloc(n, rp, col, lab, vl, out)
            best = min(best, time.perf_counter() - t)
        took.append(best)
    assert took[0] < 2.5 * took[1], took
