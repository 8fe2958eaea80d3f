"""Timed cases of the k-bisimulation library, each run through its public calls.

A case is a dict of plain values. `kind` says which calls a pass makes:

  summarize   one-off request on a graph in device memory: summarize_init (CSR)
              or summarize_init_coo, bisim_iterate, get_partition,
              summarize_destroy
  refine      bisim_iterate and get_partition on a context that stays resident
  batched     summarize_init_batched over many small graphs, bisim_iterate,
              get_partition, summarize_destroy
  updates     a batch of update operations from pinned host memory on a
              resident context, the new partition read, then the batch that
              takes it back and the partition again (so a state can be passed
              over any number of times)
  summary     get_summary_edges and get_block_sizes of a resident context's
              partition
  round       one allocation-free refinement round over caller-owned arrays

Graphs are drawn on the GPU with the distributions of
paper_2111_12493_gb300.graphgen (uniform; power-law out-degrees with copy-model
targets and Zipf labels; directed paths with extra edges; batches of small
power-law graphs). All results are integers and must agree exactly.
"""

import math

import torch

from paper_2111_12493_gb300 import bisim

FIX = bisim.FIXPOINT
DIRECTIONS = {"forward": bisim.DIR_FORWARD, "backward": bisim.DIR_BACKWARD, "both": bisim.DIR_BOTH}


def listed():
    return [
        # one refinement round inside a host that may not allocate: the smallest call, all latency
        dict(name="round_10k", kind="round", graph="uniform", n=10_000, m=50_000),
        # a small graph summarized once, start to end: context set-up, launches and synchronisations
        dict(name="summarize_uniform_1k", kind="summarize", graph="uniform", n=1_000, m=5_000, k=2, input="coo",
             order="sorted", direction="forward", labels=0),
        # the 10k / 50k configuration refined again and again on a resident context
        dict(name="refine_uniform_10k", kind="refine", graph="uniform", n=10_000, m=50_000, k=2, direction="forward"),
        # a serving request of ordinary size, from a CSR
        dict(name="summarize_csr_400k", kind="summarize", graph="powerlaw", n=400_000, m=4_000_000, k=FIX, input="csr",
             order="sorted", direction="forward", labels=0),
        # forward-backward signatures over an edge list in no order, odd sizes
        dict(name="summarize_both_1M", kind="summarize", graph="powerlaw", n=1_000_003, m=8_000_021, k=FIX, input="coo",
             order="shuffled", direction="both", labels=0),
        # the headline workload: 10M vertices, 100M edges, to the fixpoint
        dict(name="summarize_powerlaw_10M", kind="summarize", graph="powerlaw", n=10_000_000, m=100_000_000, k=FIX,
             input="coo", order="sorted", direction="forward", labels=0),
        # k-chaining on a resident graph: paths with random extra edges
        dict(name="refine_chain_1M", kind="refine", graph="chain", n=1_000_000, m=2_999_000, paths=1000, k=FIX,
             direction="forward"),
        # long k-chaining: pure paths, hundreds of rounds with every vertex listed
        dict(name="refine_paths_300k", kind="refine", graph="chain", n=300_000, m=299_500, paths=500, k=FIX,
             direction="forward"),
        # many independent small graphs in one call
        dict(name="batched_512", kind="batched", graphs=512, nmin=100, nmax=100_000, k=3),
        # serving a graph under small update batches: latency
        dict(name="updates_1k", kind="updates", graph="powerlaw", n=5_000_000, m=50_000_000, ops=1_000),
        # large update batches: throughput
        dict(name="updates_100k", kind="updates", graph="powerlaw", n=1_000_000, m=10_000_000, ops=100_000),
        # the summary graph and its payload, the product handed to the next program
        dict(name="summary_1M", kind="summary", graph="powerlaw", n=1_000_000, m=10_000_000, k=2, direction="forward"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["summarize", "summarize", "refine", "refine", "batched", "updates", "updates", "summary", "round"])
    if kind == "round":
        n = _log(rng, 500, 60_000)
        return dict(kind=kind, graph="uniform", n=n, m=n * rng.randint(2, 12) + rng.randint(0, 99))
    if kind == "batched":
        return dict(kind=kind, graphs=_log(rng, 8, 1024), nmin=rng.randint(20, 400), nmax=_log(rng, 1_000, 100_000),
                    k=rng.choice([1, 2, 3, FIX]))
    if kind == "updates":
        n = _log(rng, 20_000, 5_000_000)
        return dict(kind=kind, graph="powerlaw", n=n, m=10 * n + rng.randint(0, 99), ops=min(n // 10, _log(rng, 10, 300_000)))
    graph = rng.choice(["uniform", "powerlaw", "powerlaw", "chain"])
    n = _log(rng, 1_000, 5_000_000)
    c = dict(kind=kind, graph=graph, n=n, m=n * rng.randint(2, 10) + rng.randint(0, 99), k=rng.choice([1, 2, 3, FIX, FIX]),
             direction="forward")
    if graph == "chain":
        thin = rng.random() < 0.5                          # few extra edges or none: as many rounds as the paths are long
        if thin:
            c["n"] = n = min(n, _log(rng, 1_000, 300_000))
        c["paths"] = max(1, n // rng.randint(5, 400))
        c["m"] = n - c["paths"] + (rng.choice([0, n // 100]) if thin else 2 * n)
    if kind == "summarize":
        c.update(input=rng.choice(["coo", "csr"]), order=rng.choice(["sorted", "sorted", "shuffled"]), labels=0)
        if c["m"] <= 20_000_000:
            c["direction"] = rng.choice(["forward", "backward", "both"])
            c["labels"] = rng.choice([0, 0, 3])            # 3: only edges with one of the three first labels
    return c


# ----------------------------------------------------------------------------- graphs


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(0x5EED + 7919 * int(seed))
    return g


def _ints(g, hi, count):
    return torch.randint(0, int(hi), (int(count),), generator=g, device="cuda", dtype=torch.int64)


def _unit(g, count):
    return torch.rand(int(count), generator=g, device="cuda", dtype=torch.float64)


def _zipf(g, count, values, s):
    w = torch.arange(1, values + 1, device="cuda", dtype=torch.float64).pow(-s)
    cdf = torch.cumsum(w, 0)
    cdf /= cdf[-1].clone()
    out = torch.searchsorted(cdf, _unit(g, count), right=True)
    return out.clamp_(max=values - 1).to(torch.int32)


def _pareto(g, n, exponent, dmax):
    """Floored Pareto on [1, dmax]; dmax a number or a tensor."""
    a = exponent - 1.0
    dmax = torch.as_tensor(dmax, device="cuda", dtype=torch.float64)
    tail = dmax.pow(-a)
    return torch.minimum((1.0 - _unit(g, n) * (1.0 - tail)).pow(-1.0 / a).floor(), dmax).clamp_(min=1.0)


def _degrees(g, n, m, exponent=2.1, dmax=1_000_000):
    """Power-law out-degrees with sum m."""
    d = _pareto(g, n, exponent, min(dmax, m))
    d = d * (m / d.sum())
    fl = d.floor()
    d = (fl + (_unit(g, n) < d - fl)).to(torch.int64)
    diff = m - int(d.sum())
    while diff != 0:
        at = _ints(g, n, abs(diff))
        if diff > 0:
            d.index_add_(0, at, torch.ones_like(at))
        else:
            at = at.unique()
            d[at] -= (d[at] > 0).to(torch.int64)
        diff = m - int(d.sum())
    return d


def _copied_targets(g, n, m, p_copy=0.8):
    """Targets of m edges in order: copied from a uniform earlier edge, or uniform."""
    j = torch.arange(m, device="cuda")
    copy = _unit(g, m) < p_copy
    if m > 0:
        copy[0] = False
    parent = torch.where(copy, (_unit(g, m) * j).to(torch.int64), j)
    del copy, j
    while True:
        up = parent[parent]
        if torch.equal(up, parent):
            break
        parent = up
    return _ints(g, n, m)[parent]


def _graph(case, g):
    """n, src, dst, edge label, vertex label (int32, on the GPU), sources ascending where the generator's are."""
    n, m = case["n"], case["m"]
    i32 = torch.int32
    if case["graph"] == "uniform":
        src = _ints(g, n, m).sort().values.to(i32)
        return n, src, _ints(g, n, m).to(i32), _ints(g, 8, m).to(i32), _ints(g, 4, n).to(i32)
    if case["graph"] == "powerlaw":
        src = torch.repeat_interleave(torch.arange(n, device="cuda", dtype=i32), _degrees(g, n, m))
        dst = torch.empty(m, device="cuda", dtype=i32)
        dst[torch.randperm(m, generator=g, device="cuda")] = _copied_targets(g, n, m).to(i32)
        lab = _zipf(g, m, 1000, 1.1)
        vl = _zipf(g, n, 200, 1.0)
        vl[_unit(g, n) < 0.1] = -1
        return n, src, dst, lab, vl
    # paths of equal length (path-major ids; the last one takes the rest) and uniform extra edges
    paths = case["paths"]
    length = max(1, n // paths)
    v = torch.arange(n, device="cuda")
    v = v[(v % length != length - 1) & (v < n - 1)]
    extra = max(0, m - (n - paths))
    src = torch.cat([v, _ints(g, n, extra)])
    dst = torch.cat([v + 1, _ints(g, n, extra)])
    pure = extra == 0
    lab = _ints(g, 1 if pure else 16, len(src))
    vl = _ints(g, 1 if pure else 2, n)
    if pure:                                               # a few marked vertices, so that no two draws are alike
        vl[_ints(g, n, max(1, n // 100_000))] = 1
    return n, src.to(i32), dst.to(i32), lab.to(i32), vl.to(i32)


def _batch(case, g):
    """Vertex and edge offsets and the union's local edges of `graphs` power-law graphs of mean degree 5."""
    G = case["graphs"]
    q = (torch.arange(G, device="cuda", dtype=torch.float64) + 0.5) / G      # sizes: log-uniform quantiles in random order
    lo, hi = math.log(case["nmin"]), math.log(case["nmax"])
    ng = torch.exp(lo + q * (hi - lo)).floor().to(torch.int64).clamp_(min=2)
    ng = ng[torch.randperm(G, generator=g, device="cuda")]
    vo = torch.zeros(G + 1, device="cuda", dtype=torch.int64)
    vo[1:] = torch.cumsum(ng, 0)
    n = int(vo[-1])
    gid = torch.repeat_interleave(torch.arange(G, device="cuda"), ng)
    d = _pareto(g, n, 2.3, (ng - 1).to(torch.float64)[gid])
    total = torch.zeros(G, device="cuda", dtype=torch.float64).index_add_(0, gid, d)
    d = torch.minimum(d * (5.0 * ng.to(torch.float64) / total)[gid], (ng - 1).to(torch.float64)[gid])
    fl = d.floor()
    d = (fl + (_unit(g, n) < d - fl)).to(torch.int64)
    eg = torch.zeros(G, device="cuda", dtype=torch.int64).index_add_(0, gid, d)
    eo = torch.zeros(G + 1, device="cuda", dtype=torch.int64)
    eo[1:] = torch.cumsum(eg, 0)
    m = int(eo[-1])
    src = torch.repeat_interleave(torch.arange(n, device="cuda"), d)
    ge = gid[src]
    dst = (_unit(g, m) * ng[ge]).to(torch.int64)
    return dict(vo=vo, eo=eo, src=(src - vo[ge]).to(torch.int32), dst=dst.to(torch.int32), lab=_zipf(g, m, 64, 1.1),
                vl=_ints(g, 16, n).to(torch.int32), gid=gid, ge=ge)


def _row_ptr(n, src):
    rp = torch.zeros(n + 1, device="cuda", dtype=torch.int64)
    rp[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    return rp


def _by_source(src, dst, lab):
    src, o = torch.sort(src, stable=True)
    return src, dst[o].contiguous(), lab[o].contiguous()


def _arranged(case, g, src, dst, lab):
    """The edges in the order a case wants them in; a CSR's are grouped by source."""
    if case["order"] == "shuffled":
        o = torch.randperm(len(src), generator=g, device="cuda")
        src, dst, lab = src[o], dst[o], lab[o]
    if case["input"] == "csr" or (case["order"] == "sorted" and case["graph"] == "chain"):
        src, dst, lab = _by_source(src, dst, lab)
    return src, dst, lab


def _batches(g, n, src, dst, lab, vl, ops):
    """An update batch (70% edge adds, 25% edge deletes, 5% vertex deletes) and the batch that takes it back.

    As graphgen.update_batches draws them; deleted vertices have at most 256
    edges, which bounds the second batch. Also the edited edge list (for
    exact()) as a mask over the base edges and the added edges that stay."""
    m = len(src)
    na, nd, nv = int(0.7 * ops), int(0.25 * ops), max(1, int(0.05 * ops))
    a_src = _ints(g, n, na)
    a_dst = torch.where(_unit(g, na) < 0.8, dst[_ints(g, m, na)].to(torch.int64), _ints(g, n, na))
    a_lab = _zipf(g, na, 1000, 1.1).to(torch.int64)
    de = _ints(g, m, nd).unique()
    degree = torch.bincount(src, minlength=n) + torch.bincount(dst, minlength=n)
    dv = _ints(g, n, nv).unique()
    dv = dv[degree[dv] <= 256]
    dead = torch.zeros(n, device="cuda", dtype=torch.bool)
    dead[dv] = True
    keep = ~(dead[src.long()] | dead[dst.long()])
    keep[de] = False
    stay = ~(dead[a_src] | dead[a_dst])

    def rows(kind, s, d=None, l=None):
        z = torch.zeros_like(s)
        return torch.stack([torch.full_like(s, kind), s, z if d is None else d, z if l is None else l], 1)

    def mixed(r):
        return r[torch.randperm(len(r), generator=g, device="cuda")]

    b = [src[~keep].long(), dst[~keep].long(), lab[~keep].long()]
    do = torch.cat([mixed(torch.cat([rows(bisim.OP_EDGE_ADD, a_src, a_dst, a_lab),
                                     rows(bisim.OP_EDGE_DEL, src[de].long(), dst[de].long(), lab[de].long())])),
                    rows(bisim.OP_VERTEX_DEL, dv)])
    undo = torch.cat([rows(bisim.OP_VERTEX_ADD, dv, None, vl[dv].long()),
                      mixed(torch.cat([rows(bisim.OP_EDGE_ADD, *b),
                                       rows(bisim.OP_EDGE_DEL, a_src[stay], a_dst[stay], a_lab[stay])]))])
    host = [x.to(torch.int32).cpu().pin_memory() for x in (do, undo)]
    return host, keep, (a_src[stay], a_dst[stay], a_lab[stay]), dead


# ----------------------------------------------------------------------------- the calls


def _options(case):
    o = dict(direction=DIRECTIONS[case.get("direction", "forward")])
    if case.get("labels"):
        o["label_filter"] = list(range(case["labels"]))
    return bisim.default_options(**o)


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "batched":
        b = _batch(case, g)
        return dict(case=case, args=(b["vo"], b["eo"], b["src"], b["dst"], b["lab"], b["vl"]))
    n, src, dst, lab, vl = _graph(case, g)
    if kind == "round":
        return dict(case=case, n=n, rp=_row_ptr(n, src), col=dst, lab=lab, vl=vl, out=torch.empty_like(vl))
    if kind == "summarize":
        src, dst, lab = _arranged(case, g, src, dst, lab)
        return dict(case=case, n=n, src=_row_ptr(n, src) if case["input"] == "csr" else src, dst=dst, lab=lab, vl=vl,
                    options=_options(case))
    ctx = bisim.summarize_init_coo(n, src, dst, lab, vl, options=_options(case))
    if kind == "updates":
        bisim.bisim_iterate(ctx, 2)
        bisim.apply_updates(ctx, torch.zeros((0, 4), dtype=torch.int32, device="cuda"))     # builds the incremental state
        return dict(case=case, ctx=ctx, batches=_batches(g, n, src, dst, lab, vl, case["ops"])[0])
    if kind == "summary":
        bisim.bisim_iterate(ctx, case["k"])
        return dict(case=case, ctx=ctx, edges=torch.full((3, len(src)), -1, device="cuda", dtype=torch.int32))
    return dict(case=case, ctx=ctx)


def _cap(case):
    return 1000 if case["graph"] == "chain" else 10


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "round":
        blocks = bisim.bisim_refine_round_noalloc(state["n"], state["rp"], state["col"], state["lab"], state["vl"],
                                                  state["out"])
        return dict(partition=state["out"], blocks=blocks)
    if kind == "summarize":
        init = bisim.summarize_init if case["input"] == "csr" else bisim.summarize_init_coo
        with init(state["n"], state["src"], state["dst"], state["lab"], state["vl"], options=state["options"]) as ctx:
            rounds, blocks = bisim.bisim_iterate(ctx, case["k"], _cap(case))
            return dict(partition=bisim.get_partition(ctx), rounds=rounds, blocks=blocks)
    if kind == "batched":
        with bisim.summarize_init_batched(*state["args"]) as ctx:
            rounds, blocks = bisim.bisim_iterate(ctx, case["k"])
            return dict(partition=bisim.get_partition(ctx), rounds=rounds, blocks=blocks)
    ctx = state["ctx"]
    if kind == "refine":
        rounds, blocks = bisim.bisim_iterate(ctx, case["k"], _cap(case))
        return dict(partition=bisim.get_partition(ctx), rounds=rounds, blocks=blocks)
    if kind == "updates":
        do, undo = state["batches"]
        bisim.apply_updates(ctx, do)
        edited = bisim.get_partition(ctx)
        bisim.apply_updates(ctx, undo)
        return dict(edited=edited, restored=bisim.get_partition(ctx))
    # summary: the edges go into the caller's own array of fixed size
    edges = bisim.get_summary_edges(ctx)
    count = len(edges[0])
    for row, e in zip(state["edges"], edges):
        row[:count].copy_(e)
    return dict(edges=state["edges"], count=count, sizes=bisim.get_block_sizes(ctx))


def work(case):
    """Bytes: inputs read once (12 an edge as source, target, label; 8 an edge
    where the graph is resident), labels read and results written once (4 each)."""
    kind = case["kind"]
    if kind == "batched":
        lo, hi = case["nmin"], case["nmax"]
        n = case["graphs"] * (hi - lo) / math.log(hi / lo)
        return dict(bytes=12.0 * 5 * n + 8.0 * n, flops=0.0)
    n, m = case["n"], case["m"]
    if kind == "updates":
        return dict(bytes=3 * 16.0 * case["ops"] + 8.0 * n, flops=0.0)       # the second batch has about twice the operations
    if kind == "summarize":
        return dict(bytes=12.0 * m + 8.0 * n, flops=0.0)
    if kind == "summary":
        return dict(bytes=20.0 * m + 8.0 * n, flops=0.0)
    return dict(bytes=8.0 * m + 8.0 * n, flops=0.0)


def tolerance(case):
    return "exact"


# ----------------------------------------------------------------------------- reference


def _mix(x, salt):
    """A 64-bit mix of int64 values (two multiply-xorshift steps), for the reference only."""
    x = x ^ salt
    for mul, sh in ((-0x61C8864680B583EB, 32), (0x2545F4914F6CDD1D, 29)):
        x = x * mul
        x = x ^ ((x >> sh) & ((1 << (64 - sh)) - 1))
    return x


def _smallest_alike(n, keys):
    """For every vertex the smallest one with the same keys (a list of int64 [n])."""
    o = torch.arange(n, device="cuda")
    for k in reversed(keys):
        o = o[torch.sort(k[o], stable=True).indices]
    head = torch.ones(n, device="cuda", dtype=torch.bool)
    if n > 1:
        head[1:] = False
        for k in keys:
            head[1:] |= k[o][1:] != k[o][:-1]
    first = o[head]
    out = torch.empty(n, device="cuda", dtype=torch.int64)
    out[o] = first[torch.cumsum(head, 0) - 1]
    return out, int(head.sum())


def _round(n, src, dst, lab, P):
    pair = (lab.long() << 32) | P[dst.long()]
    o = torch.sort(pair, stable=True).indices
    o = o[torch.sort(src[o], stable=True).indices]
    s, p = src[o].long(), pair[o]
    if len(s):
        new = torch.ones(len(s), device="cuda", dtype=torch.bool)
        new[1:] = (s[1:] != s[:-1]) | (p[1:] != p[:-1])
        s, p = s[new], p[new]
    keys = [P]
    for salt in (0x1234567, 0x7654321ABCD):
        keys.append(torch.zeros(n, device="cuda", dtype=torch.int64).index_add_(0, s, _mix(p, salt)))
    return _smallest_alike(n, keys)


def _refined(n, src, dst, lab, first, k, cap):
    """Canonical partition, rounds and block count after k rounds (or at the fixpoint) from the vertex keys `first`."""
    P, blocks = _smallest_alike(n, first)
    limit, r = (cap if k == FIX else k), 0
    while r < limit:
        nxt, b = _round(n, src, dst, lab, P)
        if b == blocks:
            return nxt, (r if k == FIX else k), b
        P, blocks, r = nxt, b, r + 1
    return P, limit, blocks


def exact(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    i32 = torch.int32
    if kind == "batched":
        b = _batch(case, g)
        n = len(b["vl"])
        base = b["vo"][:-1]
        P, rounds, blocks = _refined(n, (b["src"] + base[b["ge"]]).to(i32), b["dst"] + base[b["ge"]], b["lab"],
                                     [b["gid"], b["vl"].long()], case["k"], 10)
        return dict(partition=(P - base[b["gid"]]).to(i32), rounds=rounds, blocks=blocks)
    if case["graph"] == "chain" and case.get("k") == FIX and case["n"] > 20_000 and case["m"] < 2 * case["n"]:
        return None                                        # hundreds of rounds of sorts: too slow
    n, src, dst, lab, vl = _graph(case, g)
    vkey = [vl.long()]
    if kind == "round":
        P, blocks = _round(n, src, dst, lab, vl.long())
        return dict(partition=P.to(i32), blocks=blocks)
    if kind == "updates":
        _, keep, added, dead = _batches(g, n, src, dst, lab, vl, case["ops"])
        before = _refined(n, src, dst, lab, vkey, 2, 0)[0].to(i32)
        a, b, l = (torch.cat([x[keep].long(), y]) for x, y in zip((src, dst, lab), added))
        # a deleted vertex belongs to no block: kept apart by its id, then -1
        ids = torch.where(dead, torch.arange(n, device="cuda"), torch.full((n,), -1, device="cuda"))
        after = _refined(n, a, b, l, [ids] + vkey, 2, 0)[0].to(i32)
        after[dead] = -1
        return dict(edited=after, restored=before)
    if kind == "summarize":
        src, dst, lab = _arranged(case, g, src, dst, lab)
        if case["labels"]:
            f = lab < case["labels"]
            src, dst, lab = src[f], dst[f], lab[f]
        if case["direction"] == "backward":
            src, dst = dst, src
        elif case["direction"] == "both":
            src, dst, lab = torch.cat([src, dst]), torch.cat([dst, src]), torch.cat([2 * lab, 2 * lab + 1])
    P, rounds, blocks = _refined(n, src, dst, lab, vkey, case["k"], _cap(case))
    if kind != "summary":
        return dict(partition=P.to(i32), rounds=rounds, blocks=blocks)
    t = [P[src.long()], lab.long(), P[dst.long()]]
    o = torch.arange(len(src), device="cuda")
    for k in reversed(t):
        o = o[torch.sort(k[o], stable=True).indices]
    t = torch.stack([k[o] for k in t])
    new = torch.ones(t.shape[1], device="cuda", dtype=torch.bool)
    new[1:] = (t[:, 1:] != t[:, :-1]).any(0)
    count = int(new.sum())
    edges = torch.full((3, len(src)), -1, device="cuda", dtype=i32)
    edges[:, :count] = t[:, new].to(i32)
    return dict(edges=edges, count=count, sizes=torch.bincount(P, minlength=n).to(i32))
