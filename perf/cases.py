"""Performance cases of the truss library: what its users call, through the
Python binding of the C ABI, over the range of sizes and input forms they use.

A case is a dict of plain values: the call, the kind of graph and its sizes.
``prepare`` makes the rows of that graph on the GPU from the seed (or in host
memory, where the path starts from host buffers) and the output buffers;
``run`` is one call.  The library's context and its request server are kept
for the life of the process, as a program that decomposes one graph after
another keeps them.

Graphs (the kinds the benchmark and the tests use):

* ``rmat``: 2^scale vertices, raw samples with (a, b, c, d) = (.57, .19, .19,
  .05); duplicate rows, reversed rows and self-loops stay in.
* ``chung_lu``: power-law expected degrees of exponent 2.1, mean 2 rows / n,
  capped; endpoints drawn independently, duplicates and self-loops stay in.
* ``er_cliques``: uniform random pairs plus cliques on disjoint random vertices.

All outputs are whole numbers.
"""
from __future__ import annotations

import numpy as np
import torch

from paper_1205_6693_gb300 import truss as T

DEV = "cuda:0"


def listed():
    return [
        # Support of one small graph by a program that may not allocate
        # device memory (an allocator callback, a device handed out whole).
        dict(name="noalloc_60k", call="support_noalloc", graph="rmat", scale=13, rows=60_001),
        # The smallest ordinary call: the 4,096-vertex random graph with six
        # planted cliques; latency and launches count.
        dict(name="decompose_tiny", call="decompose", graph="er_cliques", n=4096, rows=32_768,
             cliques="8,12,16,20,24,32"),
        # A small social graph with the defects of a raw edge list.
        dict(name="decompose_small", call="decompose", graph="rmat", scale=15, rows=500_009),
        # The benchmark's R-MAT graph: 16.8 M raw rows, hubs above 10^4.
        dict(name="decompose_mid", call="decompose", graph="rmat", scale=20, rows=16_777_216),
        # The benchmark's power-law graph at a quarter of its size: more edges
        # than L2 holds states for, deep peel levels.
        dict(name="decompose_large", call="decompose", graph="chung_lu", n=1 << 22,
             rows=41_943_040, cap=32_768),
        # Edges and results in pinned host memory, as a program that loads a
        # graph from disk and writes its truss numbers back has them.
        dict(name="decompose_pinned", call="decompose", graph="chung_lu", n=1 << 20,
             rows=10_485_760, cap=16_384, host=True),
        # Triangle counts per edge only, at sizes that are no power of two.
        dict(name="support_odd", call="support", graph="chung_lu", n=1_000_003, rows=9_999_991,
             cap=10_000),
        # Thousands of small uneven graphs (ego networks, molecules, windows
        # of a stream) in one call: the 4,096-graph mixed batch.
        dict(name="batch_4096", call="batch", graphs=4096, lo=64, hi=65_536),
        # A burst of requests of mixed sizes to the request server, from host
        # memory and back: small ones batched, large ones alone.
        dict(name="serve_burst", call="serve", requests=24, lo=1_000, hi=2_000_000),
        # The densest classes only (community cores): top-10 truss.
        dict(name="top10", call="top", graph="rmat", scale=18, rows=4_194_304, t=10),
        # Core numbers of a graph's vertices.
        dict(name="core_mid", call="core", graph="rmat", scale=20, rows=16_777_216),
        # Decomposition under a working-set budget, subgraph by subgraph.
        dict(name="budget_14", call="budget", graph="rmat", scale=14, rows=262_144,
             budget=40_000),
    ]


def _log(rng, lo, hi):
    """A whole number spread evenly over the logarithm of [lo, hi]."""
    x = int(round(lo * (hi / lo) ** rng.random()))
    return max(lo, min(hi, x))


def _graph(rng, lo, hi, graphs=("rmat", "chung_lu", "er_cliques")):
    """Kind and sizes of one graph of lo..hi rows, 8 to 24 rows per vertex."""
    kind = rng.choice(graphs)
    rows = _log(rng, lo, hi)
    if kind == "rmat":
        scale = max(6, (rows // rng.randint(8, 24)).bit_length())
        return dict(graph=kind, scale=scale, rows=rows)
    n = max(64, rows // rng.randint(8, 24) + rng.randint(0, 13))
    if kind == "chung_lu":
        return dict(graph=kind, n=n, rows=rows, cap=max(32, min(32_768, n // 100)))
    sizes = [s for s in (5, 9, 13, 17, 26, 33) if rng.random() < 0.6] or [7]
    while sum(sizes) > n:
        sizes.pop()
    return dict(graph=kind, n=n, rows=rows, cliques=",".join(map(str, sizes)))


def draw(rng):
    call = rng.choice(("decompose", "decompose", "decompose", "support", "support_noalloc",
                       "batch", "serve", "top", "core", "budget"))
    if call == "support_noalloc":
        return dict(call=call, **_graph(rng, 1_000, 64_000))
    if call == "batch":
        return dict(call=call, graphs=_log(rng, 16, 4096), lo=64, hi=_log(rng, 1_000, 60_000))
    if call == "serve":
        return dict(call=call, requests=rng.randint(4, 30), lo=1_000,
                    hi=_log(rng, 20_000, 1_500_000))
    if call == "budget":
        c = _graph(rng, 5_000, 100_000)
        return dict(call=call, **c, budget=c["rows"] // rng.randint(2, 5))
    c = _graph(rng, 2_000, 20_000_000)
    if call == "top":
        return dict(call=call, **c, t=rng.randint(1, 20))
    if call == "decompose" and rng.random() < 0.3:
        c["host"] = True
    return dict(call=call, **c)


# ------------------------------------------------------------------ graphs ---
def _gen(seed, device=DEV):
    return torch.Generator(device=device).manual_seed(seed)


def _rmat(gen, scale, rows):
    """Raw R-MAT samples; `scale` is a number or one number per row."""
    src = torch.zeros(rows, dtype=torch.int32, device=DEV)
    dst = torch.zeros(rows, dtype=torch.int32, device=DEV)
    per_row = isinstance(scale, torch.Tensor)
    for b in range(int(scale.max()) if per_row else scale):
        r = torch.rand(rows, generator=gen, device=DEV)
        s = (r >= 0.76).to(torch.int32)
        d = (((r >= 0.57) & (r < 0.76)) | (r >= 0.95)).to(torch.int32)
        if per_row:
            more = scale > b
            src = torch.where(more, 2 * src + s, src)
            dst = torch.where(more, 2 * dst + d, dst)
        else:
            src.mul_(2).add_(s)
            dst.mul_(2).add_(d)
    return src, dst


def _chung_lu(gen, n, rows, cap):
    """Endpoints drawn with weights min(c (i+1)^(-1/1.1), cap) of the mean 2 rows / n."""
    base = torch.arange(1, n + 1, dtype=torch.float64, device=DEV).pow_(-1.0 / 1.1)
    want = 2.0 * rows
    lo, hi = 0.0, 1.0
    while hi < 1e15 and float(base.mul(hi).clamp_(max=cap).sum()) < want:
        hi *= 2.0
    for _ in range(40):
        mid = 0.5 * (lo + hi)
        if float(base.mul(mid).clamp_(max=cap).sum()) < want:
            lo = mid
        else:
            hi = mid
    cdf = base.mul_(hi).clamp_(max=cap).cumsum_(0)
    ends = []
    for _ in range(2):
        x = torch.rand(rows, dtype=torch.float64, generator=gen, device=DEV).mul_(cdf[-1])
        ends.append(torch.searchsorted(cdf, x).clamp_(max=n - 1).to(torch.int32))
    return ends[0], ends[1]


def _clique_pairs(verts):
    a, b = np.triu_indices(len(verts), 1)
    i = torch.from_numpy(np.stack([a, b])).to(DEV)
    return verts[i[0]], verts[i[1]]


def _er_cliques(gen, n, rows, cliques):
    src = [torch.randint(0, n, (rows,), dtype=torch.int32, generator=gen, device=DEV)]
    dst = [torch.randint(0, n, (rows,), dtype=torch.int32, generator=gen, device=DEV)]
    perm = torch.randperm(n, generator=gen, device=DEV).to(torch.int32)
    at = 0
    for size in (int(x) for x in cliques.split(",") if x):
        a, b = _clique_pairs(perm[at:at + size])
        src.append(a)
        dst.append(b)
        at += size
    return torch.cat(src), torch.cat(dst)


def _rows_of(case, seed):
    """(n, src, dst) of a single-graph case, on the GPU."""
    gen = _gen(seed)
    if case["graph"] == "rmat":
        return (1 << case["scale"], *_rmat(gen, case["scale"], case["rows"]))
    if case["graph"] == "chung_lu":
        return (case["n"], *_chung_lu(gen, case["n"], case["rows"], float(case["cap"])))
    return (case["n"], *_er_cliques(gen, case["n"], case["rows"], case["cliques"]))


def _log_spread(rng, lo, hi, count):
    """`count` whole numbers evenly spread over the logarithm of [lo, hi], in
    random order (so another seed asks as much)."""
    at = (rng.permutation(count) + 0.5) / count
    return np.rint(lo * (hi / lo) ** at).astype(np.int64)


def _batch_rows(case, seed):
    """The mixed batch: a third random, a third R-MAT, a third random with a
    planted clique; edge counts spread over the logarithm of [lo, hi].
    Returns n[G], row_off[G+1], src, dst with ids local to each graph."""
    G = case["graphs"]
    rng = np.random.default_rng(seed)
    gen = _gen(seed)
    m = _log_spread(rng, case["lo"], case["hi"], G)
    kind = np.arange(G) % 3
    clique = np.zeros(G, np.int64)
    clique[kind == 2] = rng.permutation(np.count_nonzero(kind == 2)) % 37 + 4
    scale = np.maximum(4, np.ceil(np.log2(np.maximum(m / 8.0, 1.0))).astype(np.int64))
    n = np.where(kind == 1, 1 << scale, np.maximum(np.maximum(16, clique), -(-m // 4)))
    rows = m + clique * (clique - 1) // 2
    off = np.zeros(G + 1, np.int64)
    np.cumsum(rows, out=off[1:])
    total = int(off[-1])
    g = torch.repeat_interleave(torch.arange(G, device=DEV), torch.from_numpy(rows).to(DEV))
    nd = torch.from_numpy(n).to(DEV)
    ends = []
    for _ in range(2):
        x = torch.rand(total, dtype=torch.float64, generator=gen, device=DEV)
        ends.append((x * nd[g]).to(torch.int32))
    src, dst = ends
    rmat = torch.from_numpy(kind == 1).to(DEV)[g]
    sc = torch.from_numpy(scale).to(DEV).to(torch.int32)[g]
    rs, rd = _rmat(gen, torch.where(rmat, sc, torch.zeros_like(sc)), total)
    src = torch.where(rmat, rs, src)
    dst = torch.where(rmat, rd, dst)
    # cliques on the vertices c, c+step, c+2 step, ... of their graph
    for i in np.nonzero(clique)[0]:
        c, step = int(clique[i]), max(1, int(n[i]) // int(clique[i]))
        a, b = np.triu_indices(c, 1)
        ab = torch.from_numpy((np.stack([a, b]) * step).astype(np.int32)).to(DEV, non_blocking=True)
        src[int(off[i] + m[i]):int(off[i + 1])] = ab[0]
        dst[int(off[i] + m[i]):int(off[i + 1])] = ab[1]
    return n, off, src, dst


def _requests(case, seed):
    """R-MAT requests, sizes spread over the logarithm of [lo, hi], in host
    memory: (n[R], row_off[R+1], src, dst)."""
    R = case["requests"]
    rng = np.random.default_rng(seed)
    m = _log_spread(rng, case["lo"], case["hi"], R)
    scale = np.maximum(4, np.ceil(np.log2(m / 8.0)).astype(np.int64))
    off = np.zeros(R + 1, np.int64)
    np.cumsum(m, out=off[1:])
    sc = torch.repeat_interleave(torch.from_numpy(scale).to(DEV).to(torch.int32),
                                 torch.from_numpy(m).to(DEV))
    src, dst = _rmat(_gen(seed), sc, int(off[-1]))
    return 1 << scale, off, src.cpu().numpy(), dst.cpu().numpy()


# ------------------------------------------------------------------ passes ---
_kept = {}


def _context():
    """The program's one context: its workspace serves every graph."""
    if "ctx" not in _kept:
        _kept["ctx"] = T.Context(0)
    return _kept["ctx"]


def _server():
    """The program's one request server."""
    if "server" not in _kept:
        o = T.truss_serve_opts()
        o.hbm_budget_bytes = 24 << 30
        _kept["server"] = T.truss_serve_start(_context().ctx, o)
    return _kept["server"]


def prepare(case, seed):
    call = case["call"]
    if call == "serve":
        n, off, src, dst = _requests(case, seed)
        return dict(call=call, server=_server(), n=n, off=off, src=src, dst=dst,
                    support=np.empty(len(src), np.int32), truss=np.empty(len(src), np.int32))
    st = dict(call=call, ctx=_context())
    if call == "batch":
        st["n"], st["off"], st["src"], st["dst"] = _batch_rows(case, seed)
        st["kmax"] = torch.empty(case["graphs"], dtype=torch.int32, device=DEV)
    else:
        st["n"], st["src"], st["dst"] = _rows_of(case, seed)
    if case.get("host"):
        for x in ("src", "dst"):
            st[x] = st[x].cpu().pin_memory()
    rows = st["src"].shape[0]
    for x in (["core"] if call == "core" else ["truss"] if call == "top" else
              ["support"] if call.startswith("support") else ["support", "truss"]):
        st[x] = torch.empty(st["n"] if x == "core" else rows, dtype=torch.int32,
                            device=st["src"].device, pin_memory=bool(case.get("host")))
    st["t"], st["budget"] = case.get("t"), case.get("budget")
    return st


def run(s):
    call = s["call"]
    if call == "serve":
        srv, off = s["server"], s["off"]
        tickets = [T.truss_serve_submit(srv, int(s["n"][i]), s["src"][off[i]:off[i + 1]],
                                        s["dst"][off[i]:off[i + 1]]) for i in range(len(s["n"]))]
        kmax = [T.truss_serve_wait(srv, t, -1, s["support"][off[i]:off[i + 1]],
                                   s["truss"][off[i]:off[i + 1]])["kmax"]
                for i, t in enumerate(tickets)]
        return {"support": s["support"], "truss": s["truss"], "kmax": np.array(kmax, np.int32)}
    if call == "support_noalloc":
        T.truss_support_noalloc(s["n"], s["src"], s["dst"], s["support"])
        return {"support": s["support"]}
    c = s["ctx"]
    if call == "support":
        c.support(s["n"], s["src"], s["dst"], s["support"])
        return {"support": s["support"]}
    if call == "core":
        return {"core": s["core"], "kmax": c.core(s["n"], s["src"], s["dst"], s["core"])}
    if call == "top":
        return {"truss": s["truss"],
                "kmax": c.top(s["n"], s["src"], s["dst"], s["t"], s["truss"])}
    if call == "batch":
        c.decompose_batch(s["n"], s["off"], s["src"], s["dst"], s["support"], s["truss"],
                          s["kmax"])
        return {"support": s["support"], "truss": s["truss"], "kmax": s["kmax"]}
    if call == "budget":
        kmax = c.decompose_budget(s["n"], s["src"], s["dst"], s["budget"], s["support"],
                                  s["truss"])
    else:
        kmax = c.decompose(s["n"], s["src"], s["dst"], s["support"], s["truss"])
    return {"support": s["support"], "truss": s["truss"], "kmax": kmax}


def _row_count(case):
    """Rows of a case (for a batch or a burst, of its size distribution's mean)."""
    if "rows" in case:
        extra = sum(int(x) * (int(x) - 1) // 2 for x in case.get("cliques", "").split(",") if x)
        return case["rows"] + extra
    lo, hi = case["lo"], case["hi"]
    mean = (hi - lo) / np.log(hi / lo) if hi > lo else lo
    return int(case.get("graphs", case.get("requests")) * mean)


def work(case):
    """Two words read per row and the outputs written: the walk over the
    triangles between them is what the library is for, and has no fixed cost."""
    rows = _row_count(case)
    if case["call"] == "core":
        out = 4 * (case["n"] if "n" in case else 1 << case["scale"])
    else:
        out = 4 * rows * (1 if case["call"] in ("support", "support_noalloc", "top") else 2)
    return {"bytes": 8 * rows + out, "flops": 0}


# ------------------------------------------------------------------- exact ---
def _edges(n, src, dst):
    """Distinct edges (u, v) with u < v and each row's edge (-1: self-loop)."""
    src, dst = src.to(torch.int64), dst.to(torch.int64)
    key = torch.minimum(src, dst) * n + torch.maximum(src, dst)
    loop = src == dst
    uniq, inv = torch.unique(key[~loop], return_inverse=True)
    row2e = torch.full_like(src, -1)
    row2e[~loop] = inv
    return uniq // n, uniq % n, row2e


def _triangles(n, u, v):
    """Edge-id triples of all triangles of the edges (u, v)."""
    m = len(u)
    deg = torch.bincount(torch.cat([u, v]), minlength=n)
    rank = torch.empty_like(deg)
    rank[torch.argsort(deg, stable=True)] = torch.arange(n, device=u.device)
    a, b = torch.minimum(rank[u], rank[v]), torch.maximum(rank[u], rank[v])
    key, eid = torch.sort(a * n + b)
    a, b = key // n, key % n
    end = torch.searchsorted(a, a, right=True)
    after = end - torch.arange(m, device=u.device) - 1
    cum = torch.cumsum(after, 0)
    parts, i0 = [], 0
    while i0 < m:
        done = int(cum[i0 - 1]) if i0 else 0
        i1 = max(i0 + 1, int(torch.searchsorted(cum, done + (1 << 24), right=True)))
        i = torch.repeat_interleave(torch.arange(i0, i1, device=u.device), after[i0:i1])
        start = torch.repeat_interleave(cum[i0:i1] - after[i0:i1], after[i0:i1])
        j = i + 1 + (torch.arange(len(i), device=u.device) + done - start)
        want = b[i] * n + b[j]
        p = torch.searchsorted(key, want).clamp_(max=m - 1)
        hit = key[p] == want
        parts.append(torch.stack([eid[i[hit]], eid[j[hit]], eid[p[hit]]]))
        i0 = i1
    return torch.cat(parts, 1) if parts else torch.empty(3, 0, dtype=torch.int64, device=u.device)


def _truss(m, tri):
    """Support and truss number of each edge: edges of at most k - 2 triangles
    are removed, with their triangles, for k = 2, 3, ..."""
    sup = torch.bincount(tri.reshape(-1), minlength=m)
    res, truss = sup.clone(), torch.zeros_like(sup)
    alive = torch.ones(m, dtype=torch.bool, device=sup.device)
    left, k = m, 2
    while left:
        gone = alive & (res <= k - 2)
        count = int(gone.sum())
        if not count:
            k = int(res[alive].min()) + 2
            continue
        truss[gone] = k
        alive &= ~gone
        left -= count
        dead = gone[tri].any(0)
        res -= torch.bincount(tri[:, dead].reshape(-1), minlength=m)
        tri = tri[:, ~dead]
    return sup, truss


def _core(n, u, v):
    deg = torch.bincount(torch.cat([u, v]), minlength=n)
    core = torch.zeros_like(deg)
    alive = torch.ones(n, dtype=torch.bool, device=u.device)
    left, k = n, 0
    while left:
        gone = alive & (deg <= k)
        count = int(gone.sum())
        if not count:
            k = int(deg[alive].min())
            continue
        core[gone] = k
        alive &= ~gone
        left -= count
        dead = gone[u] | gone[v]
        deg -= torch.bincount(torch.cat([u[dead], v[dead]]), minlength=n)
        u, v = u[~dead], v[~dead]
    return core


def exact(case, seed):
    """The same outputs from their definitions, in plain torch on 64-bit whole
    numbers; None where that would take long."""
    call = case["call"]
    if _row_count(case) > 600_000 and not (call == "core" and case["graph"] == "rmat"):
        return None
    if call in ("batch", "serve"):
        n, off, src, dst = (_batch_rows if call == "batch" else _requests)(case, seed)
        G = len(n)
        g = torch.repeat_interleave(torch.arange(G), torch.from_numpy(np.diff(off))).to(DEV)
        base = torch.from_numpy(np.concatenate([[0], np.cumsum(n)[:-1]])).to(DEV)[g]
        n = int(n.sum())
        src = torch.as_tensor(src).to(DEV).to(torch.int64) + base
        dst = torch.as_tensor(dst).to(DEV).to(torch.int64) + base
    else:
        n, src, dst = _rows_of(case, seed)
    u, v, row2e = _edges(n, src, dst)
    if call == "core":
        core = _core(n, u, v)
        return {"core": core.to(torch.int32), "kmax": int(core.max())}
    sup, truss = _truss(len(u), _triangles(n, u, v))
    loop = row2e < 0
    per_row = [torch.where(loop, -1, x[row2e.clamp(min=0)]).to(torch.int32) for x in (sup, truss)]
    if call.startswith("support"):
        return {"support": per_row[0]}
    if call in ("batch", "serve"):
        kmax = torch.zeros(G, dtype=torch.int32, device=DEV)
        kmax.scatter_reduce_(0, g, per_row[1].clamp(min=0), "amax")
        out = {"support": per_row[0], "truss": per_row[1], "kmax": kmax}
        return out if call == "batch" else {k: x.cpu().numpy() for k, x in out.items()}
    kmax = int(truss.max()) if len(truss) else 0
    if call == "top":
        t = per_row[1]
        return {"truss": torch.where((t >= 0) & (t < kmax - case["t"] + 1), 0, t), "kmax": kmax}
    out = {"support": per_row[0], "truss": per_row[1], "kmax": kmax}
    return {k: x.cpu() if case.get("host") and k != "kmax" else x for k, x in out.items()}
