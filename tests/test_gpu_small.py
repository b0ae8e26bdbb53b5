"""The launches that build small graphs in one kernel, and the support walk's
mixed runs of short out-lists, at the sizes where they can go wrong: edges of
tiles and warps, degrees around the counted ones, the largest size taken and
one more.  Against the CPU oracle, or against the general path (which a context
with a wait limit takes); all outputs are integers and compared exactly."""
import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SMALL_ROWS = 5 << 19  # csrc/small.cu: kSmallRows


@pytest.fixture(scope="module")
def ctx():
    from paper_1205_6693_gb300 import truss as T
    c = T.Context(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def general():
    from paper_1205_6693_gb300 import truss as T
    c = T.Context(0, wait_limit_ns=4_000_000_000)
    yield c
    c.close()


def run(ctx, n, s, d):
    sup, tr = torch.full_like(s, -7), torch.full_like(s, -7)
    k = ctx.decompose(n, s, d, sup, tr)
    only = torch.full_like(s, -7)
    ctx.support(n, s, d, only)
    assert torch.equal(only, sup)
    return sup.cpu().numpy(), tr.cpu().numpy(), k


def check(ctx, n, src, dst):
    s = torch.from_numpy(np.ascontiguousarray(src, np.int32)).cuda()
    d = torch.from_numpy(np.ascontiguousarray(dst, np.int32)).cuda()
    ref = oracle.truss(n, src, dst)
    sup, tr, k = run(ctx, n, s, d)
    assert np.array_equal(sup, ref.support) and np.array_equal(tr, ref.truss) and k == ref.kmax


@pytest.mark.parametrize("rows", [1, 2, 31, 33, 511, 512, 513, 1023, 1025, 8191, 60_001])
def test_row_counts_around_tiles(ctx, rows):
    # random pairs of a dense and a sparse graph, self-loops and reversed
    # duplicates among them
    for n in (max(2, rows // 6), rows + 3):
        rng = np.random.default_rng(rows)
        check(ctx, n, rng.integers(0, n, rows), rng.integers(0, n, rows))


@pytest.mark.parametrize("hub", [254, 255, 256, 257, 600])
def test_degrees_around_the_counted_ones(ctx, hub):
    # hubs of equal degree, joined in a clique, with leaves of their own
    h = 6
    a, b = np.triu_indices(h, 1)
    leaves = hub - (h - 1)
    src = np.concatenate([a, np.repeat(np.arange(h), leaves)])
    dst = np.concatenate([b, h + np.arange(h * leaves)])
    perm = graphgen.permutation(h + h * leaves, seed=hub, stream=1)
    check(ctx, h + h * leaves, perm[src], perm[dst])


@pytest.mark.parametrize("sizes", [[31, 32, 33], [34, 64, 66], [3, 4, 5, 150, 170]])
def test_out_lists_around_the_mixed_limit(ctx, sizes):
    # a clique K_s has out-lists of every length below s: runs of heads on
    # both sides of the staging limit, and walks longer than 128 entries
    n = 4000
    src, dst = graphgen.er(n, 9000, seed=sizes[0])
    perm = graphgen.permutation(n, seed=sizes[0], stream=1)
    check(ctx, n, *graphgen.add_cliques(src, dst, perm[: sum(sizes)], sizes))


@pytest.mark.parametrize("rows", [SMALL_ROWS, SMALL_ROWS + 1])
@pytest.mark.parametrize("kind", ["rmat", "random"])
def test_largest_size_and_one_more(ctx, general, rows, kind):
    if kind == "rmat":
        n, (s, d) = 1 << 18, graphgen.rmat_raw_cuda(18, rows, seed=5)
    else:
        n, g = SMALL_ROWS, torch.Generator(device="cuda").manual_seed(5)
        s = torch.randint(0, n, (rows,), dtype=torch.int32, generator=g, device="cuda")
        d = torch.randint(0, n, (rows,), dtype=torch.int32, generator=g, device="cuda")
    a, b = run(ctx, n, s, d), run(general, n, s, d)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]) and a[2] == b[2]
    assert ctx.stats()["triangles"] == general.stats()["triangles"]


def test_small_batch_and_bad_ids(ctx):
    from paper_1205_6693_gb300 import truss as T
    G = 30
    ns, off, src, dst = graphgen.batch(G)
    assert off[-1] <= SMALL_ROWS
    s, d = torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda()
    sup, tr = torch.empty_like(s), torch.empty_like(s)
    kmax = torch.empty(G, dtype=torch.int32, device="cuda")
    ctx.decompose_batch(ns, off, s, d, sup, tr, kmax)
    sup, tr, kmax = sup.cpu().numpy(), tr.cpu().numpy(), kmax.cpu().numpy()
    for g in range(G):
        a, b = off[g], off[g + 1]
        ref = oracle.truss(int(ns[g]), src[a:b], dst[a:b])
        assert np.array_equal(sup[a:b], ref.support) and np.array_equal(tr[a:b], ref.truss)
        assert kmax[g] == ref.kmax
    # an id beyond its own graph is refused though it lies in the union
    bad = src.copy()
    bad[off[3]] = ns[3]
    sb = torch.from_numpy(bad).cuda()
    with pytest.raises(T.TrussError) as ei:
        ctx.decompose_batch(ns, off, sb, d, torch.empty_like(s), torch.empty_like(s))
    assert ei.value.code == T.TRUSS_EINVAL


@pytest.mark.parametrize("name", ["empty graphs", "one graph", "too wide to rank by graph"])
def test_batch_ranked_by_graph_on_the_general_path(general, name):
    # vertices ordered by (graph, degree, id), and by (degree, id) where graph
    # number and degree do not fit one word; empty graphs at both ends
    sizes = {"empty graphs": [0, 0, 700, 0, 1, 2, 3, 90, 0], "one graph": [500],
             "too wide to rank by graph": [60] * 2047 + [1 << 21] + [60] * 10}[name]
    rng = np.random.default_rng(3)
    n = np.array(sizes, np.int64)
    rows = np.where(n > 1, np.minimum(4 * n, 3000), 0)
    off = np.concatenate([[0], np.cumsum(rows)]).astype(np.int64)
    g = np.repeat(np.arange(len(n)), rows)
    # ends drawn from the first 300 vertices: graphs dense in triangles
    src, dst = (np.minimum((rng.random(len(g)) * np.minimum(n[g], 300)).astype(np.int32),
                           n[g] - 1).astype(np.int32) for _ in range(2))
    s, d = torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda()
    sup, tr = torch.full_like(s, -7), torch.full_like(s, -7)
    kmax = torch.full((len(n),), -7, dtype=torch.int32, device="cuda")
    general.decompose_batch(n, off, s, d, sup, tr, kmax)
    sup, tr, kmax = sup.cpu().numpy(), tr.cpu().numpy(), kmax.cpu().numpy()
    for i in range(len(n)):
        a, b = off[i], off[i + 1]
        if a == b:
            assert kmax[i] == 0
            continue
        ref = oracle.truss(int(n[i]), src[a:b], dst[a:b])
        assert np.array_equal(sup[a:b], ref.support) and np.array_equal(tr[a:b], ref.truss)
        assert kmax[i] == ref.kmax


def _give_up_graphs():
    s, d = graphgen.rmat_raw(13, 60_001, seed=8)
    yield "rmat", 1 << 13, s, d
    yield "tiny", *graphgen.tiny()


@pytest.mark.parametrize("build,offsets", [("1", None), ("-1", None), (None, "-1"), (None, "1")])
def test_general_path_when_the_blocks_cannot_meet(ctx, monkeypatch, build, offsets):
    # limits that run out in the build's launch, or in the one after the walk of
    # a graph that was built in one launch: the general path takes over there
    graphs = list(_give_up_graphs())
    want = {}
    for name, n, s, d in graphs:
        ds, dd = torch.from_numpy(s).cuda(), torch.from_numpy(d).cuda()
        ctx.decompose(n, ds, dd, torch.empty_like(ds), torch.empty_like(ds))
        want[name] = ctx.stats()["launches"]
    G = 30
    ns, off, src, dst = graphgen.batch(G)
    sb, db = torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda()
    ref = [torch.empty_like(sb), torch.empty_like(sb),
           torch.empty(G, dtype=torch.int32, device="cuda")]
    ctx.decompose_batch(ns, off, sb, db, *ref)
    if build:
        monkeypatch.setenv("TRUSS_SMALL_BUILD_WAIT_NS", build)
    if offsets:
        monkeypatch.setenv("TRUSS_SMALL_OFFSETS_WAIT_NS", offsets)
    for name, n, s, d in graphs:
        check(ctx, n, s, d)
        ds, dd = torch.from_numpy(s).cuda(), torch.from_numpy(d).cuda()
        ctx.decompose(n, ds, dd, torch.empty_like(ds), torch.empty_like(ds))
        if "-1" in (build, offsets):  # within 1 ns, or 16 polls, the blocks may meet
            assert ctx.stats()["launches"] > want[name]
    got = [torch.full_like(x, -7) for x in ref]
    ctx.decompose_batch(ns, off, sb, db, *got)
    assert all(torch.equal(a, b) for a, b in zip(got, ref))
    monkeypatch.undo()
    for name, n, s, d in graphs:
        check(ctx, n, s, d)
        assert ctx.stats()["launches"] <= want[name]


def both(ctx, general, n, s, d):
    a, b = run(ctx, n, s, d), run(general, n, s, d)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]) and a[2] == b[2]
    return ctx.stats()["launches"], general.stats()["launches"]


@pytest.mark.parametrize("length", [383, 384, 385, 511, 512, 513, 1024, 1025])
def test_long_out_lists(ctx, general, length):
    # `length` heads, each joined to length + 40 tails and some to one another:
    # a tail's list holds every head; two such parts, apart in the ids
    n, parts = 100_000, []
    for k in range(2):
        o = k * 4000
        a = np.repeat(np.arange(length) + o, length + 40)
        b = np.tile(np.arange(length + 40) + 2000 + o, length)
        ex, ey = graphgen.er(length, 2000, seed=length + k)
        parts += [(a, b), (ex + o, ey + o)]
    perm = graphgen.permutation(n, seed=length, stream=1)
    src, dst = (perm[np.concatenate(x)].astype(np.int32) for x in zip(*parts))
    order = np.random.default_rng(length).permutation(len(src))
    for rows in (np.arange(len(src)), order):  # a tail's edges together, and scattered
        s, d = torch.from_numpy(src[rows]).cuda(), torch.from_numpy(dst[rows]).cuda()
        few, many = both(ctx, general, n, s, d)
        assert few < many  # the launches of support alone: the small path was taken


def test_longest_out_list(ctx):
    # K_2290 fills the rows: its first vertex has the longest list there can be
    k, n = 2290, 30_000
    a = torch.triu_indices(k, k, 1, device="cuda").to(torch.int32)
    s, d = a[0].contiguous(), a[1].contiguous()
    assert s.numel() <= SMALL_ROWS
    sup = torch.full_like(s, -7)
    ctx.support(n, s, d, sup)
    assert ctx.stats()["launches"] < 10
    assert bool((sup == k - 2).all())


@pytest.mark.parametrize("name", ["hub", "four hubs in turn", "one edge", "runs of an edge",
                                  "three edges in turn"])
def test_rows_that_share_a_counter_or_a_slot(ctx, name):
    # neighbouring lanes with the same end, or the same edge, and lanes apart
    k = 5000
    i = np.arange(k)
    src, dst = {"hub": (np.zeros(k, int), i), "four hubs in turn": (i % 4, i + 4),
                "one edge": (np.ones(k, int), np.full(k, 7)),
                "runs of an edge": (i // 40, i // 40 + 1),
                "three edges in turn": (i % 3, (i + 1) % 3)}[name]
    n = 6000
    es, ed = graphgen.er(300, 2000, seed=1)
    src, dst = np.concatenate([src, es]), np.concatenate([dst, ed])
    flip = np.random.default_rng(2).random(len(src)) < 0.5
    check(ctx, n, np.where(flip, dst, src), np.where(flip, src, dst))


@pytest.mark.parametrize("n,rows,small", [
    (1 << 10, 1 << 20, True), (1 << 10, (1 << 20) + 1, False),
    (1 << 14, 1 << 21, True), (1 << 14, (1 << 21) + 1, False)])
def test_densest_rows_taken_and_one_more(ctx, general, n, rows, small):
    g = torch.Generator(device="cuda").manual_seed(6)
    s, d = (torch.randint(0, n, (rows,), dtype=torch.int32, generator=g, device="cuda")
            for _ in range(2))
    few, many = both(ctx, general, n, s, d)
    assert few < many if small else few == many


@pytest.mark.parametrize("spare", [0, 1])
def test_batch_of_as_many_vertices_as_rows(general, spare):
    # ranked graph by graph up to there, in one order with a vertex more
    G, rows = 60, 200
    n = np.full(G, rows, np.int64)
    n[-1] += spare
    off = np.arange(G + 1, dtype=np.int64) * rows
    rng = np.random.default_rng(spare)
    src, dst = (rng.integers(0, 40, G * rows).astype(np.int32) for _ in range(2))
    s, d = torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda()
    sup, tr = torch.full_like(s, -7), torch.full_like(s, -7)
    general.decompose_batch(n, off, s, d, sup, tr)
    sup, tr = sup.cpu().numpy(), tr.cpu().numpy()
    for i in range(G):
        a, b = off[i], off[i + 1]
        ref = oracle.truss(int(n[i]), src[a:b], dst[a:b])
        assert np.array_equal(sup[a:b], ref.support) and np.array_equal(tr[a:b], ref.truss)
