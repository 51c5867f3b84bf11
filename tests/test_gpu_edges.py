"""Edges of the kernels' tiles, splits and dispatch rules: the exact sum (target
tiles of 128 and 256, source stages of 1,024, one block for all stages above
65,536 nodes, attraction by lane, warp and block), the allocation-free
iteration (cluster sizes 1 to 8), the FMM's small-tree paths (cluster sort up
to 32,768 points, rows of leaves, trees of up to 128 tiles), the radix sorts of
the graph build (tiles of 4,096 keys) and the k-hop kernels (hubs, many hops,
caps).  Against the oracle at the tolerances of the other tests: exact forces
1e-5 of the sum of the terms' sizes, FMM forces within the truncation ceiling
of their order (floor 2e-5), whole numbers equal."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

RHO = 2 ** 0.5 / (4 - 2 ** 0.5)


def _bgl():
    import paper_2403_03504_gb300 as bgl
    return bgl


@pytest.fixture(scope="module")
def ctx():
    c = _bgl().Context(0)
    yield c
    c.close()


def _hub_graph(n, hub_degree):
    """A path of n nodes and a hub (node 0) joined to hub_degree others."""
    u = np.arange(n - 1, dtype=np.int32)
    v = u + 1
    k = np.arange(2, min(n, hub_degree + 2), dtype=np.int32)
    return np.concatenate([u, np.zeros(len(k), np.int32)]), np.concatenate([v, k])


def _component(ctx, n, u, v):
    g = _bgl().Graph.from_edges(ctx, n, u, v)
    g.components(labels=False)
    off, adj = g.csr()
    return g, off, adj, np.diff(off) + 1.0


@pytest.mark.parametrize("n,hub", [(2, 0), (127, 9), (128, 120), (129, 128), (257, 129), (1023, 40), (1024, 700),
                                   (1025, 1000), (2049, 2048), (5000, 4500), (65536, 300), (65537, 300)])
def test_exact_forces_at_tile_and_stage_edges(ctx, n, hub):
    bgl = _bgl()
    g, off, adj, mass = _component(ctx, n, *_hub_graph(n, hub))
    xy = synth.points(n, n, "uniform", scale=40.0)
    f = g.fa2_forces(0, bgl.params(repulsion=bgl.REP_EXACT), xy).astype(np.float64)
    tg = np.arange(n) if n <= 5000 else np.random.default_rng(n).choice(n, 600, replace=False)
    tg[0] = 0
    o = oracle.fa2_forces(xy[:, 0], xy[:, 1], mass, off, adj, 1.0, 1.0, targets=tg)
    ref = o["frep"] + o["fatt"] + o["fgrav"]
    assert np.max(np.hypot(*(f[tg] - ref).T) / o["sabs"]) <= 1e-5
    g.destroy()


def test_exact_component_is_the_same_alone_and_among_many(ctx):
    """Many components take two targets a lane, one takes one: the same bits."""
    bgl = _bgl()
    sizes, u, v = synth.forest(5, 220, 1500.0, 5000.0)
    g = bgl.Graph.from_edges(ctx, int(sizes.sum()), u, v)
    g.components(labels=False)
    off, _, nodes = g.component_nodes()
    p = bgl.params(seed=3, fa2_iters=3, repulsion=bgl.REP_EXACT, kk_max_nodes=50)
    xy = g.layout(p)
    for c in (0, 219):
        ids = nodes[off[c]:off[c + 1]]
        x, y = oracle.init_positions(3, ids)
        alone, _ = g.fa2_step(c, p, 3, np.stack([x, y], 1).astype(np.float32))
        assert np.array_equal(alone, xy[ids])
    g.destroy()


@pytest.mark.parametrize("n,hub", [(1, 0), (2, 0), (128, 60), (129, 100), (1024, 9), (1025, 1000), (7168, 7000),
                                   (7169, 33), (8193, 50)])
def test_noalloc_forces_at_cluster_edges(ctx, n, hub):
    import torch
    bgl = _bgl()
    u, v = _hub_graph(n, hub) if n > 1 else (np.zeros(0, np.int32), np.zeros(0, np.int32))
    g, off, adj, mass = _component(ctx, n, u, v)
    xy = synth.points(n, n, "uniform", scale=30.0)
    dev = [torch.from_numpy(a).cuda() for a in (off, np.append(adj, 0).astype(np.int32), mass.astype(np.float32), xy)]
    f, fp = torch.zeros(n, 2, device="cuda"), torch.zeros(n, 2, device="cuda")
    sg = torch.ones(1, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    ctx.fa2_iteration_noalloc(n, dev[0], dev[1], dev[2], dev[3], fp, f, sg, bgl.params(repulsion=bgl.REP_EXACT))
    ctx.sync()
    o = oracle.fa2_forces(xy[:, 0], xy[:, 1], mass, off, adj)
    ref = o["frep"] + o["fatt"] + o["fgrav"]
    assert np.max(np.hypot(*(f.cpu().numpy() - ref).T) / np.maximum(o["sabs"], 1e-30)) <= 1e-5
    if n > 1:
        assert float(sg.cpu()[0]) == 1.0        # swing equals traction when F_{-1} = 0
    g.destroy()


@pytest.mark.parametrize("kind", ["uniform", "clustered"])
@pytest.mark.parametrize("n", [65, 4095, 4096, 4097, 12289, 32768, 32769, 131072, 131073])
def test_fmm_at_small_tree_edges(ctx, n, kind):
    bgl = _bgl()
    g, off, adj, mass = _component(ctx, n, *_hub_graph(n, 0))
    xy = synth.points(n, n, kind, scale=25.0)
    p = bgl.params(repulsion=bgl.REP_FMM, fmm_p=8)
    tg = np.random.default_rng(n).choice(n, min(n, 300), replace=False)
    o = oracle.fa2_forces(xy[:, 0], xy[:, 1], mass, off, adj, 1.0, 1.0, targets=tg)
    ceiling = max(2 * (1 + RHO) * RHO ** 9 / (1 - RHO), 2e-5)
    f = g.fa2_repulsion(0, p, xy)
    assert np.max(np.hypot(*(f[tg] - o["frep"]).T) / o["srep"]) <= ceiling
    # an iteration whose sort skips passes, and one that follows it, stay within it as well
    st = g.fmm_stats(0, p, xy, reps=2)
    assert st["sortmode_rel_diff"] <= 1e-5
    g.destroy()


@pytest.mark.parametrize("m", [1, 4095, 4096, 4097, 8193, 70000])
def test_graph_of_edges_at_sort_tile_edges(ctx, m):
    bgl = _bgl()
    rng = np.random.default_rng(m)
    n = max(2, m // 3)
    u, v = rng.integers(0, n, m).astype(np.int32), rng.integers(0, n, m).astype(np.int32)
    g = bgl.Graph.from_edges(ctx, n, u, v)
    src, dst = g.edges()
    key = np.unique(u.astype(np.int64) * n + v)
    assert np.array_equal(src, key // n) and np.array_equal(dst, key % n)
    both = np.concatenate([u, v]).astype(np.int64) * n + np.concatenate([v, u])
    both = np.unique(both[np.concatenate([u != v, u != v])])
    off, adj = g.csr()
    assert np.array_equal(adj, both % n)
    assert np.array_equal(off, np.searchsorted(both // n, np.arange(n + 1)))
    lab, nc = g.components()
    olab, onc = oracle.components(off, adj)
    assert nc == onc and np.array_equal(lab, olab)
    coff, clab, nodes = g.component_nodes()
    size = np.bincount(olab, minlength=n)
    order = np.lexsort((np.flatnonzero(size), -size[size > 0]))
    assert np.array_equal(np.diff(coff), size[size > 0][order]) and np.array_equal(clab, np.flatnonzero(size)[order])
    assert np.array_equal(np.sort(nodes), np.arange(n))
    g.destroy()


@pytest.mark.parametrize("seed,hops", [(0, 0), (0, 1), (0, 2), (1, 1), (3999, 7), (3999, 9), (3999, 40), (1500, 3)])
def test_khop_hubs_many_hops_and_caps(ctx, seed, hops):
    """A path of 4,000 nodes whose node 0 is also joined to 2..1401 (a hub of
    more than 1,024 entries)."""
    bgl = _bgl()
    n = 4000
    u, v = _hub_graph(n, 1400)
    g = bgl.Graph.from_edges(ctx, n, u, v)
    off, adj = g.csr()
    ids, edges = oracle.khop(off, adj, seed, hops)
    got = g.khop(seed, hops, 1 << 30)
    assert np.array_equal(got[0], ids)
    assert sorted(zip(np.minimum(got[1], got[2]).tolist(), np.maximum(got[1], got[2]).tolist())) == edges
    assert np.array_equal(g.khop(seed, hops, len(ids))[0], ids)
    if len(ids) > 1:
        assert g.khop(seed, hops, len(ids) - 1) is None
    g.destroy()


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("n", [255, 2048, 2049, 16384, 16385])
def test_noalloc_speed_and_update_at_tile_and_cluster_edges(ctx, n, variant):
    """Up to eight tiles of 2,048 nodes the sums and the update are one cluster
    kernel, above it two kernels: s_G of the second call against the FP64 sums
    of the GPU's own forces (1e-5), positions against bgl_fa2_step (1e-3 of the
    diagonal)."""
    import torch
    bgl = _bgl()
    g, off, adj, mass = _component(ctx, n, *_hub_graph(n, 20))
    xy = synth.points(n, n, "uniform", scale=30.0)
    dev = [torch.from_numpy(a).cuda() for a in (off, adj, mass.astype(np.float32), xy)]
    f, fp = torch.zeros(n, 2, device="cuda"), torch.zeros(n, 2, device="cuda")
    sg = torch.ones(1, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    p = bgl.params(repulsion=bgl.REP_EXACT, swing_variant=variant)
    forces = []
    for _ in range(2):
        ctx.fa2_iteration_noalloc(n, dev[0], dev[1], dev[2], dev[3], fp, f, sg, p)
        ctx.sync()
        forces.append(f.cpu().numpy().astype(np.float64))
        assert np.array_equal(fp.cpu().numpy(), f.cpu().numpy())
    f1, f2 = forces
    w = mass if variant else np.ones(n)
    swg, trc = np.sum(w * np.hypot(*(f2 - f1).T)), np.sum((0.5 if variant else 1.0) * w * np.hypot(*(f2 + f1).T))
    first = 0.5 if variant else 1.0                 # of the first call, where swing equals traction
    assert float(sg.cpu()[0]) == pytest.approx(min(trc / swg, 1.5 * first), rel=1e-5)
    want, _ = g.fa2_step(0, p, 2, xy)
    err = np.max(np.hypot(*(dev[3].cpu().numpy() - want).T))
    assert err <= 1e-3 * np.hypot(*np.ptp(want, axis=0))
    g.destroy()
