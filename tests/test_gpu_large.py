"""Dispatch rules whose line lies above the sizes of the other tests.

* bgl_fa2_iteration_noalloc: from 262,144 nodes on a block has two targets a
  thread and all stages; below, the stages are spread over a cluster.  Forces
  against the oracle on sampled nodes, to the 1e-5 of the sum of the terms'
  sizes that the exact forces are held to elsewhere.
* k-hop neighbourhoods in a resident graph of 2^24 nodes and more come from a
  sort of the visited nodes, in smaller ones from scans over the marks of all:
  equal to the oracle's on both sides of the line.  A sort that gives up
  (BGL_TEST_SORT_STALL=1, see test_gpu_recovery.py) is reported.
  Either way a hop may meet several hubs.
* The partial sums of exact components above 8,192 nodes take at most 512 MiB
  a run, whatever their number (64 bytes a node below), with the same bits as
  when a component has them all to itself; and a server's footprint estimate
  bounds what a request of one such component takes.
* Kamada-Kawai classes of 608 blocks and more fill the chip, and beside them the
  FMM of up to 32,768 points has its separate sort; beside classes the exact
  iterations' kernels ask for their shared-memory split: every component gets
  the layout that it gets alone."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _bgl():
    import paper_2403_03504_gb300 as bgl
    return bgl


@pytest.fixture(scope="module")
def ctx():
    c = _bgl().Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n", [262143, 262144, 262273, 262401])
def test_noalloc_forces_of_large_components(ctx, n):
    """One node short of the line, on it, and last blocks of 129 and 257 - 256
    targets; a hub of 3,000 entries and, last, a node of one."""
    import torch
    bgl = _bgl()
    u, v = np.arange(n - 1), np.arange(1, n)
    hub = np.arange(2, 3000)
    g = bgl.Graph.from_edges(ctx, n, np.concatenate([u, np.zeros_like(hub)]), np.concatenate([v, hub]))
    off, adj = g.csr()
    g.destroy()
    mass = np.diff(off) + 1.0
    xy = synth.points(n, n, "uniform", scale=200.0)
    dev = [torch.from_numpy(a).cuda() for a in (off, adj, mass.astype(np.float32), xy)]
    f, fp = torch.zeros(n, 2, device="cuda"), torch.zeros(n, 2, device="cuda")
    sg = torch.ones(1, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    ctx.fa2_iteration_noalloc(n, dev[0], dev[1], dev[2], dev[3], fp, f, sg, bgl.params(repulsion=bgl.REP_EXACT))
    ctx.sync()
    tg = np.unique(np.concatenate([np.random.default_rng(n).choice(n, 200, replace=False),
                                   [0, 1, 2999, 3000, 127, 128, 255, 256, n - 130, n - 129, n - 2, n - 1]]))
    o = oracle.fa2_forces(xy[:, 0], xy[:, 1], mass, off, adj, targets=tg)
    ref = o["frep"] + o["fatt"] + o["fgrav"]
    assert np.max(np.hypot(*(f.cpu().numpy()[tg] - ref).T) / o["sabs"]) <= 1e-5


@pytest.mark.parametrize("n", [(1 << 24) - 1, 1 << 24])
def test_khop_in_a_large_graph(ctx, monkeypatch, n):
    """A path whose node 0 is also joined to 2..1401 and to the last nodes."""
    bgl = _bgl()
    u, v = np.arange(n - 1, dtype=np.int32), np.arange(1, n, dtype=np.int32)
    hub = np.concatenate([np.arange(2, 1402), np.arange(n - 40, n)]).astype(np.int32)
    g = bgl.Graph.from_edges(ctx, n, np.concatenate([u, np.zeros_like(hub)]), np.concatenate([v, hub]))
    off, adj = g.csr()
    for seed, hops in ((0, 0), (0, 1), (n - 1, 2), (700, 2), (n // 2, 1), (n // 2, 2500), (n - 50, 11)):
        ids, edges = oracle.khop(off, adj, seed, hops)
        got = g.khop(seed, hops, 1 << 30)
        assert np.array_equal(got[0], ids)
        assert sorted(zip(np.minimum(got[1], got[2]).tolist(), np.maximum(got[1], got[2]).tolist())) == edges
        assert np.array_equal(g.khop(seed, hops, len(ids))[0], ids)
        if len(ids) > 1:
            assert g.khop(seed, hops, len(ids) - 1) is None
    if n >= 1 << 24:
        monkeypatch.setenv("BGL_TEST_SORT_STALL", "1")
        with pytest.raises(bgl.BglError) as e:
            g.khop(n // 2, 2500, n)                  # 5,001 nodes: two tiles
        assert e.value.status == -4
        monkeypatch.delenv("BGL_TEST_SORT_STALL")
        assert len(g.khop(n // 2, 2500, n)[0]) == 5001
    g.destroy()


def _trees(comps, n, arity):
    """Trees of n nodes, the parent of a tree's node i being (i - 1) // arity."""
    i = np.arange(1, n)
    base = np.arange(comps)[:, None] * n
    return comps * n, (base + (i - 1) // arity).ravel(), (base + i).ravel()


def test_partial_sums_of_many_exact_components_are_bounded():
    import torch
    bgl = _bgl()
    comps, size = 30, 60000
    n, u, v = _trees(comps, size, 3)
    with bgl.Context(0) as c:
        g = bgl.Graph.from_edges(c, n, u, v)
        g.components(labels=False)
        p = bgl.params(seed=5, fa2_iters=1, repulsion=bgl.REP_EXACT)
        free = torch.cuda.mem_get_info()[0]
        xy = g.layout(p)
        taken = free - torch.cuda.mem_get_info()[0]
        # positions, forces and tiles: some 70 bytes a node; unbounded partial sums would take 470 more
        assert taken <= (512 << 20) + 128 * n, taken
        off, _, nodes = g.component_nodes()
        for k in (0, comps - 1):
            ids = nodes[off[k]:off[k + 1]]
            x, y = oracle.init_positions(5, ids)
            alone, _ = g.fa2_step(k, p, 1, np.stack([x, y], 1).astype(np.float32))
            assert np.array_equal(alone, xy[ids])
        g.destroy()


def test_footprint_estimate_bounds_an_exact_request(ctx):
    bgl = _bgl()
    n, u, v = _trees(1, 65536, 50)
    g = bgl.Graph.from_edges(ctx, n, u, v)
    srv = bgl.Server(g, slots=1)
    for size, hops in ((n, 3), (2551, 2)):
        status, k, _, nbytes = srv.wait(srv.submit(0, hops, bgl.params(fa2_iters=1, repulsion=bgl.REP_EXACT)))
        assert status == 0 and k == size
        assert 0 < nbytes[1] <= nbytes[0]
    srv.close()
    g.destroy()


@pytest.mark.parametrize("rep,size", [("exact", 3000), ("fmm", 10000)])
def test_layout_beside_classes_that_fill_the_chip(ctx, rep, size):
    """20,000 components of 3 to 50 nodes (some 900 blocks) beside a large one."""
    bgl = _bgl()
    sizes, u, v = synth.forest(8, 20000, 3.0, 50.0)
    base = int(sizes.sum())
    n, gu, gv = _trees(1, size, 3)
    g = bgl.Graph.from_edges(ctx, base + n, np.concatenate([u, base + gu]), np.concatenate([v, base + gv]))
    g.components(labels=False)
    p = bgl.params(seed=6, fa2_iters=30, kk_sweeps=20, ksmax=0.05,
                   repulsion=bgl.REP_EXACT if rep == "exact" else bgl.REP_FMM)
    xy = g.layout(p)
    x, y = oracle.init_positions(6, np.arange(base, base + n))
    alone, _ = g.fa2_step(0, p, 30, np.stack([x, y], 1).astype(np.float32))
    assert np.array_equal(xy[base:], alone)
    p.fa2_iters = 0                                  # the classes without iterations beside them
    assert np.array_equal(xy[:base], g.layout(p)[:base])
    g.destroy()


@pytest.mark.parametrize("hops", [1, 2, 3, 4])
def test_khop_over_several_hubs_in_several_hops(ctx, hops):
    """Hubs of 1,100 to 5,100 entries (more than a block's 1,024), two of them
    met in the first hop and two more in each of the next ones."""
    bgl = _bgl()
    rng = np.random.default_rng(3)
    n, hubs = 30000, 8
    degree = 1100 + 570 * np.arange(hubs)
    u = np.concatenate([np.repeat(np.arange(hubs), degree), np.arange(hubs - 2), [hubs, hubs]])
    v = np.concatenate([rng.integers(hubs + 1, n, degree.sum()), np.arange(2, hubs), [0, 1]])
    g = bgl.Graph.from_edges(ctx, n, u, v)
    off, adj = g.csr()
    ids, edges = oracle.khop(off, adj, hubs, hops)
    got = g.khop(hubs, hops, n)
    assert np.array_equal(got[0], ids)
    assert sorted(zip(np.minimum(got[1], got[2]).tolist(), np.maximum(got[1], got[2]).tolist())) == edges
    g.destroy()
