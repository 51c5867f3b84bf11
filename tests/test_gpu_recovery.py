"""What a handle is worth after one of its calls has failed, and failures that
only a later call would meet.

* bgl_components on a graph that has components rebuilds their arrays in
  place: a call that fails partway (a refused allocation) leaves the graph
  without components, so that the calls that need them return BGL_ESTATE
  until bgl_components has succeeded again.
* A serving worker keeps its k-hop scratch between requests: after a request
  that a refused allocation ended, while the scratch was made or grown, the
  next requests get the same neighbourhoods and layouts as ever.
* The radix sorts of the graph build, the components and the assembly wait
  for each other's tiles, with a bound.  With BGL_TEST_SORT_STALL=1 the first
  tile withholds its counts and the waits on it give up after 4,096 polls: the
  call returns BGL_ETIMEOUT before a sorted value indexes anything (in each of
  the sorts, inputs of two tiles and more), and the same call without the aid
  gives what it gave before."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

ENOMEM, ETIMEOUT, ESTATE = -2, -4, -6


def _bgl():
    import paper_2403_03504_gb300 as bgl
    return bgl


@pytest.fixture(scope="module")
def ctx():
    c = _bgl().Context(0)
    yield c
    c.close()


def _forest(ctx, seed, comps, lo, hi):
    sizes, u, v = synth.forest(seed, comps, lo, hi)
    return _bgl().Graph.from_edges(ctx, int(sizes.sum()), u, v)


def _refused(ctx, call, status):
    with pytest.raises(_bgl().BglError) as e:
        call()
    assert e.value.status == status, e.value


def test_failed_components_leave_the_graph_without_any(ctx):
    bgl = _bgl()
    g = _forest(ctx, 3, 40, 3.0, 300.0)
    p = bgl.params(seed=2, fa2_iters=3, kk_sweeps=3)
    g.components(labels=False)
    want = g.layout(p)
    refused = 0
    for after in range(64):
        ctx.debug_fail_alloc(after)
        try:
            g.components(labels=False)
        except bgl.BglError as e:
            assert e.status == ENOMEM
            ctx.debug_fail_alloc(-1)
            _refused(ctx, lambda: g.layout(p, out=np.empty_like(want)), ESTATE)
            g.components(labels=False)
            assert np.array_equal(g.layout(p), want), after
            refused += 1
        else:
            break
    ctx.debug_fail_alloc(-1)
    assert refused >= 15                 # every allocation of the call was refused once
    g.destroy()


def test_serving_worker_goes_on_after_a_refused_allocation(ctx):
    bgl = _bgl()
    n = 3000
    u, v = np.arange(n - 1), np.arange(1, n)
    hub = np.arange(2, 1300)                                # node 0: more than 1,024 entries
    g = bgl.Graph.from_edges(ctx, n, np.concatenate([u, np.zeros_like(hub)]), np.concatenate([v, hub]))
    p = bgl.params(seed=4, fa2_iters=1, kk_sweeps=1)
    # (the visit list of the third and fourth is larger than those before)
    requests = [(2500, 3, 10), (2000, 5, 20), (1290, 2, n), (0, 1, n), (2500, 3, 10)]

    def serve(after):
        ctx.debug_fail_alloc(after)
        srv = bgl.Server(g, slots=1)
        ctx.debug_fail_alloc(-1)
        out = []
        for seed, hops, cap in requests:
            rid = srv.submit(seed, hops, p, cap)
            status, k, _, _ = srv.wait(rid)
            out.append(srv.fetch(rid, k) if status == 0 else status)
        srv.close()
        return out

    want = serve(-1)
    for (seed, hops, cap), w in zip(requests, want):
        assert np.array_equal(w[0], g.khop(seed, hops, cap)[0])
    after, refused = 0, len(requests)
    while refused:
        refused = 0
        for w, got in zip(want, serve(after)):
            if isinstance(got, int):
                assert got == ENOMEM
                refused += 1
            else:
                assert np.array_equal(got[0], w[0]) and np.array_equal(got[1], w[1]), after
        assert refused <= 1
        after += 1
    assert 100 < after < 2000            # every allocation of the five requests was refused once
    g.destroy()


def _build(ctx):
    tx = synth.tx_lists(**dict(synth.C1, n_tx=3000))
    g = _bgl().Graph.build(ctx, tx.in_off, tx.in_addr, tx.out_off, tx.out_addr)
    out = [g.addresses(), *g.edges(), *g.csr()]
    g.destroy()
    return out


def _from_edges(ctx, n, u, v):
    g = _bgl().Graph.from_edges(ctx, n, u, v)
    out = [*g.edges(), *g.csr()]
    g.destroy()
    return out


def _pairs(comps, size):
    """Paths of `size` nodes."""
    u = np.setdiff1d(np.arange(comps * size), np.arange(1, comps + 1) * size - 1)
    return comps * size, u, u + 1


def _components(ctx, g):
    labels, n_comp = g.components()
    return [labels, np.array(n_comp), *g.component_nodes()]


def _assembled(ctx, g, out):
    return [g.layout(_bgl().params(seed=1, kk_sweeps=2, assemble=1), out=out)]


@pytest.mark.parametrize("sort", ["addresses", "directed edges", "undirected edges", "component sizes", "nodes",
                                  "assembly order"])
def test_a_sort_that_gives_up_is_reported_before_its_output_is_used(ctx, monkeypatch, sort):
    bgl = _bgl()
    g, out = None, np.zeros((0, 2), np.float32)
    if sort == "addresses":
        call = lambda: _build(ctx)
    elif sort == "directed edges":
        rng = np.random.default_rng(1)
        u, v = rng.integers(0, 9000, (2, 20000))
        call = lambda: _from_edges(ctx, 9000, u, v)
    elif sort == "undirected edges":                # one tile of edges, two of both directions
        n, u, v = _pairs(1, 3001)
        call = lambda: _from_edges(ctx, n, u, v)
    else:
        n, u, v = _pairs(*((2, 4000) if sort == "nodes" else (5000, 2)))
        g = bgl.Graph.from_edges(ctx, n, u, v)
        if sort == "assembly order":
            g.components(labels=False)
            out = np.zeros((n, 2), np.float32)
            call = lambda: _assembled(ctx, g, out)
        else:
            call = lambda: _components(ctx, g)
    want = [a.copy() for a in call()]
    out[:] = 7.5
    monkeypatch.setenv("BGL_TEST_SORT_STALL", "1")
    for _ in range(2):
        _refused(ctx, call, ETIMEOUT)
    assert np.all(out == 7.5)
    if g is not None and sort != "assembly order":
        _refused(ctx, lambda: g.layout(bgl.params()), ESTATE)
    monkeypatch.delenv("BGL_TEST_SORT_STALL")
    got = call()
    assert len(got) == len(want) and all(np.array_equal(a, b) for a, b in zip(got, want))
    if g is not None:
        g.destroy()
