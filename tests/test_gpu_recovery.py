"""What a handle is worth after one of its calls has failed, and failures that
only a later call would meet.

* bgl_components on a graph that has components rebuilds their arrays in
  place: a call that fails partway (a refused allocation) leaves the graph
  without components, so that the calls that need them return BGL_ESTATE
  until bgl_components has succeeded again."""
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
