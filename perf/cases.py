"""Performance cases of the layout library: the calls a program makes, over the range of graphs it makes them on.

Graphs are transaction graphs of the recipe that the tests and the benchmark use (inputs and outputs per transaction
geometric, two outputs with probability 0.7, 40 % of the endpoints reuse an address chosen by Zipf(1.2)), and forests
of random recursive trees with 10 % extra edges, drawn here with numpy from the case's seed.  Positions stand for a
layout under way: ForceAtlas2's gravity spreads the mass evenly over a disc of radius sqrt(kr M / kg), a transaction
anywhere in it and an address near the transaction that it first appears in ("disc"); or dense clusters of very
different widths, whose quadtree is deep and uneven ("clustered").

Sessions and layouts take ForceAtlas2's steps small (ksmax = 0.05), as the last iterations of a layout are: with the
default 10 any rounding grows tenfold an iteration, so that after a few nothing could be compared with anything.

kinds:
  noalloc   Context.fa2_iteration_noalloc on device arrays, `iters` calls on a run that goes on
  session   Graph.session_advance(iters) on a run that goes on, and its positions
  forces    Graph.fa2_forces, one evaluation with host arrays
  whole     transaction lists on the device to coordinates on the device: Graph.build_dev, components, layout_dev
  layout    Graph.layout_dev of a graph in memory: Kamada-Kawai on the small components, ForceAtlas2 on the others
  build     Graph.build from host arrays, components, and the CSR and labels read back
  khop      Graph.khop neighbourhoods of a graph in memory, what a serving program asks for first
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2403_03504_gb300 as bgl

STEP = 0.05
_device = {}


def _context():
    """The program's one context, on a stream of its own."""
    if not _device:
        _device["stream"] = torch.cuda.Stream()
        _device["ctx"] = bgl.Context(torch.cuda.current_device())
        _device["ctx"].set_stream(_device["stream"])
    return _device["ctx"]


# ------------------------------------------------------------------ graphs and positions (numpy, from the seed alone)


def _endpoints(n_tx):
    """The structure of a transaction graph: inputs and outputs per transaction, and of every endpoint in scan order its
    transaction and its address (numbered by creation)."""
    rng = np.random.default_rng(n_tx)
    n_in = np.minimum(rng.geometric(0.5, n_tx), 20)
    n_out = np.where(rng.random(n_tx) < 0.7, 2, np.minimum(rng.geometric(0.5, n_tx), 50))
    tx = np.repeat(np.arange(n_tx), n_in + n_out)
    new = rng.random(len(tx)) >= 0.4
    new[0] = True
    before = np.cumsum(new) - new
    # Zipf(1.2) over the creation ranks so far: the continuous law's inverse, rounded down
    zipf = np.floor((1.0 - rng.random(len(tx)) * (1.0 - (before + 1.0) ** -0.2)) ** -5.0).astype(np.int64)
    return n_in, n_out, tx, np.where(new, before, np.clip(zipf, 1, np.maximum(before, 1)) - 1)


def _forest(rng, n_comp, lo, hi):
    """Components of log-uniform sizes in [lo, hi]: random recursive trees and 10 % extra edges, their nodes numbered in
    an order of rng's: (n, u, v, component of every node)."""
    fix = np.random.default_rng([n_comp, int(lo), int(hi)])
    size = np.rint(np.exp(fix.uniform(math.log(lo), math.log(hi), n_comp))).astype(np.int64)
    base = np.cumsum(size) - size
    comp = np.repeat(np.arange(n_comp), size)
    local = np.arange(size.sum()) - base[comp]
    child = np.flatnonzero(local > 0)
    parent = base[comp[child]] + (fix.random(len(child)) * local[child]).astype(np.int64)
    extra = np.repeat(np.arange(n_comp), np.rint(0.1 * (size - 1)).astype(np.int64))
    eu = base[extra] + (fix.random(len(extra)) * size[extra]).astype(np.int64)
    ev = base[extra] + (fix.random(len(extra)) * size[extra]).astype(np.int64)
    keep = eu != ev
    name = rng.permutation(len(comp)).astype(np.int32)
    u, v = np.concatenate([parent, eu[keep]]), np.concatenate([child, ev[keep]])
    of = np.empty_like(comp)
    of[name] = comp
    return len(comp), name[u], name[v], of


def _positions(rng, kind, n_tx, home, mass):
    """A position (FP32) for every node of a transaction graph, in node-id order (home: each address's first
    transaction)."""
    n = n_tx + len(home)
    if kind == "clustered":
        k = max(1, n // 500)
        w = rng.pareto(1.2, k) + 1e-3
        lab = rng.choice(k, size=n, p=w / w.sum())
        scale = math.sqrt(float(mass.sum()))
        widths = scale * 10.0 ** rng.uniform(-3.0, -1.0, k)
        centre = rng.uniform(-scale, scale, (k, 2))
        return (centre[lab] + rng.normal(size=(n, 2)) * widths[lab, None]).astype(np.float32)
    # transactions and, behind each, the addresses that first appear in it, along a Hilbert curve that fills the square
    # around the disc, each node given an area in proportion to its mass; then the square mapped onto the disc
    place = rng.permutation(n_tx)
    order = np.argsort(np.concatenate([place, place[home]]) * 2 + (np.arange(n) >= n_tx), kind="stable")
    area = mass[order]
    at = np.empty(n)
    at[order] = (np.cumsum(area) - rng.uniform(0.3, 0.7, n) * area) / area.sum()
    q = _hilbert(at) + rng.normal(0.0, 0.2 / math.sqrt(n), (n, 2))
    a, b = 2.0 * q[:, 0] - 1.0, 2.0 * q[:, 1] - 1.0
    disc = np.stack([a * np.sqrt(1.0 - 0.5 * b * b), b * np.sqrt(1.0 - 0.5 * a * a)], 1)
    return (disc * math.sqrt(float(mass.sum()))).astype(np.float32)


def _hilbert(t, bits=16):
    """Points of the unit square on the Hilbert curve at parameters t in [0, 1)."""
    d = (np.clip(t, 0.0, 1.0 - 2.0 ** -40) * 4.0 ** bits).astype(np.int64)
    x, y = np.zeros(len(t), np.int64), np.zeros(len(t), np.int64)
    for k in range(bits):
        s = 1 << k
        rx, ry = 1 & (d >> 1), 1 & (d ^ (d >> 1))
        flip = (ry == 0) & (rx == 1)
        x, y = np.where(flip, s - 1 - x, x), np.where(flip, s - 1 - y, y)
        x, y = np.where(ry == 0, y, x) + s * rx, np.where(ry == 0, x, y) + s * ry
        d >>= 2
    return (np.stack([x, y], 1) + 0.5) / float(1 << bits)


class _Tx:
    """A transaction graph of a case in numpy: lists and positions, and its components and CSR for exact().  The number
    of transactions gives the structure, and so every size; the seed gives the order of the transactions (and with it
    every id), the address keys and the positions."""

    def __init__(self, case, seed):
        n_tx = self.n_tx = case["n_tx"]
        n_in, n_out, tx, addr = _endpoints(n_tx)
        rng = np.random.default_rng([seed, n_tx])
        place = rng.permutation(n_tx)
        order = np.argsort(place[tx], kind="stable")
        tx, addr = place[tx[order]], addr[order]
        back = np.argsort(place)
        n_in, n_out = n_in[back], n_out[back]
        # addresses by first appearance
        m, self.n_addr = len(tx), int(addr.max()) + 1
        first = np.empty(self.n_addr, np.int64)
        first[addr[::-1]] = np.arange(m)[::-1]
        appears = np.zeros(m, bool)
        appears[first] = True
        self.ids = (np.cumsum(appears) - 1)[first]
        addr = self.ids[addr]
        key = (addr.astype(np.uint64) + np.uint64(seed + 1)) * np.uint64(0x9E3779B97F4A7C15)
        key = (key ^ (key >> np.uint64(29))) * np.uint64(0xBF58476D1CE4E5B9)
        start = np.cumsum(n_in + n_out) - (n_in + n_out)
        is_in = np.arange(m) - start[tx] < n_in[tx]
        self.lists = [np.concatenate([[0], np.cumsum(n_in)]).astype(np.int64), key[is_in],
                      np.concatenate([[0], np.cumsum(n_out)]).astype(np.int64), key[~is_in]]
        self.n = n_tx + self.n_addr
        if case.get("where"):
            # distinct (transaction, address) pairs: the undirected edges
            pair = np.sort(tx * self.n_addr + addr)
            pair = pair[np.concatenate([[True], pair[1:] != pair[:-1]])]
            self.u, self.v = pair // self.n_addr, n_tx + pair % self.n_addr
            self.mass = 1.0 + np.bincount(self.u, minlength=self.n) + np.bincount(self.v, minlength=self.n)
            self.xy = _positions(rng, case["where"], n_tx, tx[appears], self.mass)

    def giant(self):
        """Node ids of the largest component (the one with the smallest id of equals), ascending."""
        lab = np.arange(self.n)
        u, v = self.u, self.v
        while True:
            m = np.minimum(lab[u], lab[v])
            if np.array_equal(m, lab[u]) and np.array_equal(m, lab[v]):
                break
            np.minimum.at(lab, lab[u], m)
            np.minimum.at(lab, lab[v], m)
            while not np.array_equal(lab, lab[lab]):
                lab = lab[lab]
        return np.flatnonzero(lab == np.argmax(np.bincount(lab)))

    def local(self, nodes):
        """(off, adj, mass, xy) of the component `nodes`, local ids in node order."""
        off, adj = _local_csr(self.n, self.u, self.v, nodes)
        return off, adj, self.mass[nodes], self.xy[nodes]


def _local_csr(n, u, v, nodes):
    """Undirected CSR of the component `nodes` in local ids, from edges of a graph of n nodes: duplicates and self-loops
    left out."""
    where = np.full(n, -1, np.int64)
    where[nodes] = np.arange(len(nodes))
    a, b = where[np.concatenate([u, v])], where[np.concatenate([v, u])]
    key = np.unique((a * len(nodes) + b)[(a >= 0) & (a != b)])
    off = np.zeros(len(nodes) + 1, np.int64)
    np.cumsum(np.bincount(key // len(nodes), minlength=len(nodes)), out=off[1:])
    return off, (key % len(nodes)).astype(np.int32)


def _params(case, **kw):
    for k in ("fmm_p", "leaf_size", "swing_variant", "kk_max_nodes", "fa2_iters"):
        if k in case:
            kw[k] = case[k]
    kw["repulsion"] = bgl.REP_FMM if case.get("repulsion") == "fmm" else bgl.REP_AUTO
    return bgl.params(ksmax=STEP, **kw)


# ------------------------------------------------------------------ the cases


def listed():
    return [
        # A loop on the layout of a day's small graph (1,000 transactions, giant component of some 2,900 nodes) in a
        # process that owns all device memory: four short kernels a call, latency and nothing else.
        dict(name="noalloc-1k-tx", kind="noalloc", n_tx=1000, where="disc", iters=4),
        # The same graph advanced by the 50 iterations that a metrics log takes at a time: below 8,192 nodes the default
        # is the exact sum.
        dict(name="session-1k-tx", kind="session", n_tx=1000, where="disc", iters=50),
        # Just over 8,192 nodes, where the default becomes the FMM: every kernel of its chain on a few blocks.
        dict(name="session-3.1k-tx-fmm", kind="session", n_tx=3100, where="disc", iters=50),
        # A mid-size graph at the high expansion order, with ForceAtlas2's weighted swing.
        dict(name="session-25k-tx-fmm-p16", kind="session", n_tx=25_000, where="disc", iters=10, fmm_p=16,
             swing_variant=1),
        # The benchmark's graph (200,000 transactions, giant component of some 560,000 nodes), default options.
        dict(name="session-200k-tx-fmm", kind="session", n_tx=200_000, where="disc", iters=10),
        # One evaluation of the forces of a clustered layout with host arrays, as an analysis of a layout asks for it:
        # uneven tree, long lists, odd size.
        dict(name="forces-61k-tx-clustered", kind="forces", n_tx=61_003, where="clustered", repulsion="fmm", fmm_p=12,
             leaf_size=48),
        # The largest: the giant component of 600,000 transactions (1.7 million nodes), beyond what the L2 holds.
        dict(name="session-600k-tx-fmm", kind="session", n_tx=600_000, where="disc", iters=6),
        # The whole call on an ordinary day's graph, default numbers of iterations and sweeps.
        dict(name="whole-10k-tx", kind="whole", n_tx=10_000, fa2_iters=50),
        # The exact sum over many components at once, as a graph without a giant one has them: 200 to 5,000 nodes.
        dict(name="layout-300-mid-components", kind="layout", comps=300, lo=200.0, hi=5000.0, kk_max_nodes=199,
             fa2_iters=20),
        # Kamada-Kawai on many components of 3 to 200 nodes.
        dict(name="layout-kk-20k-components", kind="layout", comps=20_000, lo=3.0, hi=200.0, kk_max_nodes=200,
             fa2_iters=0),
        # Host transaction lists to a graph with labelled components, read back.
        dict(name="build-200k-tx", kind="build", n_tx=200_000),
        # Neighbourhoods of a graph in memory: the first half of a serving request.
        dict(name="khop-200k-tx", kind="khop", n_tx=200_000, seeds=4, hops=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["noalloc", "session", "session", "session", "session", "forces", "whole", "layout", "layout",
                       "build", "khop"])
    if kind == "noalloc":
        return dict(kind=kind, n_tx=_log(rng, 300, 10_000), where="disc", iters=rng.randint(1, 4))
    if kind == "session":
        n_tx = _log(rng, 300, 400_000)
        return dict(kind=kind, n_tx=n_tx, where="disc", iters=rng.randint(2, 40 if n_tx < 10_000 else 8),
                    fmm_p=rng.choice([6, 8, 8, 8, 12, 16]), leaf_size=rng.choice([48, 64, 64, 64, 96]),
                    swing_variant=rng.randint(0, 1))
    if kind == "forces":
        return dict(kind=kind, n_tx=_log(rng, 300, 100_000), where=rng.choice(["disc", "clustered"]),
                    fmm_p=rng.choice([8, 8, 12, 16]), leaf_size=rng.choice([32, 64, 64, 96]))
    if kind == "whole":
        return dict(kind=kind, n_tx=_log(rng, 300, 100_000), fa2_iters=rng.randint(10, 50))
    if kind == "layout":
        if rng.random() < 0.5:
            return dict(kind=kind, comps=_log(rng, 20, 300), lo=200.0, hi=5000.0, kk_max_nodes=199,
                        fa2_iters=rng.randint(5, 20))
        return dict(kind=kind, comps=_log(rng, 200, 20_000), lo=3.0, hi=float(rng.choice([50, 120, 200])),
                    kk_max_nodes=200, fa2_iters=0)
    if kind == "build":
        return dict(kind=kind, n_tx=_log(rng, 1000, 400_000))
    return dict(kind=kind, n_tx=_log(rng, 1000, 400_000), seeds=rng.randint(1, 8), hops=rng.randint(1, 4))


def _graph(t):
    g = bgl.Graph.build(_context(), *t.lists)
    g.components(labels=False)
    return g


def _component_xy(g, t):
    off, _, nodes = g.component_nodes()
    return np.ascontiguousarray(t.xy[nodes[off[0]:off[1]]])


def prepare(case, seed):
    kind, ctx = case["kind"], _context()
    if kind == "noalloc":
        t = _Tx(case, seed)
        off, adj, mass, xy = t.local(t.giant())
        dev = [torch.from_numpy(a).cuda() for a in (off, adj, mass.astype(np.float32), xy)]
        f = [torch.zeros(len(mass), 2, device="cuda") for _ in range(2)]
        return dict(kind=kind, n=len(mass), iters=case["iters"], p=_params(case), arrays=dev, fprev=f[0], f=f[1],
                    sg=torch.ones(1, dtype=torch.float64, device="cuda"))
    if kind in ("session", "forces"):
        t = _Tx(case, seed)
        g = _graph(t)
        xy, p = _component_xy(g, t), _params(case)
        if kind == "session":
            g.session_begin(0, p, xy)
        return dict(kind=kind, g=g, p=p, xy=xy, iters=case.get("iters", 0))
    if kind == "layout":
        rng = np.random.default_rng([seed, case["comps"]])
        n, u, v, _ = _forest(rng, case["comps"], case["lo"], case["hi"])
        g = bgl.Graph.from_edges(ctx, n, u, v)
        g.components(labels=False)
        return dict(kind=kind, g=g, p=_params(case, seed=seed), out=torch.empty(n, 2, device="cuda"))
    if kind == "whole":
        t = _Tx(case, seed)
        dev = [torch.from_numpy(a.view(np.int64)).cuda() for a in t.lists]
        return dict(kind=kind, lists=dev, sizes=(t.n_tx, len(t.lists[1]), len(t.lists[3])), p=_params(case, seed=seed),
                    out=torch.empty(t.n, 2, device="cuda"))
    t = _Tx(case, seed)
    if kind == "build":
        return dict(kind=kind, lists=t.lists)
    fix = np.random.default_rng([case["n_tx"], case["seeds"], case["hops"]])
    return dict(kind=kind, g=_graph(t), hops=case["hops"], n=t.n,
                seeds=[int(t.n_tx + t.ids[a]) for a in fix.integers(0, t.n_addr, case["seeds"])])


def run(state):
    kind = state["kind"]
    if kind == "noalloc":
        off, adj, mass, xy = state["arrays"]
        ctx = _context()
        for _ in range(state["iters"]):
            ctx.fa2_iteration_noalloc(state["n"], off, adj, mass, xy, state["fprev"], state["f"], state["sg"],
                                      state["p"])
        # s_G is a quotient of sums of FP32 terms: handed on as FP32
        with torch.cuda.stream(_device["stream"]):
            return [xy, state["fprev"], state["sg"].float()]
    if kind == "session":
        stats = state["g"].session_advance(state["iters"])
        # swing, traction and s_G of every iteration: sums of FP32 terms, handed on as FP32
        return [state["g"].session_positions(len(state["xy"]))[0], stats.astype(np.float32)]
    if kind == "forces":
        return state["g"].fa2_forces(0, state["p"], state["xy"])
    if kind == "layout":
        state["g"].layout_dev(state["p"], state["out"])
        return state["out"]
    if kind == "whole":
        g = bgl.Graph.build_dev(_context(), *state["sizes"], *state["lists"])
        g.components(labels=False)
        g.layout_dev(state["p"], state["out"])
        g.destroy()
        return state["out"]
    if kind == "build":
        g = bgl.Graph.build(_context(), *state["lists"])
        labels, n_comp = g.components()
        off, adj = g.csr()
        g.destroy()
        return [labels, n_comp, off, adj]
    out = []
    for s in state["seeds"]:
        out += list(state["g"].khop(s, state["hops"], state["n"]))
    return out


def _nodes(case):
    """Typical sizes of a case: nodes and adjacency entries of what it lays out (2.77 nodes per transaction and 2.5
    adjacency entries per node in the giant component of a transaction graph)."""
    if "n_tx" in case:
        n = 2.77 * case["n_tx"]
        return n, 2.5 * n
    lo, hi = case["lo"], case["hi"]
    n = case["comps"] * (hi - lo) / math.log(hi / lo)
    return n, 2.2 * n


def work(case):
    n, m = _nodes(case)
    kind, iters = case["kind"], case.get("iters", case.get("fa2_iters", 1))
    if kind in ("noalloc", "session", "forces", "whole"):
        exact = kind == "noalloc" or (case.get("repulsion") != "fmm" and n < 8192)
        if exact:
            flops = 10.0 * n * n
        else:
            # near field: nine leaves of 0.6 times their capacity around a point; far: P2M, L2P and 27 M2L per leaf
            leaf, p = case.get("leaf_size", 64), case.get("fmm_p", 8)
            flops = n * (9 * 0.6 * leaf * 10.0 + 16.0 * (p + 1)) + n / (0.6 * leaf) * 27 * 8.0 * (p + 1) ** 2
        # positions and previous forces read and written, masses and adjacency read, once an iteration
        return dict(bytes=iters * (36.0 * n + 12.0 * m), flops=iters * (flops + 4.0 * m))
    if kind == "layout":
        lo, hi = case["lo"], case["hi"]
        pairs = case["comps"] * (hi * hi - lo * lo) / 2 / math.log(hi / lo)
        steps = case["fa2_iters"] * 10.0 if case["fa2_iters"] else 200 * 17.0
        return dict(bytes=16.0 * n + 8.0 * m, flops=pairs * steps)
    if kind == "build":
        return dict(bytes=16.0 * 5.4 * case["n_tx"] + 12.0 * n + 4.0 * m, flops=0.0)
    return dict(bytes=case["seeds"] * (12.0 * n + 8.0 * m) * 0.25, flops=0.0)


# ------------------------------------------------------------------ the same results in 64 bits


def _repulsion64(x, y, m):
    """sum_j m_i m_j (p_i - p_j) / |p_i - p_j|^2 over all pairs, coincident ones adding nothing."""
    fx, fy = torch.empty_like(x), torch.empty_like(y)
    step = max(1, min(len(x), (1 << 26) // len(x)))
    for i in range(0, len(x), step):
        dx, dy = x[i:i + step, None] - x, y[i:i + step, None] - y
        r2 = dx * dx + dy * dy
        w = torch.where(r2 > 0, m / r2, 0.0)
        fx[i:i + step], fy[i:i + step] = (w * dx).sum(1), (w * dy).sum(1)
    return m * fx, m * fy


def _forces64(x, y, m, src, dst):
    fx, fy = _repulsion64(x, y, m)
    fx.index_add_(0, src, x[dst] - x[src])
    fy.index_add_(0, src, y[dst] - y[src])
    return fx - m * x, fy - m * y


def _iterate64(case, iters, off, adj, mass, xy):
    """`iters` iterations with kr = kg = tau = 1, ks = 0.1, ksmax = STEP from F = 0, s_G = 1: positions, F, and swing,
    traction and s_G of each."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    x, y, m = (torch.from_numpy(np.array(a, np.float64)).to(dev) for a in (xy[:, 0], xy[:, 1], mass))
    src = torch.from_numpy(np.repeat(np.arange(len(mass)), np.diff(off))).to(dev)
    dst = torch.from_numpy(adj.astype(np.int64)).to(dev)
    px, py, sg, stats = torch.zeros_like(x), torch.zeros_like(y), 1.0, []
    for _ in range(iters):
        fx, fy = _forces64(x, y, m, src, dst)
        sw, tr = torch.hypot(fx - px, fy - py), torch.hypot(fx + px, fy + py)
        w = m if case.get("swing_variant") else torch.ones_like(m)
        swing, trac = float((w * sw).sum()), float((w * tr).sum()) * (0.5 if case.get("swing_variant") else 1.0)
        sg = min(trac / swing, 1.5 * sg)
        s = torch.minimum(0.1 * sg / (1 + sg * torch.sqrt(sw)), STEP / torch.hypot(fx, fy))
        x, y, px, py = x + s * fx, y + s * fy, fx, fy
        stats.append([swing, trac, sg])
    return torch.stack([x, y], 1), torch.stack([px, py], 1), np.array(stats)


def _start(seed, n):
    """The library's start positions of nodes 0..n-1: x and y in [-1, 1) from two SplitMix64 outputs each."""
    with np.errstate(over="ignore"):
        s = np.uint64(seed) ^ (np.arange(n, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15))
        xy = np.empty((n, 2))
        for k in range(2):
            s = s + np.uint64(0x9E3779B97F4A7C15)
            z = (s ^ (s >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            xy[:, k] = ((z ^ (z >> np.uint64(31))) >> np.uint64(40)).astype(np.float64) * 2.0 ** -23 - 1.0
    return xy


def exact(case, seed):
    kind = case["kind"]
    if kind == "layout" and case["fa2_iters"]:
        # every component is above kk_max_nodes: ForceAtlas2 on each, exact sums
        n, u, v, of = _forest(np.random.default_rng([seed, case["comps"]]), case["comps"], case["lo"], case["hi"])
        xy = torch.from_numpy(_start(seed, n)).to("cuda" if torch.cuda.is_available() else "cpu")
        nodes, edges = np.argsort(of, kind="stable"), np.argsort(of[u], kind="stable")
        nodes = np.split(nodes, np.cumsum(np.bincount(of))[:-1])
        edges = np.split(edges, np.cumsum(np.bincount(of[u], minlength=case["comps"]))[:-1])
        for c, e in zip(nodes, edges):
            off, adj = _local_csr(n, u[e], v[e], c)
            xy[c] = _iterate64(case, case["fa2_iters"], off, adj, np.diff(off) + 1.0, xy[c].cpu().numpy())[0]
        return xy
    if kind not in ("noalloc", "session", "forces"):
        return None      # whole numbers, or Kamada-Kawai's sweeps: minutes here
    # the all-pairs sum in 64 bits: some 1e10 pairs a second
    if (2.77 * case["n_tx"]) ** 2 * case.get("iters", 1) > 6e10:
        return None
    t = _Tx(case, seed)
    off, adj, mass, xy = t.local(t.giant())
    if kind == "forces":
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        x, y, m = (torch.from_numpy(np.array(a, np.float64)).to(dev) for a in (xy[:, 0], xy[:, 1], mass))
        src = torch.from_numpy(np.repeat(np.arange(len(mass)), np.diff(off))).to(dev)
        return torch.stack(_forces64(x, y, m, src, torch.from_numpy(adj.astype(np.int64)).to(dev)), 1)
    pos, f, stats = _iterate64(case, case["iters"], off, adj, mass, xy)
    if kind == "noalloc":
        return [pos, f, torch.tensor([stats[-1, 2]], dtype=torch.float64)]
    return [pos, stats]
