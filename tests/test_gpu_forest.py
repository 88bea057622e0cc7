"""Certificate forests (the marking step that leads a default solve's rounds)
at the sizes where they can go wrong: fewer vertices than a warp, rows beyond
one chunk, weights beyond the levels, several components, 64-bit weights, long
paths, cliques.  Every value against the oracle or a closed form, every side
against the cut weight."""
import numpy as np
import pytest

import oracle
import synth
from tests import graphs as G
from tests.test_gpu_parity import _check_solve, canon, mc

pytestmark = pytest.mark.gpu

def _hub_and_cycle(n, hub_w):
    """A hub joined to every vertex of a random cycle (rows of n - 1 entries)."""
    rng = np.random.default_rng(n)
    e = [(0, i) for i in range(1, n)] + [(i, i % (n - 1) + 1) for i in range(1, n)]
    w = [int(x) for x in rng.integers(1, hub_w + 1, n - 1)] + \
        [int(x) for x in rng.integers(1, 8, n - 1)]
    return G.from_edges(n, e, w)

@pytest.mark.parametrize("n", [3, 4, 5, 31, 32, 33, 255, 257, 700])
def test_small_random(n):
    rng = np.random.default_rng(n)
    for hi in (1, 10, 1000, 2_000_000):
        g = G.random_graph(n, min(1.0, 8.0 / n), rng, 1, hi, connected=True)
        _check_solve(n, canon(n, *g))

@pytest.mark.parametrize("n,hub_w", [(258, 1), (513, 40), (1025, 400), (2050, 3)])
def test_long_rows(n, hub_w):
    c = canon(n, *_hub_and_cycle(n, hub_w))
    _check_solve(n, c, expect=oracle.noi(n, *c)[0])

@pytest.mark.parametrize("n", [600, 5000, 70_001])
def test_long_cycles(n):
    """Θ(n) diameter: the last batch takes what the others left."""
    rng = np.random.default_rng(n)
    w = rng.integers(3, 50, n)
    two = np.sort(w)[:2].sum()
    _check_solve(n, canon(n, *G.cycle(n, [int(x) for x in w])), expect=int(two))

def test_components_and_cliques():
    a = G.complete(60, 7)
    _check_solve(60, canon(60, *a), expect=59 * 7)
    # two components: cut 0
    rp, col, w = a
    both = (np.concatenate([rp, rp[1:] + rp[-1]]), np.concatenate([col, col + 60]).astype(np.int32),
            np.concatenate([w, w]))
    _check_solve(120, canon(120, *both), expect=0)

def test_planted_cut_64bit_weights():
    """Unit weights scaled past a total of 2^31: the same rounds in 64 bits."""
    s = synth.planted(1 << 10, 21 << 10, 30, 9, 1, 11)
    c = (s.row_ptr, s.col, s.w.astype(np.int64))
    lam = oracle.noi(s.n, *c)[0]
    assert _check_solve(s.n, c, expect=lam)["seq_passes"] == 0
    big = (s.row_ptr, s.col, s.w.astype(np.int64) * 60_000)
    _check_solve(s.n, big, expect=lam * 60_000)

@pytest.mark.parametrize("log_nb,cross,seed", [(10, 9, 11), (11, 9, 5), (12, 25, 3)])
def test_small_planted_cuts(log_nb, cross, seed):
    """The forests join enough of them, in every round, that no whole-graph
    pass runs."""
    nb = 1 << log_nb
    s = synth.planted(nb, 21 * nb, 30, cross, 1, seed)
    c = (s.row_ptr, s.col, s.w.astype(np.int64))
    lam = oracle.noi(s.n, *c)[0]
    for _ in range(5):
        assert _check_solve(s.n, c, expect=lam)["seq_passes"] == 0


def test_weak_forests_on_a_large_graph():
    """A unit cycle, of which the forests join one vertex and the other marks
    none: every round runs the whole-graph passes, the first one too."""
    n = 12_000
    p = np.random.default_rng(1).permutation(n)
    c = canon(n, *G.from_edges(n, np.stack([p, np.roll(p, -1)], 1)))
    _check_solve(n, c, expect=2)
    g = mc.mincut_graph_from_csr(n, *c)
    mc.mincut_solve(g, mc.default_options(profile=1))
    prof = mc.mincut_profile_read(g)
    g.destroy()
    assert prof["capforest_seq"]["launches"] == prof["pr_marks"]["launches"]


@pytest.mark.parametrize("w", [3, 1000, 60_000])
def test_weights_nearly_alike(w):
    """Equal weights with a few heavier ones among them: half their mean lies
    above half of most, which must not cost the forests half of each edge
    (64-bit sums with the largest)."""
    s = synth.planted(1 << 13, 21 << 13, 20, 25, 1, 3)
    src = np.repeat(np.arange(s.n), np.diff(s.row_ptr))
    ww = np.where((src + s.col) % 97 == 0, w + w // 2, w)  # by the sum of the ends: symmetric
    c = (s.row_ptr, s.col, ww.astype(np.int64))
    assert _check_solve(s.n, c, expect=oracle.noi(s.n, *c)[0])["seq_passes"] == 0


@pytest.mark.parametrize("seed", range(3))
def test_random_sparse_20000(seed):
    g = synth.er_connected(20_000, 100_000, 1, 30, 50 + seed)
    c = (g.row_ptr, g.col, g.w.astype(np.int64))
    _check_solve(g.n, c, expect=oracle.noi(g.n, *c)[0])

@pytest.mark.parametrize("clusters,size,hub", [(2, 1200, 0), (300, 8, 0), (300, 8, 700),
                                               (1023, 4, 0), (1025, 4, 0), (1700, 4, 1500),
                                               (2040, 3, 0), (2300, 3, 0)])
def test_what_the_forests_leave(clusters, size, hub):
    """Heavy clusters joined by light edges: the forests leave one vertex per
    cluster, summed in a matrix, listed, or too many for either; hubs with rows
    of several pieces stay vertices of their own."""
    rng = np.random.default_rng(clusters + size)
    n = clusters * size
    first = np.arange(clusters) * size
    e, w = [], []
    for i in range(size):  # a heavy cycle within each cluster
        j = (i + 1) % size
        if size > 2 or i < j:
            e += list(zip(first + i, first + j))
            w += [500] * clusters
    order = rng.permutation(clusters)  # a light cycle through the clusters, and chords
    for a, b in [(order, np.roll(order, 1)),
                 (rng.integers(0, clusters, 3 * clusters), rng.integers(0, clusters, 3 * clusters))]:
        u = first[a] + rng.integers(0, size, len(a))
        v = first[b] + rng.integers(0, size, len(b))
        k = a != b
        e += list(zip(u[k], v[k]))
        w += [int(x) for x in rng.integers(1, 9, int(k.sum()))]
    for h in range(2 if hub else 0):  # hubs: one light edge to each of many vertices
        e += [(n + h, int(v)) for v in rng.choice(n, hub, replace=False)]
        w += [1] * hub
    n += 2 if hub else 0
    perm = rng.permutation(n)
    c = canon(n, *G.from_edges(n, [(perm[a], perm[b]) for a, b in e], w))
    _check_solve(n, c, expect=oracle.noi(n, *c)[0])


@pytest.mark.parametrize("deg", [255, 256, 257, 1000, 2900])
@pytest.mark.parametrize("w", [1, 300])
def test_hub_in_a_batch(deg, w):
    """A vertex whose row is listed by its own thread (up to four pieces of 64)
    or by its warp, met inside the graph and not only as the first vertex; light
    edges, and edges of many units at once."""
    n = 3000
    rng = np.random.default_rng(deg + w)
    hub = 1234
    spokes = rng.choice(np.setdiff1d(np.arange(n), [hub]), deg, replace=False)
    e = [(i, (i + d) % n) for i in range(n) for d in (1, 2, 7)]
    ww = [int(x) for x in rng.integers(1, 4, len(e))]
    e += [(hub, int(v)) for v in spokes]
    ww += [w] * deg
    c = canon(n, *G.from_edges(n, e, ww))
    _check_solve(n, c, expect=oracle.noi(n, *c)[0])


def _torus(a, b, w, rng):
    i = np.arange(a * b).reshape(a, b)
    e = np.concatenate([np.stack([i.ravel(), np.roll(i, -1, k).ravel()], 1) for k in (0, 1)])
    return a * b, G.from_edges(a * b, e, [int(x) for x in rng.integers(1, w + 1, len(e))])


def _ladder(n, w, rng):
    i = np.arange(n)
    j = (i + 1) % n
    e = np.concatenate([np.stack([i, j], 1), np.stack([n + i, n + j], 1), np.stack([i, n + i], 1)])
    return 2 * n, G.from_edges(2 * n, e, [int(x) for x in rng.integers(1, w + 1, len(e))])


def _forest_ms(n, c, expect):
    """Device time of the forest kernel in a default solve."""
    _check_solve(n, c, expect=expect)
    g = mc.mincut_graph_from_csr(n, *c)
    mc.mincut_solve(g)
    mc.mincut_solve(g, mc.default_options(profile=1))
    prof = mc.mincut_profile_read(g)
    g.destroy()
    return prof["forest"]["ms"]


@pytest.mark.parametrize("name,limit", [("torus", 1.0), ("ladder", 1.0), ("wheel", 0.7),
                                        ("tree", 0.5)])
def test_thin_frontiers(name, limit):
    """Graphs on which a batch is a handful of vertices: the forests do not
    take a hundred batches for them (1.6 ms and more; the tree 0.8)."""
    rng = np.random.default_rng(5)
    if name == "wheel":
        s = synth.wheel(4097, seed=1)
        n, g, expect = s.n, (s.row_ptr, s.col, s.w.astype(np.int64)), 8192
    elif name == "tree":
        n = 50_000
        w = rng.integers(1, 51, n - 1)
        p = rng.permutation(n)
        e = np.stack([p[1:], p[(rng.random(n - 1) * np.arange(1, n)).astype(np.int64)]], 1)
        g, expect = G.from_edges(n, e, [int(x) for x in w]), int(w.min())
    else:
        n, g = _torus(60, 60, 50, rng) if name == "torus" else _ladder(3000, 20, rng)
        expect = oracle.noi(n, *canon(n, *g))[0]
    assert _forest_ms(n, canon(n, *g), expect) < limit


def _cube(a, rng):
    """Periodic a x a x a grid, weights 1 to 20."""
    i = np.arange(a ** 3).reshape(a, a, a)
    e = np.concatenate([np.stack([i.ravel(), np.roll(i, -1, d).ravel()], 1) for d in range(3)])
    p = rng.permutation(a ** 3)
    return a ** 3, G.from_edges(a ** 3, p[e], [int(x) for x in rng.integers(1, 21, len(e))])


@pytest.mark.parametrize("a,limit", [(15, 0.6), (40, 0.9)])
def test_frontiers_that_grow_slowly(a, limit):
    """Balls in a 3-d grid: frontiers of hundreds that grow by less than half
    (0.8 and 1.5 ms by batches)."""
    n, g = _cube(a, np.random.default_rng(6))
    c = canon(n, *g)
    assert _forest_ms(n, c, oracle.noi(n, *c)[0]) < limit


@pytest.mark.parametrize("n", [2050, 4097, 40_001])
def test_nothing_to_join(n):
    """A wheel's spokes have no units and its rim too few for the last level:
    no batch is scanned (0.3 ms with)."""
    s = synth.wheel(n, seed=1)
    c = (s.row_ptr, s.col, s.w.astype(np.int64))
    assert _forest_ms(n, c, 2 * (n - 2) + 2) < 0.15


@pytest.mark.parametrize("d,n,cross", [(4, 8000, 1), (10, 5000, 5), (30, 3000, 9)])
def test_cut_between_regular_graphs(d, n, cross):
    """Two random regular graphs, degrees at the bound: a prefix cut is the
    minimum cut, and the forests need no whole-graph pass after it."""
    rng = np.random.default_rng(d)
    e = []
    for half in (0, n):
        for _ in range(d // 2):
            p = half + rng.permutation(n)
            e.append(np.stack([p, np.roll(p, 1)], 1))
    e.append(np.stack([rng.integers(0, n, cross), n + rng.integers(0, n, cross)], 1))
    c = canon(2 * n, *G.from_edges(2 * n, np.concatenate(e)))
    st = _check_solve(2 * n, c, expect=oracle.noi(2 * n, *c)[0])
    assert st["seq_passes"] == 0


@pytest.mark.parametrize("n,deg,whi", [(2500, 150, 100), (2500, 200, 20)])
def test_too_few_units_for_the_levels(n, deg, whi):
    """Degrees close to the bound once the units are rounded: the last level
    cannot join much, and no batch of the first round is scanned (2 ms and more
    with)."""
    s = synth.cycle_plus(n, deg, 1, whi, 3)
    c = (s.row_ptr, s.col, s.w.astype(np.int64))
    _check_solve(n, c, expect=oracle.noi(n, *c)[0])
    g = mc.mincut_graph_from_csr(n, *c)
    ro = mc.default_options(profile=1)
    mc.mincut_solve(g, ro)
    prof = mc.mincut_profile_read(g)["forest"]
    assert prof["ms"] < 0.25 * prof["launches"], prof
    g.destroy()


def test_small_graphs_use_several_blocks():
    """A wheel of unit weights, which the forests do not help: they stay cheap
    (0.2 ms by one block)."""
    s = synth.wheel(4097, seed=1)
    c = (s.row_ptr, s.col, np.ones_like(s.w, dtype=np.int64))
    assert _forest_ms(s.n, c, 3) < 0.15


@pytest.mark.parametrize("m", [3071, 3072, 3073, 9999, 10_000, 10_001, 57_343, 57_344, 57_345])
def test_block_counts(m):
    """Entries around the numbers at which the kernel's grid changes (10,000
    edges: eight entries per vertex)."""
    n = 2500
    rng = np.random.default_rng(m)
    p = rng.permutation(n)  # a random cycle, then other pairs up to m
    pair = np.minimum(p, np.roll(p, 1)) * n + np.maximum(p, np.roll(p, 1))
    u, v = rng.integers(0, n, (2, 3 * m))
    extra = np.setdiff1d((np.minimum(u, v) * n + np.maximum(u, v))[u != v], pair)
    pair = np.concatenate([pair, rng.choice(extra, m - n, replace=False)])
    c = canon(n, *G.from_edges(n, np.stack([pair // n, pair % n], 1), rng.integers(1, 10, m)))
    assert c[0][-1] == 2 * m
    _check_solve(n, c, expect=oracle.noi(n, *c)[0])


@pytest.mark.parametrize("kind", ["cliques", "random"])
def test_wait_that_runs_out(kind):
    """A limit of one poll, which the grid barriers run into at once: the kernel
    returns an error status, the solve goes on without the forests, and the
    graph and the context stay usable."""
    if kind == "cliques":
        k = 100  # a ring of cliques of 25
        n = 25 * k
        e = [(25 * i + a, 25 * i + b) for i in range(k) for a in range(25) for b in range(a)]
        w = [10] * len(e) + [2] * k
        e += [(25 * i, (25 * i + 26) % n) for i in range(k)]
        c = canon(n, *G.from_edges(n, e, w))
    else:
        s = synth.cycle_plus(2600, 40, 1, 1, 3)
        n, c = s.n, (s.row_ptr, s.col, s.w.astype(np.int64))
    expect = oracle.noi(n, *c)[0]
    g = mc.mincut_graph_from_csr(n, *c)
    for opts in (mc.default_options(spin_limit=1, profile=1), mc.default_options(spin_limit=1 << 22)):
        value, bitmap, _ = mc.mincut_solve(g, opts)
        side = mc.bitmap_to_side(bitmap, n)
        assert value == expect and oracle.cut_weight(n, *c, side) == expect
        assert mc.mincut_last_error() == ""
        if opts.profile:  # tried once, and not again in the solve
            assert mc.mincut_profile_read(g)["forest"]["launches"] == 1
    g.destroy()


@pytest.mark.parametrize("kw", [dict(max_rounds=1 << 30), dict(lp_every_round=1),
                                dict(seq_passes=2, seed=7), dict(lp_min_n=2, max_rounds=1 << 30)])
def test_solves_without_forests(kw):
    """Whole solves by label propagation, PR tests and the passes, which the
    options that ask for them still reach."""
    for s in (synth.workload_rmat_core(14, 5, 2), synth.planted(1 << 10, 21 << 10, 30, 9, 1, 11),
              synth.cycle_plus(12_000, 7, 1, 40, 3)):
        c = (s.row_ptr, s.col, s.w.astype(np.int64))
        expect = oracle.noi(s.n, *c)[0]
        _check_solve(s.n, c, mc.default_options(**kw), expect=expect)
        g = mc.mincut_graph_from_csr(s.n, *c)
        mc.mincut_solve(g, mc.default_options(profile=1, **kw))
        prof = mc.mincut_profile_read(g)
        assert "forest" not in prof and "small_solve" not in prof and "capforest_passes" in prof
        assert "lp_sweep" in prof or s.n < 10_000 and kw.get("lp_min_n") != 2
        g.destroy()


@pytest.mark.parametrize("refused", [1, 2, 3])
def test_allocations_refused(refused, monkeypatch):
    """The first requests of a solve refused by the caller's allocator: buffers
    that come as one block are asked for one by one, and a round without room
    for the forests does without them."""
    class Refusing(mc._TorchAllocator):
        def __init__(self, device):
            super().__init__(device)
            self.refuse = 0
            give = self._alloc

            def _alloc(nbytes, stream, ctx):
                if self.refuse > 0:
                    self.refuse -= 1
                    return None
                return give(nbytes, stream, ctx)

            self._give, self._alloc = give, type(give)(_alloc)
            self.struct = mc.MincutAllocator(self._alloc, self._free, None)

    monkeypatch.setattr(mc, "_TorchAllocator", Refusing)
    n = 3000
    rng = np.random.default_rng(refused)
    g = G.random_graph(n, 10.0 / n, rng, 1, 20, connected=True)
    c = canon(n, *g)
    dev = [mc_dev(x) for x in (np.asarray(c[0], np.int64), np.asarray(c[1], np.int32),
                               np.asarray(c[2], np.int32))]
    h = mc.mincut_graph_from_csr(n, *dev, use_torch_allocator=True)
    expect = oracle.noi(n, *c)[0]
    for _ in range(2):
        h._allocator.refuse = refused
        value, bitmap, _ = mc.mincut_solve(h)
        h._allocator.refuse = 0
        side = mc.bitmap_to_side(bitmap, n)
        assert value == expect and oracle.cut_weight(n, *c, side) == expect
    h.destroy()


def test_refusal_is_no_error(monkeypatch):
    """Both requests for the forests' buffers refused: the solve does without
    them to its end, asks no more for them, and leaves no message."""
    class Refusing(mc._TorchAllocator):
        def __init__(self, device):
            super().__init__(device)
            self.refuse = 0
            give = self._alloc

            def _alloc(nbytes, stream, ctx):
                if self.refuse > 0:
                    self.refuse -= 1
                    return None
                return give(nbytes, stream, ctx)

            self._give, self._alloc = give, type(give)(_alloc)
            self.struct = mc.MincutAllocator(self._alloc, self._free, None)

    monkeypatch.setattr(mc, "_TorchAllocator", Refusing)
    nb = 1 << 11
    s = synth.planted(nb, 21 * nb, 30, 9, 1, 5)
    h = mc.mincut_graph_from_csr(s.n, mc_dev(s.row_ptr.astype(np.int64)),
                                 mc_dev(s.col.astype(np.int32)), mc_dev(s.w.astype(np.int32)),
                                 use_torch_allocator=True)
    h._allocator.refuse = 2
    value, _, st = mc.mincut_solve(h, mc.default_options(profile=1))
    assert value == oracle.noi(s.n, s.row_ptr, s.col, s.w.astype(np.int64))[0]
    assert st["rounds"] > 1 and mc.mincut_last_error() == ""
    assert "forest" not in mc.mincut_profile_read(h)
    h.destroy()


def mc_dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()
