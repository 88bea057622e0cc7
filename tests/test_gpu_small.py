"""The one-block solver of small graphs (single solves, batches) at its edges:
its largest vertex count and the first beyond, more entries than it takes,
graphs whose rounds it leaves to the others, heavy weights, closed forms."""
import numpy as np
import pytest

import oracle
import synth
from tests import graphs as G
from tests.test_gpu_parity import _check_solve, canon, mc
from tests.test_gpu_batch import _check_batch

pytestmark = pytest.mark.gpu


def _graph(s):
    return s.row_ptr, s.col, s.w.astype(np.int64)


@pytest.mark.parametrize("n,m", [(2047, 9000), (2048, 20_000), (2049, 9000), (2048, 70_000),
                                 (700, 66_000)])
def test_size_limits(n, m):
    s = synth.er_connected(n, m, 1, 50, n + m)
    c = _graph(s)
    _check_solve(n, c, expect=oracle.noi(n, *c)[0])


@pytest.mark.parametrize("n", [2, 3, 5, 33, 130])
def test_closed_forms(n):
    _check_solve(n, canon(n, *G.complete(n, 3)), expect=3 * (n - 1))
    if n > 2:
        _check_solve(n, canon(n, *G.cycle(n, list(range(5, 5 + n)))), expect=11)


def test_rounds_it_leaves():
    """Interleaved heavy cycles: no forest joins anything, the other rounds
    take over; alone, and in a batch among ordinary graphs."""
    hard = [synth.dblcyc(n, seed=n) for n in (34, 66, 130)]
    easy = [synth.batch_graph(4, i) for i in range(12)]
    graphs = [(s.n, *_graph(s)) for s in hard + easy]
    expect = [oracle.noi(*g)[0] for g in graphs]
    for g, e in zip(graphs[:3], expect):
        _check_solve(g[0], g[1:], expect=e)
    for kw in (dict(), dict(deterministic=1), dict(pr_mask=0)):
        _check_batch(graphs, expect, mc.default_options(batch_small_n=2048, **kw))


def test_heavy_and_light_weights():
    rng = np.random.default_rng(3)
    for n in (40, 400):
        g = G.random_graph(n, 8.0 / n, rng, 1, 1, connected=True)
        c = canon(n, *g)
        w = c[2].copy()
        src = np.repeat(np.arange(n), np.diff(c[0]))
        heavy = ((src + c[1]) % 7 == 0)
        w[heavy] *= 900_000  # by the sum of the ends: symmetric
        _check_solve(n, (c[0], c[1], w))


@pytest.mark.parametrize("whi", [1, 3, 40])
@pytest.mark.parametrize("n", [17, 200, 1023, 1500])
def test_level_counts(n, whi):
    """Least degrees from 2 to 12 (as many levels under unit weights, one lane
    per edge and level up to 8, the general insertion beyond), with fewer edges
    than a block's threads and with more; alone and as a batch."""
    rng = np.random.default_rng(n + whi)
    graphs = []
    for k in range(1, 12):
        d = k if n * k % 2 == 0 else k + 1
        u = np.repeat(np.arange(n), (d + 1) // 2)
        v = (u + np.tile(np.arange(1, (d + 1) // 2 + 1), n)) % n
        x = rng.integers(0, n, 2 * n if k % 3 == 0 else 3)
        y = rng.integers(0, n, len(x))
        u, v = np.concatenate([u, x]), np.concatenate([v, y])
        keep = u != v
        pair = np.unique(np.minimum(u, v)[keep] * n + np.maximum(u, v)[keep])
        w = rng.integers(1, whi + 1, len(pair))
        graphs.append((n, *canon(n, *G.from_edges(n, np.stack([pair // n, pair % n], 1), w))))
    expect = [oracle.noi(*g)[0] for g in graphs]
    for g, e in zip(graphs, expect):
        _check_solve(g[0], g[1:], expect=e)
    _check_batch(graphs, expect)


@pytest.mark.parametrize("n,whi", [(50_000, 100), (1500, 2)])
def test_rounds_that_join_next_to_nothing(n, whi):
    """Cycles whose minimum weights repeat: once only those are left (500 and
    more), a round here joins a single vertex, and the others take over, until 63
    vertices are left: at most 61 such rounds, and those before them, which join
    an eighth or a vertex per whole-graph pass."""
    rng = np.random.default_rng(n)
    w = rng.integers(1, whi + 1, n)
    st = _check_solve(n, canon(n, *G.cycle(n, [int(x) for x in w])), expect=int(np.sort(w)[:2].sum()))
    assert st["rounds"] <= 61 + 40


@pytest.mark.parametrize("n", [1025, 2048])
def test_given_up_once(n):
    """A wheel that the block solver gives up: the grid-wide forests, whose
    certificate is the same, do not try it again; and a clique ring whose rest
    it gives up is not taken again at once."""
    s = synth.wheel(n, seed=1)
    c = _graph(s)
    _check_solve(n, c, expect=2 * (n - 2) + 2)
    g = mc.mincut_graph_from_csr(n, *c)
    mc.mincut_solve(g, mc.default_options(profile=1))
    assert "forest" not in mc.mincut_profile_read(g)
    g.destroy()
    k = 100  # cliques of 25 in a ring of light edges: a unit cycle of 100 is left
    e = [(25 * i + a, 25 * i + b) for i in range(k) for a in range(25) for b in range(a)]
    w = [10] * len(e) + [2] * k
    e += [(25 * i, (25 * i + 26) % (25 * k)) for i in range(k)]
    c = canon(25 * k, *G.from_edges(25 * k, e, w))
    _check_solve(25 * k, c, expect=4)
    g = mc.mincut_graph_from_csr(25 * k, *c)
    mc.mincut_solve(g, mc.default_options(profile=1))
    prof = mc.mincut_profile_read(g)
    # once led by the forests with the rest behind them, and once when a quarter is left
    assert prof["forest"]["launches"] == 1 and prof["small_solve"]["launches"] <= 2
    g.destroy()


def test_one_slow_round():
    """A 3-regular graph with a few doubled edges: PR2 joins only their ends,
    and the next degree bound is the minimum cut; no whole-graph pass is needed."""
    n = 1500
    rng = np.random.default_rng(5)
    p, q = rng.permutation(n), rng.permutation(n)
    pair = np.sort(np.concatenate([np.stack([p, np.roll(p, 1)], 1), q.reshape(-1, 2)]), 1)
    pair, w = np.unique(np.concatenate([pair, np.sort(np.stack([p[:9], np.roll(p, 1)[:9]], 1), 1)]),
                        axis=0, return_counts=True)
    c = canon(n, *G.from_edges(n, pair, [int(x) for x in w]))
    st = _check_solve(n, c, expect=oracle.noi(n, *c)[0])
    assert st["seq_passes"] == 0


def test_too_few_levels():
    """A dense small graph: the block solver has too few levels for it and the
    forests too few units per level, both see so at once, and the block solver
    takes over when half the vertices are left."""
    s = synth.cycle_plus(500, 200, 1, 20, 5)
    c = _graph(s)
    _check_solve(s.n, c, expect=oracle.noi(s.n, *c)[0])
    g = mc.mincut_graph_from_csr(s.n, *c)
    mc.mincut_solve(g)
    mc.mincut_solve(g, mc.default_options(profile=1))
    prof = mc.mincut_profile_read(g)
    g.destroy()
    assert prof["forest"]["launches"] == 1 and prof["forest"]["ms"] < 0.25, prof
    assert prof["small_solve"]["launches"] == 2, prof


@pytest.mark.parametrize("kind", ["wheel", "unit cycle", "ladder"])
def test_thin_and_slow_in_a_batch(kind):
    """The same graphs in a batch, where what the block solver gives up goes to
    the one-warp solver."""
    graphs, expect = [], []
    for i, n in enumerate((20, 63, 64, 65, 200, 600)):
        if kind == "wheel":
            s = synth.wheel(n, seed=i)
            graphs.append((s.n, *canon(s.n, *_graph(s))))
        elif kind == "unit cycle":
            graphs.append((n, *canon(n, *G.cycle(n))))
        else:
            e = [(j, (j + 1) % n) for j in range(n)]
            e += [(n + a, n + b) for a, b in e] + [(j, n + j) for j in range(n)]
            w = np.random.default_rng(i).integers(1, 20, len(e))
            graphs.append((2 * n, *canon(2 * n, *G.from_edges(2 * n, e, [int(x) for x in w]))))
        expect.append(oracle.noi(*graphs[-1])[0])
    for kw in (dict(), dict(pr_mask=0)):
        _check_batch(graphs, expect, mc.default_options(**kw))
