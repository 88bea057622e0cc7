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
