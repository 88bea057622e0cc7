"""Packed batch solve (many independent graphs in one CSR) against the oracle:
every graph's value equals the oracle's, and every graph's side (from the
shared bitmap) has that cut weight with both sides non-empty."""
import numpy as np
import pytest

import oracle
import synth
from tests import graphs as G

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2609_07204_gb300 as mc  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    mc.load_library()


def _check_batch(graphs, expect, opts=None):
    vo, rp, col, w = mc.pack_graphs(graphs)
    B = mc.mincut_batch_from_csr(vo, rp, col, w)
    vals, bm, st = mc.mincut_batch_solve(B, opts)
    side_all = mc.bitmap_to_side(bm, int(vo[-1]))
    for i, (n, grp, gcol, gw) in enumerate(graphs):
        assert vals[i] == expect[i], (i, n, vals[i], expect[i])
        side = side_all[vo[i]:vo[i + 1]]
        assert side[0] == 0 and 0 < side.sum() < n, i
        assert oracle.cut_weight(n, grp, gcol, gw, side) == vals[i], i
    B.destroy()
    return st


def test_batch_random_small_graphs():
    rng = np.random.default_rng(91)
    graphs, expect = [], []
    for i in range(300):
        n = int(rng.integers(2, 50))
        g = G.random_graph(n, float(rng.uniform(0.05, 0.9)), rng, 1, int(rng.integers(1, 60)))
        c = oracle.canonicalize(n, *g)
        graphs.append((n, c[0], c[1], c[2]))
        expect.append(oracle.stoer_wagner(n, *c)[0])
    _check_batch(graphs, expect)
    _check_batch(graphs, expect, mc.default_options(deterministic=1))
    # every graph in the shared round kernels; every graph on its own warp;
    # both at once
    for small in (-1, 2048, 20):
        _check_batch(graphs, expect, mc.default_options(batch_small_n=small))


def test_batch_closed_forms_and_disconnected():
    cases = [(G.cycle(30), 30, 2), (G.complete(9), 9, 8), (G.hypercube(5), 32, 5),
             (G.grid(6, 7), 42, 2), (G.two_cliques(7, 1, 6, 2), 14, 2),
             (G.from_edges(5, [(0, 1), (2, 3)], [4, 4]), 5, 0),
             (G.from_edges(2, [(0, 1)], [7]), 2, 7)]
    graphs = []
    for c, n, lam in cases:
        cc = oracle.canonicalize(n, *c)
        graphs.append((n, cc[0], cc[1], cc[2]))
    for small in (0, -1, 2048, 10):
        _check_batch(graphs, [lam for _, _, lam in cases], mc.default_options(batch_small_n=small))


def test_batch_workload_subset_vs_noi():
    graphs, expect = [], []
    for i in range(256):
        s = synth.batch_graph(4, i)
        graphs.append((s.n, s.row_ptr, s.col, s.w.astype(np.int64)))
        expect.append(oracle.noi(s.n, s.row_ptr, s.col, s.w)[0])
    _check_batch(graphs, expect)  # threshold chosen by timing
    st = _check_batch(graphs, expect, mc.default_options(batch_small_n=-1))
    assert st["rounds"] >= 1
    st = _check_batch(graphs, expect, mc.default_options(batch_small_n=2048))
    assert st["rounds"] == 0  # every graph solved by its own warp
    _check_batch(graphs, expect, mc.default_options(batch_small_n=300))


def test_batch_warp_path_weighted_and_pr_variants():
    """The one-warp-per-graph solver on weighted graphs up to its size
    limit, with and without the PR tests (it applies PR1 / PR2 of the mask),
    against Stoer-Wagner."""
    rng = np.random.default_rng(17)
    graphs, expect = [], []
    for i in range(24):
        n = int(rng.integers(100, 700)) if i % 4 else 2048
        s = synth.er_connected(n, int(n * rng.uniform(2.0, 7.0)), 1, 100, 300 + i)
        c = (s.row_ptr, s.col, s.w.astype(np.int64))
        graphs.append((n, *c))
        expect.append(oracle.stoer_wagner(n, *c)[0])
    for mask in (0xF, 0x1, 0x0):
        _check_batch(graphs, expect, mc.default_options(batch_small_n=2048, pr_mask=mask))


def test_warp_solver_weighted_and_pr_variants():
    """The one-warp solver itself (deterministic mode) on weighted graphs up to
    its size limit, with and without the PR tests, against NOI; twice each, so
    that its launches are also captured."""
    rng = np.random.default_rng(18)
    graphs, expect = [], []
    for i in range(24):
        n = int(rng.integers(100, 700)) if i % 4 else 2048
        s = synth.cycle_plus(n, rng.uniform(4.0, 14.0), 1, 100, 300 + i)
        graphs.append((n, s.row_ptr, s.col, s.w.astype(np.int64)))
        expect.append(oracle.noi(*graphs[-1])[0])
    vo, rp, col, w = mc.pack_graphs(graphs)
    B = mc.mincut_batch_from_csr(vo, rp, col, w)
    for mask in (0xF, 0x3, 0x1, 0x0):
        for _ in range(2):
            _solve_and_check(B, vo, graphs, expect, mc.default_options(
                deterministic=1, batch_small_n=2048, pr_mask=mask))
    B.destroy()


def test_replay_follows_the_mode():
    """Captured launches of the block and of the warp solver on one batch: a
    change of mode takes the other's launches, not the captured ones."""
    graphs, expect = [], []
    for i in range(60):
        s = synth.batch_graph(4, 2000 + i)
        graphs.append((s.n, s.row_ptr, s.col, s.w.astype(np.int64)))
        expect.append(oracle.noi(s.n, s.row_ptr, s.col, s.w)[0])
    vo, rp, col, w = mc.pack_graphs(graphs)
    B = mc.mincut_batch_from_csr(vo, rp, col, w)
    launches = {0: set(), 1: set()}
    for det in (0, 0, 0, 1, 1, 1, 0, 1, 0, 0, 0):
        st = _solve_and_check(B, vo, graphs, expect, mc.default_options(deterministic=det))
        launches[det].add(st["kernel_launches"])
    assert len(launches[0]) == len(launches[1]) == 1 and launches[0] != launches[1]
    B.destroy()


def _solve_and_check(B, vo, graphs, expect, opts):
    vals, bm, st = mc.mincut_batch_solve(B, opts)
    side_all = mc.bitmap_to_side(bm, int(vo[-1]))
    for i, (n, grp, gcol, gw) in enumerate(graphs):
        assert vals[i] == expect[i], (i, n, vals[i], expect[i])
        side = side_all[vo[i]:vo[i + 1]]
        assert side[0] == 0 and 0 < side.sum() < n, i
        assert oracle.cut_weight(n, grp, gcol, gw, side) == vals[i], i
    return st


@pytest.mark.parametrize("own_stream", [False, True])
def test_batch_repeated_solves_replay_captured_launches(own_stream):
    """Solving the same batch again (every graph on its own warp) replays the
    launches captured as a CUDA graph at the second solve; a changed PR mask,
    a round-kernel solve in between (which swaps the offsets buffer) and a
    profiled solve take the direct launches or a new capture.  Every solve
    matches the oracle."""
    graphs, expect = [], []
    for i in range(160):
        s = synth.batch_graph(4, 1000 + i)
        graphs.append((s.n, s.row_ptr, s.col, s.w.astype(np.int64)))
        expect.append(oracle.noi(s.n, s.row_ptr, s.col, s.w)[0])
    vo, rp, col, w = mc.pack_graphs(graphs)
    strm = torch.cuda.Stream() if own_stream else None
    B = mc.mincut_batch_from_csr(vo, rp, col, w, stream=strm)
    warp = mc.default_options(batch_small_n=2048)
    launches = set()
    for _ in range(4):
        launches.add(_solve_and_check(B, vo, graphs, expect, warp)["kernel_launches"])
    assert len(launches) == 1  # the replayed graph launches the same kernels
    for _ in range(3):
        _solve_and_check(B, vo, graphs, expect, mc.default_options(batch_small_n=2048, pr_mask=0x1))
    _solve_and_check(B, vo, graphs, expect, mc.default_options(batch_small_n=-1))
    for _ in range(3):
        _solve_and_check(B, vo, graphs, expect, warp)
    _solve_and_check(B, vo, graphs, expect, mc.default_options(batch_small_n=2048, profile=1))
    _solve_and_check(B, vo, graphs, expect, warp)
    B.destroy()


@pytest.mark.parametrize("det", [0, 1])
def test_batch_tiny_graphs(det):
    """Around the sizes at which a graph goes to a warp instead of a block
    (32 vertices; 64 with six entries per vertex), alone and mixed."""
    rng = np.random.default_rng(5)
    graphs = []
    for n in (3, 4, 31, 32, 33, 63, 64, 65):
        for deg in (2.2, 5.8, 6.2, 12):
            s = synth.cycle_plus(n, min(deg, n - 1), 1, 50, int(rng.integers(1 << 30)))
            graphs.append((s.n, *oracle.canonicalize(s.n, s.row_ptr, s.col, s.w.astype(np.int64))))
    expect = [oracle.stoer_wagner(*g)[0] for g in graphs]
    opts = mc.default_options(deterministic=det)
    _check_batch(graphs, expect, opts)
    tiny = [i for i, g in enumerate(graphs) if g[0] <= 32]
    big = [i for i, g in enumerate(graphs) if g[0] > 64]
    for part in (tiny, big):
        _check_batch([graphs[i] for i in part], [expect[i] for i in part], opts)


def test_batch_tiny_graphs_are_no_slower_than_warps():
    """4,096 dense graphs of 8 vertices: the default batch takes the time of
    the one-warp solver (2.8 times that by a block each)."""
    rng = np.random.default_rng(7)
    g = [(8, *G.complete(8, int(w))) for w in rng.integers(1, 100, 4096)]
    B = mc.mincut_batch_from_csr(*mc.pack_graphs(g))
    ms = []
    for det in (0, 1):
        opts = mc.default_options(deterministic=det)
        times = [mc.mincut_batch_solve(B, opts)[2]["ms_total"] for _ in range(9)]
        ms.append(sorted(times)[4])
    B.destroy()
    assert ms[0] < 1.5 * ms[1], ms


@pytest.mark.parametrize("det", [0, 1])
def test_batch_dense_graphs(det):
    """Graphs of 20,000 entries and 24 per vertex, and just below either: the
    former take the round kernels, alone and among others, and a batch of them
    no longer than by warps."""
    rng = np.random.default_rng(3)
    dense, other = [], []
    for n, m, part in ((600, 24_000, dense), (300, 10_000, dense), (800, 10_000, dense),
                       (833, 9_999, other), (860, 10_100, other), (100, 4_950, other)):
        u, v = np.triu_indices(n, 1)
        pick = rng.choice(len(u), m, replace=False)
        w = rng.integers(1, 21, m)
        c = oracle.canonicalize(n, *G.from_edges(n, np.stack([u[pick], v[pick]], 1), w))
        part.append((n, *c))
    for graphs in (dense, other, other + dense):
        expect = [oracle.noi(*g)[0] for g in graphs]
        st = _check_batch(graphs, expect, mc.default_options(deterministic=det))
        assert st["rounds"] > 0 or graphs is other
    B = mc.mincut_batch_from_csr(*mc.pack_graphs(dense))
    ms = []
    for small in (0, 2048):
        opts = mc.default_options(deterministic=det, batch_small_n=small)
        ms.append(min(mc.mincut_batch_solve(B, opts)[2]["ms_total"] for _ in range(5)))
    B.destroy()
    assert ms[0] < ms[1], ms


@pytest.mark.parametrize("det", [0, 1])
@pytest.mark.parametrize("kind", ["wheels", "interleaved cycles", "unit cycles", "mixed"])
def test_batch_graphs_given_up(kind, det):
    """Graphs that the block and the warp solver give up share rounds with all
    the PR tests, then take a warp each where those do not help; alone, among
    ordinary ones, repeatedly (captured launches) and with fewer PR tests."""
    graphs = []
    if kind in ("wheels", "mixed"):
        graphs += [synth.wheel(n, seed=n) for n in (40, 63, 64, 65, 66, 200, 301, 600)]
    if kind in ("interleaved cycles", "mixed"):
        graphs += [synth.dblcyc(n, seed=n) for n in (34, 66, 130)]
    if kind == "mixed":
        graphs += [synth.batch_graph(4, i) for i in range(40)]
    graphs = [(s.n, s.row_ptr, s.col, s.w.astype(np.int64)) for s in graphs]
    if kind in ("unit cycles", "mixed"):
        graphs += [(n, *oracle.canonicalize(n, *G.cycle(n))) for n in (64, 65, 300)]
    expect = [oracle.noi(*g)[0] for g in graphs]
    vo, rp, col, w = mc.pack_graphs(graphs)
    B = mc.mincut_batch_from_csr(vo, rp, col, w)
    opts = mc.default_options(deterministic=det)
    for _ in range(4):
        st = _solve_and_check(B, vo, graphs, expect, opts)
        assert st["rounds"] > 0
    _solve_and_check(B, vo, graphs, expect, mc.default_options(deterministic=1 - det))
    for mask in (0x7, 0x3, 0):
        _solve_and_check(B, vo, graphs, expect, mc.default_options(deterministic=det, pr_mask=mask))
    _solve_and_check(B, vo, graphs, expect, opts)
    B.destroy()


def test_ordinary_graphs_take_no_shared_rounds():
    """What the blocks leave of an ordinary batch a warp each finishes: rounds
    over the whole batch would cost more than all the rest."""
    graphs = [synth.batch_graph(4, 5000 + i) for i in range(1200)]
    B = mc.mincut_batch_from_csr(*mc.pack_graphs([(s.n, s.row_ptr, s.col, s.w) for s in graphs]))
    for _ in range(8):
        assert mc.mincut_batch_solve(B, bitmap=False)[2]["rounds"] == 0
    B.destroy()


@pytest.mark.parametrize("det", [0, 1])
@pytest.mark.parametrize("kind", ["given up", "dense"])
def test_no_room_for_rounds(kind, det):
    """No memory for the contractions of shared rounds: a warp each finishes
    the graphs that were given up, and the dense ones, as it needs none."""
    import ctypes

    class Limited(mc._TorchAllocator):
        def __init__(self, device):
            super().__init__(device)
            self.left, self.refuse = 1 << 30, 0
            give = self._alloc

            def _alloc(nbytes, stream, ctx):
                self.left -= 1
                self.refuse -= 1
                return None if self.left < 0 or self.refuse >= 0 else give(nbytes, stream, ctx)

            self._give, self._alloc = give, type(give)(_alloc)
            self.struct = mc.MincutAllocator(self._alloc, self._free, None)

    graphs = ([synth.wheel(n, seed=n) for n in (70, 90, 130)] if kind == "given up" else
              [synth.cycle_plus(500, 50, 1, 20, i) for i in range(3)])
    graphs = [(s.n, s.row_ptr, s.col, s.w.astype(np.int64)) for s in graphs]
    expect = [oracle.noi(*g)[0] for g in graphs]
    vo, rp, col, w = mc.pack_graphs(graphs)
    keep = [np.ascontiguousarray(vo, np.int64), np.ascontiguousarray(rp, np.int64),
            np.ascontiguousarray(col, np.int32), np.ascontiguousarray(w, np.int32)]
    alloc, out = Limited(0), ctypes.c_void_p(0)
    rc = mc.load_library().mincut_batch_from_csr(
        len(vo) - 1, *(a.ctypes.data for a in keep), mc.MINCUT_HOST_PTRS, ctypes.c_void_p(0),
        ctypes.byref(alloc.struct), ctypes.byref(out))
    assert rc == 0
    B = mc.Graph(out.value, int(vo[-1]), keep, alloc)
    B.G, B.vertex_offsets = len(vo) - 1, keep[0]
    alloc.left = 4 if kind == "given up" else 1 << 30  # the small-graph solvers' lists and scratch
    for _ in range(3):
        alloc.refuse = 2 if kind == "dense" else 0  # the buffers as one block, then the first
        _solve_and_check(B, vo, graphs, expect, mc.default_options(deterministic=det))
        assert mc.mincut_last_error() == ""
    alloc.left = 1 << 30
    _solve_and_check(B, vo, graphs, expect, mc.default_options(deterministic=det))
    B.destroy()


@pytest.mark.parametrize("det", [0, 1])
def test_batch_of_wheels_is_no_slower_than_rounds(det):
    """40 wheels of about 250 vertices: no more than twice the time of the
    round kernels, which solve them in one round (60 times by warps)."""
    graphs = [synth.wheel(230 + i, seed=i) for i in range(40)]
    B = mc.mincut_batch_from_csr(*mc.pack_graphs([(s.n, s.row_ptr, s.col, s.w) for s in graphs]))
    ms = []
    for small in (0, -1):
        opts = mc.default_options(deterministic=det, batch_small_n=small)
        ms.append(sorted(mc.mincut_batch_solve(B, opts)[2]["ms_total"] for _ in range(7))[3])
    B.destroy()
    assert ms[0] < 2 * ms[1], ms


def test_batch_rejects_cross_graph_edge_and_tiny_graph():
    c1 = oracle.canonicalize(3, *G.cycle(3))
    c2 = oracle.canonicalize(3, *G.cycle(3))
    vo, rp, col, w = mc.pack_graphs([(3, *c1), (3, *c2)])
    col = col.copy()
    col[0] = 4  # 0 -> 4 crosses into the second graph (and breaks symmetry)
    with pytest.raises(mc.MincutError) as e:
        mc.mincut_batch_from_csr(vo, rp, col, w, skip_validate=True)
    assert e.value.status == mc.MINCUT_ERR_INVALID
    vo2 = np.array([0, 1, 6], np.int64)
    with pytest.raises(mc.MincutError):
        mc.mincut_batch_from_csr(vo2, rp, col, w)
