"""Contraction to few vertices through a dense triangle: bit-exact against the
oracle at the sizes where its branches change (one vertex, triangles with many
copies, one copy, none; the largest vertex count the rule takes and the next),
uneven groups, 64-bit totals, and the degrees the next round reads."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")

import paper_2609_07204_gb300 as mc  # noqa: E402
from tests.test_gpu_parity import _cuda, assert_csr_equal, make  # noqa: E402,F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,whi,n2,skew", [
    (60, 511, 9, 12, 0), (60, 512, 9, 32, 0), (60, 512, 9, 33, 0), (300, 2047, 9, 63, 0),
    (300, 2047, 9, 64, 0), (5000, 60_000, 100, 1, 0), (5000, 60_000, 100, 2, 0),
    (5000, 60_000, 100, 23, 0), (5000, 60_000, 100, 24, 0), (5000, 60_000, 100, 346, 0),
    (5000, 60_000, 100, 347, 0), (20_001, 230_001, 1, 128, 0), (20_001, 230_001, 1, 129, 0),
    (20_001, 230_001, 10, 150, 1), (20_001, 230_001, 10, 6, 1), (20_001, 230_001, 1, 600, 1),
    (20_001, 230_001, 1 << 20, 5, 0), (20_001, 230_001, 1 << 20, 64, 0),
    (20_001, 230_001, 1 << 20, 200, 1)])
def test_contract_to_few_vertices(n, m, whi, n2, skew):
    rng = np.random.default_rng(n + n2)
    g0 = synth.er(n, m, 1, whi, 5)
    groups = rng.integers(0, n2, n).astype(np.int32)
    groups[:n2] = np.arange(n2)
    if skew:  # most vertices in two groups
        groups[n2:] = np.where(rng.random(n - n2) < 0.9, rng.integers(0, 2, n - n2), groups[n2:])
    g = make(n, g0.row_ptr, g0.col, g0.w)
    ro = mc.default_round_options()
    ro.groups = groups.ctypes.data
    assert mc.mincut_contract_round(g, ro)["n_out"] == n2
    _, L = oracle.labels_from_groups(groups)
    exp = oracle.contract(n, g0.row_ptr, g0.col, g0.w, L, n2)
    assert_csr_equal(mc.mincut_graph_export_csr(g), exp)
    if n2 > 2:  # a round that only looks at the degrees
        ro = mc.default_round_options()
        ro.lp_iters = 0
        ro.pr_mask = 0
        ro.capforest = 0
        ro.lambda_in = mc.INT64_MAX
        deg = np.add.reduceat(exp[2].astype(np.int64), exp[0][:-1])
        assert mc.mincut_contract_round(g, ro)["lambda_out"] == deg.min()
    g.destroy()


@pytest.mark.parametrize("whi", [1, 4000])
def test_own_triangles_of_many_tiles(whi):
    """Enough entries that a block sums several tiles in triangles of its own:
    the vertex counts around which the copies that fit beside the tile's rows
    change (91: one copy fewer, or none), 32-bit and 64-bit totals."""
    n, m = 200_000, 5_100_000
    g0 = synth.er(n, m, 1, whi, 5)
    g = make(n, g0.row_ptr, g0.col, g0.w)
    rng = np.random.default_rng(whi)
    for n2 in (90, 91, 92, 128, 129):
        groups = rng.integers(0, n2, n).astype(np.int32)
        groups[:n2] = np.arange(n2)
        ro = mc.default_round_options()
        ro.groups = groups.ctypes.data
        mc.mincut_graph_reset(g)
        assert mc.mincut_contract_round(g, ro)["n_out"] == n2
        exp = oracle.contract(n, g0.row_ptr, g0.col, g0.w, oracle.labels_from_groups(groups)[1], n2)
        assert_csr_equal(mc.mincut_graph_export_csr(g), exp)
    g.destroy()


def test_refused_groups_leave_the_graph():
    g0 = synth.er(5000, 60_000, 1, 9, 5)
    g = make(5000, g0.row_ptr, g0.col, g0.w)
    groups = np.zeros(5000, np.int32)
    groups[17] = 5000
    ro = mc.default_round_options()
    ro.groups = groups.ctypes.data
    with pytest.raises(mc.MincutError) as e:
        mc.mincut_contract_round(g, ro)
    assert e.value.status == mc.MINCUT_ERR_INVALID
    assert_csr_equal(mc.mincut_graph_export_csr(g), (g0.row_ptr, g0.col, g0.w))
    g.destroy()
