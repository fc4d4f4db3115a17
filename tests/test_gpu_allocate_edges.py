"""pair_allocate's interior-point solver at the edges of its kernel shapes (the
padded group sizes 8, 16, 32, 64, 128) and of its linear solver: dense graphs,
where the Newton system is nearly diagonal, and sparse ones, whose off-diagonal
row sums reach half the diagonal (the bound its Chebyshev iteration relies on),
at edge-proxy scales far from 1.

Each group is held to the KKT conditions at its returned fp32 pi (1e-5, as in
test_gpu_allocate.py: the rounding of pi), the duality gap to 1e-12 Phi (the
contract), and the expected cost to the budget."""
import numpy as np
import pytest

from oracle import allocation as al
from paper_2608_11368_gb300 import synth
from tests.test_gpu_allocate import _run

pytestmark = pytest.mark.gpu


def _check(inp, a, st, pi, stats):
    assert st == 0
    c = inp["c_hat"].astype(np.float64)
    budget = inp["budget"].astype(np.float64)
    b = al.shared_vertex_b(a)
    assert np.all(stats[:, 4] == al.ALLOC_OK)
    assert np.all(stats[:, 1] <= budget)
    assert np.all(stats[:, 2] <= 1e-12 * stats[:, 0])
    assert np.all(pi >= np.float32(inp["pi_min"])) and np.all(pi <= 1.0)
    for g in range(pi.shape[0]):
        k = al.kkt_residual(pi[g].astype(np.float64), a[g], b[g], c[g], float(budget[g]),
                            float(inp["pi_min"]), bound_tol=1e-6)
        assert k["stat"] <= 1e-5, (g, k)


@pytest.mark.parametrize("G", [2, 7, 8, 9, 16, 17, 32, 33, 64, 65, 127])
@pytest.mark.parametrize("frac,pi_min", [(0.12, 0.08), (0.5, 1e-3), (0.97, 0.05)])
def test_allocate_shapes(G, frac, pi_min):
    inp = synth.make_alloc_inputs(100 + G, 5, G, budget_frac=frac, pi_min=pi_min,
                                  score_norms=G % 2 == 0)
    a = al.edge_proxy(inp["p_hat"], inp["m_hat"])
    _check(inp, a, *_run(inp))


@pytest.mark.parametrize("G", [3, 8, 24, 64, 100])
@pytest.mark.parametrize("scale", [1e-20, 1.0, 1e12])
def test_allocate_sparse_proxy(G, scale):
    inp = synth.make_alloc_inputs(200 + G, 4, G, budget_frac=0.4)
    rng = np.random.default_rng(G)
    keep = np.triu(rng.random((4, G, G)) < 1.5 / G, 1)
    for i in range(G):  # no vertex without an edge
        j = i + 1 if i + 1 < G else 0
        keep[:, min(i, j), max(i, j)] = True
    a = np.where(keep, rng.uniform(0.1, 2.0, (4, G, G)) * scale, 0.0)
    a = (a + np.swapaxes(a, 1, 2)).astype(np.float32)
    st, pi, stats = _run(inp, explicit_a=a)
    _check(inp, a.astype(np.float64), st, pi, stats)
    assert np.array_equal(pi, _run(inp, explicit_a=a)[1])
