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
from tests.gpu_util import dev, dev_err_word
from tests.test_gpu_allocate import _binding, _run

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


def _groups(kind, B, G, cost_sd, rng):
    """Predicted success probabilities, or an explicit sparse proxy (about two
    edges a vertex, none without one; "isolated": some without), and costs."""
    c = np.exp(cost_sd * rng.standard_normal((B, G))).astype(np.float32)
    if kind == "predicted":
        return dict(p_hat=rng.random((B, G)).astype(np.float32)), c
    keep = np.triu(rng.random((B, G, G)) < 1.5 / G, 1)
    i = np.arange(G - 1)
    if kind == "sparse":
        keep[:, i, i + 1] = True
    else:  # but for one edge, so that the objective is not flat
        keep[:, 0, 1] = True
    a = np.where(keep, rng.uniform(0.1, 2.0, (B, G, G)), 0.0).astype(np.float32)
    return dict(a=a + np.swapaxes(a, 1, 2)), c


def _solved(proxy, c, budget, pi_min):
    """Every group between its limits is solved, within its budget and to the
    duality gap of the contract. Returns the stats."""
    B = _binding()
    err = dev_err_word()
    pi, stats = B.pair_allocate(dev(c), dev(budget), pi_min, dev_err=err,
                                **{k: dev(v) for k, v in proxy.items()})
    pi, st = pi.cpu().numpy(), stats.cpu().numpy()
    total = np.add.accumulate(c.astype(np.float64), axis=1)[:, -1]
    b = budget.astype(np.float64)
    inside = (b > np.float64(np.float32(pi_min)) * total) & (b < total)
    assert inside.mean() > 0.5
    assert np.count_nonzero(st[inside, 4] != al.ALLOC_OK) == 0
    assert np.all(st[inside, 1] <= b[inside])
    assert np.all(st[inside, 2] <= 1e-12 * st[inside, 0])
    assert np.all(pi[inside] >= np.float32(pi_min)) and np.all(pi[inside] <= 1.0)
    return st


@pytest.mark.parametrize("G", [2, 3, 4, 8])
@pytest.mark.parametrize("kind", ["predicted", "sparse"])
@pytest.mark.parametrize("pi_min", [0.02, 0.08, 0.5])
def test_allocate_solves_every_ordinary_group(G, kind, pi_min):
    """100,000 groups: where the Newton system's off-diagonal row sums come near
    half its diagonal, the inner solves have to be tight enough that the steps
    go on (a tenth of the residual left 40 to 70 of 100,000 groups of 2 at the
    uniform fallback)."""
    B = 100000
    rng = np.random.default_rng(1000 * G + int(100 * pi_min))
    proxy, c = _groups(kind, B, G, 0.6, rng)
    frac = rng.uniform(max(0.15, 1.05 * pi_min), 0.9, B)
    _solved(proxy, c, (frac * c.sum(1, dtype=np.float64)).astype(np.float32), pi_min)


def test_allocate_stalled_group_of_two():
    """A group of 2 that such solves left at the fallback."""
    p = np.array([[0.97856975, 0.0509815]], np.float32)
    c = np.array([[0.79262024, 0.51749206]], np.float32)
    st = _solved(dict(p_hat=p), c, np.array([1.0323904], np.float32), 0.08)
    assert st[0, 0] < 1.4315 and st[0, 3] <= 20  # 1.497 at the uniform pi


@pytest.mark.parametrize("G", [2, 4, 8, 16])
@pytest.mark.parametrize("kind", ["predicted", "sparse"])
def test_allocate_near_the_limits_with_costs_over_decades(G, kind):
    """Budgets within 1e-6 to 1/2 of the range's ends, costs exp(3 N): the dual
    residual's rounding is above 1e-12 of the objective in some of these."""
    B, pi_min = 40000, 0.3
    rng = np.random.default_rng(77 + G)
    proxy, c = _groups(kind, B, G, 3.0, rng)
    eps = np.exp(rng.uniform(np.log(1e-6), np.log(0.5), B))
    frac = np.where(rng.random(B) < 0.5, pi_min + (1 - pi_min) * eps, 1 - (1 - pi_min) * eps)
    _solved(proxy, c, (frac * c.sum(1, dtype=np.float64)).astype(np.float32), pi_min)


@pytest.mark.parametrize("G", [3, 6, 12])
@pytest.mark.parametrize("cost_sd", [0.6, 3.0, 6.0])
def test_allocate_vertices_without_an_edge(G, cost_sd):
    """Vertices whose only curvature is the bounds' (any budget they take is as
    good as any other), budgets and costs as in the test above."""
    B, pi_min = 40000, 0.01
    rng = np.random.default_rng(99 + G)
    proxy, c = _groups("isolated", B, G, cost_sd, rng)
    eps = np.exp(rng.uniform(np.log(1e-6), np.log(0.5), B))
    frac = np.where(rng.random(B) < 0.5, pi_min + (1 - pi_min) * eps, 1 - (1 - pi_min) * eps)
    _solved(proxy, c, (frac * c.sum(1, dtype=np.float64)).astype(np.float32), pi_min)
