"""The streaming coefficient kernel's form for group sizes that are no multiple
of 4 and for inputs without the alignment of bulk copies (clipped and
self-normalised weighting): every G up to 64 against the fp64 oracle beside the
HT forms (coefficients to 1e-6 of 1/2 sum |term|, counts exact), misaligned
arrays, quotients of any rho > 0 (a subnormal or a huge one is accepted), the
error bit only for completed edges, and the dense estimator's coefficients,
which are pair_coeffs' bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_11368_gb300 import synth
from tests.gpu_util import dev, dev_err_word
from tests.test_gpu_audit import _binding

pytestmark = pytest.mark.gpu


def _inputs(G, B=37):
    wl = synth.WORKLOADS["coeffs_dense_stress"]
    inp = synth.draw_group_inputs(wl, 300 + G, B, G)
    inp["J"][0], inp["J"][1] = 0, 1
    return inp


def _shifted(x):
    """A copy of x that starts one element past an aligned address."""
    t = torch.empty(x.numel() + 1, dtype=x.dtype, device="cuda")[1:].view(x.shape)
    return t.copy_(x)


@pytest.mark.parametrize("G", list(range(2, 65)))
def test_every_group_size(G):
    B = _binding()
    inp = _inputs(G)
    r, J, rho = dev(inp["r"]), dev(inp["J"]), dev(inp["rho"])
    if G % 4 == 0:
        r, J, rho = _shifted(r), _shifted(J), _shifted(rho)
    ref = oracle.coeffs(inp["r"], inp["J"], inp["rho"], scale=0.5)
    err = dev_err_word()
    for wmode in (None, B.PAIR_W_HT, B.PAIR_W_CLIPPED, B.PAIR_W_HAJEK):
        if wmode is None:
            out = B.pair_coeffs(r, J, rho, scale=0.5, dev_err=err)
        else:
            out = B.pair_coeffs_weighted(r, J, rho, wmode=wmode, w_max=5.0, scale=0.5, dev_err=err)
        assert B.pair_status_sync(err) == 0
        a = out[0].cpu().numpy().astype(np.float64)
        for k, name in enumerate(("active", "edges", "contrast")):
            assert np.array_equal(out[1 + k].cpu().numpy(), ref[name]), name
        if wmode in (None, B.PAIR_W_HT):
            assert (np.abs(a - ref["a"]) <= 1e-6 * ref["a_mag"]).all()
        else:
            w = oracle.coeffs_w(inp["r"], inp["J"], inp["rho"], scale=0.5, wmode=wmode, w_max=5.0)
            lim = 2e-6 * np.abs(w["a"]).max(axis=1, keepdims=True) * np.sqrt(G)
            assert (np.abs(a - w["a"]) <= lim + 1e-30).all()
            np.testing.assert_allclose(out[4].cpu().numpy(), w["ess"], rtol=2e-5)
    g, a2 = B.pair_estimate_dense(r, J, rho, torch.ones(37, G, 5, device="cuda"), scale=0.5,
                                  a=torch.empty(37, G, device="cuda"))
    assert torch.equal(a2, B.pair_coeffs(r, J, rho, scale=0.5)[0])


def test_subnormal_and_invalid_rho():
    B = _binding()
    G = 6
    r = np.array([[1, 0, 1, 0, 1, 0]], np.float32)
    rho = np.full((1, G, G), 0.5, np.float32)
    rho[0, 1, 3], rho[0, 2, 5], rho[0, 0, 1] = 2e-38, 0.0, 3e37
    for J, want in (([1, 1, 1, 1, 0, 0], 0), ([1, 1, 1, 1, 0, 1], 4)):
        err = dev_err_word()
        J = np.array([J], np.uint8)
        a = B.pair_coeffs(dev(r), dev(J), dev(rho), dev_err=err)[0].cpu().numpy()
        assert B.pair_status_sync(err) == want
        b = B.pair_coeffs_weighted(dev(r), dev(J), dev(rho), wmode=B.PAIR_W_CLIPPED, w_max=3e38,
                                   dev_err=err)[0].cpu().numpy()
        assert B.pair_status_sync(err) == want
        if not want:
            ref = oracle.coeffs(r, J, rho)
            assert (np.abs(a - ref["a"]) <= 1e-6 * ref["a_mag"]).all()
            assert (np.abs(b - ref["a"]) <= 1e-6 * ref["a_mag"]).all()


@pytest.mark.parametrize("dr,p01", [(1e5, 1e-36), (3e38, 0.25), (np.inf, 0.5), (1e-38, 0.3),
                                    (1e30, 1e-12), (7e-20, 1e25)])
def test_quotients_beyond_the_range(dr, p01):
    """Terms that overflow are infinite, not NaN, and tiny ones are rounded like
    the IEEE quotient: one contrast edge, whose coefficients are +-1/2 of it."""
    B = _binding()
    G = 3
    r = np.array([[dr, 0.0, 0.0]], np.float32)
    rho = np.full((1, G, G), p01, np.float32)
    J = np.array([[1, 1, 0]], np.uint8)
    with np.errstate(over="ignore"):
        want = np.float32(0.5) * (np.float32(dr) / np.float32(p01))
    err = dev_err_word()
    a = B.pair_coeffs_weighted(dev(r), dev(J), dev(rho), wmode=B.PAIR_W_CLIPPED, w_max=3e38,
                               dev_err=err)[0].cpu().numpy()
    assert B.pair_status_sync(err) == 0
    assert a.tolist() == [[float(want), -float(want), 0.0]]
