"""pair_audit's draws kernel at the edges of its batches and teams, against the
explicit fp64 oracle: 32 draws per batch (a last batch of 1, 31, 32, 33), one
warp per batch up to G = 32 and the block's eight above, several batches per
team, weighted draws, centring, and the error bit of an invalid weight only
where a draw completes its edge. Tolerance as in test_gpu_audit.py."""
import math

import numpy as np
import pytest
import torch

import oracle
from tests.gpu_util import dev, dev_err_word
from tests.test_gpu_audit import _binding, _check, _population

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G,N", [(2, 1), (5, 31), (16, 32), (31, 33), (32, 4000), (33, 1),
                                 (64, 33), (127, 95), (128, 6000), (16, 60000)])
@pytest.mark.parametrize("wmode,center", [(oracle.W_HT, True), (oracle.W_HAJEK, False),
                                          (oracle.W_HAJEK, True)])
def test_audit_batches(G, N, wmode, center):
    B = _binding()
    D = 300 if N < 10000 else 8
    r, S, p, rho, Jd = _population(900 + G, G, D, N)
    w = np.random.default_rng(G).uniform(0.2, 1.0, N)
    M = math.comb(G, 2)
    err = dev_err_word()
    stats, bias = B.pair_audit(dev(r), dev(rho), dev(S), dev(Jd), draw_weight=dev(w), wmode=wmode,
                               scale=1.0 / M, flags=1 if center else 0, dev_err=err)
    assert B.pair_status_sync(err) == 0
    ref = oracle.audit(r, rho, S, Jd, w, scale=1.0 / M, center=center, wmode=wmode)
    _check(stats, bias, ref, rtol=2e-5)


@pytest.mark.parametrize("G,N,scale", [(2, 40, 1.0), (3, 64, 1.0), (16, 100, 120.0), (50, 70, 1.0)])
def test_audit_self_normalised_forms(G, N, scale):
    """Self-normalised estimates are about 1 / C(G, 2) of the target, and equal to it
    for complete draws of two (one edge, rho = 1): neither ||ghat||^2 nor the error
    is left to a difference that cancels. 1e-6: the fp32 sum of the weights."""
    B = _binding()
    r, S, p, rho, Jd = _population(1100 + G, G, 9, N)
    if G < 4:
        rho[:] = 1.0
        Jd[: N // 2] = 1
    err = dev_err_word()
    stats = B.pair_audit(dev(r), dev(rho), dev(S), dev(Jd), wmode=oracle.W_HAJEK, scale=scale,
                         dev_err=err)[0].cpu().numpy()
    assert B.pair_status_sync(err) == 0
    ref = oracle.audit(r, rho, S, Jd, scale=scale, wmode=oracle.W_HAJEK)
    assert abs(stats[2] - ref["cos"]) <= 1e-6
    assert abs(stats[1] - ref["mse"]) <= 1e-6 * ref["mse"]
    if G == 2:  # complete draws alone: the estimate is the target
        one = B.pair_audit(dev(r), dev(rho), dev(S), dev(Jd[:1]), wmode=oracle.W_HAJEK,
                           scale=scale)[0].cpu().numpy()
        assert one[1] <= 1e-24 * one[6] and abs(one[2] - 1.0) <= 1e-12


@pytest.mark.parametrize("G", [12, 40])
def test_audit_standardize_is_a_scale_per_draw(G):
    """One draw: standardised coefficients are the plain ones over the sample
    standard deviation of the completed rewards, so the estimate's cosine is
    unchanged and ||ghat|| scales (fp32 rounding of the coefficients)."""
    B = _binding()
    r, S, p, rho, Jd = _population(950 + G, G, 20, 1)
    Jd[:] = 1
    Jd[0, G // 2] = 0
    sd = r[Jd[0] != 0].astype(np.float64).std(ddof=1)
    out = []
    for flags in (0, 2):
        stats, bias = B.pair_audit(dev(r), dev(rho), dev(S), dev(Jd), flags=flags)
        out.append((stats.cpu().numpy(), bias.cpu().numpy()))
    M = G * r.astype(np.float64) - r.sum()
    g = (0.5 * M) @ S.astype(np.float64)
    h0, h2 = out[0][1] + g, out[1][1] + g
    assert np.linalg.norm(h2 - h0 / sd) <= 1e-5 * np.linalg.norm(h2)
    assert abs(out[0][0][2] - out[1][0][2]) <= 1e-5


@pytest.mark.parametrize("G", [9, 50])
def test_audit_invalid_weight_needs_a_completed_edge(G):
    B = _binding()
    r, S, p, rho, Jd = _population(970 + G, G, 4, 70)
    rho[2, 5] = rho[5, 2] = 0.0
    for both, want in ((0, 0), (1, 4)):
        Jd[:, 2] = 1
        Jd[:, 5] = 0
        Jd[66, 5] = both
        err = dev_err_word()
        B.pair_audit(dev(r), dev(rho), dev(S), dev(Jd), dev_err=err)
        assert B.pair_status_sync(err) == want


@pytest.mark.parametrize("G,tiny", [(8, 1e-9), (16, 1e-9), (16, 1e-39), (60, 1e-9)])
def test_audit_clipped_with_one_tiny_rho(G, tiny):
    """Clipped terms keep their split when one 1 / rho is far above w_max: the bias to
    1e-8 of itself. (With scale a power of two split terms leave some 2^-48 G of the
    largest one, fp32 sums of whole terms left 2e-8 to 7e-8 of this bias from G = 16 on.)"""
    B = _binding()
    N, w_max = 40000, 200.0
    r, S, p, rho, Jd = _population(990 + G, G, 16, N)
    r[2], r[3] = 1.0, 0.0
    rho[2, 3] = rho[3, 2] = tiny
    Jd[:, 2] = Jd[:, 3] = 0  # never completed: only the split sees it
    scale = 1.0 / 2 ** int(math.log2(math.comb(G, 2)))  # exact in fp32
    _, bias = B.pair_audit(dev(r), dev(rho), dev(S), dev(Jd), wmode=oracle.W_CLIPPED, w_max=w_max,
                           scale=scale)
    ref = oracle.audit(r, rho, S, Jd, scale=scale, wmode=oracle.W_CLIPPED, w_max=w_max)
    err = np.linalg.norm(bias.cpu().numpy() - ref["bias"]) / np.linalg.norm(ref["bias"])
    assert err <= 1e-8, err


@pytest.mark.parametrize("G,N", [(6, 40), (32, 100), (50, 64), (125, 40)])
@pytest.mark.parametrize("size", [1e-3, 1e-5, 1e-7])
def test_audit_cosine_of_small_estimates(G, N, size):
    """Coefficients far below the target's (weights clipped at `size`; every edge
    clipped): the cosine does not depend on their size, and ||ghat||^2 is not
    left to the difference of terms of the target's size. The coefficients' own
    rounding beside the target leaves 2^-53 / size of a."""
    B = _binding()
    r, S, p, rho, Jd = _population(1000 + G, G, 9, N)
    scale = 1.0 / math.comb(G, 2)
    st = [B.pair_audit(dev(r), dev(rho), dev(S), dev(Jd), wmode=oracle.W_CLIPPED, w_max=w,
                       scale=scale)[0].cpu().numpy() for w in (1.0, size)]
    ref = oracle.audit(r, rho, S, Jd, scale=scale, wmode=oracle.W_CLIPPED, w_max=np.float32(size))
    assert abs(st[1][2] - ref["cos"]) <= 1e-6 * abs(ref["cos"])
    assert abs(st[1][2] - st[0][2]) <= 1e-6 * abs(ref["cos"])
    assert abs(st[1][1] - ref["mse"]) <= 1e-6 * ref["mse"]


@pytest.mark.parametrize("G", [7, 32, 100])
def test_audit_standardize_by_the_exact_deviation(G):
    """Rewards around 1000: the coefficients are the plain ones over the fp64 sample
    standard deviation (two-pass fp32 sums left 1e-8 to 2e-7 of it)."""
    B = _binding()
    r, S, p, rho, Jd = _population(960 + G, G, 20, 1)
    r = (1000.0 + np.random.default_rng(G).standard_normal(G)).astype(np.float32)
    Jd[:] = 1
    Jd[0, G // 2] = 0
    sd = r[Jd[0] != 0].astype(np.float64).std(ddof=1)
    g = 0.5 * (G * r.astype(np.float64) - r.astype(np.float64).sum()) @ S.astype(np.float64)
    h = [B.pair_audit(dev(r), dev(rho), dev(S), dev(Jd), flags=f)[1].cpu().numpy() + g
         for f in (0, 2)]
    assert np.linalg.norm(h[1] - h[0] / sd) <= 1e-11 * np.linalg.norm(g)


def test_audit_largest_draw_count():
    """N = 2^31 - 1 draws (4.3 GB of flags): the batch count is formed beyond 32 bits."""
    B = _binding()
    N = 2 ** 31 - 1
    r, S, p, rho, _ = _population(991, 2, 3, 1)
    Jd = torch.ones(N, 2, dtype=torch.uint8, device="cuda")
    Jd[N - 1] = 0
    stats, _ = B.pair_audit(dev(r), dev(rho), dev(S), Jd)
    st = stats.cpu().numpy()
    assert abs(st[7] - 1.0) <= 1e-6 and abs(st[3] - 2.0 * (N - 1) / N) <= 1e-6
    assert abs(st[4] - (N - 1) / N) <= 1e-6 and st[1] > 0
