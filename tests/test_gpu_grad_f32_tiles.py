"""The fp32 head's tiled kernels at their edges, against the fp64 oracle: one
column slice and several per cluster (d up to 2048, and beyond, where the
row-by-row form runs), slices of unequal width, vocabularies below, at and
past a tile of 32 rows, fewer tokens than a tile, more parts than tiles, and
a target that many tokens share.

Tolerance: a logit is a sum over d in 16-term pieces, so it is off by at most
(16 + d / 16 / C) 2^-24 sum |h_k w_k| <= 5e-5 for d <= 2048 and logits of unit
variance, and p = exp(z - lse) by twice that; the one-hot parts and the sums
over tokens or vocabulary add a few 2^-24. Hence 1e-4 of the softmax part (its
own norm) and of the whole."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_11368_gb300 import synth
from tests.gpu_util import rel_fro
from tests.test_gpu_grad import _coeffs, _run

pytestmark = pytest.mark.gpu

TOL = 1e-4


def _case(d, V, B, G, ls, seed=3):
    inp = synth.make_head_workload(synth.WORKLOADS["pr1_ref_fp32"], seed, B=B, G=G, d=d, V=V,
                                   len_scale=ls)
    a = _coeffs(inp)
    a[0] = 0.75
    return inp, a


@pytest.mark.parametrize("d,V,B,G,ls", [
    (16, 1, 1, 2, 0.02), (48, 31, 1, 4, 0.1), (256, 32, 2, 4, 0.3), (256, 33, 2, 8, 1.0),
    (256, 5000, 1, 2, 0.05), (272, 500, 2, 4, 0.5), (528, 777, 2, 4, 0.4), (1040, 300, 1, 4, 0.3),
    (2032, 257, 1, 4, 0.3), (2048, 700, 2, 4, 0.2), (2064, 100, 1, 4, 0.1)])
def test_f32_tiles(d, V, B, G, ls):
    inp, a = _case(d, V, B, G, ls)
    st, J, dH, dW, lps, _ = _run(inp, a)
    assert st == 0
    ref = oracle.pair_grad_ref(inp, a.astype(np.float64), full=True)
    dHn, dWn = dH.cpu().numpy().astype(np.float64), dW.cpu().numpy().astype(np.float64)
    assert abs(J - ref["J"]) <= TOL * max(ref["J_abs"], 1e-30)
    np.testing.assert_allclose(lps.cpu().numpy(), ref["logp_seq"], rtol=1e-5, atol=1e-4)
    if V > 1:  # with one vocabulary row both gradients are exactly 0
        assert rel_fro(dHn, ref["dH"]) <= TOL
        assert rel_fro(dWn, ref["dW"]) <= TOL
    idx, c, _ = oracle.compact_tokens(inp["cu_seqlens"], inp["mask"], a)
    Wf, y = inp["W"].astype(np.float64), inp["y"][idx]
    one_h = c[:, None] * Wf[y]
    one_w = np.zeros_like(Wf)
    np.add.at(one_w, y, c[:, None] * inp["H"][idx].astype(np.float64))
    assert rel_fro(dHn[idx] - one_h, ref["dH"][idx] - one_h) <= TOL
    assert rel_fro(dWn - one_w, ref["dW"] - one_w) <= TOL
    again = _run(inp, a)
    assert again[1] == J and torch.equal(again[2], dH) and torch.equal(again[3], dW)


def test_f32_tiles_no_active_token_and_shared_target():
    inp, a = _case(272, 200, 2, 4, 0.5)
    st, J, dH, dW, lps, _ = _run(inp, np.zeros_like(a))
    assert st == 0 and J == 0.0 and (dH == 0).all() and (dW == 0).all() and (lps == 0).all()
    inp["y"][inp["mask"] != 0] = 70
    st, J, dH, dW, _, _ = _run(inp, a)
    ref = oracle.pair_grad_ref(inp, a.astype(np.float64), full=True)
    assert st == 0
    assert rel_fro(dW.cpu().numpy(), ref["dW"]) <= TOL
    assert rel_fro(dH.cpu().numpy(), ref["dH"]) <= TOL
