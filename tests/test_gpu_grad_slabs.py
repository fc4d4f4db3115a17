"""The backward by slabs (bf16 hidden sizes whose workspace holds no image):
gradient tiles in the ring for both products, in dW for dH by token chunks and
for dW by vocabulary slabs, and by token chunks within a slab; one product by slabs
and the other recomputed; last 512-column
units of one and two halves, ragged vocabularies and token blocks. Checked as in
test_gpu_grad.py; reruns are bit-identical, and pair_grad_clipped (whose
coefficients come after the log-sum-exp) at ratio 1 equals pair_grad."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_11368_gb300 import synth
from tests.gpu_util import dev_err_word
from tests.test_gpu_grad import _binding, _coeffs, _full_check, _run

pytestmark = pytest.mark.gpu

CASES = [
    # d, V, B, G, len_scale: the launches the model of the dispatch picks
    (2496, 2050, 1, 4, 0.45),  # all tiles in the ring; last unit 448 columns: two halves
    (1216, 7000, 1, 8, 0.25),  # dH in one chunk, dW recomputed; last unit 192 columns: one half
    (2496, 5000, 2, 8, 0.28),  # one dH chunk and three dW slabs
    (1216, 9000, 2, 8, 0.6),   # five dH chunks, narrow last units split in half as many parts
    (4096, 3000, 1, 8, 0.25),  # d beyond the cluster form, minimum workspace
    (320, 777, 2, 4, 0.1),     # too small for either
]


def _inputs(d, V, B, G, ls):
    inp = synth.make_head_workload(synth.WORKLOADS["qwen3_1p7b_head"], 13, B=B, G=G, d=d, V=V,
                                   len_scale=ls, w_std_mult=3.0)
    a = _coeffs(inp)
    a[:2] = (0.75, -0.5)
    return inp, a


@pytest.mark.parametrize("d,V,B,G,ls", CASES)
def test_slabs(d, V, B, G, ls):
    inp, a = _inputs(d, V, B, G, ls)
    blocks = 0 if d % 512 == 0 else None
    J, dH, dW = _full_check(inp, a, image_blocks=blocks)
    st, J2, dH2, dW2, lps, t = _run(inp, a, blocks)
    assert st == 0 and J2 == J and torch.equal(dH, dH2) and torch.equal(dW, dW2)
    B_ = _binding()
    err = dev_err_word()
    _, dH3, dW3, _, _ = B_.pair_grad_clipped(t["H"], t["W"], t["y"], t["mask"], t["cu_seqlens"],
                                             t["a"], lps, 0.2, dev_err=err)
    assert B_.pair_status_sync(err) == 0
    # The ratio is exp of the fp64 sum minus its fp32 rounding.
    assert (dH3 - dH).norm() <= 1e-3 * dH.norm() and (dW3 - dW).norm() <= 1e-3 * dW.norm()


def test_slabs_token_chunks():
    """More than 192 token blocks: the last slabs, of two vocabulary blocks each,
    do not fit the ring with all tokens, which then run in two chunks."""
    d, V = 4032, 2600
    inp = synth.make_head_workload(synth.WORKLOADS["qwen3_1p7b_head"], 13, B=3, G=8, d=d, V=V)
    a = np.linspace(-1.0, 1.0, inp["R"]).astype(np.float32)
    idx, _, _ = oracle.compact_tokens(inp["cu_seqlens"], inp["mask"], a)
    assert idx.size > 193 * 128
    _full_check(inp, a)
