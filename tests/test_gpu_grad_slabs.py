"""The backward by slabs (bf16 hidden sizes whose workspace holds no image):
gradient tiles in the ring for both products, in dW for dH by token chunks and
for dW by vocabulary slabs, and by token chunks within a slab; one product by slabs
and the other recomputed; last 512-column
units of one and two halves, ragged vocabularies and token blocks. Each case says
how many gradient images and GEMMs its products take (0: recomputed), so that a
change of the dispatch's model shows; the narrow units' parts are checked by the
rule of the work list. Checked as in test_gpu_grad.py; reruns are bit-identical, and pair_grad_clipped (whose
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
    # d, V, B, G, len_scale: the launches the model of the dispatch picks (of the
    # gradient's image, of dH's GEMM, of dW's)
    (2496, 2050, 1, 4, 0.45, (1, 1, 1)),  # all tiles in the ring; last unit 448 columns: two halves
    (1216, 7000, 1, 8, 0.25, (1, 1, 0)),  # dH in one chunk, dW recomputed; last unit 192 columns: one half
    (2496, 5000, 2, 8, 0.28, (4, 1, 3)),  # one dH chunk and three dW slabs
    (2112, 1500, 2, 8, 0.45, (4, 2, 2)),  # two dH chunks; last units of 64 columns in half as many parts
    (3136, 9750, 1, 8, 0.1, (3, 1, 2)),   # narrow last units in half as many parts, in both products
    (1664, 2250, 1, 8, 0.05, (1, 1, 0)),  # the same in dH, tiles in the ring
    (1216, 9000, 2, 8, 0.6, (0, 0, 0)),   # chunks and slabs would cost as much: recomputed
    (4096, 3000, 1, 8, 0.25, (1, 1, 1)),  # d beyond the cluster form, minimum workspace
    (320, 777, 2, 4, 0.1, (0, 0, 0)),     # too small for either
]


def _inputs(d, V, B, G, ls, draw_hw=True):
    inp = synth.make_head_workload(synth.WORKLOADS["qwen3_1p7b_head"], 13, B=B, G=G, d=d, V=V,
                                   len_scale=ls, w_std_mult=3.0, draw_hw=draw_hw)
    a = _coeffs(inp)
    a[:2] = (0.75, -0.5)
    return inp, a


def _timed_run(inp, a, blocks):
    """_run, with the counts of its launches of (grad_image, dh_gemm_tc,
    dw_gemm_tc) and of (bwd_dh_tc, bwd_dw_tc)."""
    B = _binding()
    B.pair_timing_enable(True)
    try:
        out = _run(inp, a, blocks)
        names = [n for n, _ in B.pair_timing_read()]
    finally:
        B.pair_timing_enable(False)
    return out, tuple(names.count(n) for n in ("grad_image", "dh_gemm_tc", "dw_gemm_tc")), \
        tuple(names.count(n) for n in ("bwd_dh_tc", "bwd_dw_tc"))


def _parts(d, row_blocks, cap, nks, overhead, ncl=76):
    """Parts of the wide and the narrow units of a GEMM's last round over
    row_blocks blocks of 128 rows (tail_split in tc_kernels.cuh; 76 pairs)."""
    nq = -(-d // 512)
    n_units = (row_blocks + 1) // 2 * nq
    R = n_units % ncl
    h0 = nq - 1 - (n_units - R) % nq
    Rh = 1 + (R - 1 - h0) // nq if 0 < d % 512 <= 256 and R > h0 else 0
    best = None
    for S in range(1, min(64, nks) + 1):
        Sh = (S + 1) // 2 if Rh else S
        n = R * Sh + (R - Rh) * (S - Sh)
        if S == 1 or n <= cap:
            cost = 64 * -(-n // ncl) * (-(-nks // S) + overhead) + (16 * n if S > 1 else 0)
            best = min(best or (cost, S, Sh), (cost, S, Sh))
    return best[1:]


def _active_blocks(d, V, B, G, ls):
    inp, a = _inputs(d, 1000, B, G, ls, draw_hw=False)
    return -(-oracle.compact_tokens(inp["cu_seqlens"], inp["mask"], a)[0].size // 128)


def test_slabs_narrow_units_have_half_the_parts():
    """That the narrow cases above are split as they say (scratch tiles: what the
    first dH chunk, or all rows, leave of dW, and the ring's 24)."""
    nrb = _active_blocks(2112, 1500, 2, 8, 0.45)
    assert nrb > 32 and _parts(2112, 32, 24, 2 * 12, 20) == (6, 3)
    nrb = _active_blocks(3136, 9750, 1, 8, 0.1)
    assert _parts(3136, nrb, 199, 2 * 77, 20) == (3, 2)
    assert _parts(3136, 66, 24, 4 * nrb, 40) == (5, 3)
    assert _parts(1664, _active_blocks(1664, 2250, 1, 8, 0.05), 28, 2 * 18, 20) == (4, 2)


@pytest.mark.parametrize("d,V,B,G,ls,launches", CASES)
def test_slabs(d, V, B, G, ls, launches):
    inp, a = _inputs(d, V, B, G, ls)
    blocks = 0 if d % 512 == 0 else None
    J, dH, dW = _full_check(inp, a, image_blocks=blocks)
    (st, J2, dH2, dW2, lps, t), slabs, whole = _timed_run(inp, a, blocks)
    assert slabs == launches and whole == (int(launches[1] == 0), int(launches[2] == 0))
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
    do not fit the ring with all tokens, which then run in two chunks: four dH
    chunks, five slabs of one and five of two."""
    d, V = 4032, 2600
    inp = synth.make_head_workload(synth.WORKLOADS["qwen3_1p7b_head"], 13, B=3, G=8, d=d, V=V)
    a = np.linspace(-1.0, 1.0, inp["R"]).astype(np.float32)
    idx, _, _ = oracle.compact_tokens(inp["cu_seqlens"], inp["mask"], a)
    assert idx.size > 193 * 128
    _full_check(inp, a)
    _, slabs, whole = _timed_run(inp, a, None)
    assert slabs == (19, 4, 15) and whole == (0, 0)
