"""The recomputing backward of bf16 hidden sizes without an image (a row block
and 256 columns of d per CTA; two row blocks and 384 columns per CTA pair): last
slices of 64 to 256 and 64 to 384 columns, one, odd and even numbers of token and vocabulary
blocks, ragged ends of both, units split over parts of the other side (scratch
in the ring and in dW), and more units than CTAs. Checked as in
test_gpu_grad.py; reruns are bit-identical."""
import pytest
import torch

from paper_2608_11368_gb300 import synth
from tests.test_gpu_grad import _coeffs, _full_check, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,V,B,G,ls", [
    (64, 100, 1, 4, 0.01),      # less than one block of either side
    (64, 300, 1, 2, 0.05),      # one column of K per tile, three vocabulary blocks
    (128, 1111, 1, 4, 0.1),
    (192, 640, 2, 4, 0.1),      # whole vocabulary blocks, an odd number
    (320, 777, 2, 4, 0.2),      # a second slice of 64 columns
    (448, 257, 1, 8, 0.3),      # of 192
    (640, 2000, 1, 4, 0.06),
    (128, 24000, 1, 4, 0.2),    # dW: more units than pairs
    (256, 16000, 1, 4, 0.3),    # dH split, its scratch in dW
    (320, 2100, 2, 8, 0.3),     # pairs with one slice
    (384, 4001, 1, 8, 0.4),     # a whole one
    (704, 2100, 2, 8, 0.3),     # pairs, an odd number of vocabulary blocks, dW split
    (960, 1024, 2, 8, 0.3),     # dW in pairs; three slices, the last of 192
    (768, 2048, 1, 8, 0.3),     # two whole slices
    (832, 2500, 1, 8, 0.3),     # a last slice of 64
    (640, 5000, 2, 8, 0.5),     # of 256
])
def test_recompute(d, V, B, G, ls):
    inp = synth.make_head_workload(synth.WORKLOADS["qwen3_1p7b_head"], 17, B=B, G=G, d=d, V=V,
                                   len_scale=ls, w_std_mult=2.0)
    a = _coeffs(inp)
    a[:2] = (0.75, -0.5)
    J, dH, dW = _full_check(inp, a)
    st, J2, dH2, dW2, _, _ = _run(inp, a, None)
    assert st == 0 and J2 == J and torch.equal(dH, dH2) and torch.equal(dW, dW2)
