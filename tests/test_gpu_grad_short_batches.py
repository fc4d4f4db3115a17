"""Short token batches on wide vocabularies: the log-sum-exp pass with the
split count its makespan rule picks (up to 64, any number), and the backward
GEMMs whose last, or only, round deals the K steps of a few units to all
clusters, in one or two segments per cluster; with the scratch in dW (first
chunk) and in the workspace (later chunks, vocabularies smaller than that).
Checked as in test_gpu_grad.py, and reruns are bit-identical."""
import pytest
import torch

import oracle
from paper_2608_11368_gb300 import synth
from tests.test_gpu_grad import _coeffs, _full_check, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,V,B,G,ls,blocks", [
    (512, 40000, 1, 4, 0.05, None),   # one pair of token blocks, one unit
    (512, 40000, 1, 8, 0.12, None),   # a few pairs
    (512, 9999, 2, 8, 0.3, 2),        # chunks of one pair: workspace scratch
    (1024, 20001, 1, 6, 0.15, None),
    (1536, 12345, 2, 4, 0.2, None),   # three 512-column units per pair
    (4096, 5000, 1, 4, 0.1, None),    # no tail rows in the workspace: the ring alone
    (320, 30000, 1, 4, 0.1, None),    # no image: the plain log-sum-exp pass
])
def test_short_batches(d, V, B, G, ls, blocks):
    inp = synth.make_head_workload(synth.WORKLOADS["qwen3_1p7b_head"], 11, B=B, G=G, d=d, V=V,
                                   len_scale=ls, w_std_mult=2.0)
    a = _coeffs(inp)
    a[:2] = (0.75, -0.5)
    idx, _, _ = oracle.compact_tokens(inp["cu_seqlens"], inp["mask"], a)
    if blocks:
        assert idx.size > 128 * blocks
    J, dH1, dW1 = _full_check(inp, a, image_blocks=blocks)
    st, J2, dH, dW, _, _ = _run(inp, a, blocks)
    assert st == 0 and J2 == J
    assert torch.equal(dH, dH1) and torch.equal(dW, dW1)
