"""pair_grad's bookkeeping kernels at the edges of their dispatch: rollout
offsets summed inside the gather kernel up to 2048 rollouts and by the scan
kernel above, rollouts shorter and longer than a gather block, many tokens in
one target bucket, and a target out of range (reported, and no kernel reads
past W). Against the fp64 oracle, tolerances as in test_gpu_grad.py."""
import numpy as np
import pytest
import torch

from paper_2608_11368_gb300 import synth
from tests.test_gpu_grad import _coeffs, _full_check, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [256, 257])
@pytest.mark.parametrize("name,d", [("pr1_ref_fp32", 32), ("qwen3_1p7b_head", 64)])
def test_many_rollouts(B, name, d):
    inp = synth.make_head_workload(synth.WORKLOADS[name], 9, B=B, G=8, d=d, V=60,
                                   len_scale=0.04 if name == "pr1_ref_fp32" else 0.002)
    assert inp["R"] == 8 * B
    _full_check(inp, _coeffs(inp))


def test_long_rollouts_and_one_bucket():
    inp = synth.make_head_workload(synth.WORKLOADS["qwen3_1p7b_head"], 9, B=1, G=3, d=512, V=700,
                                   len_scale=1.2)
    a = _coeffs(inp)
    a[:] = (0.75, 0.0, -0.5)
    assert inp["lengths"].max() > 1024
    on = np.nonzero(inp["mask"])[0]
    inp["y"][on[::2]] = 33   # more than the ranked bucket size
    inp["y"][on[1::8]] = 34  # and a second row of the same bucket
    _full_check(inp, a)


@pytest.mark.parametrize("bad", [-7, 700, 2 ** 31 - 1])
def test_target_out_of_range_reads_nothing(bad):
    inp = synth.make_head_workload(synth.WORKLOADS["qwen3_1p7b_head"], 9, B=1, G=4, d=512, V=700,
                                   len_scale=0.05)
    a = np.array([0.5, -0.5, 0.25, 0.0], np.float32)
    inp["y"][np.nonzero(inp["mask"])[0][3]] = bad
    st, _, dH, dW, _, _ = _run(inp, a)
    assert st == _run(inp, a)[0] == 5
    torch.cuda.synchronize()
