"""Packed batches with long runs of empty sequences (offsets padded to a fixed number of slots) on the default bf16 path.

With more (sequence, head) units than SMs a CTA takes several, empty ones among them, and its roles pass items through a
ring of four: whatever a role holds back of one item must not wait for an item four further on.  The heads of a sequence
are neighbouring items, so every run here is many times that long.
"""
import numpy as np
import pytest
import torch

from paper_2404_07904_b200 import binding
from tests import gpu_util as G
from tests import test_gpu_varlen as TV

pytestmark = pytest.mark.gpu

TOL = 2e-2
H = 8
RUNS = {
    "in front, between and behind": [0] * 13 + [130] + [0] * 40 + [64, 1, 200] + [0] * 5 + [65] + [0] * 30,
    "every other": [0, 70] * 40,
    "all but one": [0] * 60 + [193],
}


def _inputs(lengths):
    assert len(lengths) * H > torch.cuda.get_device_properties(0).multi_processor_count
    return TV._packed_inputs(lengths, H=H, d=128, io="bf16", seed=41)


@pytest.mark.parametrize("name", RUNS)
def test_forward_over_runs_of_empty_sequences(name):
    inp = _inputs(RUNS[name])
    t = {k: torch.from_numpy(inp[k]).cuda().to(torch.bfloat16) for k in ("o", "f", "i")}
    cu, S0 = torch.from_numpy(inp["cu"]).cuda(), torch.from_numpy(inp["S0"]).cuda()
    y, SN, _, ws, _ = binding.hgrn2_fwd_varlen(t["o"], t["f"], t["i"], cu, S0)
    torch.cuda.synchronize()
    assert binding.hgrn2_poll(ws) == 0
    want = TV._oracle(inp)
    G.assert_close({"y": y.float().cpu().numpy(), "SN": SN.cpu().numpy()}, {k: want[k] for k in ("y", "SN")}, TOL, name)
    empty = [b for b, n in enumerate(RUNS[name]) if n == 0]
    np.testing.assert_array_equal(SN.cpu().numpy()[empty], inp["S0"][empty])


@pytest.mark.parametrize("use_saved", [True, False])
@pytest.mark.parametrize("name", RUNS)
def test_backward_over_runs_of_empty_sequences(name, use_saved):
    inp = _inputs(RUNS[name])
    got, _ = TV._run_gpu(inp, "bf16", use_saved=use_saved)
    G.assert_close(got, TV._oracle(inp), TOL, name)
    empty = [b for b, n in enumerate(RUNS[name]) if n == 0]
    np.testing.assert_array_equal(got["dS0"][empty], inp["dSN"][empty])
