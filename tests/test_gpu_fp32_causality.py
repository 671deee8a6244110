"""Inf and NaN on the fp32 kernels: a token's outputs depend on no later token, a token's gradients on no earlier one, whatever is
in it (a right-padded batch may hold anything in its padding)."""
import numpy as np
import pytest
import torch

from paper_2404_07904_b200 import binding, workloads as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu

SHAPES = [("f32", 128, 0), ("f32", 64, 0), ("bf16", 64, 0), ("bf16", 128, binding.FLAG_FORCE_ALU)]


def _run(inp, io, flags):
    return G.gpu_fwd_bwd(inp, io, flags=flags)


def _same(got, clean, rows, names):
    # bit for bit: what is left out is a product with a zero of the masked matrix
    for k in names:
        assert np.isfinite(got[k][:, :, rows]).all(), k
        np.testing.assert_array_equal(got[k][:, :, rows], clean[k][:, :, rows], err_msg=k)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("t", [10, 70, 110])                              # both halves of a chunk, chunks 0 and 1 of 3
@pytest.mark.parametrize("io,d,flags", SHAPES)
def test_no_output_sees_a_later_token_no_gradient_an_earlier_one(io, d, flags, t, bad):
    inp = W.make_inputs(W.scaled(W.CONFIGS["tiny_f32"], B=1, H=2, N=150, dk=d, dv=d, io=io, has_S0=True, has_dSN=True,
                                 seed=60, gamma=0.5, scale=d ** -0.5))
    clean = _run(inp, io, flags)
    for name, rows, outputs in (("i", slice(0, t), ("y",)), ("o", slice(t + 1, None), ("d_i", "d_f")),
                                ("dy", slice(t + 1, None), ("d_i", "d_f"))):
        x = dict(inp, **{name: inp[name].copy()})
        x[name][:, :, t, 5] = bad
        _same(_run(x, io, flags), clean, rows, outputs)
