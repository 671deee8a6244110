"""Small values on the fp32 path beside gates that forget fast: with f around 0.12 to 0.13 the decay of half a chunk is 2^-98 to 2^-94,
close to what the kernels' operands carry, whatever the size of the gradients, values or queries it is multiplied into."""
import numpy as np
import pytest

from paper_2404_07904_b200 import workloads as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu

# Sums of float32 products: 64 to 128 terms of 2^-24 each, and d_f's sum over time divided by an f of 0.12; measured 4e-7, d_f 2e-6.
TOL = {"f32": 1e-5, "bf16": G.TOL["bf16"]}
SHAPES = [("f32", 64, 64), ("f32", 128, 128), ("f32", 128, 64), ("f32", 32, 128), ("bf16", 64, 64)]


def _inputs(io, dk, dv, f, **factors):
    w = W.scaled(W.CONFIGS["tiny_f32"], B=1, H=2, N=150, dk=dk, dv=dv, io=io, has_S0=True, has_dSN=True, seed=81)
    inp = W.make_inputs(w)
    inp["S0"] *= 50
    inp["dSN"] *= 50
    inp["f"][:] = f + 0.08 * f * (2 * np.random.default_rng(82).random(inp["f"].shape) - 1) * (f > 0.12)
    if io == "bf16":
        inp["f"] = W.round_to_bf16(inp["f"])
    for name, x in factors.items():
        inp[name] = inp[name] * np.float32(x)
        if io == "bf16" and name not in ("S0", "dSN"):
            inp[name] = W.round_to_bf16(inp[name])
    return inp


def _check(inp, io, outputs):
    got, want = G.gpu_fwd_bwd(inp, io), G.oracle_fwd_bwd(inp)
    G.assert_close({k: got[k] for k in outputs}, {k: want[k] for k in outputs}, TOL[io])


@pytest.mark.parametrize("scale", [1e-6, 1e-8, 1e-10])
@pytest.mark.parametrize("f", [0.118, 0.13])
@pytest.mark.parametrize("io,dk,dv", SHAPES)
def test_small_gradients_and_values(io, dk, dv, f, scale):
    _check(_inputs(io, dk, dv, f, dy=scale, dSN=scale), io, ("d_i", "dS0"))
    _check(_inputs(io, dk, dv, f, i=scale, S0=scale), io, ("y", "SN"))


@pytest.mark.parametrize("scale", [1e-6, 1e-9])
@pytest.mark.parametrize("io,dk,dv", SHAPES)
def test_small_queries(io, dk, dv, scale):
    _check(_inputs(io, dk, dv, 0.118, o=scale), io, ("y", "SN", "d_o", "d_f", "d_i"))


# dA, X and their products with the decays reach the end of float32's range.  Bound: as above where the float32 terms themselves are
# normal numbers (1e-8, decays of 2^-98); with 1e-14 the terms lie below 2^-126 unless they are lifted.
@pytest.mark.parametrize("scale", [1e-8, 1e-14, 1e-20])
@pytest.mark.parametrize("io,dk,dv", SHAPES)
def test_small_gradients_of_the_gates(io, dk, dv, scale):
    inp = _inputs(io, dk, dv, 0.118, dy=scale, dSN=scale)
    _check(inp, io, ("d_o", "d_f") if scale > 1e-12 else ("d_o",))
