"""Values on the fp32 path that the parts of a tensor-core operand cannot hold: Inf, NaN, and the largest floats, whose
leading part would round to Inf."""
import numpy as np
import pytest

from oracle import ref
from paper_2404_07904_b200 import workloads as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


# Bound of the finite case: that of the configuration, as for any other column.
@pytest.mark.parametrize("bad", [np.inf, np.nan, np.finfo(np.float32).max, np.finfo(np.float32).min])
@pytest.mark.parametrize("t", [10, 100])
@pytest.mark.parametrize("io,d,flags", [("f32", 128, 0), ("f32", 64, 0), ("bf16", 64, 0)])
def test_forward_with_one_odd_value(io, d, flags, t, bad):
    inp = W.make_inputs(W.scaled(W.CONFIGS["tiny_f32"], B=1, H=2, N=150, dk=d, dv=d, io=io, has_S0=True, has_dSN=True,
                                 seed=70, gamma=0.5, scale=d ** -0.5))
    clean = G.gpu_fwd_bwd(inp, io, flags=flags)
    if io == "bf16" and np.isfinite(bad):
        bad = np.float32(np.sign(bad) * 2.0 ** 127 * (2 - 2.0 ** -7))          # bf16's largest
    x = dict(inp, i=inp["i"].copy())
    x["i"][0, 1, t, 5] = bad
    got = G.gpu_fwd_bwd(x, io, flags=flags)
    others = [c for c in range(d) if c != 5]
    for k in ("y", "SN"):                                                      # nobody else's value
        np.testing.assert_array_equal(got[k][:, :1], clean[k][:, :1])
        np.testing.assert_array_equal(got[k][..., others], clean[k][..., others])
    np.testing.assert_array_equal(got["y"][:, :, :t], clean["y"][:, :, :t])
    y, SN = got["y"][0, 1, t:, 5], got["SN"][0, 1, :, 5]
    if not np.isfinite(bad):
        assert not np.isfinite(y).any() and not np.isfinite(SN).any()
        return
    want_y, want_SN = ref.hgrn2_fwd(x["o"], x["f"], x["i"], x["S0"])
    assert G.rel_err(y, want_y[0, 1, t:, 5]) <= G.TOL[io]
    assert G.rel_err(SN, want_SN[0, 1, :, 5]) <= 1e-4


# Bound of the finite values: the path's.
@pytest.mark.parametrize("gamma", [0.5, 0.0])                                  # 0.0 with a hard gate: the pairwise form
@pytest.mark.parametrize("t,s", [(100, 97), (100, 100), (20, 18)])            # (further apart, d_f before s cancels to less than its rounding)
@pytest.mark.parametrize("io,d,flags", [("f32", 128, 0), ("f32", 64, 0), ("bf16", 64, 0)])
def test_an_overflow_in_the_backward_stays_with_what_depends_on_it(io, d, flags, t, s, gamma):
    # dY_t . V_s leaves float32 although every element of dY and V is finite
    inp = W.make_inputs(W.scaled(W.CONFIGS["tiny_f32"], B=1, H=2, N=150, dk=d, dv=d, io=io, has_S0=True, has_dSN=True,
                                 seed=71, gamma=gamma, scale=d ** -0.5))
    if gamma == 0.0:
        inp["f"][..., 3] = 0.03125
    clean = G.gpu_fwd_bwd(inp, io, flags=flags)
    big = W.round_to_bf16(np.float32([1e25]))[0]
    x = dict(inp, i=inp["i"].copy(), dy=inp["dy"].copy())
    x["i"][0, 1, s, 5] = big
    x["dy"][0, 1, t, 5] = big
    got, want = G.gpu_fwd_bwd(x, io, flags=flags), G.oracle_fwd_bwd(x)
    keys = [c for c in range(d) if gamma or c != 3]                            # (the hard gate forgets V_s before t)
    assert not np.isfinite(got["d_o"][0, 1, t, keys]).any()
    assert not np.isfinite(got["d_f"][0, 1, s:t + 1, keys]).any()
    for k in ("d_o", "d_f"):
        np.testing.assert_array_equal(got[k][:, 0], clean[k][:, 0])
    np.testing.assert_array_equal(got["d_o"][0, 1, :s], clean["d_o"][0, 1, :s])
    rest = {"d_o": [n for n in range(150) if n != t], "d_f": [n for n in range(150) if not s <= n <= t]}
    for k, rows in rest.items():
        assert np.isfinite(got[k][0, 1, rows]).all(), k
        assert G.rel_err(got[k][0, 1, rows], want[k][0, 1, rows]) <= G.TOL[io], k
