"""Values on the fp32 path that the parts of a tensor-core operand cannot hold: Inf, NaN, and the largest floats, whose
leading part would round to Inf."""
import numpy as np
import pytest
import torch

from oracle import ref
from paper_2404_07904_b200 import binding, workloads as W
from tests import gpu_util as G, test_gpu_gated as gated, test_gpu_varlen as varlen

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


def _classes(x):
    return np.where(np.isnan(x), 3, np.where(np.isinf(x), np.where(x > 0, 1, 2), 0))


# What an Inf makes of the outputs, by the recurrence in float64: NaN, Inf and its sign where it is a sum of Inf alone.
@pytest.mark.parametrize("name,t", [("i", 10), ("i", 100), ("o", 10), ("o", 100), ("dy", 10), ("dy", 100), ("S0", None), ("dSN", None)])
@pytest.mark.parametrize("io,dk,dv", [("f32", 128, 128), ("f32", 64, 64), ("f32", 32, 128), ("bf16", 64, 64)])
def test_one_inf_and_what_depends_on_it(io, dk, dv, name, t):
    inp = W.make_inputs(W.scaled(W.CONFIGS["tiny_f32"], B=1, H=2, N=150, dk=dk, dv=dv, io=io, has_S0=True, has_dSN=True,
                                 seed=73, gamma=0.5, scale=dk ** -0.5))
    for k in ("o", "dy", "i"):
        inp[k] = np.abs(inp[k])                                                # no two Inf of opposite sign meet in y, SN, d_o, d_i, dS0
    x = dict(inp, **{name: inp[name].copy()})
    if t is None:
        x[name][0, 1, 7, 5] = np.inf
    else:
        x[name][0, 1, t, 5] = -np.inf
    got, want = G.gpu_fwd_bwd(x, io), G.oracle_fwd_bwd(x)
    for k in want:
        np.testing.assert_array_equal(np.isfinite(got[k]), np.isfinite(want[k]), err_msg=k)
        if k != "d_f":
            np.testing.assert_array_equal(_classes(got[k]), _classes(want[k]), err_msg=k)
        ok = np.isfinite(want[k])
        assert G.rel_err(got[k][ok], want[k][ok]) <= G.TOL[io], k


def test_an_inf_in_every_sequence_does_not_hold_the_call_up():
    # with every output that depends on it summed in full such a call took 300 times as long
    w = W.scaled(W.CONFIGS["tiny_f32"], B=2, H=16, N=1024, dk=128, dv=128, gamma=0.5, scale=128 ** -0.5)
    t = G.to_dev(W.make_inputs(w), "f32")
    bad = t["i"].clone()
    bad[:, :, 10, 5] = float("inf")

    def once(i):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        _, _, saved, ws, _ = binding.hgrn2_fwd(t["o"], t["f"], i, None)
        binding.hgrn2_bwd(t["o"], t["f"], i, None, t["dy"], None, saved, ws=ws)
        b.record()
        torch.cuda.synchronize()
        return a.elapsed_time(b)

    clean = min(once(t["i"]) for _ in range(5))
    assert min(once(bad) for _ in range(3)) <= 40 * clean


def _check(got, want, clean, want_clean, tol):
    """Every output of a call with one odd value: Inf or NaN where the recurrence in float64 has it, what the value does not reach as
    without it, the rest to the path's bound.  Beyond 1e37 (sums of the largest floats) it is Inf, NaN or at least large."""
    for k in want:
        g, w = got[k], want[k]
        large = np.isfinite(w) & (np.abs(w) >= 1e37)
        assert (~np.isfinite(g[large]) | (np.abs(g[large]) > 1e36)).all(), k
        np.testing.assert_array_equal(np.isfinite(g[~large]), np.isfinite(w[~large]), err_msg=k)
        same = w == want_clean[k]
        assert np.abs(g[same] - clean[k][same]).max(initial=0) <= tol * np.abs(want_clean[k]).max(), k
        rest = ~same & ~large & np.isfinite(w)
        assert np.abs(g[rest] - w[rest]).max(initial=0) <= tol * np.abs(w[rest]).max(initial=0), k


BAD = [np.inf, np.nan, np.finfo(np.float32).max, np.finfo(np.float32).min]
SHAPES = [(io, dk, dv, bad) for io, dk, dv in (("f32", 128, 128), ("f32", 64, 64), ("f32", 32, 128), ("bf16", 64, 64), ("bf16", 128, 16))
          for bad in BAD if io == "f32" or not np.isfinite(bad)]             # (the tiles hold every finite bf16)


@pytest.mark.parametrize("name,t", [("i", 10), ("i", 100), ("o", 10), ("o", 100), ("dy", 10), ("dy", 100), ("S0", None), ("dSN", None)])
@pytest.mark.parametrize("io,dk,dv,bad", SHAPES)
def test_every_output_with_one_odd_value(io, dk, dv, name, t, bad):
    inp = W.make_inputs(W.scaled(W.CONFIGS["tiny_f32"], B=1, H=2, N=150, dk=dk, dv=dv, io=io, has_S0=True, has_dSN=True,
                                 seed=74, gamma=0.5, scale=dk ** -0.5))
    inp["dy"] = inp["dy"] * np.float32(0.125)                                  # (below 1: no product with the largest float overflows)
    x = dict(inp, **{name: inp[name].copy()})
    x[name][(0, 1, 7, 5) if t is None else (0, 1, t, 5)] = bad
    _check(G.gpu_fwd_bwd(x, io), G.oracle_fwd_bwd(x), G.gpu_fwd_bwd(inp, io), G.oracle_fwd_bwd(inp), G.TOL[io])


@pytest.mark.parametrize("name,bad", [("zi", np.inf), ("zi", np.nan), ("zo", np.inf), ("zo", np.nan), ("zf", np.inf), ("dy", np.inf), ("dy", np.nan)])
@pytest.mark.parametrize("io,d", [("f32", 128), ("bf16", 64)])
def test_every_output_of_the_gated_call_with_one_odd_value(io, d, name, bad):
    inp = gated._inputs(1, 2, 150, d, io, 75, 0.5, 0.9)
    x = dict(inp, **{name: inp[name].copy()})
    x[name][0, 1, 70, 5] = bad
    _check(gated._run(x, io)[0], gated._oracle(x), gated._run(inp, io)[0], gated._oracle(inp), G.TOL[io])


@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("name", ["i", "o", "dy"])
def test_every_output_of_a_packed_batch_with_one_odd_value(name, bad):
    inp = varlen._packed_inputs([70, 0, 130, 1, 64], 2, 64, "f32", 76, gamma=0.5)
    x = dict(inp, **{name: inp[name].copy()})
    x[name][1, 150, 5] = bad
    _check(varlen._run_gpu(x, "f32")[0], varlen._oracle(x), varlen._run_gpu(inp, "f32")[0], varlen._oracle(inp), G.TOL["f32"])
