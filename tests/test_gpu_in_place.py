"""Outputs in the place of inputs on the fp32 kernels: the same results as into buffers of their own."""
import pytest
import torch

from paper_2404_07904_b200 import binding, workloads as W
from tests import gpu_util as G
from tests import test_gpu_gated as TG

pytestmark = pytest.mark.gpu

SHAPES = [("f32", 128, 0), ("f32", 32, 0), ("bf16", 64, 0), ("bf16", 128, binding.FLAG_FORCE_ALU)]


def _host(x):
    return {k: v.float().cpu().numpy() for k, v in x.items()}


@pytest.mark.parametrize("save", [True, False])
@pytest.mark.parametrize("io,d,flags", SHAPES)
def test_sequence_calls(io, d, flags, save):
    inp = W.make_inputs(W.scaled(W.CONFIGS["tiny_f32"], B=1, H=3, N=200, dk=d, dv=d, io=io, has_S0=True, has_dSN=True, seed=61,
                                 gamma=0.5, scale=d ** -0.5))
    want = G.oracle_fwd_bwd(inp)
    for name in ("o", "f", "i"):
        t = G.to_dev(inp, io)
        y, SN, saved, ws, _ = binding.hgrn2_fwd(t["o"], t["f"], t["i"], t["S0"], y=t[name], save_for_backward=save, flags=flags)
        G.assert_close(_host({"y": y, "SN": SN}), {k: want[k] for k in ("y", "SN")}, G.TOL[io], f"y in the place of {name}")
        t = G.to_dev(inp, io)                                                # its saved states serve an ordinary backward
        d_o, d_f, d_i, dS0, _ = binding.hgrn2_bwd(t["o"], t["f"], t["i"], t["S0"], t["dy"], t["dSN"], saved, ws=ws, flags=flags)
        got = _host({"d_o": d_o, "d_f": d_f, "d_i": d_i, "dS0": dS0})
        G.assert_close(got, {k: want[k] for k in got}, G.TOL[io], f"backward behind y in the place of {name}")
    for places in (dict(d_o="o", d_f="f", d_i="i"), dict(d_i="dy"), dict(d_o="dy", d_f="i")):
        t = G.to_dev(inp, io)
        _, _, saved, ws, _ = binding.hgrn2_fwd(t["o"], t["f"], t["i"], t["S0"], save_for_backward=save, flags=flags)
        d_o, d_f, d_i, dS0, _ = binding.hgrn2_bwd(t["o"], t["f"], t["i"], t["S0"], t["dy"], t["dSN"], saved, ws=ws, flags=flags,
                                                  **{k: t[v] for k, v in places.items()})
        got = _host({"d_o": d_o, "d_f": d_f, "d_i": d_i, "dS0": dS0})
        G.assert_close(got, {k: want[k] for k in got}, G.TOL[io], str(places))


def test_gated_calls():
    inp = TG._inputs(1, 2, 150, 64, "f32", seed=62, beta_lo=0.0, beta_hi=0.9)
    want = TG._oracle(inp)
    t = {k: torch.from_numpy(v).cuda() for k, v in inp.items()}
    _, _, saved, ws, _ = binding.hgrn2_fwd_gated(t["zo"], t["zf"], t["zi"], t["beta"], t["S0"])
    d_zo, d_zf, d_zi, d_beta, dS0, _ = binding.hgrn2_bwd_gated(t["zo"], t["zf"], t["zi"], t["beta"], t["S0"], t["dy"], t["dSN"],
                                                               saved, d_zo=t["zo"], d_zf=t["zf"], d_zi=t["zi"], ws=ws)
    got = _host({"d_zo": d_zo, "d_zf": d_zf, "d_zi": d_zi, "d_beta": d_beta, "dS0": dS0})
    G.assert_close(got, {k: want[k] for k in got}, 1e-4, "gradients in the place of pre-activations")
    t = {k: torch.from_numpy(v).cuda() for k, v in inp.items()}
    y, SN, _, _, _ = binding.hgrn2_fwd_gated(t["zo"], t["zf"], t["zi"], t["beta"], t["S0"], y=t["zi"])
    G.assert_close(_host({"y": y, "SN": SN}), {k: want[k] for k in ("y", "SN")}, 1e-4, "y in the place of zi")


@pytest.mark.parametrize("T", [1, 3, 21])
@pytest.mark.parametrize("io,d,H", [("bf16", 128, 8), ("f32", 128, 400), ("bf16", 64, 8), ("f32", 64, 8)])
def test_decode_calls(io, d, H, T):
    # few units (one token: several CTAs per unit) and many; bit for bit what goes into a buffer of its own
    inp = W.make_inputs(W.scaled(W.CONFIGS["tiny_f32"], B=1, H=H, N=T, dk=d, dv=d, io=io, has_S0=True, seed=63, gamma=0.5))

    def call(place):
        t = G.to_dev(inp, io)
        if T == 1:
            t.update({k: t[k][:, :, 0].contiguous() for k in ("o", "f", "i")})
        y = t[place] if place else None
        y = (binding.hgrn2_step if T == 1 else binding.hgrn2_step_multi)(t["o"], t["f"], t["i"], t["S0"], y=y)
        return y, t["S0"]

    want = call(None)
    for place in ("o", "f", "i"):
        for got, w in zip(call(place), want):
            assert torch.equal(got, w), place
