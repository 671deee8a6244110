"""The time-out exit of the fp32 path's kernels: with HGRN2_FLAG_DEBUG_EXPIRE_WAITS every wait for products gives up at once.  The calls must
return, report HGRN2_ERR_TIMEOUT and write inside the caller's buffers only, and the next ordinary call on the same buffers must be
correct."""
import pytest
import torch

from paper_2404_07904_b200 import binding, workloads as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("io,dk,dv", [("f32", 64, 64), ("f32", 128, 128), ("f32", 128, 16), ("bf16", 64, 64)])
@pytest.mark.parametrize("f", [None, 0.01])                                    # framed and pairwise decays
def test_expired_waits_of_the_fp32_kernels(io, dk, dv, f):
    w = W.scaled(W.CONFIGS["tiny_f32"], B=1, H=2, N=150, dk=dk, dv=dv, io=io, has_S0=True, has_dSN=True, seed=92, scale=dk ** -0.5)
    inp = W.make_inputs(w)
    if f is not None:
        inp["f"][..., ::2] = W.round_to_bf16(inp["f"][..., ::2] * 0 + f)
    t = G.to_dev(inp, io)
    bufs, outs = {}, {}
    for name, like in (("y", "i"), ("SN", "S0"), ("d_o", "o"), ("d_f", "f"), ("d_i", "i"), ("dS0", "S0")):
        bufs[name], outs[name] = G.canary(tuple(t[like].shape), t[like].dtype)
    grads = {k: outs[k] for k in ("d_o", "d_f", "d_i", "dS0")}

    def fwd(saved, ws, flags):
        r = binding.hgrn2_fwd(t["o"], t["f"], t["i"], t["S0"], y=outs["y"], SN=outs["SN"], saved=saved, ws=ws, flags=flags)
        torch.cuda.synchronize()
        return r[2], r[3]

    def bwd(saved, ws, flags):
        binding.hgrn2_bwd(t["o"], t["f"], t["i"], t["S0"], t["dy"], t["dSN"], saved, ws=ws, flags=flags, **grads)
        torch.cuda.synchronize()

    saved, ws = fwd(None, None, binding.FLAG_DEBUG_EXPIRE_WAITS)
    assert binding.hgrn2_poll(ws) == 6
    fwd(saved, ws, 0)
    assert binding.hgrn2_poll(ws) == 0
    bwd(saved, ws, binding.FLAG_DEBUG_EXPIRE_WAITS)
    assert binding.hgrn2_poll(ws) == 6
    for name, b in bufs.items():
        assert G.canary_ok(b), f"out-of-bounds write next to {name}"
    bwd(saved, ws, 0)
    assert binding.hgrn2_poll(ws) == 0
    G.assert_close({k: v.float().cpu().numpy() for k, v in outs.items()}, G.oracle_fwd_bwd(inp), G.TOL[io], "after the timed-out calls")
