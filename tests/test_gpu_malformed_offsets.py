"""Malformed offsets of packed batches: the sequences they belong to write nothing, the others come out as ever, and on the
tensor-core path the status word says so."""
import numpy as np
import pytest
import torch

from paper_2404_07904_b200 import binding, workloads as W
from oracle import ref
from tests import gpu_util as G

pytestmark = pytest.mark.gpu

INT_MIN = -2 ** 31


def _check(cu, good, T, H, io, d, flags, status):
    """Forward with offsets `cu`: rows and states of the sequences `good` against the oracle, all other rows untouched."""
    inp = W.make_inputs(W.scaled(W.CONFIGS["lm_2048"], B=1, H=H, N=T, dk=d, dv=d, io=io, seed=51))
    o, f, i = (np.ascontiguousarray(inp[k][0]) for k in ("o", "f", "i"))
    tdt = torch.float32 if io == "f32" else torch.bfloat16
    t = [torch.from_numpy(x).cuda().to(tdt) for x in (o, f, i)]
    buf, y = G.canary((H, T, d), tdt)
    _, SN, _, ws, _ = binding.hgrn2_fwd_varlen(*t, torch.tensor(cu, dtype=torch.int32, device="cuda"), None, y=y, flags=flags)
    torch.cuda.synchronize()
    assert binding.hgrn2_poll(ws) == status and G.canary_ok(buf)
    y, SN, untouched = y.float().cpu().numpy(), SN.cpu().numpy(), np.ones(T, bool)
    for b in good:
        s, e = cu[b], cu[b + 1]
        want = ref.hgrn2_fwd(o[None, :, s:e], f[None, :, s:e], i[None, :, s:e], None)
        G.assert_close({"y": y[None, :, s:e], "SN": SN[b:b + 1]}, dict(zip(("y", "SN"), want)), G.TOL[io], f"sequence {b} of {cu}")
        untouched[s:e] = False
    assert (y[:, untouched] == np.float32(torch.tensor(12345.0).to(tdt).float())).all()


PATHS = [("bf16", 128, 0, 1), ("bf16", 128, binding.FLAG_FORCE_ALU, 0), ("f32", 64, 0, 0)]


@pytest.mark.parametrize("io,d,flags,status", PATHS)
@pytest.mark.parametrize("T", [400, 900])                                # 900 rows, few units: cut into segments
def test_lengths_beyond_the_integer_range(T, io, d, flags, status):
    # INT_MIN - 60 wraps to a length of 2^31 - 60, and start + length to a negative row
    _check([0, 60, INT_MIN, 100, 300], [0, 3], T, 2, io, d, flags, status)


@pytest.mark.parametrize("B,T", [(2, 400), (20, 900), (700, 900)])       # whole, in segments, several per CTA
def test_the_report_is_not_lost(B, T):
    # the malformed sequence is the last one: its CTA has nothing to do and must not race the clearing of the status word
    H, cu = 2, [0] * B + [T + 1]
    x = torch.randn(H, T, 128, device="cuda").bfloat16().sigmoid()
    cu = torch.tensor(cu, dtype=torch.int32, device="cuda")
    junk = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    for turn in range(20):
        _, _, saved, ws, _ = binding.hgrn2_fwd_varlen(x, x, x, cu)
        torch.cuda.synchronize()
        assert binding.hgrn2_poll(ws) == 1, turn
        junk.fill_(turn)
        for s in (saved, None):
            binding.hgrn2_bwd_varlen(x, x, x, cu, None, x, None, s, ws=ws)
            torch.cuda.synchronize()
            assert binding.hgrn2_poll(ws) == 1, turn


@pytest.mark.parametrize("io,d,flags,status", PATHS)
@pytest.mark.parametrize("cu,good", [
    ([0, 130, -5, 130, 330], [0, 3]),                # an offset that a search by value takes for an early one
    ([0, 64, 500, 64, 200, 330], [0, 3, 4]),         # ... for a late one
    ([-1, 70, 100, 200, 401], [1, 2]),               # the first and the last sequence
])
def test_other_sequences_are_unaffected(cu, good, io, d, flags, status):
    _check(cu, good, 400, 2, io, d, flags, status)
