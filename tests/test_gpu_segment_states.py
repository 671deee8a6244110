"""Accuracy of sequences that run as segments on the default bf16 path.

S_N and dS_0 of such a sequence come out of the chaining of its segments, whose state-only pass rounds a token's decay from
the segment's end (its start in the backward), where it is 1.
"""
import numpy as np
import pytest
import torch

from paper_2404_07904_b200 import workloads as W
from tests import gpu_util as G
from tests import test_gpu_small_f as TS
from tests import test_gpu_varlen as TV

pytestmark = pytest.mark.gpu

# With f = sigmoid(normal), E[f^2] = 0.29: the last two tokens hold 91 % of S_N's energy (the first holds 71 % of dS_0's),
# their decay factors 1 and f_N (f_1) are bf16 as they are, and so their terms are rounded once; the others twice.
# One bf16 rounding is 2^-8 / sqrt(3) * sqrt(E[m^-2] = 1/2) = 1.6e-3 rms, so 1.67e-3 and 1.81e-3 are to be expected (fp32
# sums do not count); two roundings of every term, as the mid-chunk frame has them, are 2.26e-3.
BOUND = 2.1e-3


def _norm_err(got, want):
    return float(np.linalg.norm(got.astype(np.float64) - want) / np.linalg.norm(want))


@pytest.mark.parametrize("H,N", [(8, 1088), (4, 1100)])                  # whole chunks; a partial last segment
def test_final_states_of_cut_sequences(H, N):
    inp = W.make_inputs(W.scaled(W.CONFIGS["long_16k"], B=1, H=H, N=N, has_S0=True, has_dSN=True, seed=31, gamma=0.0))
    got, want = G.gpu_fwd_bwd(inp, "bf16"), G.oracle_fwd_bwd(inp)
    assert {k: e for k in ("SN", "dS0") if not (e := _norm_err(got[k], want[k])) <= BOUND} == {}


def test_final_states_of_cut_packed_sequences():
    inp = TV._packed_inputs([1100, 0, 700, 200], H=4, d=128, io="bf16", seed=32, gamma=0.0)
    (got, _), want, full = TV._run_gpu(inp, "bf16"), TV._oracle(inp), [0, 2, 3]
    assert {k: e for k in ("SN", "dS0") if not (e := _norm_err(got[k][full], want[k][full])) <= BOUND} == {}
    np.testing.assert_array_equal(got["SN"][1], inp["S0"][1])            # no tokens: the state passes through
    np.testing.assert_array_equal(got["dS0"][1], inp["dSN"][1])


def _sms_and_three():
    return torch.cuda.get_device_properties(0).multi_processor_count + 3


# few units, cut all; more units than SMs, the last three cut, several items per CTA
@pytest.mark.parametrize("units,N", [(lambda: 4, 2048), (_sms_and_three, 1024)])
@pytest.mark.parametrize("use_saved", [True, False])
def test_a_cut_unit_with_hard_gates_is_redone_whole(units, N, use_saved):
    # One segment of whole chunks leaves the operands' range: the unit's states come out as exactly as those of a unit that is
    # not cut.  1e-5: fp32 sums of 2048 terms that decay (1e-7 each); segments redone on their own start from states
    # with bf16 operands in them, 1.5e-3 and more.
    H = units()
    inp = W.make_inputs(W.scaled(W.CONFIGS["long_16k"], B=1, H=H, N=N, has_S0=True, has_dSN=True, seed=33, gamma=0.9))
    hard = H - 2
    inp["f"][0, hard, N // 2 + 5:N // 2 + 60, 7] = W.round_to_bf16(np.float32(0.02))
    got, n_fwd, n_bwd = TS._run(inp, use_saved)
    assert (n_fwd, n_bwd) == (1, 1 if use_saved else 2)
    for (b, h), want in G.oracle_fwd_bwd(inp, [(0, hard), (0, H - 1)]).items():
        mine = {k: got[k][b:b + 1, h:h + 1] for k in want}
        G.assert_close(mine, want, 2e-2, f"unit {h} of {H}")
        if h == hard:
            assert {k: e for k in ("SN", "dS0") if not (e := _norm_err(mine[k], want[k])) <= 1e-5} == {}
