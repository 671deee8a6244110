"""GPU parity of many short sequences on the default bf16 path.

With more (batch, head) units than SMs a CTA takes several of them, one after the other, in kernels of their own (the
forward always, the backward up to 6 chunks per sequence).  A unit's results must not depend on which CTA took it, or
after which other unit: every output is compared bit for bit with a call on that unit alone, and some with the oracle.
"""
import numpy as np
import pytest
import torch

from paper_2404_07904_b200 import binding, workloads as W
from tests import gpu_util as G
from tests import test_gpu_small_f as TS
from tests import test_gpu_varlen as TV

pytestmark = pytest.mark.gpu

TOL = 2e-2


# 1 chunk (partial, whole), 2 with a one-token rest, 4 partial, 7 (backward beyond the rule's line); 3 units more than
# SMs, and so many that every CTA takes several
@pytest.mark.parametrize("N,per_sm,extra", [(1, 3, 0), (64, 3, 1), (65, 2, 5), (200, 1, 3), (200, 4, 0), (448, 2, 0)])
def test_many_short_sequences(N, per_sm, extra):
    H = torch.cuda.get_device_properties(0).multi_processor_count * per_sm + extra
    w = W.scaled(W.CONFIGS["lm_2048"], B=1, H=H, N=N, has_S0=True, has_dSN=True, seed=70 + N % 9)
    inp = W.make_inputs(w)
    hard = [2, H - 1] if N >= 64 else []                                # redone on the exact path, and only they
    for h in hard:
        inp["f"][0, h, 10:60, 7] = W.round_to_bf16(np.float32(0.02))
    got, n_fwd, n_bwd = TS._run(inp)
    assert n_fwd == len(hard) and n_bwd == len(hard)
    some = sorted({0, 2, H // 2, H - 2, H - 1})
    for h in some:
        alone, _, _ = TS._run({k: v[:, h:h + 1] for k, v in inp.items()})
        if N <= 384:                                                    # longer ones are cut into segments when alone
            for k in alone:
                np.testing.assert_array_equal(got[k][:, h:h + 1], alone[k], err_msg=f"{k} of unit {h}")
    for (b, h), want in G.oracle_fwd_bwd(inp, [(0, 0), (0, 2), (0, H - 1)]).items():
        G.assert_close({k: got[k][:, h:h + 1] for k in want}, want, TOL, f"N = {N}, unit {h} of {H}")


def test_many_short_packed_sequences():
    # more items than SMs in a packed batch, empty sequences among them
    H = 4
    B = torch.cuda.get_device_properties(0).multi_processor_count // 2
    lengths = [(0, 1, 64, 130, 63, 200)[b % 6] for b in range(B)]
    inp = TV._packed_inputs(lengths, H=H, d=128, io="bf16", seed=78)
    got, _ = TV._run_gpu(inp, "bf16")
    G.assert_close(got, TV._oracle(inp), TOL, "many packed sequences")
