"""The chunk-parallel fp32 kernels at the sizes where their tiling can go wrong: chunk edges, blocks of 32 and 64 columns
that the head size fills only partly, several value and key blocks, states re-created in rounds (odd and even unit
counts; one unit falls back to the serial kernels) and gates that leave the range of the mid-chunk operands."""
import numpy as np
import pytest

from oracle import ref
from paper_2404_07904_b200 import workloads as W
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


# Bound: the fp32 configuration's 1e-4.  A term carries the rounding of two products of at most 32 factors
# (64 * 2^-24 = 4e-6), sums of up to 128 such terms add a few ulp, and d_f = dg / f - dk amplifies what is left of
# dg's terms by 1 / f <= 100 only in the columns whose dg is itself that much smaller than the tensor's largest.
@pytest.mark.parametrize("N,dk,dv,H,saved,forget", [
    (64, 16, 64, 2, True, False),
    (193, 128, 16, 2, True, False),
    (130, 32, 32, 3, True, True),
    (65, 128, 128, 1, True, True),
    (257, 64, 128, 1, True, True),
    (200, 64, 64, 1, False, False),
    (200, 64, 64, 2, False, True),
    (200, 128, 64, 3, False, False),
])
def test_chunk_and_block_edges(N, dk, dv, H, saved, forget):
    w = W.scaled(W.CONFIGS["tiny_f32"], B=1, H=H, N=N, dk=dk, dv=dv, has_S0=True, has_dSN=True, seed=N + dk, gamma=0.5,
                 scale=dk ** -0.5)
    inp = W.make_inputs(w)
    if forget:                            # 0.05 over half a chunk is 2^-138: below what the mid-chunk operands carry
        inp["f"][:, :, N // 3:, 3::7] = np.float32(0.05)
        inp["f"][:, :, :40, 1] = np.float32(0.01)
    G.assert_close(G.gpu_fwd_bwd(inp, "f32", use_saved=saved), G.oracle_fwd_bwd(inp), 1e-4, f"N={N} dk={dk} dv={dv}")


# The final state of gates that forget fast is a sum of few terms, the last tokens' the largest.  Bound on the norm: float32's rounding of
# the sum (0.29 ulp: 2.5e-8 on average over a binade) and of the terms before it; FMAs in float32 measure 4.35e-8 with gates around 0.5.
@pytest.mark.parametrize("f", [None, 0.13])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("n", [128, 129, 131, 150, 3])                         # rows of the last chunk: 64, 1, 3, 22; one short chunk
def test_final_state_of_gates_that_forget_fast(n, d, f):
    inp = W.make_inputs(W.scaled(W.CONFIGS["tiny_f32"], B=2, H=8, N=n, dk=d, dv=d, io="f32", seed=72, gamma=0.0))
    if f is not None:
        inp["f"] = np.float32(f) + np.float32(0.02) * (inp["f"] - np.float32(0.5))
    got, want = G.gpu_fwd_bwd(inp, "f32")["SN"].astype(np.float64), ref.hgrn2_fwd(inp["o"], inp["f"], inp["i"], None)[1]
    assert np.linalg.norm(got - want) <= 4.8e-8 * np.linalg.norm(want)
