"""The chunk-parallel fp32 kernels at the sizes where their tiling can go wrong: chunk edges, blocks of 32 and 64 columns
that the head size fills only partly, several value and key blocks, states re-created in rounds (odd and even unit
counts; one unit falls back to the serial kernels) and gates that leave the range of the mid-chunk operands."""
import numpy as np
import pytest

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
