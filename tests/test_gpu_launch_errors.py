"""Calls whose launches cannot be made: refused, with nothing launched, and without a trace in the calls behind them."""
import ctypes

import pytest
import torch

from paper_2404_07904_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("packed", [False, True])
def test_more_units_than_a_grid_has_blocks(packed):
    # 2^32 units (slots of a packed batch): the host refuses the call; the outputs' addresses, well away from the inputs, are
    # those of no memory
    B, H = ((1 << 16) - 2, 1 << 16) if packed else (1 << 16, 1 << 16)
    d = binding.make_desc(B, H, 1, 16, 16, binding.HGRN2_F32)
    buf = torch.zeros(1 << 12, dtype=torch.uint8, device="cuda")
    p, far, lib = ctypes.c_void_p(buf.data_ptr()), ctypes.c_void_p(1 << 56), binding.load()
    ref, cu = ctypes.byref(d), [p] if packed else []
    fwd, bwd = (lib.hgrn2_fwd_varlen, lib.hgrn2_bwd_varlen) if packed else (lib.hgrn2_fwd, lib.hgrn2_bwd)
    assert fwd(ref, p, p, p, *cu, None, far, None, None, p, None) == 5
    assert bwd(ref, p, p, p, *cu, None, p, None, p, far, far, far, None, p, None) == 5
    o = torch.rand(1, 2, 64, device="cuda")
    binding.hgrn2_step(o, o, o, torch.zeros(1, 2, 64, 64, device="cuda"))    # asks for the error of its own launch
    torch.cuda.synchronize()
    assert not buf.any()
