"""What the C++ marshalling of the binding's calls takes and refuses (no GPU: every call ends at its first CPU tensor)."""
import numpy as np
import pytest
import torch

import __graft_entry__ as entry
from paper_2404_07904_b200 import binding


@pytest.fixture(scope="module")
def t():
    entry.build()
    return torch.zeros(1, 2, 4, 64)


@pytest.mark.parametrize("value", [64, 64.0, np.float32(64), np.int64(64), torch.tensor(64), "64", 2 ** 70 + 64])
def test_chunk_and_flags_are_whatever_int_takes(t, value):
    # the CPU tensor is what is refused, not the number
    with pytest.raises(ValueError, match="not on a CUDA device"):
        binding.hgrn2_fwd(t, t, t, chunk=value, ws=None, saved=None, save_for_backward=False)
    with pytest.raises(ValueError, match="not on a CUDA device"):
        binding.hgrn2_bwd(t, t, t, None, t, flags=value)


def test_numbers_that_int_refuses(t):
    with pytest.raises(TypeError):
        binding.hgrn2_fwd(t, t, t, chunk=None)
    with pytest.raises(ValueError):
        binding.hgrn2_fwd(t, t, t, flags="many")


def test_f_may_be_missing_where_its_gradient_has_a_buffer(t):
    # a NULL f is the library's to refuse (or, without tokens, to accept); only the shape of a new d_f comes from it
    with pytest.raises(ValueError, match="not on a CUDA device"):
        binding.hgrn2_bwd(t, None, t, None, t, d_f=t)
    with pytest.raises(TypeError):
        binding.hgrn2_bwd(t, None, t, None, t)
