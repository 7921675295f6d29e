"""The Python binding's argument conversion and prepared passes, without a GPU: every call here is refused by the library's host
checks, or by the binding itself, before anything is launched."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2303_11257_b200 import _binding
from paper_2303_11257_b200 import lib as L

cast = _binding.calls["us_cast_fp8"]
F32, F8 = torch.zeros(4, 16), torch.zeros(4, 16, dtype=torch.float8_e4m3fn)


@pytest.mark.parametrize("bad,error", [(5, TypeError), (np.zeros((4, 16), np.float32), TypeError), ([F32], TypeError), (torch.zeros(16), ValueError),
                                       (torch.zeros(16, 4).t(), ValueError), (torch.zeros(4, 16, dtype=torch.int64), KeyError)])
def test_what_is_no_matrix_is_refused_by_the_binding(bad, error):
    with pytest.raises(error):
        cast(bad, 1.0, F8, 0)


def test_argument_counts_and_numbers_are_checked():
    for args in ((F32, 1.0, F8), (F32, 1.0, F8, 0, 0), (F32, "1", F8, 0), (F32, 1.0, F8, "0")):
        with pytest.raises(TypeError):
            cast(*args)
    with pytest.raises(KeyError):
        _binding.prepare("us_nothing", ())


@pytest.mark.parametrize("t", [F32, F32[:, :5], F32[:1, :5], torch.zeros(1, 1), F32.to(torch.bfloat16)[1:3]])
def test_a_tensor_is_described_as_by_the_python_side(t):
    """A slot of a program gets what describe() says (the call itself is refused: its output has another shape)."""
    m, out = L.us_mat(), L.mat(torch.zeros(7, 3, dtype=torch.float8_e4m3fn))
    prog = _binding.program([(0, _binding.prepare("us_cast_fp8", (m, 1.0, out)))], [(0, m)])
    assert _binding.run(prog, 0, (t,), 0, 0, 0, 0) == L.US_ERR_INVALID_ARG
    assert (m.ptr, m.dtype, m.rows, m.cols, m.ld) == L.describe(t)


def test_a_pass_stops_at_a_refused_call_and_goes_on_behind_it():
    bad, good = L.mat(F32), L.mat(torch.zeros(4, 16, dtype=torch.bfloat16))
    empty = L.us_mat(None, L.US_F32, 0, 16, 16)
    nothing = _binding.prepare("us_cast_fp8", (empty, 1.0, L.us_mat(None, L.US_E4M3, 0, 16, 16)))      # no rows: succeeds, launches nothing
    refused = _binding.prepare("us_cast_fp8", (bad, 1.0, good))                                        # no 8-bit output
    prog = _binding.program([(0, nothing), (0, refused), (2, None), (0, nothing), (1, refused)], [])
    assert _binding.run(prog, 0, (), 0, 0, 0, 0) == 1 << 8 | L.US_ERR_UNSUPPORTED
    assert _binding.run(prog, 2, (), 0, 0, 0, 0) == 4 << 8 | L.US_ERR_UNSUPPORTED
    assert _binding.run(prog, 5, (), 0, 0, 0, 0) == -1


def test_unchanged_compares_objects_and_addresses():
    own = (F32, F8)
    at = tuple(t.data_ptr() for t in own)
    assert _binding.unchanged(own, own, at)
    assert not _binding.unchanged((F32, F8.clone()), own, at) and not _binding.unchanged(own, own, (at[0], at[1] + 16)) and not _binding.unchanged(own[:1], own, at)
