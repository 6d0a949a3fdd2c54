"""Calls made in loops pass packed bytes instead of filled ctypes structures:
the same bytes, and whatever the structures took is still taken -- scales
beyond FP32 (infinity), paddings with fewer than four numbers (zeros follow)."""
import ctypes

import pytest
import torch

from paper_2307_16080_gb300 import nk


def _bytes(arg, size):
    return arg[:size] if isinstance(arg, bytes) else ctypes.string_at(arg if isinstance(arg, int) else ctypes.addressof(arg), size)


@pytest.mark.parametrize("scales", [(1.0, 1.0), (0.1, -2.5e-40), (1e39, 1.0), (1.0, -1e300), (float("inf"), float("nan"))])
def test_epilogue(scales):
    bias = torch.zeros(4)
    e, owner = nk._epilogue_arg(bias, True, False, *scales, None, None, None)
    want = nk._epi(bias, True, False, *scales)
    n = ctypes.sizeof(nk.nk_epilogue)
    assert _bytes(e, n) == ctypes.string_at(ctypes.addressof(want), n)
    del owner


@pytest.mark.parametrize("t", [torch.zeros(3), torch.zeros(2, 5).t(), torch.zeros(2, 3, 4, 5, dtype=torch.bfloat16)[:, 1:],
                               torch.zeros(0, 4), torch.zeros(4, 6, dtype=torch.uint8).expand(4, 6)])
def test_tensor(t):
    n = ctypes.sizeof(nk.nk_tensor)
    want = nk.as_nk_tensor(t)
    assert nk._tensor_bytes(t) == ctypes.string_at(ctypes.addressof(want), n)


@pytest.mark.parametrize("args", [((1, 1), (1, 1), (0, 0, 0, 0)), ((2, 1), (1, 3), (1, 2, 3, 4)), ((1, 1), (1, 1), (1, 1)),
                                  ((2,), (1, 1), ()), ([1, 2], [3, 4], [-1, 0, 2 ** 62, 5])])
def test_convolution_arguments(args):
    got, want = nk._conv_bytes(*args), nk._conv_args(*args)
    for g, w, n in zip(got, want, (16, 16, 32)):
        assert _bytes(g, n) == ctypes.string_at(ctypes.addressof(w), n)


def test_too_many_numbers_are_refused():
    with pytest.raises((ValueError, IndexError)):
        nk._conv_bytes((1, 1, 1), (1, 1), (0, 0, 0, 0))
