"""Ratios, shares and reductions of a call reach the library as float() gives them, whatever kind of sequence holds them."""
import array
import ctypes
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_2509_22323_b200 import binding

NUMBERS = [0.5, 1, 0.1, 1e-9, 3e38, 1e300, -0.0, float("inf"), 0.30000000000000004]


@pytest.mark.parametrize("n", [0, 1, 4, 5, 9])
@pytest.mark.parametrize("kind", [list, tuple, np.array, np.float32, torch.tensor, lambda x: array.array("d", x),
                                  lambda x: [np.float32(v) for v in x], lambda x: [torch.tensor(v) for v in x],
                                  lambda x: [str(v) for v in x], lambda x: [Fraction(1, 3) for v in x],
                                  lambda x: bytes(range(len(x))), lambda x: bytearray(range(len(x))), lambda x: "1" * len(x)])
def test_every_kind_of_sequence(kind, n):
    with np.errstate(over="ignore"):
        xs = kind(NUMBERS[:n])
    got = binding._f32(xs)
    want = [ctypes.c_float(float(x)).value for x in xs]
    assert len(got) == n and list(got) == want
    assert isinstance(got, ctypes.Array)


@pytest.mark.parametrize("bad,error", [((x for x in [0.5] * 8), TypeError), ([None] * 8, TypeError), (["a"] * 8, ValueError),
                                       ([10 ** 400] * 8, OverflowError), ([[0.5]] * 8, TypeError)])
def test_what_is_no_list_of_numbers_is_refused(bad, error):
    with pytest.raises(error):
        binding._f32(bad)
