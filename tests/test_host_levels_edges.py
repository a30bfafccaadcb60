"""Activation levels at the edges of their shortcuts (oddness, saturation), against math.tanh."""
import math

import numpy as np
import pytest

from paper_2604_17109_gb300 import build as pkg_build

pkg_build.build()
from paper_2604_17109_gb300 import pim  # noqa: E402


@pytest.mark.parametrize("imax", [1, 63, 511])
@pytest.mark.parametrize("b", [0.0, 1e-30, 1e-3, 0.0195, 0.02, 0.1587, 1.0, 9.9999, 10.0, 3e5, 3e38])
def test_tanh_levels(b, imax):
    b = float(np.float32(b))
    got = pim.pim_activation_levels(b, imax)
    want = np.array([math.tanh(b * i) for i in range(-imax, imax + 1)]).astype(np.float32)
    assert np.array_equal(got.view(np.uint32) & 0x7FFFFFFF, want.view(np.uint32) & 0x7FFFFFFF)
    assert np.array_equal(got, want)
