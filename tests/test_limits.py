"""The size limits that include/lddmm.h states and that are checked before any CUDA call."""

import ctypes

import pytest


@pytest.mark.parametrize("grid,band", [((64, 600), (8, 514)), ((64, 600), (66, 8)), ((16, 600, 16), (4, 514, 4)),
                                       ((16, 16, 600), (4, 4, 514))])
def test_bands_above_the_limits_are_refused_without_a_gpu(grid, band):
    from paper_1807_11560_gb300 import lddmm
    h = ctypes.c_void_p()
    arr = ctypes.c_int * len(grid)
    assert lddmm.lib().lddmm_create(ctypes.byref(h), len(grid), arr(*grid), arr(*band), 0.01, 2, 0.1, 4, None) == 1
    assert h.value is None
