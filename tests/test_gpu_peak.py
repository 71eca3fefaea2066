"""mt_imad_peak: the integer multiply-add rate that the benchmark holds the
fixed-point kernels against."""
from __future__ import annotations

import ctypes

import pytest


@pytest.mark.gpu
def test_integer_multiply_add_rate():
    """Repeatable, and between 8 and 64 lanes of an SM and clock (152 SMs, up to
    2070 MHz): neither a chain that waits for its own result nor one that the
    compiler has folded."""
    import paper_2402_06083_gb300 as mt
    a, b = mt.imad_peak(), mt.imad_peak()
    assert abs(a / b - 1) < 0.05
    assert 152 * 8 * 1.4e9 / 1e12 < a < 152 * 64 * 2.07e9 / 1e12


def test_invalid_arguments_fail_before_any_launch():
    from paper_2402_06083_gb300 import _lib
    from paper_2402_06083_gb300 import build as b
    b.build()
    L = _lib.load()
    out = ctypes.c_double(0.0)
    assert L.mt_imad_peak(None, 1 << 30, None, None) == _lib.MT_EINVAL
    assert L.mt_imad_peak(None, 1 << 30, ctypes.byref(out), None) == _lib.MT_ENOMEM
