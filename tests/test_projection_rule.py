"""Which way the tensor path's projection over many columns takes x: converted
inside, two row tiles per CTA, or by a pass before (host only; the lines are
those measured beside the rule)."""
import ctypes

import pytest

from paper_1905_00689_gb300 import _binding


@pytest.mark.parametrize("columns,D,K,inside", [
    (2400, 4096, 64, False), (4800, 4096, 128, False), (8000, 4096, 64, True),   # one wave; two against one
    (2400, 4096, 256, False), (2800, 4096, 256, True),
    (2800, 4096, 512, False), (4000, 4096, 512, True),                           # three against two; four against two
    (2400, 1024, 64, False), (2400, 256, 64, True),                              # the pass costs a launch
    (65536, 2048, 128, True), (65536, 2048, 512, True), (5120, 1024, 512, True),
])
def test_conversion(columns, D, K, inside):
    f = _binding.load()._ZN16lstm_approx_impl16tc_rows_convertsEiii
    f.argtypes, f.restype = [ctypes.c_int] * 3, ctypes.c_bool
    assert f(columns, 4 * ((K + 127) // 128), D) == inside
