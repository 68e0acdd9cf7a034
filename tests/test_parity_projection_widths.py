"""GPU parity of the few-column input projection (fp32) where x's rows do not
lie on 16-byte boundaries, against the oracle (elementwise 1e-4)."""
import ctypes

import numpy as np
import pytest

from parity_util import FP32_TOL, assert_parity, oracle_run, run_gpu
from paper_1905_00689_gb300 import LSTMApprox, Q_PERSISTENT_VARIANT, _binding
from workloads import draw_factor_set, draw_inputs


def few_column_kernel(columns, D, x=4096, v=4096, ldv=None, ldx=None, bf16=False):
    """Whether the rule the run applies gives this projection to the
    few-column kernel (v, x: addresses of the factor rows and of the input)."""
    f = _binding.load()._ZN16lstm_approx_impl18xproj_cluster_fitsEiiPKviPKfib
    f.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p, ctypes.c_int, ctypes.c_bool]
    f.restype = ctypes.c_bool
    return f(columns, D, v, ldv or (D + 7) // 8 * 8, x, ldx or D, bf16)


@pytest.mark.parametrize("columns,D,kw,fits", [
    (1, 1, {}, True), (256, 301, {}, True), (257, 301, {}, False), (40, 2046, {"x": 4100}, True),
    (9, 300, {"ldv": 300}, True), (9, 302, {"ldv": 302}, False),   # caller's own factor rows off the 16 bytes
    (9, 304, {"v": 4100}, False), (9, 304, {"bf16": True}, True), (9, 300, {"bf16": True}, False),
])
def test_rule(columns, D, kw, fits):
    assert few_column_kernel(columns, D, **kw) == fits


@pytest.mark.gpu
@pytest.mark.parametrize("D,T,B,K,variant", [
    (4, 3, 1, 70, 0), (12, 2, 3, 70, 0),       # off the 8s
    (1, 2, 1, 70, 0), (127, 3, 2, 65, 0), (129, 2, 1, 66, 1),  # around one staged group
    (1027, 3, 3, 80, 1), (2046, 2, 20, 130, 1),  # D split over a cluster, 40 columns (two chunks)
    (301, 32, 8, 40, 1),                        # 256 columns, the most
])
def test_widths(cuda_device, D, T, B, K, variant):
    assert few_column_kernel(T * B, D)
    H = 144
    gates = [draw_factor_set(H, D + H, K, max(1, (D + H) // 3), 9500 + g) for g in range(4)]
    x = draw_inputs(T, B, D, "uniform", 95)
    got, m = run_gpu([gates], x, K, checkpoints=[K // 2], variant=variant)
    assert m.query(Q_PERSISTENT_VARIANT) in (1, 2)
    assert_parity(got, oracle_run([gates], x, K, checkpoints=[K // 2]), FP32_TOL)


@pytest.mark.gpu
@pytest.mark.parametrize("offset", [1, 2, 3])
def test_views(cuda_device, offset):
    """x starting `offset` floats into its buffer, recurrence before the projection (one stream, K = 200)."""
    import torch
    D, H, T, B, K = 64, 512, 4, 1, 200
    gates = [draw_factor_set(H, D + H, K, 100, 9600 + g) for g in range(4)]
    x = draw_inputs(T, B, D, "uniform", 96)
    buf = torch.full((T * B * D + 8,), float("nan"), device="cuda")
    xv = buf[offset:offset + T * B * D].view(T, B, D)
    assert few_column_kernel(T * B, D, x=xv.data_ptr())
    xv.copy_(torch.from_numpy(x.astype(np.float32)))
    m = LSTMApprox(1, [D], H, K, B, "fp32")
    m.set_layer(0, gates)
    out = torch.empty((T, B, H), device="cuda")
    m.run(xv, K, out)
    m.sync()
    assert m.query(Q_PERSISTENT_VARIANT) == 1
    assert_parity({"h": out.double().cpu().numpy()}, oracle_run([gates], x, K), FP32_TOL, keys=("h",))
