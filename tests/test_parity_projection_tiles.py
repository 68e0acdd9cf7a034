"""GPU parity of the tensor path's projection over many columns (two 128-row
tiles per CTA, x read in fp32 or from its pair) against the oracle on sampled
streams."""
import numpy as np
import pytest

from parity_util import BF16_TOL, assert_parity, oracle_run, run_gpu
from workloads import draw_factor_set, draw_inputs

pytestmark = pytest.mark.gpu


def _check(D, T, B, K, layers, H=64):
    lay = [[draw_factor_set(H, (D if l == 0 else H) + H, K, 30, 9700 + 10 * l + g) for g in range(4)]
           for l in range(layers)]
    x = draw_inputs(T, B, D, "uniform", 97)
    got, m = run_gpu(lay, x, K, dtype="bf16", checkpoints=[K // 2])
    streams = [0, 63, B - 1]
    ref = oracle_run(lay, x[:, streams], K, dtype="bf16", checkpoints=[K // 2])
    cut = {k: v[:, streams] if k in ("h", "c_last") else v[:, :, streams] for k, v in got.items()}
    assert_parity(cut, ref, BF16_TOL)


@pytest.mark.parametrize("D,T,B,K", [
    (2052, 8, 300, 40),    # one wave either way: one row tile per CTA, x converted by a pass
    (2050, 8, 303, 128),   # the same with rows of x TMA cannot map
    (1024, 8, 350, 512),   # three waves against two
    (65, 66, 97, 300),     # five against three: two row tiles, an odd number per gate, from the pair
])
def test_tiles_by_waves(cuda_device, D, T, B, K):
    _check(D, T, B, K, layers=2)


@pytest.mark.parametrize("D,T,B,K", [
    (72, 40, 130, 40),     # one row tile per gate (a CTA's two tiles are two gates), ragged columns, D off the 64s
    (42, 40, 130, 40),     # rows of x TMA cannot map: converted by a pass before
    (4, 37, 128, 130),     # two row tiles per gate, the second nearly empty; one short chunk of D
    (260, 33, 97, 300),    # an odd number of row tiles per gate (pairs across gates)
    (65, 33, 97, 300),     # the same from the pair
    (2044, 64, 512, 96),   # many turns of the ring in every CTA, all SMs busy
])
@pytest.mark.parametrize("layers", [1, 2])
def test_many_columns(cuda_device, D, T, B, K, layers):
    H = 64
    lay = [[draw_factor_set(H, (D if l == 0 else H) + H, K, 30, 9700 + 10 * l + g) for g in range(4)]
           for l in range(layers)]
    x = draw_inputs(T, B, D, "uniform", 97)
    got, m = run_gpu(lay, x, K, dtype="bf16", checkpoints=[K // 2])
    streams = [0, 63, B - 1]
    ref = oracle_run(lay, x[:, streams], K, dtype="bf16", checkpoints=[K // 2])
    cut = {k: v[:, streams] if k in ("h", "c_last") else v[:, :, streams] for k, v in got.items()}
    assert_parity(cut, ref, BF16_TOL)
    again, _ = run_gpu(lay, x, K, dtype="bf16", checkpoints=[K // 2])
    for k, v in got.items():  # the order of every sum is fixed
        assert np.array_equal(again[k], v), k
