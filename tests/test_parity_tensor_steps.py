"""GPU parity of the tensor path's launches per timestep (tau' GEMM, gate GEMM,
reduce) at the shapes whose tiles and splits `test_parity_tensor.py` names:
most of them take a launch for all timesteps by themselves, so these runs
force the launches per step."""
import numpy as np
import pytest

import test_parity_tensor as shapes
from parity_util import BF16_TOL, WORKLOADS, assert_parity, oracle_run, run_gpu, synthetic_layer, workload_inputs
from paper_1905_00689_gb300 import BF16, PATH_TENSOR, Q_LAST_PATH, Q_TENSOR_LOOP, Q_TENSOR_SEQ, plan
from workloads import draw_factor_set, draw_inputs

pytestmark = pytest.mark.gpu


def _parameters(test):
    mark = [m for m in test.pytestmark if m.name == "parametrize"][0]
    return pytest.mark.parametrize(*mark.args, **mark.kwargs)


def _run(layers, x, K, **kw):
    got, m = run_gpu(layers, x, K, dtype="bf16", tensor_seq=1, **kw)
    assert m.query(Q_LAST_PATH) == PATH_TENSOR and m.query(Q_TENSOR_LOOP) == 0 and m.query(Q_TENSOR_SEQ) == 0
    return got


@_parameters(shapes.test_tensor_path_small_shapes)
def test_small_shapes(cuda_device, D, H, T, B, K, nz, cps):
    gates = [draw_factor_set(H, D + H, K, nz, 5100 + 7 * D + g) for g in range(4)]
    rng = np.random.default_rng(H)
    for g in gates:
        g["bias"] = 0.2 * rng.standard_normal(H)
    x = draw_inputs(T, B, D, "uniform", 66)
    h0 = 0.3 * rng.standard_normal((1, B, H))
    c0 = 0.3 * rng.standard_normal((1, B, H))
    if H >= 1000:  # the cases meant to split tau'
        assert plan(BF16, H, T, B, K, cps, PATH_TENSOR)["tau_splits"] == 4
    got = _run([gates], x, K, h0=h0, c0=c0, checkpoints=cps)
    assert_parity(got, oracle_run([gates], x, K, dtype="bf16", h0=h0, c0=c0, checkpoints=cps), BF16_TOL)


@_parameters(shapes.test_prefix_of_stored_terms)
def test_prefix_of_stored_terms(cuda_device, K, cps):
    D, H, T, B, KS = 72, 128, 3, 24, 96
    gates = [draw_factor_set(H, D + H, KS, 60, 6100 + g) for g in range(4)]
    x = draw_inputs(T, B, D, "uniform", 8)
    got = _run([gates], x, K, checkpoints=cps, max_rank=KS)
    assert_parity(got, oracle_run([gates], x, K, dtype="bf16", checkpoints=cps), BF16_TOL)


def test_widest_stream_tile(cuda_device):
    D, H, T, B, K = 64, 1280, 2, 1000, 48
    gates = [draw_factor_set(H, D + H, K, 200, 6300 + g) for g in range(4)]
    x = draw_inputs(T, B, D, "uniform", 31)
    assert plan(BF16, H, T, B, K, [16, 32])["gate_tile_streams"] == 128
    got = _run([gates], x, K, checkpoints=[16, 32])
    streams = [0, 517, 895, 999]
    ref = oracle_run([gates], x[:, streams], K, dtype="bf16", checkpoints=[16, 32])
    assert_parity(shapes._sample(got, streams), ref, BF16_TOL)


def test_two_layers(cuda_device):
    """The sequence between layers as its pair, a depth off the 16-term slices."""
    D, H, T, B, K = 72, 96, 4, 12, 48
    layers = [[draw_factor_set(H, (D if l == 0 else H) + H, K, int(0.4 * ((D if l == 0 else H) + H)),
                               6600 + 10 * l + g) for g in range(4)] for l in range(2)]
    x = draw_inputs(T, B, D, "uniform", 9)
    got = _run(layers, x, K, checkpoints=[5, K])
    assert_parity(got, oracle_run(layers, x, K, dtype="bf16", checkpoints=[5, K]), BF16_TOL)


@pytest.mark.parametrize("K,cps", [(32, [16, 19, 32]), (512, []), (512, [16, 259, 512])])
def test_throughput_workload_full_size(cuda_device, K, cps):
    """D=1024, H=512, T=20, B=256, keep 50%, the terms split four ways at K = 512."""
    layers = [list(synthetic_layer("c3", 0, 512, 0.5))]
    x = workload_inputs(WORKLOADS["c3"])
    got = _run(layers, x, K, max_rank=512, checkpoints=cps)
    streams = [0, 77, 255]
    assert_parity(shapes._sample(got, streams), oracle_run(layers, x[:, streams], K, dtype="bf16", checkpoints=cps),
                  BF16_TOL)
