"""GPU parity of the one-CTA persistent kernel (fp32 factors in one CTA's
registers, the input projection inside where it is small; automatic runs
only), and the rule that chooses it (CPU).

Against the oracle (elementwise 1e-4, as every fp32 kernel), and against the
one-exchange or per-unit-block kernel on the same inputs: both sum the same
fp32 products in another order, so their outputs differ by a few unit
roundoffs of sums of at most D + H + K terms; 2e-5 of the largest value
allows 300 of them.
"""
import numpy as np
import pytest

from parity_util import FP32_TOL, assert_parity, oracle_run, run_gpu
from paper_1905_00689_gb300 import FP32, PATH_SIMT, Q_LAST_PATH, Q_LAUNCHES, Q_PERSISTENT_VARIANT, plan
from workloads import draw_factor_set, draw_inputs


@pytest.mark.gpu
@pytest.mark.parametrize("D,H,T,B,K,nz,cps,L,launches", [
    (1, 4, 1, 1, 1, 1, [], 1, 1),                 # the smallest of everything
    (64, 64, 8, 1, 16, 64, [4, 8], 1, 1),         # 256 threads, dense projection inside
    (64, 64, 9, 1, 16, 128, [1, 2, 3, 15, 16], 1, 1),  # a second pass of timesteps, two rounds of depth sets
    (35, 28, 17, 3, 5, 20, [4], 1, 1),            # D off the 16-byte rows, three passes, several streams
    (8256, 64, 1, 1, 16, 130, [], 1, 1),          # compressed rows inside
    (1000, 64, 3, 2, 4, 20, [2], 1, 1),           # the same, several streams and timesteps
    (1024, 64, 4, 1, 32, 300, [13], 1, 2),        # 512 threads; projection by its own launch
    (300, 128, 3, 2, 16, 100, [15], 1, 2),        # the largest H
    (20, 8, 5, 2, 128, 10, [100, 127], 1, 1),     # the largest K
    (48, 64, 4, 2, 20, 30, [7], 2, 2),            # two layers
    (12, 32, 3, 200, 8, 12, [], 1, 2),            # more streams than SMs: projection by its own launch
])
def test_one_cta_kernel(cuda_device, D, H, T, B, K, nz, cps, L, launches):
    layers = [[draw_factor_set(H, (D if l == 0 else H) + H, K, min(nz, (D if l == 0 else H) + H), 9100 + 10 * l + g)
               for g in range(4)] for l in range(L)]
    rng = np.random.default_rng(D + K)
    for la in layers:
        for g in la:
            g["bias"] = 0.3 * rng.standard_normal(H)
    x = draw_inputs(T, B, D, "uniform", 91)
    h0 = 0.5 * rng.standard_normal((L, B, H))
    c0 = 0.5 * rng.standard_normal((L, B, H))
    got, m = run_gpu(layers, x, K, h0=h0, c0=c0, checkpoints=cps)
    assert m.query(Q_PERSISTENT_VARIANT) == 3 and m.query(Q_LAUNCHES) == launches
    assert plan(FP32, H, T, B, K, cps)["one_cta"] == 1
    assert_parity(got, oracle_run(layers, x, K, h0=h0, c0=c0, checkpoints=cps), FP32_TOL)
    other, m2 = run_gpu(layers, x, K, h0=h0, c0=c0, checkpoints=cps, variant=1)
    assert m2.query(Q_PERSISTENT_VARIANT) == 1
    for k in got:
        assert np.abs(got[k] - other[k]).max() <= 2e-5 * np.abs(other[k]).max(), k


@pytest.mark.gpu
def test_depths_ignore_later_terms_that_are_not_finite(cuda_device):
    """A term whose coefficient is infinite leaves the depths that end before
    it what they are without it."""
    D, H, T, K = 16, 16, 1, 6
    gates = [draw_factor_set(H, D + H, K, D, 9300 + g) for g in range(4)]
    x = draw_inputs(T, 1, D, "uniform", 93)
    plain, _ = run_gpu([gates], x, K, checkpoints=[2, 5])
    for g in gates:
        g["sigma"] = g["sigma"].copy()
        g["sigma"][K - 1] = np.inf
    got, m = run_gpu([gates], x, K, checkpoints=[2, 5])
    assert m.query(Q_PERSISTENT_VARIANT) == 3
    assert not np.array_equal(got["h"], plain["h"])
    for k in ("ckpt_h", "ckpt_c"):
        assert np.isfinite(plain[k]).all() and np.array_equal(got[k], plain[k]), k


@pytest.mark.gpu
@pytest.mark.parametrize("H,K,term", [(8, 8, 5), (8, 40, 37), (4, 104, 101), (64, 8, 7)])
def test_lanes_past_a_row_meet_no_infinity(cuda_device, H, K, term):
    """Lanes without values of their own add nothing, also where the row's
    last coefficients are infinite: the gate saturates, as for a very large
    coefficient."""
    D, T = 12, 2
    gates = [draw_factor_set(H, D + H, K, 10, 9350 + g) for g in range(4)]
    gates[2]["sigma"] = gates[2]["sigma"].copy()
    x = draw_inputs(T, 1, D, "uniform", 94)
    gates[2]["sigma"][term] = 1e30
    ref = oracle_run([gates], x, K, checkpoints=[4])
    gates[2]["sigma"][term] = np.inf
    got, m = run_gpu([gates], x, K, checkpoints=[4])
    assert m.query(Q_PERSISTENT_VARIANT) == 3
    assert_parity(got, ref, FP32_TOL)


@pytest.mark.parametrize("H,K,one", [(64, 16, 1), (64, 32, 1), (64, 33, 0), (128, 16, 1), (128, 17, 0), (132, 4, 0),
                                     (32, 64, 1), (32, 65, 0), (4, 128, 1), (4, 129, 0), (512, 16, 0)])
def test_rule(H, K, one):
    """H, K <= 128 and at most 16 values of either factor per thread of 512."""
    assert plan(FP32, H, 4, 1, K)["one_cta"] == one


@pytest.mark.gpu
def test_widths_off_the_quads_take_the_per_timestep_kernels(cuda_device):
    """H not a multiple of 4: no persistent kernel, whatever the size."""
    D, H, T, B, K = 20, 62, 3, 2, 6
    gates = [draw_factor_set(H, D + H, K, 20, 9400 + g) for g in range(4)]
    x = draw_inputs(T, B, D, "uniform", 95)
    got, m = run_gpu([gates], x, K, checkpoints=[3])
    assert m.query(Q_LAST_PATH) == PATH_SIMT == plan(FP32, H, T, B, K, [3])["path"]
    assert_parity(got, oracle_run([gates], x, K, checkpoints=[3]), FP32_TOL)


@pytest.mark.parametrize("H,K,T,cps,one", [
    (64, 32, 12, [], 1), (64, 32, 13, [], 0), (64, 32, 13, [8], 1), (64, 32, 13, [32], 0),
    (128, 16, 20, [], 1), (128, 16, 21, [], 0), (64, 16, 100, [], 1), (128, 8, 100, [], 1), (8, 96, 32, [], 1),
])
def test_rule_for_many_timesteps(H, K, T, cps, one):
    """512 threads of 16 values: a longer step than the cluster kernel's without depths below K."""
    assert plan(FP32, H, T, 1, K, cps)["one_cta"] == one


@pytest.mark.gpu
@pytest.mark.parametrize("H,K,T,variant", [(64, 32, 12, 3), (64, 32, 13, 2), (128, 16, 21, 2)])
def test_many_timesteps_run_what_the_plan_says(cuda_device, H, K, T, variant):
    gates = [draw_factor_set(H, 24 + H, K, 40, 9380 + g) for g in range(4)]
    x = draw_inputs(T, 2, 24, "uniform", 96)
    got, m = run_gpu([gates], x, K)
    assert m.query(Q_PERSISTENT_VARIANT) == variant
    assert_parity(got, oracle_run([gates], x, K), FP32_TOL)
