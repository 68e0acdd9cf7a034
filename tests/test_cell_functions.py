"""GPU accuracy of the gate nonlinearities and the cell update (Sec. II) of
every kernel family over the whole fp32 range of pre-activations, against
fp64.  All coefficients are zero (sigma = 0), so a gate's pre-activation is its
bias exactly and one timestep evaluates the cell at chosen arguments.

Bounds: the logistic function and tanh are formed from ex2.approx and
rcp.approx (each within 2^-22 relative, PTX ISA) and a few fp32 roundings of
values up to 2: absolute error of either below 1e-6.  c_t sums two products of
them with c_{t-1} and 1, so it errs by at most 1e-6 (1 + |c_{t-1}|) and the
rounding of the sum; h_t by 1.5e-6 and c_t's error times the slope of tanh.
"""
import numpy as np
import pytest

from parity_util import run_gpu

pytestmark = pytest.mark.gpu

# around 0, the series' end at 1/4, saturation, where e^z leaves the normal and
# then the whole fp32 range (87.3, 88.7, 103.3), and far past it
EDGES = [0.0, 1e-30, 1e-8, 1e-4, 0.2499, 0.25, 0.2501, 1.0, 8.0, 16.6, 19.9, 20.1, 43.6, 44.4, 51.6, 87.3, 87.4, 88.7,
         88.8, 103.2, 104.0, 127.0, 200.0, 1e4, 1e30]


@pytest.mark.parametrize("dtype,H,kw", [
    ("fp32", 64, {}),                       # one CTA per stream
    ("fp32", 512, {"variant": 1}), ("fp32", 512, {"variant": 2}),
    ("fp32", 130, {}),                      # per-timestep CUDA-core kernels
    ("bf16", 512, {}),                      # one launch per stream tile
    ("bf16", 640, {}),                      # resident-factor launch
    ("bf16", 640, {"tensor_seq": 1}),       # launches per timestep
])
def test_cell_over_the_whole_range(cuda_device, dtype, H, kw):
    D, B, K = 8, 24, 4
    rng = np.random.default_rng(H)
    edges = np.array(EDGES + [-e for e in EDGES])
    z = rng.uniform(-110.0, 110.0, (4, H)) * rng.choice([1.0, 0.1, 0.01], (4, H))
    z = np.where(rng.random((4, H)) < 0.5, rng.choice(edges, (4, H)), z).astype(np.float32).astype(np.float64)
    z[:, :8] = np.array([-200.0, 40.0, 0.0, 40.0])[:, None]  # h = tanh(c0): i = 0, f = o = 1
    c0 = np.where(rng.random((1, B, H)) < 0.5, rng.choice(edges[np.abs(edges) <= 1e4], (1, B, H)),
                  rng.standard_normal((1, B, H))).astype(np.float32).astype(np.float64)
    gates = [{"sigma": np.zeros(K), "u": rng.standard_normal((K, H)), "idx": np.tile(np.arange(3, dtype=np.int32), (K, 1)),
              "val": np.ones((K, 3)), "bias": z[g]} for g in range(4)]
    got, _ = run_gpu([gates], np.zeros((1, B, D)), K, dtype=dtype, c0=c0, **kw)
    with np.errstate(over="ignore"):
        s = 1.0 / (1.0 + np.exp(-z))
    c = s[1] * c0[0] + s[0] * np.tanh(z[2])
    h = s[3] * np.tanh(c)
    dc = 1e-6 * (1.0 + np.abs(c0[0])) + 2.0 ** -23 * np.abs(c)
    slope = 1.0 - np.tanh(np.maximum(np.abs(c) - dc, 0.0)) ** 2
    assert np.all(np.abs(got["c_last"][0] - c) <= dc)
    assert np.all(np.abs(got["h"][0] - h) <= 1.5e-6 + dc * slope)
    if dtype == "fp32":  # tanh keeps its relative accuracy towards 0
        want = np.tanh(c0[0][:, :8])
        assert np.all(np.abs(got["h"][0][:, :8] - want) <= 2e-6 * np.abs(want))
