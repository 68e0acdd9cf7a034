"""GPU parity of the tensor path's launch over all stream tiles and timesteps
with the factors resident on chip (bf16 factors; k_tensor_loop.cu), and the
rule that chooses it (CPU).

Each GPU case is checked against the oracle on the factors as the library
stores them, and against the two-launches-per-step kernels on the same inputs.
The second bound, 4e-4 of the largest value, is derived: both form the same
products of the same bf16 pairs (2^-17 relative each), K + H terms of fp32 sums
in another order (relative 2^-24 each), over T steps of a contracting cell.
"""
import numpy as np
import pytest

from parity_util import BF16_TOL, assert_parity, oracle_run, run_gpu
from paper_1905_00689_gb300 import (BF16, LSTMApprox, LSTMApproxError, OPT_TEST_STALL, OPT_WAIT_LIMIT, Q_TENSOR_LOOP,
                                    Q_TENSOR_SEQ, plan)
from workloads import draw_factor_set, draw_inputs


def _gates(H, C, K, nz, seed):
    gates = [draw_factor_set(H, C, K, nz, seed + g) for g in range(4)]
    rng = np.random.default_rng(seed)
    for g in gates:
        g["bias"] = 0.2 * rng.standard_normal(H)
    return gates


@pytest.mark.gpu
@pytest.mark.parametrize("H,T,B,K,cps", [
    (64, 3, 1, 1, []),                      # one term, one stream: 16 packed rows per gate
    (72, 2, 17, 16, [16]),                  # the largest K of 16 rows; a depth at K
    (301, 3, 33, 17, [1, 16]),              # odd H (a padding column), 32 rows; a depth of one term
    (640, 2, 40, 33, [3, 9, 20]),           # 64 rows, H over two CTAs, two depths in one slice
    (128, 4, 32, 64, []),                   # whole tiles
    (512, 3, 65, 65, [64]),                 # 128 rows, a depth at a chunk boundary
    (1000, 2, 31, 128, [17, 100]),          # largest K with all gates in a CTA
    (512, 3, 33, 129, [128]),               # one gate per CTA: the gate exchange
    (1100, 2, 20, 200, [5, 48, 199]),       # H over four CTAs, both exchanges
    (1024, 2, 40, 512, [32, 511]),          # both exchanges, groups of two and four
    (2048, 2, 64, 1024, [16, 64, 256, 1024]),  # terms of U in shared memory, several tiles per CTA
    (256, 2, 300, 1000, []),                # many row tiles: several stream tiles per CTA
    (512, 3, 40, 513, []),                  # the shortest sum cut into segments
    (512, 3, 40, 902, [9, 451]),            # depths among the segments, one inside a slice
    (512, 3, 40, 800, [640]),               # a segment after the last depth
])
def test_small_shapes(cuda_device, H, T, B, K, cps):
    D = 48
    gates = _gates(H, D + H, K, min(60, D + H), 8100 + H + K)
    rng = np.random.default_rng(B)
    x = draw_inputs(T, B, D, "uniform", 80 + B)
    h0 = 0.3 * rng.standard_normal((1, B, H))
    c0 = 0.3 * rng.standard_normal((1, B, H))
    got, m = run_gpu([gates], x, K, dtype="bf16", h0=h0, c0=c0, checkpoints=cps)
    assert m.query(Q_TENSOR_LOOP) == 1 == plan(BF16, H, T, B, K, cps)["tensor_loop"]
    step, m2 = run_gpu([gates], x, K, dtype="bf16", h0=h0, c0=c0, checkpoints=cps, tensor_seq=1)
    assert m2.query(Q_TENSOR_LOOP) == 0
    for k in got:
        assert np.abs(got[k] - step[k]).max() <= 4e-4 * np.abs(step[k]).max(), k
    streams = sorted({0, B // 2, B - 1})
    ref = oracle_run([gates], x[:, streams], K, dtype="bf16", h0=h0[:, streams], c0=c0[:, streams], checkpoints=cps)
    cut = {k: v[:, streams] if k in ("h", "c_last") else v[:, :, streams] for k, v in got.items()}
    assert_parity(cut, ref, BF16_TOL)


@pytest.mark.gpu
def test_two_layers_and_graph_replay(cuda_device):
    """Layer 0 hands its sequence on as the pair; a captured run replayed on
    new inputs equals an eager one (the counters are left at zero)."""
    import torch
    D, H, T, B, K = 72, 136, 4, 40, 48
    layers = [_gates(H, (D if l == 0 else H) + H, K, 60, 8300 + 10 * l) for l in range(2)]
    x = draw_inputs(T, B, D, "uniform", 83)
    got, m = run_gpu(layers, x, K, dtype="bf16", checkpoints=[10])
    assert m.query(Q_TENSOR_LOOP) == 1
    assert_parity(got, oracle_run(layers, x, K, dtype="bf16", checkpoints=[10]), BF16_TOL)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        m = LSTMApprox(2, [D, H], H, K, B, "bf16", stream=s)
        for l in range(2):
            m.set_layer(l, layers[l])
        xt = torch.zeros(T, B, D, device="cuda")
        out = torch.empty(T, B, H, device="cuda")
        m.run(xt, K, out)
        m.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            m.run(xt, K, out)
        xt.copy_(torch.from_numpy(x.astype(np.float32)))
        for _ in range(2):
            g.replay()
        m.sync()
    eager, _ = run_gpu(layers, x, K, dtype="bf16")  # the same call: no depths, so the same order of sums
    assert np.array_equal(out.double().cpu().numpy(), eager["h"])


@pytest.mark.gpu
@pytest.mark.parametrize("H,B,K,T,warm", [
    (256, 64, 1000, 2, (9, 1000)),    # few timesteps after many
    (1024, 128, 1000, 9, (9, 512)),   # past this launch's limits after a shape within them
])
def test_capture_needs_no_storage_of_the_other_launches(cuda_device, H, B, K, T, warm):
    """Where the launches per step are the faster way but would have to
    allocate while the stream is captured, this launch is captured instead; an
    eager run of the same call takes them."""
    import torch
    D = 40
    gates = _gates(H, D + H, K, 60, 8900 + H)
    x = torch.from_numpy(draw_inputs(warm[0], B, D, "uniform", 89).astype(np.float32)).cuda()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        m = LSTMApprox(1, [D], H, K, B, "bf16", stream=s)
        m.set_layer(0, gates)
        out = torch.empty(warm[0], B, H, device="cuda")
        m.run(x, warm[1], out)
        m.sync()
        assert m.query(Q_TENSOR_LOOP) == 1
        got = torch.empty(T, B, H, device="cuda")
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            m.run(x[:T], K, got)
        assert m.query(Q_TENSOR_LOOP) == 1
        g.replay()
        m.sync()
        eager = torch.empty(T, B, H, device="cuda")
        m.run(x[:T], K, eager)
        m.sync()
        assert m.query(Q_TENSOR_LOOP) == 0 == plan(BF16, H, T, B, K, [])["tensor_loop"]
    assert float((got - eager).abs().max()) <= 4e-4 * float(eager.abs().max())


@pytest.mark.gpu
def test_two_handles_on_two_streams(cuda_device):
    """Launches of two handles on two streams, each needing most of the SMs
    at once, complete and agree."""
    import torch
    D, H, T, B, K = 64, 512, 6, 256, 200
    gates = _gates(H, D + H, K, 100, 8400)
    x = torch.from_numpy(draw_inputs(T, B, D, "uniform", 84).astype(np.float32)).cuda()
    runs = []
    for _ in range(2):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            m = LSTMApprox(1, [D], H, K, B, "bf16", stream=s)
            m.set_layer(0, gates)
            runs.append((s, m, torch.empty(T, B, H, device="cuda")))
    torch.cuda.synchronize()
    for _ in range(10):
        for s, m, out in runs:
            with torch.cuda.stream(s):
                m.run(x, K, out)
    for s, m, out in runs:
        m.sync()
        assert m.query(Q_TENSOR_LOOP) == 1
    assert torch.equal(runs[0][2], runs[1][2])


@pytest.mark.gpu
@pytest.mark.parametrize("H,K", [(136, 40), (1024, 200)])
def test_bounded_wait_reports_timeout(cuda_device, H, K):
    """CTA 0 withholds its first h: the waits run out after the short limit,
    the run reports ETIMEOUT, and the next run on the handle is correct."""
    import torch
    D, T, B = 32, 3, 20
    gates = _gates(H, D + H, K, 40, 8500)
    x = draw_inputs(T, B, D, "uniform", 85)
    ref, m = run_gpu([gates], x, K, dtype="bf16")
    m.set_option(OPT_WAIT_LIMIT, 50_000)  # 50 ms
    m.set_option(OPT_TEST_STALL, 1)
    xt = torch.from_numpy(x.astype(np.float32)).cuda()
    out = torch.zeros((T, B, H), device="cuda")
    m.run(xt, K, out)
    with pytest.raises(LSTMApproxError) as ei:
        m.sync()
    assert ei.value.code == 4  # LSTM_APPROX_ETIMEOUT
    m.set_option(OPT_WAIT_LIMIT, 2_000_000)
    m.run(xt, K, out)
    m.sync()
    assert np.array_equal(out.double().cpu().numpy(), ref["h"])


@pytest.mark.gpu
@pytest.mark.parametrize("T", [1, 2])
@pytest.mark.parametrize("H,B,K,cps", [
    (136, 40, 40, [10, 32]),    # all gates in a CTA
    (512, 70, 200, [64, 100]),  # one gate per CTA
    (512, 256, 640, [320]),     # segments
    (512, 1000, 100, [50]),     # several stream tiles per CTA
])
def test_state_in_place(cuda_device, H, B, K, cps, T):
    """The same buffers as initial and final state (a caller that resumes one
    call after another): every output as with separate buffers."""
    import torch
    D = 40
    gates = _gates(H, D + H, K, 50, 8600 + H + K)
    rng = np.random.default_rng(86)
    x = torch.from_numpy(draw_inputs(T, B, D, "uniform", 86).astype(np.float32)).cuda()
    h0, c0 = (torch.from_numpy(rng.standard_normal((1, B, H)).astype(np.float32)).cuda() for _ in range(2))
    m = LSTMApprox(1, [D], H, K, B, "bf16")
    m.set_layer(0, gates)
    res = []
    for in_place in (False, True):
        h_in, c_in = h0.clone(), c0.clone()
        c_out = c_in if in_place else torch.empty_like(c_in)
        out = h_in if in_place and T == 1 else torch.empty(T, B, H, device="cuda")
        ck = torch.empty(2, len(cps), T, B, H, device="cuda")
        m.run(x, K, out, h0=h_in, c0=c_in, out_c=c_out, checkpoints=cps, ckpt_h=ck[0], ckpt_c=ck[1])
        m.sync()
        assert m.query(Q_TENSOR_LOOP) == 1
        res.append((out, c_out, ck))
    for apart, same in zip(*res):
        assert torch.equal(apart, same)


@pytest.mark.gpu
@pytest.mark.parametrize("H,B,K,cps,term", [
    (72, 20, 48, [10, 45], 12),      # all gates in a CTA; the term shares the first depth's slice
    (72, 20, 48, [10, 32, 45], 46),  # ... the last depth's; the others end before it
    (1024, 300, 128, [20, 64], 21),  # several stream tiles per CTA
    (512, 40, 200, [100, 133], 143),  # one gate per CTA
    (512, 40, 902, [451, 455], 453),  # segments; one depth before the term, one past it
])
def test_depths_ignore_later_terms_that_are_not_finite(cuda_device, H, B, K, cps, term):
    """A term whose coefficient is infinite leaves the depths that end before
    it what they are without it, also inside its 16-term slice; everything
    agrees with the two-launches-per-step kernels, which stop at the depth."""
    D, T = 32, 3
    gates = _gates(H, D + H, K, 50, 8700 + H + K)
    x = draw_inputs(T, B, D, "uniform", 87)
    plain, _ = run_gpu([gates], x, K, dtype="bf16", checkpoints=cps)
    gates[1]["sigma"] = gates[1]["sigma"].copy()
    gates[1]["sigma"][term] = np.inf
    got, m = run_gpu([gates], x, K, dtype="bf16", checkpoints=cps)
    assert m.query(Q_TENSOR_LOOP) == 1
    step, m2 = run_gpu([gates], x, K, dtype="bf16", checkpoints=cps, tensor_seq=1)
    assert m2.query(Q_TENSOR_LOOP) == 0
    for k in got:
        assert np.isfinite(step[k]).all() and np.abs(got[k] - step[k]).max() <= 4e-4 * np.abs(step[k]).max(), k
    for i, c in enumerate(cps):
        if c <= term:  # the first step starts from the same state
            assert np.abs(got["ckpt_h"][i, 0] - plain["ckpt_h"][i, 0]).max() <= 1e-5


@pytest.mark.parametrize("H,B,K,cps,loop", [
    (512, 256, 512, [], 1), (512, 256, 32, [], 0),             # K <= 32 at H = 512: one launch per stream tile
    (600, 100, 32, [10], 1), (2048, 64, 1024, [16, 256], 1),
    (2049, 16, 64, [], 0), (2048, 16, 1025, [], 0),             # outside its limits
    (1024, 1024, 128, [], 1), (1024, 1024, 512, [], 0),         # too many streams per CTA
    (1024, 256, 640, [], 1), (1024, 256, 1000, [], 0),
    (512, 400, 200, [], 1), (512, 600, 256, [], 0), (512, 600, 256, [100], 1), (2048, 256, 200, [], 1),
])
def test_rule(H, B, K, cps, loop):
    p = plan(BF16, H, 2, B, K, cps)
    assert p["tensor_loop"] == loop
    assert p["tensor_seq"] == (1 if K <= 32 and H == 512 else 0)


@pytest.mark.parametrize("H,B,K,cps,loop", [
    (1024, 256, 448, [], 1), (1024, 300, 448, [], 0), (1024, 300, 512, [], 1),    # 128, 160, 160 streams per CTA
    (512, 500, 384, [], 1), (512, 600, 384, [], 0), (512, 600, 448, [], 1),
    (1024, 128, 800, [], 1), (1024, 160, 800, [], 0), (512, 400, 800, [], 1),
    (1024, 64, 1000, [], 1), (1024, 96, 1000, [], 0),                             # tiles of 16 for want of room
    (2048, 64, 1000, [64, 320], 1), (2048, 96, 1000, [64, 320], 0),
])
def test_limits(H, B, K, cps, loop):
    """Either side of the measured lines between this launch and two launches per step."""
    assert plan(BF16, H, 12, B, K, cps)["tensor_loop"] == loop


@pytest.mark.parametrize("H,B,K,cps,T,loop", [
    (256, 64, 1000, [], 1, 0), (256, 64, 1000, [], 2, 0), (256, 64, 1000, [], 9, 1),
    (136, 40, 48, [], 1, 0), (136, 40, 48, [], 4, 1),
    (1024, 256, 200, [], 1, 1), (600, 100, 90, [10, 45], 1, 1),
    (1024, 1024, 128, [], 1, 0), (1024, 1024, 128, [], 2, 1),      # many streams: from two steps on
])
def test_few_timesteps(H, B, K, cps, T, loop):
    """A run too short to pay for loading the factors takes the launches per step."""
    assert plan(BF16, H, T, B, K, cps)["tensor_loop"] == loop


@pytest.mark.gpu
@pytest.mark.parametrize("H,B,K,cps", [(256, 64, 1000, []), (136, 40, 48, [10]), (512, 33, 129, [128])])
def test_few_timesteps_run_what_the_plan_says(cuda_device, H, B, K, cps):
    D = 40
    gates = _gates(H, D + H, K, 60, 8800 + H)
    for T in (1, 2, 9):
        x = draw_inputs(T, B, D, "uniform", 88)
        got, m = run_gpu([gates], x, K, dtype="bf16", checkpoints=cps)
        assert m.query(Q_TENSOR_LOOP) == plan(BF16, H, T, B, K, cps)["tensor_loop"]
        streams = sorted({0, B // 2, B - 1})
        ref = oracle_run([gates], x[:, streams], K, dtype="bf16", checkpoints=cps)
        cut = {k: v[:, streams] if k in ("h", "c_last") else v[:, :, streams] for k, v in got.items()}
        assert_parity(cut, ref, BF16_TOL)
