"""The calls whose speed matters to a user of this library, as plain cases.

A case is one call of `lstm_approx_run` (or `lstm_approx_run_host`, the
host-buffer entry) through the package's public class, on a handle whose
factors are set once, as a program that serves a model does.  The sizes are
those of the workloads in `workloads/`, the benchmark and the tests, plus
odd ones of the same ranges:

- one stream (or a few) with fp32 factors: the latency path, from a call of
  8 timesteps at H = 64 to 20 timesteps at D = 1024, H = 512, K = 256;
- many streams with bf16 factors: the throughput path, from B = 16 to 1024
  streams, K = 8 to 1024, one or two layers;
- with and without intermediate depths, on and off the 16-term slices of
  the tensor-core path; with and without an initial state and final cells.

Factors are random draws with the structure of a pruned residual expansion
(decreasing sigma, unit u, unit v on `nz` random columns), as in
`workloads.draw_factor_set`, drawn on the GPU and already representable in
the storage type, so that the 64-bit result below is of the same factors.
"""
import math

import numpy as np
import torch

from paper_1905_00689_gb300 import LSTMApprox


def _case(name, dtype, D, H, T, B, K, keep, depths=(), L=1, x="uniform", state=False, host=False):
    return {"name": name, "dtype": dtype, "D": D, "H": H, "T": T, "B": B, "K": K, "keep": keep,
            "depths": ",".join(str(d) for d in depths), "L": L, "x": x, "state": state, "host": host}


def listed():
    return [
        # the smallest call: the D = H = 64 model, one stream, two outputs cut
        # short at 4 and 8 terms (launches and set-up are most of it)
        _case("small-one-stream", "fp32", 64, 64, 8, 1, 16, 0.5, (4, 8)),
        # the paper's case-study LSTM (Sec. VI), one timestep per call: a
        # control loop that feeds one video frame at a time
        _case("frame-by-frame", "fp32", 8256, 64, 1, 1, 16, 130 / 8320, x="relu", state=True),
        # the benchmark's latency workload: a clip of 20 frames, all 256
        # terms, outputs at 16 and 64 for a time budget that may be cut
        _case("clip-k256", "fp32", 1024, 512, 20, 1, 256, 0.25, (16, 64), x="relu"),
        # the same model at 64 terms through the host-buffer call (copies in
        # and out inside the call), as an application without device tensors
        _case("clip-k64-host", "fp32", 1024, 512, 20, 1, 64, 0.25, x="relu", host=True),
        # eight cameras at once on the fp32 model
        _case("eight-streams", "fp32", 1024, 512, 20, 8, 64, 0.25, x="relu"),
        # a small two-layer model of odd sizes, resumed from a state
        _case("odd-two-layer", "fp32", 300, 200, 15, 3, 50, 0.3, (7, 20), L=2, state=True),
        # the batched models: 256 streams of clips, all terms with two early outputs
        _case("batch256-k512", "bf16", 1024, 512, 20, 256, 512, 0.5, (32, 128), x="relu"),
        # odd sizes on the batched path, depths off the 16-term slices, resumed
        _case("odd-batch", "bf16", 1000, 600, 13, 100, 90, 0.4, (10, 45), state=True),
        # 1024 streams at a coarse, a middle and a fine depth
        _case("batch1024-k8", "bf16", 2048, 1024, 64, 1024, 8, 0.5),
        _case("batch1024-k128", "bf16", 2048, 1024, 64, 1024, 128, 0.1),
        _case("batch1024-k512", "bf16", 2048, 1024, 64, 1024, 512, 0.5),
        # two wide layers, outputs at four depths in one run
        _case("two-layer-progressive", "bf16", 4096, 2048, 16, 64, 1024, 0.3, (16, 64, 256, 1024), L=2),
    ]


def _log_int(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))
    return max(lo, min(hi, int(v) // step * step if v >= step else lo))


def _cost(c):
    return 8.0 * c["L"] * c["T"] * c["B"] * c["K"] * (c["D"] + 2 * c["H"])


def draw(rng):
    """One more case of the same ranges, at most the largest listed one's work."""
    most = max(_cost(c) for c in listed())
    c = {"L": 2 if rng.random() < 0.25 else 1, "x": rng.choice(["uniform", "relu"]), "state": rng.random() < 0.4,
         "host": rng.random() < 0.2}
    if rng.random() < 0.4:  # latency: fp32, one stream or a few
        c.update(dtype="fp32", D=_log_int(rng, 32, 8256, rng.choice([1, 4, 64])), H=_log_int(rng, 32, 768, rng.choice([4, 32])),
                 T=_log_int(rng, 1, 32), B=rng.choice([1, 1, 1, 2, 3, 8, 16]), K=_log_int(rng, 1, 256),
                 keep=rng.choice([0.05, 0.25, 0.5]))
    else:  # throughput: bf16, many streams
        c.update(dtype="bf16", D=_log_int(rng, 64, 4096, rng.choice([1, 8, 64])),
                 H=rng.choice([256, 512, 1024, _log_int(rng, 128, 2048, rng.choice([1, 8, 64]))]),
                 T=_log_int(rng, 2, 64), B=_log_int(rng, 16, 1024, rng.choice([1, 16])),
                 K=rng.choice([8, 32, 128, 512, _log_int(rng, 4, 1024)]), keep=rng.choice([0.1, 0.3, 0.5]), host=False)
    while _cost(c) > most and c["T"] > 1:
        c["T"] //= 2
    while _cost(c) > most and c["B"] > 1:
        c["B"] //= 2
    n = rng.choice([0, 0, 1, 2])
    depths = sorted({max(1, min(c["K"], rng.choice([16, c["K"] // 2, rng.randint(1, c["K"])]))) for _ in range(n)})
    c["depths"] = ",".join(str(d) for d in depths)
    return c


def _depths(c):
    return [int(d) for d in c["depths"].split(",")] if c["depths"] else []


def _nz(c, C):
    return max(1, int(math.floor(c["keep"] * C + 0.5)))


def _inputs(c, seed):
    """Factors per layer and gate, the sequence and the state, on the GPU (64-bit values that the
    storage types hold exactly)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1000003 + 17)
    store = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32

    def rand(*s):
        return torch.rand(*s, device="cuda", generator=g)

    def randn(*s):
        return torch.randn(*s, device="cuda", generator=g)

    H, K = c["H"], c["K"]
    layers = []
    for l in range(c["L"]):
        C = (c["D"] if l == 0 else H) + H
        nz, r = _nz(c, C), math.sqrt(H / C)
        gates = []
        for _ in range(4):
            sigma = (rand(K) * (1 + r - max(1 - r, 0.05)) + max(1 - r, 0.05)).sort(descending=True).values
            u = randn(K, H)
            u = (u / u.norm(dim=1, keepdim=True)).to(store).double()
            val = randn(K, nz)
            val = (val / val.norm(dim=1, keepdim=True)).to(store).double()
            idx = rand(K, C).topk(nz, dim=1).indices.sort(dim=1).values
            gates.append({"sigma": sigma.double(), "u": u, "idx": idx, "val": val, "bias": (0.1 * randn(H)).double()})
        layers.append(gates)
    x = randn(c["T"], c["B"], c["D"]).clamp_(min=0) if c["x"] == "relu" else rand(c["T"], c["B"], c["D"]) * 2 - 1
    h0 = c0 = None
    if c["state"]:
        h0 = 0.3 * randn(c["L"], c["B"], H)
        c0 = 0.3 * randn(c["L"], c["B"], H)
    return layers, x, h0, c0


def prepare(case, seed):
    layers, x, h0, c0 = _inputs(case, seed)
    T, B, H, L = case["T"], case["B"], case["H"], case["L"]
    m = LSTMApprox(L, [case["D"]] + [H] * (L - 1), H, case["K"], B, case["dtype"])
    for l, gates in enumerate(layers):
        m.set_layer(l, [{"sigma": f["sigma"].cpu().numpy(), "u": f["u"].cpu().numpy(),
                         "idx": f["idx"].to(torch.int32).cpu().numpy(), "val": f["val"].cpu().numpy(),
                         "bias": f["bias"].cpu().numpy()} for f in gates])
    J = len(_depths(case))
    s = {"m": m, "K": case["K"], "depths": _depths(case), "host": case["host"], "x": x, "h0": h0, "c0": c0,
         "h": torch.empty(T, B, H, device="cuda"), "c": torch.empty(L, B, H, device="cuda") if case["state"] else None,
         "kh": torch.empty(J, T, B, H, device="cuda") if J else None}
    if case["host"]:  # page-locked buffers, as a program that calls in a loop holds them
        for k in ("x", "h0", "c0", "h", "c", "kh"):
            if s[k] is not None:
                s[k] = s[k].cpu().pin_memory().numpy()
    return s


def run(state):
    s = state
    call = s["m"].run_host if s["host"] else s["m"].run
    call(s["x"], s["K"], s["h"], h0=s["h0"], c0=s["c0"], out_c=s["c"], checkpoints=s["depths"], ckpt_h=s["kh"])
    out = {"h": s["h"]}
    if s["c"] is not None:
        out["c"] = s["c"]
    if s["kh"] is not None:
        out["depths_h"] = s["kh"]
    return out


def work(case):
    """The method's own operations, 4 K (2 NZ + 2 H + 1) per layer, timestep and stream (Sec. III), and
    its bytes: the factors as kept values with a bit per column, the inputs and the outputs, once each."""
    T, B, H, K, L = case["T"], case["B"], case["H"], case["K"], case["L"]
    size = 2 if case["dtype"] == "bf16" else 4
    flops = nbytes = 0
    for l in range(L):
        C = (case["D"] if l == 0 else H) + H
        nz = _nz(case, C)
        flops += T * B * 4 * K * (2 * nz + 2 * H + 1)
        nbytes += 4 * K * (nz * size + (C + 7) // 8 + H * size + 4) + 16 * H
    nbytes += 4 * T * B * (case["D"] + H * (1 + len(_depths(case)))) + (12 * L * B * H if case["state"] else 0)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """fp32 path: 32-bit sums, measured 1e-7 to 2.1e-7 from `exact` over the listed and drawn cases.
    bf16 path: the activations enter the products as two bf16 halves (about 2^-17 each) and all sums are
    32-bit; measured 1.1e-6 to 5.1e-6, growing with K and the widths."""
    return {"rel": 1.5e-6 if case["dtype"] == "fp32" else 2.5e-5}


def exact(case, seed):
    """The recurrence in 64 bits on the same inputs."""
    layers, x, h0, c0 = _inputs(case, seed)
    T, B, H, K = case["T"], case["B"], case["H"], case["K"]
    depths = _depths(case)
    seq = x.double()
    depths_h = torch.zeros(len(depths), T, B, H, dtype=torch.float64, device="cuda")
    last_c = []
    for l, gates in enumerate(layers):
        D = seq.shape[2]
        V = []
        for f in gates:
            v = torch.zeros(K, D + H, dtype=torch.float64, device="cuda")
            v.scatter_(1, f["idx"], f["val"])
            V.append(v)
        V = torch.cat(V)                                                   # [4K][D + H]
        P = (seq.reshape(T * B, D) @ V[:, :D].t()).reshape(T, B, 4, K)
        Vh = V[:, D:].t().contiguous()
        S = torch.stack([f["sigma"] for f in gates])
        U = torch.stack([f["u"] for f in gates])                           # [4][K][H]
        bias = torch.stack([f["bias"] for f in gates])
        h = h0[l].double() if h0 is not None else torch.zeros(B, H, dtype=torch.float64, device="cuda")
        c = c0[l].double() if c0 is not None else torch.zeros_like(h)

        def cell(y, c):
            y = y + bias[:, None, :]
            c = torch.sigmoid(y[1]) * c + torch.sigmoid(y[0]) * torch.tanh(y[2])
            return torch.sigmoid(y[3]) * torch.tanh(c), c

        out = torch.empty(T, B, H, dtype=torch.float64, device="cuda")
        for t in range(T):
            tau = (S * (P[t] + (h @ Vh).reshape(B, 4, K))).transpose(0, 1)  # [4][B][K]
            if l == case["L"] - 1:
                for j, k in enumerate(depths):
                    depths_h[j, t] = cell(tau[:, :, :k] @ U[:, :k], c)[0]
            h, c = cell(tau @ U, c)
            out[t] = h
        seq = out
        last_c.append(c)
    want = {"h": seq}
    if case["state"]:
        want["c"] = torch.stack(last_c)
    if depths:
        want["depths_h"] = depths_h
    return {k: v.cpu().numpy() for k, v in want.items()} if case["host"] else want
