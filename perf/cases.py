"""Performance cases of the mixed-bit linear layer.

Each case is one pass through the public entry points of
``paper_2607_14618_gb300.polyq`` as a user's program makes it: a decode GEMV
(``linear_gemv``, ``linear_gemv_group``, ``linear_gemv_noalloc``), one decoder
layer of a decode step (four fused calls captured as a CUDA graph, or one
chained launch), or a prefill GEMM (``linear_gemm``).  ``listed()`` names the
standing cases, ``draw()`` gives others of the same ranges, ``prepare()`` packs
the layers and makes the inputs and the buffers a program keeps, ``run()`` is
the timed pass and ``exact()`` the same result in 64 bits from the definition
of the layer (allocation, quantiser, product), written here without the
library.

Inputs follow the synthetic recipe of ``synth.py`` on the GPU: weights
N(0, 0.02^2) with 1% of the columns x10, activation magnitudes lognormal(0, 1)
with 1% of the channels x20, activations bf16(magnitude * N(0, 1)).
"""
import heapq
import math

import numpy as np
import torch

from paper_2607_14618_gb300 import polyq

DEV = "cuda"
WIDTHS = (2, 3, 4, 8, 16)
EPS = 1e-6
# hidden, q width, k/v width, FFN width
MODELS = {"llama2-13b": (5120, 5120, 5120, 13824), "qwen3-32b": (5120, 8192, 1024, 25600)}


def listed():
    """The standing cases."""
    return [
        # One small layer on its own, called eagerly: launches and the host path count.
        {"name": "gemv_2048_b1", "kind": "gemv", "N": 2048, "K": 2048, "B": 3.0, "batch": 1,
         "alloc": True, "scaled": False},
        # An odd layer with activation factors at batch 3: remainders of tiles, steps and groups.
        {"name": "gemv_odd_scaled_b3", "kind": "gemv", "N": 6001, "K": 3001, "B": 3.5, "batch": 3,
         "alloc": False, "scaled": True},
        # Two layers on one input at a wider budget, batch 2 (speculative or paired decoding).
        {"name": "gemv_gate_up_b2", "kind": "group", "N": 13824, "K": 5120, "B": 4.5, "batch": 2,
         "layers": 2},
        # One decoder layer of a batch-1 decode step, as a decode loop replays it.
        {"name": "decode_llama13b_b1", "kind": "step", "model": "llama2-13b", "B": 3.0, "batch": 1,
         "chain": False},
        # The same for four sequences on grouped-query shapes.
        {"name": "decode_qwen32b_b4", "kind": "step", "model": "qwen3-32b", "B": 3.0, "batch": 4,
         "chain": False},
        # A decoder layer as one chained launch.
        {"name": "chain_llama13b_b1", "kind": "step", "model": "llama2-13b", "B": 3.0, "batch": 1,
         "chain": True},
        # A few sequences decoded together, beyond the GEMV's batch.
        {"name": "gemm_m16", "kind": "gemm", "M": 16, "N": 5120, "K": 5120, "B": 3.0,
         "scaled": False},
        # A short prompt or a prefill chunk on the widest layer.
        {"name": "gemm_m96_gate", "kind": "gemm", "M": 96, "N": 13824, "K": 5120, "B": 3.0,
         "scaled": False},
        # Ragged in every dimension, with activation factors.
        {"name": "gemm_odd_scaled_m203", "kind": "gemm", "M": 203, "N": 4099, "K": 2501, "B": 3.5,
         "scaled": True},
        # The prefill sizes of the benchmark.
        {"name": "gemm_m512_down", "kind": "gemm", "M": 512, "N": 5120, "K": 13824, "B": 3.0,
         "scaled": False},
        {"name": "gemm_m2048_gate", "kind": "gemm", "M": 2048, "N": 13824, "K": 5120, "B": 4.5,
         "scaled": False},
        # A long prompt: the largest.
        {"name": "gemm_m8192_gate", "kind": "gemm", "M": 8192, "N": 13824, "K": 5120, "B": 3.0,
         "scaled": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(("gemv", "gemv", "group", "step", "gemm", "gemm", "gemm", "gemm"))
    B = rng.choice((2.5, 3.0, 3.0, 3.5, 4.0, 4.5, 5.0, 6.0))
    if kind == "step":
        return {"kind": "step", "model": rng.choice(sorted(MODELS)), "B": B,
                "batch": rng.randint(1, 4), "chain": rng.random() < 0.25}
    N, K = _log_int(rng, 256, 16384), _log_int(rng, 256, 16384)
    if rng.random() < 0.6:  # most layers are multiples of 64; the others keep their odd sizes
        N, K = max(64, N // 64 * 64), max(64, K // 64 * 64)
    while N * K > 13824 * 5120:
        N = max(64, N // 2)
    scaled = rng.random() < 0.2 and N * K <= 1 << 24
    if kind == "gemv":
        return {"kind": "gemv", "N": N, "K": K, "B": B, "batch": rng.randint(1, 4),
                "alloc": rng.random() < 0.5, "scaled": scaled}
    if kind == "group":
        return {"kind": "group", "N": N, "K": K, "B": B, "batch": rng.randint(1, 4),
                "layers": rng.randint(2, 3)}
    return {"kind": "gemm", "M": _log_int(rng, 1, 8192), "N": N, "K": K, "B": B, "scaled": scaled}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(DEV).manual_seed(int(seed))


def _weights(g, N, K):
    """fp32 weights [N][K] and channel magnitudes [K] on the GPU."""
    W = torch.randn(N, K, generator=g, device=DEV).mul_(0.02)
    n = round(0.01 * K)
    W[:, torch.randperm(K, generator=g, device=DEV)[:n]] *= 10.0
    m = torch.exp(torch.randn(K, generator=g, device=DEV))
    m[torch.randperm(K, generator=g, device=DEV)[:n]] *= 20.0
    return W, m


def _x(g, m, rows):
    return (m * torch.randn(rows, m.numel(), generator=g, device=DEV)).to(torch.bfloat16)


def _host(W, m, B, scaled=False):
    return polyq.HostLayer.pack(W.cpu().numpy(), m.cpu().numpy(), B, act_scaling=scaled)


def _step_layers(case):
    """(name, N, K) of a decoder layer's linears."""
    h, q, kv, f = MODELS[case["model"]]
    return [("q", q, h), ("k", kv, h), ("v", kv, h), ("o", h, q), ("gate", f, h), ("up", f, h),
            ("down", h, f)]


def _merged(case):
    """Whether attention hands v on as it stands (as many k/v as query channels)."""
    _, q, kv, _ = MODELS[case["model"]]
    return q == kv


def _step_inputs(case, seed):
    """The weights (fp32, GPU) and magnitudes by name, the stream s0 [batch][hidden] and, for
    grouped queries, the attention kernel's output [batch][q width].  q, k, v share their input's
    magnitudes, and so do gate and up."""
    g = _gen(seed)
    layers = {n: _weights(g, N, K) for n, N, K in _step_layers(case)}
    for a, b in (("k", "q"), ("v", "q"), ("up", "gate")):
        layers[a] = (layers[a][0], layers[b][1])
    s0 = torch.randn(case["batch"], MODELS[case["model"]][0], generator=g, device=DEV)
    att = None if _merged(case) else _x(g, layers["o"][1], case["batch"]).float()
    return layers, s0, att


def _prepare_step(case, seed):
    layers, s0, att = _step_inputs(case, seed)
    batch, merged = case["batch"], att is None
    hidden, qd, kv, ffn = MODELS[case["model"]]
    hosts = {n: _host(W, m, case["B"]) for n, (W, m) in layers.items()}
    # merges: gate and up emit in down's order and, where attention at position 0 over one key
    # returns v, v in o's
    p_d = hosts["down"].export()["perm"]
    hosts["gate"].permute_rows(p_d)
    hosts["up"].permute_rows(p_d)
    if merged:
        hosts["v"].permute_rows(hosts["o"].export()["perm"])
    dev = {n: polyq.DeviceLayer(hosts[n], DEV, identity_gather=n == "down" or (n == "o" and merged))
           for n in hosts}
    y = {n: torch.empty(batch, w, device=DEV)
         for n, w in (("q", qd), ("k", kv), ("v", kv), ("s1", hidden), ("gate", ffn), ("up", ffn),
                      ("s2", hidden))}
    # the four calls of the layer: layers, input kind, inputs, outputs, residuals
    calls = [(["q", "k", "v"], polyq.X_RMSNORM, s0, None, ["q", "k", "v"], None),
             (["o"], polyq.X_F32, y["v"] if merged else att, None, ["s1"], [s0]),
             (["gate", "up"], polyq.X_RMSNORM, y["s1"], None, ["gate", "up"], None),
             (["down"], polyq.X_SILU_MUL, y["gate"], y["up"], ["s2"], [y["s1"]])]
    st = {"kind": "step", "dev": dev, "s0": s0, "att": att, "y": y}
    if case["chain"]:
        st["chain"] = polyq.GemvChain(
            [dict(layers=[dev[n] for n in names], kind=kind, a=a, b=b, eps=EPS,
                  ys=[y[n] for n in outs], residuals=res)
             for names, kind, a, b, outs, res in calls], batch)
        st["step"] = st["chain"].run
        return st
    st["ws"] = ws = torch.zeros(
        max(polyq.gemv_group_workspace_bytes([dev[n] for n in c[0]], batch) for c in calls),
        dtype=torch.uint8, device=DEV)

    def layer_calls():
        for names, kind, a, b, outs, res in calls:
            polyq.linear_gemv_input([dev[n] for n in names], kind, a, b=b, eps=EPS,
                                    ys=[y[n] for n in outs], residuals=res, workspace=ws)

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        layer_calls()
    torch.cuda.current_stream().wait_stream(side)
    st["graph"] = torch.cuda.CUDAGraph()
    with torch.cuda.graph(st["graph"]):
        layer_calls()
    st["step"] = st["graph"].replay
    return st


def prepare(case, seed):
    """Packed layers on the GPU, inputs, outputs and workspaces of a case."""
    kind = case["kind"]
    if kind == "step":
        return _prepare_step(case, seed)
    g = _gen(seed)
    N, K = case["N"], case["K"]
    if kind == "gemm":
        W, m = _weights(g, N, K)
        X = _x(g, m, case["M"])
        L = polyq.DeviceLayer(_host(W, m, case["B"], case["scaled"]), DEV)
        return {"kind": kind, "L": L, "X": X, "Y": torch.empty(case["M"], N, device=DEV),
                "ws": torch.zeros(polyq.gemm_workspace_bytes(L, case["M"]), dtype=torch.uint8,
                                  device=DEV)}
    batch = case["batch"]
    if kind == "gemv":
        W, m = _weights(g, N, K)
        x = _x(g, m, batch)
        L = polyq.DeviceLayer(_host(W, m, case["B"], case["scaled"]), DEV)
        res = torch.randn(batch, N, generator=g, device=DEV)
        ws = None
        if case["alloc"]:
            ws = torch.zeros(polyq.gemv_workspace_bytes(L, batch), dtype=torch.uint8, device=DEV)
        return {"kind": kind, "L": L, "x": x, "res": res, "y": torch.empty(batch, N, device=DEV),
                "ws": ws}
    # several layers on one input
    Ls, m0 = [], None
    for _ in range(case["layers"]):
        W, m = _weights(g, N, K)
        m0 = m if m0 is None else m0
        Ls.append(polyq.DeviceLayer(_host(W, m0, case["B"]), DEV))
    x = _x(g, m0, batch)
    return {"kind": kind, "L": Ls, "x": x,
            "ys": [torch.empty(batch, N, device=DEV) for _ in Ls],
            "ws": torch.zeros(polyq.gemv_group_workspace_bytes(Ls, batch), dtype=torch.uint8,
                              device=DEV)}


def run(st):
    """One pass; the outputs are the state's own buffers."""
    kind = st["kind"]
    if kind == "gemm":
        return polyq.linear_gemm(st["L"], st["X"], Y=st["Y"], workspace=st["ws"])
    if kind == "gemv":
        if st["ws"] is None:
            return polyq.linear_gemv_noalloc(st["L"], st["x"], st["y"], residual=st["res"])
        return polyq.linear_gemv(st["L"], st["x"], y=st["y"], residual=st["res"],
                                 workspace=st["ws"])
    if kind == "group":
        return polyq.linear_gemv_group(st["L"], [st["x"]] * len(st["L"]), ys=st["ys"],
                                       workspace=st["ws"])
    st["step"]()
    return st["y"]


# ---------------------------------------------------------------------------
# work and tolerance
# ---------------------------------------------------------------------------
def _layer_bytes(N, K, B):
    return N * K * B / 8 + N * 4.0 * math.ceil(K / 64)


def work(case):
    """Packed codes and scale/zero entries once, the gather indices (and factors), activations in
    and results out once; two operations per weight and row."""
    kind = case["kind"]
    if kind == "step":
        b = case["batch"]
        h, q, kv, f = MODELS[case["model"]]
        shapes = _step_layers(case)
        nk = sum(N * K for _, N, K in shapes)
        by = sum(_layer_bytes(N, K, case["B"]) for _, N, K in shapes)
        # s0, s1, attention, gate, up read; q, k, v, s1, gate, up, s2 written; q, k, v and gate,
        # up gather (as does o where v is not merged into its order)
        by += 4.0 * b * (2 * h + q + 2 * f) + 4.0 * b * (q + 2 * kv + 2 * f + 2 * h)
        by += 4.0 * (5 * h + (0 if _merged(case) else q))
        return {"bytes": by, "flops": 2.0 * b * nk}
    N, K = case["N"], case["K"]
    rows = case["M"] if kind == "gemm" else case["batch"]
    n = case.get("layers", 1)
    by = n * (_layer_bytes(N, K, case["B"]) + 4.0 * rows * N + 4.0 * K) + 2.0 * rows * K
    if case.get("scaled"):
        by += 4.0 * K
    if kind == "gemv":
        by += 4.0 * rows * N  # the residual
    return {"bytes": by, "flops": 2.0 * n * rows * N * K}


def tolerance(case):
    """Four times what the path measures against ``exact`` (GEMV: fp16 copies of the bf16
    activations, exact codes, fp32 sums; GEMM: weights rounded once to fp16).  A decode step rounds
    activations to bf16 between its calls, so a last bit of one call moves later ones."""
    if case["kind"] == "step":
        return {"rel": 8e-3}
    return {"rel": 1.2e-3 if case["kind"] == "gemm" else 4e-4}


# ---------------------------------------------------------------------------
# the result in 64 bits
# ---------------------------------------------------------------------------
def _fp16(v):
    """Nearest fp16 value (ties to even) of non-negative float64 values, as float64."""
    _, e = torch.frexp(v)
    q = torch.exp2((e.to(torch.float64) - 11.0).clamp_min(-24.0))
    return torch.round(v / q) * q


def _allocate(W, m, B):
    """Widths by waterfilling: gain per bit of (m ||W_k|| / (2^b - 1))^2, E_16 = 0."""
    K = W.shape[1]
    sal = (m.double() * torch.sqrt((W.double() ** 2).sum(0))).cpu().numpy()
    bits = np.full(K, 2)
    left = int(math.floor(B * K + 0.5)) - 2 * K
    err = lambda k, b: 0.0 if b == 16 else (sal[k] / (2 ** b - 1)) ** 2  # noqa: E731

    def rung(k):
        b = int(bits[k])
        b2 = WIDTHS[WIDTHS.index(b) + 1]
        return (-(err(k, b) - err(k, b2)) / (b2 - b), k, b2)

    heap = [rung(k) for k in range(K)]
    heapq.heapify(heap)
    while heap and left > 0:
        _, k, b2 = heapq.heappop(heap)
        if b2 - bits[k] > left:
            continue
        left -= b2 - int(bits[k])
        bits[k] = b2
        if b2 < 16:
            heapq.heappush(heap, rung(k))
    return bits


def _quantised(V, b):
    """Dequantised values of V (float64 [N][n]) with groups of 64 columns at b bits."""
    out = torch.empty_like(V)
    n = V.shape[1]
    full = n // 64 * 64
    for part, cols in ((V[:, :full], slice(0, full)), (V[:, full:], slice(full, n))):
        if part.shape[1] == 0:
            continue
        G = part.reshape(V.shape[0], -1, min(64, part.shape[1]))
        lo, hi = G.amin(2, keepdim=True), G.amax(2, keepdim=True)
        s = _fp16((hi - lo) / (2 ** b - 1))
        alt = _fp16(torch.maximum(torch.maximum(lo.abs(), hi.abs()),
                                  torch.full_like(lo, 2.0 ** -14)))
        s = torch.where(s == 0, alt, s)
        z = torch.round(-lo / s).clamp_(0, 2 ** b - 1)
        q = (torch.round(G / s) + z).clamp_(0, 2 ** b - 1)
        out[:, cols] = ((q - z) * s).reshape(part.shape)
    return out


def _dense(W, m, bits, scaled=False):
    """The layer's effective weights in original channel order (float64)."""
    out = torch.empty(W.shape, dtype=torch.float64, device=W.device)
    for b in WIDTHS:
        idx = np.nonzero(bits == b)[0]
        if idx.size == 0:
            continue
        ix = torch.from_numpy(idx).to(W.device)
        V = W[:, ix].double()
        if b == 16:
            out[:, ix] = torch.sign(V) * _fp16(V.abs())
            continue
        if not scaled:
            out[:, ix] = _quantised(V, b)
            continue
        a = m.double().cpu().numpy()
        met = a[idx] / (float(np.cumsum(a)[-1]) / a.size)
        a2 = torch.from_numpy(a[idx] ** 2).to(W.device)
        best = None
        for j in range(11):
            t = torch.from_numpy((met ** -(j / 10)).astype(np.float32).astype(np.float64))
            t = t.to(W.device)
            Q = _quantised(V / t, b) * t
            e = float((((Q - V) ** 2).sum(0) * a2).mean())
            if best is None or e < best[0]:
                best = (e, Q)
        out[:, ix] = best[1]
    return out


def _bf16(v):
    return v.float().to(torch.bfloat16).double()


def _rms(s):
    return _bf16(s / torch.sqrt((s * s).mean(1, keepdim=True) + EPS))


def exact(case, seed):
    """What run() returns, in 64 bits, from the definition of the layer."""
    kind = case["kind"]
    if kind == "step":
        layers, s0, att = _step_inputs(case, seed)
        D, order = {}, {}
        for n in list(layers):
            W, m = layers.pop(n)
            bits = _allocate(W, m, case["B"])
            D[n] = _dense(W, m, bits)
            order[n] = torch.from_numpy(np.argsort(bits, kind="stable")).to(DEV)
        s0 = s0.double()
        h = _rms(s0)
        q, k, v = (h @ D[n].T for n in ("q", "k", "v"))
        s1 = s0 + _bf16(v if att is None else att) @ D["o"].T
        h = _rms(s1)
        g, u = h @ D["gate"].T, h @ D["up"].T
        s2 = s1 + _bf16(g / (1 + torch.exp(-g)) * u) @ D["down"].T
        if att is None:  # v is emitted in o's order, gate and up in down's
            v = v[:, order["o"]]
        return {"q": q, "k": k, "v": v, "s1": s1, "gate": g[:, order["down"]],
                "up": u[:, order["down"]], "s2": s2}
    g = _gen(seed)
    N, K = case["N"], case["K"]
    if kind == "group":
        ys, m0 = [], None
        for _ in range(case["layers"]):
            W, m = _weights(g, N, K)
            m0 = m if m0 is None else m0
            ys.append(_dense(W, m0, _allocate(W, m0, case["B"])))
        x = _x(g, m0, case["batch"]).double()
        return [x @ d.T for d in ys]
    W, m = _weights(g, N, K)
    x = _x(g, m, case["M"] if kind == "gemm" else case["batch"]).double()
    y = x @ _dense(W, m, _allocate(W, m, case["B"]), case["scaled"]).T
    if kind == "gemv":
        y = y + torch.randn(case["batch"], N, generator=g, device=DEV).double()
    return y
