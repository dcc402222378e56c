"""Timed cases of the BitDelta product and its compress step, through the package's public entry points.

A case is one call (or, for "layer", one captured decode step of four dependent calls) as a serving program makes it:
weights, packed signs, scales, workspace and output buffers are held by the program, activations are new.  Sizes are
those of `synth.WORKLOADS`, of the tests and of `bench.py`, and odd ones between them.  Inputs follow the recipe of
`synth`: X ~ N(0, 1), W_base ~ N(0, 0.02), uniform sign words, alpha ~ U(0.001, 0.01).
"""
from __future__ import annotations

import math

import torch

import paper_2609_36800_b200 as bd

MAX_BYTES = 362.0e6      # work of the largest listed cases (many_tenant_down; prefill): no drawn case exceeds either
MAX_FLOPS = 138.0e9
MAX_RAGGED_FLOPS = 4.2e9  # ... and the largest listed case whose K is not a multiple of 128


def gemm_case(name, B, m, K, N, dtype="bf16", bias=False, act="none"):
    return {"name": name, "op": "gemm", "B": B, "m": m, "K": K, "N": N, "dtype": dtype, "bias": bias, "act": act}


def listed():
    return [
        # smallest call: one tenant, a handful of tokens, a small projection (launch and host latency)
        gemm_case("tiny", 1, 16, 512, 512),
        # one tenant decoding one token on an attention projection
        gemm_case("one_token", 1, 1, 4096, 4096),
        # the headline: eight tenants, one token each, attention projection
        gemm_case("decode_attn", 8, 1, 4096, 4096),
        # sixteen tenants, four tokens each (speculative decoding), MLP up projection
        gemm_case("decode_mlp_up", 16, 4, 4096, 11008),
        # the same step as a gated MLP in fp16: gate and up rows interleaved, bias, fused gate
        gemm_case("decode_gate_fp16", 16, 4, 4096, 11008, dtype="fp16", bias=True, act="silu_gate"),
        # many tenants, eight tokens each, MLP down projection (long K): the largest in bytes
        gemm_case("many_tenant_down", 32, 8, 14336, 4096),
        # a decode step of one layer (attention in, attention out, gated MLP up, MLP down) as one CUDA graph, the way a
        # serving loop replays it
        {"name": "decode_layer", "op": "layer", "B": 8, "m": 1, "K": 4096, "N": 11008},
        # short chunks of tokens per tenant, an odd count (chunked prefill mixed with decode)
        gemm_case("chunk_mid", 8, 37, 4096, 4096),
        # prefill of four prompts: the largest in operations
        gemm_case("prefill", 4, 512, 4096, 4096),
        # ragged prompts through the gated MLP in fp16
        gemm_case("prefill_gate_fp16", 2, 300, 4096, 11008, dtype="fp16", act="silu_gate"),
        # sizes that divide nothing: K a multiple of 32 only, odd N
        gemm_case("ragged", 6, 40, 2080, 1999),
        # loading tenants: signs and scales from fine-tuned weights
        {"name": "compress", "op": "compress", "B": 8, "K": 4096, "N": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_once(rng):
    kind = rng.choice(("decode", "decode", "decode", "mid", "prefill", "prefill", "layer", "compress"))
    if kind == "compress":
        return {"op": "compress", "B": _log_int(rng, 1, 16), "K": 32 * _log_int(rng, 16, 448), "N": _log_int(rng, 128, 11008)}
    if kind == "layer":
        return {"op": "layer", "B": _log_int(rng, 1, 16), "m": rng.choice((1, 1, 2, 4)), "K": 128 * _log_int(rng, 8, 40),
                "N": 128 * _log_int(rng, 16, 90)}
    m = _log_int(rng, 1, 16) if kind == "decode" else _log_int(rng, 17, 64) if kind == "mid" else _log_int(rng, 65, 1024)
    K = 32 * _log_int(rng, 16, 448) if rng.random() < 0.2 else 128 * _log_int(rng, 4, 112)
    N = 2 * _log_int(rng, 256, 5504) - (1 if rng.random() < 0.2 else 0)
    act = rng.choice(("none", "none", "none", "silu", "silu_gate"))
    if act == "silu_gate" and N % 2:
        act = "silu"
    return {"op": "gemm", "B": _log_int(rng, 1, 32), "m": m, "K": K, "N": N, "dtype": rng.choice(("bf16", "bf16", "bf16", "fp16")),
            "bias": rng.random() < 0.25, "act": act}


def draw(rng):
    while True:
        c = _draw_once(rng)
        w = work(c)
        if w["bytes"] <= MAX_BYTES and w["flops"] <= (MAX_RAGGED_FLOPS if c["K"] % 128 and c["op"] == "gemm" else MAX_FLOPS):
            return c


def _gemm_work(B, m, K, N, bias=False, act="none"):
    n_out = N // 2 if act == "silu_gate" else N
    return {"bytes": 2 * B * m * K + 2 * N * K + B * N * K // 8 + 4 * B + (2 * N if bias else 0) + 2 * B * m * n_out,
            "flops": 4 * B * m * N * K}


def _layer_products(case):
    """(K, N, act) of the four dependent products of one layer of hidden size K and MLP size N."""
    h, f = case["K"], case["N"]
    return ((h, h, "none"), (h, h, "none"), (h, 2 * f, "silu_gate"), (f, h, "none"))


def work(case):
    B, K, N = case["B"], case["K"], case["N"]
    if case["op"] == "compress":
        return {"bytes": 2 * B * N * K + 2 * N * K + B * N * K // 8 + 4 * B, "flops": 3 * B * N * K}
    if case["op"] == "layer":
        parts = [_gemm_work(B, case["m"], k, n, act=act) for k, n, act in _layer_products(case)]
        return {key: sum(p[key] for p in parts) for key in ("bytes", "flops")}
    return _gemm_work(B, case["m"], K, N, case["bias"], case["act"])


def tolerance(case):
    # Four times the distance of each product from the same sums in 64 bits, over the listed cases and fourteen drawn ones:
    # bf16 1.67e-3 (3.9e-3 at most), the rounding of the result; fp16 2.1e-4 (5.0e-4), which also holds the delta's e5m2
    # pieces; the layer's last output, four roundings and a gate in a row, 4.1e-3 (3.6e-2); alpha 3.5e-8.
    if case["op"] == "compress":
        return {"rel": 2e-7, "max": 2e-7, "differ": 0.0}   # the sign words are exact
    if case["op"] == "layer":
        return {"rel": 1.6e-2, "max": 0.15}
    if case["dtype"] == "fp16":
        return {"rel": 9e-4, "max": 2e-3}
    return {"rel": 6.7e-3, "max": 1.6e-2}


def _weights(g, B, N, K, dtype):
    W = (torch.randn(N, K, device="cuda", generator=g) * 0.02).to(dtype)
    bits = torch.randint(-2**31, 2**31, (B, N, K // 32), device="cuda", dtype=torch.int32, generator=g)
    alpha = torch.rand(B, device="cuda", generator=g) * 0.009 + 0.001
    return W, bits, alpha


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    B, K, N = case["B"], case["K"], case["N"]
    if case["op"] == "compress":
        base = (torch.randn(N, K, device="cuda", generator=g) * 0.02).to(torch.bfloat16)
        fine = torch.empty(B, N, K, dtype=torch.bfloat16, device="cuda")
        for b in range(B):
            delta = torch.randn(N, K, device="cuda", generator=g) * 0.004
            delta *= torch.rand(N, K, device="cuda", generator=g) >= 0.01   # 1 % of the weights were not changed
            fine[b] = (base + delta).to(torch.bfloat16)
        return {"fine": fine, "base": base, "bits": torch.empty(B, N, K // 32, dtype=torch.int32, device="cuda"),
                "alpha": torch.empty(B, dtype=torch.float32, device="cuda")}
    m = case["m"]
    if case["op"] == "layer":
        x = torch.randn(B, m, K, device="cuda", generator=g).to(torch.bfloat16)
        parts = []
        for k, n, act in _layer_products(case):
            W, bits, alpha = _weights(g, B, n, k, torch.bfloat16)
            out = torch.empty(B, m, n // 2 if act == "silu_gate" else n, dtype=torch.bfloat16, device="cuda")
            parts.append((W, bits, alpha, out, bd.make_workspace(B, m, n, k), act))

        def step():
            y = x
            for W, bits, alpha, out, ws, act in parts:
                y = bd.gemm(y, W, bits, alpha, out=out, workspace=ws, act=act)

        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            step()
        torch.cuda.current_stream().wait_stream(side)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            step()
        return {"graph": graph, "x": x, "parts": parts, "outs": [p[3] for p in parts]}
    dtype = torch.float16 if case["dtype"] == "fp16" else torch.bfloat16
    W, bits, alpha = _weights(g, B, N, K, dtype)
    return {"X": torch.randn(B, m, K, device="cuda", generator=g).to(dtype), "W": W, "bits": bits, "alpha": alpha,
            "bias": (torch.randn(N, device="cuda", generator=g) * 0.5).to(dtype) if case["bias"] else None, "act": case["act"],
            "out": torch.empty(B, m, N // 2 if case["act"] == "silu_gate" else N, dtype=dtype, device="cuda"),
            "ws": bd.make_workspace(B, m, N, K)}


def run(s):
    if "fine" in s:
        return bd.compress(s["fine"], s["base"], bits=s["bits"], alpha=s["alpha"])
    if "graph" in s:
        s["graph"].replay()
        return s["outs"]
    return bd.gemm(s["X"], s["W"], s["bits"], s["alpha"], out=s["out"], workspace=s["ws"], bias=s["bias"], act=s["act"])


def _signs64(bits, b):
    """+1 / -1 of tenant b as [N, K] in 64 bits."""
    j = torch.arange(32, device="cuda", dtype=torch.int32)
    return (((bits[b].unsqueeze(-1) >> j) & 1).to(torch.float64) * 2 - 1).reshape(bits.shape[1], -1)


def _product64(X, W, bits, alpha, bias, act):
    base = W.double()
    Y = []
    for b in range(X.shape[0]):
        x = X[b].double()
        z = x @ base.t() + alpha[b].double() * (x @ _signs64(bits, b).t())
        if bias is not None:
            z = z + bias.double()
        if act == "silu":
            z = z * torch.sigmoid(z)
        elif act == "silu_gate":
            z = z[:, 0::2] * torch.sigmoid(z[:, 0::2]) * z[:, 1::2]
        Y.append(z)
    return torch.stack(Y)


def exact(case, seed):
    s = prepare(case, seed)
    if case["op"] == "compress":
        base, bits, alpha = s["base"].double(), [], []
        j = torch.arange(32, device="cuda", dtype=torch.int64)
        for fine in s["fine"]:
            delta = fine.double() - base
            word = ((delta > 0).reshape(case["N"], -1, 32).long() << j).sum(-1)
            bits.append(torch.where(word >= 2**31, word - 2**32, word).to(torch.int32))
            alpha.append(delta.abs().mean())
        return torch.stack(bits), torch.stack(alpha)
    if case["op"] == "layer":
        y, outs = s["x"], []
        for W, bits, alpha, _, _, act in s["parts"]:
            y = _product64(y, W, bits, alpha, None, act)
            outs.append(y)
        return outs
    return _product64(s["X"], s["W"], s["bits"], s["alpha"], s["bias"], s["act"])
