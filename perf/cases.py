"""The work whose speed is watched: attention layers and linear layers as a training program runs them.

A case names one call, or the forward and backward pair of a training step, through the public entry points of
``paper_2606_10415_b200.binding``: the attention forward, its backward, both on fp16 or bfloat16 tensors in
``[B,H,S,D]``, ``[B,S,H,D]`` or fused-projection layouts, the call on host buffers, and the linear-layer product.
Shapes come from ``workloads.py``, from the tests, and from the weight shapes of the linear-layer profile that the
benchmark times.  The store of probability tiles (``lt_attn_save_p``) is left out: it exists to be compared with.

Values: the named layers take the distributions ``workloads.py`` gives them.  Other attention cases take unit normal
Q, K, V (scores of order one after the 1/sqrt(D) scale, as normalised activations give) and upstream gradients of
1e-2.  Linear layers take unit normal activations and weights of variance 1/K.
"""
from __future__ import annotations

import math

import torch

from paper_2606_10415_b200 import binding as lt
from paper_2606_10415_b200 import workloads

_DTYPES = {"fp16": torch.float16, "bf16": torch.bfloat16}


def _attn(name, op, B, Hq, Hkv, S, D, causal=True, dtype="fp16", layout="bhsd", std=1.0, do_std=1e-2):
    case = {"op": op, "B": B, "Hq": Hq, "Hkv": Hkv, "S": S, "D": D, "causal": causal, "dtype": dtype,
            "layout": layout, "std": std, "do_std": do_std}
    return {"name": name, **case} if name else case


def _workload(name, op, key):
    c = workloads.ALL_CONFIGS[key]
    return _attn(name, op, c.B, c.Hq, c.Hkv, c.S, c.D, c.causal, std=c.qkv_std, do_std=c.do_std)


def _gemm(name, M, N, K, dtype="fp16"):
    case = {"op": "gemm", "M": M, "N": N, "K": K, "dtype": dtype}
    return {"name": name, **case} if name else case


def listed():
    return [
        # one head tile: the smallest backward a program issues, where launches and host work are the cost
        _workload("bwd_tiny", "bwd", "tiny"),
        # a micro-batch of short sequences of an odd length in the [B,S,H,D] layout of most training stacks
        _attn("step_short_bf16", "step", 8, 16, 16, 333, 64, dtype="bf16", layout="bshd"),
        # one 7B layer at a short context: forward and backward of a training step
        _workload("step_7b_s1024", "step", "llama2_7b_s1024"),
        # one 7B layer at its full context, the two directions by themselves (activation recomputation runs the
        # forward alone; the backward is the benchmark's metric)
        _workload("fwd_7b", "fwd", "llama2_7b"),
        _workload("bwd_7b", "bwd", "llama2_7b"),
        # grouped queries with few key/value heads: more multiprocessors than work items
        _workload("bwd_32b_gqa_s2048", "bwd", "qwen25_32b_gqa_s2048"),
        # a length that is no multiple of the tiles, bfloat16, read from and written to a fused QKV projection
        _attn("step_ragged_fused_bf16", "step", 1, 32, 32, 3000, 128, dtype="bf16", layout="fused"),
        # bidirectional attention with 64-element heads and an odd length
        _attn("step_unmasked_d64", "step", 4, 16, 16, 1531, 64, causal=False),
        # the largest layer: grouped queries, two sequences
        _workload("step_70b_gqa", "step", "llama2_70b_gqa"),
        # a linear layer of the 7B model over 2048 tokens, and one over the few rows of a short sequence
        _gemm("gemm_2048x11008x4096", 2048, 11008, 4096),
        _gemm("gemm_rows77_bf16", 77, 4096, 4096, dtype="bf16"),
        # the same 7B layer with all tensors in pinned host memory (an offloaded layer)
        _workload("host_7b", "host", "llama2_7b"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    limit = work(_workload(None, "step", "llama2_70b_gqa"))
    while True:
        kind = rng.choice(["fwd", "bwd", "step", "step", "gemm", "host"])
        if kind == "gemm":
            case = _gemm(None, _log_int(rng, 1, 8192), _log_int(rng, 128, 11008), 8 * _log_int(rng, 16, 1376),
                         rng.choice(["fp16", "bf16"]))
            if rng.random() < 0.7:
                case["N"] = max(128, case["N"] // 64 * 64)
        else:
            D = rng.choice([64, 128, 128])
            S = _log_int(rng, 48, 8192)
            if rng.random() < 0.5:
                S = max(64, S // 64 * 64)
            Hkv = rng.choice([1, 2, 4, 8, 16, 32, 40])
            G = rng.choice([1, 1, 2, 4, 5, 8])
            dtype = "fp16" if kind == "host" else rng.choice(["fp16", "bf16"])
            layout = "bhsd" if kind == "host" else rng.choice(["bhsd", "bshd", "fused"])
            case = _attn(None, kind, rng.choice([1, 1, 2, 4, 8]), Hkv * G, Hkv, S, D, rng.random() < 0.75, dtype,
                         layout)
            if case["Hq"] > 64:
                continue
            if kind == "host" and work(case)["bytes"] > 5.0e8:  # copies of a few hundred MB, not of gigabytes
                continue
        w = work(case)
        if w["flops"] <= limit["flops"] and w["bytes"] <= limit["bytes"]:
            return case


def _place(t, layout):
    """``t`` ([B,H,S,D], contiguous) as a view of the same shape in the given memory layout."""
    return t if layout == "bhsd" else t.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)


def _fused_views(buf, Hq, Hkv, D):
    """Q, K, V as [B,H,S,D] views of a [B,S,(Hq+2Hkv)*D] projection output."""
    B, S, _ = buf.shape
    heads = buf.view(B, S, Hq + 2 * Hkv, D).permute(0, 2, 1, 3)
    return heads[:, :Hq], heads[:, Hq:Hq + Hkv], heads[:, Hq + Hkv:]


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    dtype = _DTYPES[case["dtype"]]

    def randn(shape, std):
        return (torch.randn(shape, generator=gen, dtype=torch.float32, device="cuda") * std).to(dtype)

    if case["op"] == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"op": "gemm", "A": randn((M, K), 1.0), "W": randn((N, K), K ** -0.5),
                "C": torch.empty((M, N), dtype=dtype, device="cuda"),
                "ws": lt.alloc_workspace(lt.lt_gemm_f16_workspace_bytes())}

    B, Hq, Hkv, S, D = (case[k] for k in ("B", "Hq", "Hkv", "S", "D"))
    dims = (B, Hq, Hkv, S, D)
    scale = float(D) ** -0.5
    st = {"op": case["op"], "dtype": case["dtype"], "causal": case["causal"], "scale": scale,
          "strided": case["layout"] != "bhsd"}
    if case["layout"] == "fused":
        qkv = randn((B, S, (Hq + 2 * Hkv) * D), case["std"])
        st["Q"], st["K"], st["V"] = _fused_views(qkv, Hq, Hkv, D)
        st["dO"] = _place(randn((B, Hq, S, D), case["do_std"]), "bshd")
        st["dqkv"] = torch.empty_like(qkv)
        st["dQ"], st["dK"], st["dV"] = _fused_views(st["dqkv"], Hq, Hkv, D)
        st["O"] = _place(torch.empty((B, Hq, S, D), dtype=dtype, device="cuda"), "bshd")
    else:
        for name, H in (("Q", Hq), ("K", Hkv), ("V", Hkv)):
            st[name] = _place(randn((B, H, S, D), case["std"]), case["layout"])
        st["dO"] = _place(randn((B, Hq, S, D), case["do_std"]), case["layout"])
        for name, src in (("O", "Q"), ("dQ", "Q"), ("dK", "K"), ("dV", "V")):
            st[name] = torch.empty_like(st[src])  # keeps the strides
    st["LSE"] = torch.empty((B, Hq, S), dtype=torch.float32, device="cuda")
    if case["op"] == "host":
        for name in ("Q", "K", "V", "dO", "O", "dQ", "dK", "dV", "LSE"):
            t = st[name]
            host = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
            st[name] = host.copy_(t) if name in ("Q", "K", "V", "dO") else host
        st["arena"] = lt.alloc_workspace(lt.lt_attn_host_arena_bytes(*dims))
        return st
    st["fws"] = lt.alloc_workspace(lt.lt_attn_fwd_workspace_bytes(*dims))
    if case["op"] != "fwd":
        st["ws"] = lt.alloc_workspace(lt.lt_attn_bwd_workspace_bytes(*dims))
    if case["op"] == "bwd":
        _forward(st)  # the state a backward starts from: the forward's output and row log-sum-exp
    return st


def _forward(st):
    fn = lt.lt_attn_fwd_bf16 if st["dtype"] == "bf16" else lt.lt_attn_fwd_strided if st["strided"] else lt.lt_attn_fwd
    fn(st["Q"], st["K"], st["V"], st["O"], st["LSE"], st["causal"], st["scale"], st["fws"])


def _backward(st):
    fn = lt.lt_attn_bwd_bf16 if st["dtype"] == "bf16" else lt.lt_attn_bwd_strided if st["strided"] else lt.lt_attn_bwd
    fn(st["Q"], st["K"], st["V"], st["O"], st["dO"], st["LSE"], st["dQ"], st["dK"], st["dV"], st["causal"],
       st["scale"], st["ws"])


def run(state):
    st = state
    if st["op"] == "gemm":
        lt.lt_gemm_f16(st["A"], st["W"], st["C"], st["ws"])
        return st["C"]
    if st["op"] == "host":
        lt.lt_attn_fwd_bwd_host(st["Q"], st["K"], st["V"], st["dO"], st["O"], st["LSE"], st["dQ"], st["dK"],
                                st["dV"], st["causal"], st["scale"], st["arena"])
    if st["op"] in ("fwd", "step"):
        _forward(st)
    if st["op"] in ("bwd", "step"):
        _backward(st)
    out = []
    if st["op"] != "bwd":
        out += [st["O"], st["LSE"]]
    if st["op"] != "fwd":
        out += [st["dqkv"]] if "dqkv" in st else [st["dQ"], st["dK"], st["dV"]]
    return out


def work(case):
    if case["op"] == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 2 * (M * K + N * K + M * N), "flops": 2 * M * N * K}
    B, Hq, Hkv, S, D = (case[k] for k in ("B", "Hq", "Hkv", "S", "D"))
    q, kv, lse = 2 * B * Hq * S * D, 2 * B * Hkv * S * D, 4 * B * Hq * S
    pairs = B * Hq * (S * (S + 1) // 2 if case["causal"] else S * S)  # visible (query, key) pairs
    fwd = {"bytes": 2 * q + 2 * kv + lse, "flops": 4 * pairs * D}      # Q, K, V -> O, LSE; two products
    bwd = {"bytes": 4 * q + 4 * kv + lse, "flops": 10 * pairs * D}     # Q, K, V, O, dO, LSE -> dQ, dK, dV; five
    if case["op"] == "fwd":
        return fwd
    if case["op"] == "bwd":
        return bwd
    # both: Q, K, V, dO -> O, LSE, dQ, dK, dV
    return {"bytes": 4 * q + 4 * kv + lse, "flops": fwd["flops"] + bwd["flops"]}


# Four times the largest error against the same computation in 64 bits, measured on the listed cases and sixteen drawn
# ones: relative 2-norm, and largest difference over the larger of the value and the result's root mean square.
#   forward       fp16 2.9e-4 / 5.4e-3    bf16 2.3e-3 / 2.2e-2   (rounding of P and of O)
#   with backward fp16 5.4e-4 / 1.4e-2    bf16 2.8e-3 / 7.2e-2   (dS and P rounded before the products)
#   linear layer  fp16 2.1e-4 / 5.0e-4    bf16 1.7e-3 / 3.9e-3   (rounding of the result)
_TOLERANCE = {
    ("fwd", "fp16"): (1.2e-3, 2.2e-2), ("fwd", "bf16"): (9.2e-3, 8.8e-2),
    ("bwd", "fp16"): (2.2e-3, 5.6e-2), ("bwd", "bf16"): (1.1e-2, 2.9e-1),
    ("gemm", "fp16"): (8.4e-4, 2.0e-3), ("gemm", "bf16"): (6.8e-3, 1.6e-2),
}


def tolerance(case):
    op = case["op"] if case["op"] in ("fwd", "gemm") else "bwd"
    rel, most = _TOLERANCE[op, case["dtype"]]
    return {"rel": rel, "max": most}
