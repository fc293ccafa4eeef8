"""Backward on sequences of one tile (S <= 128), where a call is one or two launches and dQ is written without an
accumulator: the smallest and largest length, lengths around the sixteen-row pieces, several heads and units per CTA,
strided outputs, both head dimensions and types, against the oracle; nothing in the workspace may be expected clear."""
import pytest
import torch

from paper_2606_10415_b200 import workloads
from parity_checks import check_grads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,S,D,launches", [
    (1, 2, 2, 128, 64, 1), (1, 1, 1, 1, 64, 1), (2, 160, 160, 17, 64, 2), (1, 6, 2, 100, 64, 2), (3, 120, 60, 64, 64, 2),
    (1, 2, 2, 128, 128, 1), (1, 1, 1, 1, 128, 1), (2, 150, 150, 31, 128, 1), (3, 99, 33, 127, 128, 1), (1, 4, 2, 96, 128, 3),
])
@pytest.mark.parametrize("dtype,causal", [("fp16", True), ("bf16", False)])
def test_one_tile(oracle, B, Hq, Hkv, S, D, launches, dtype, causal):
    from paper_2606_10415_b200 import binding as lt
    assert lt.lt_attn_bwd_num_launches(B, Hq, Hkv, S, D, causal) == launches
    dt = torch.float16 if dtype == "fp16" else torch.bfloat16
    cfg = workloads.custom(B, Hq, Hkv, S, D, causal, seed=S + Hq)
    Q, K, V, dO = (t.float().to(dt) for t in workloads.make_inputs(cfg))
    Qd, Kd, Vd, dOd = (t.cuda() for t in (Q, K, V, dO))
    O, LSE = torch.empty_like(Qd), torch.empty(Q.shape[:3], dtype=torch.float32, device="cuda")
    # [B,S,H,D] outputs with a guard row behind each sequence
    outs = [torch.full((B, S + 1, H, D), float("nan"), dtype=dt, device="cuda") for H in (Hq, Hkv, Hkv)]
    dQ, dK, dV = (t[:, :S].permute(0, 2, 1, 3) for t in outs)
    dims = (B, Hq, Hkv, S, D)
    ws = lt.alloc_workspace(lt.lt_attn_bwd_workspace_bytes(*dims))
    ws.fill_(0xFF)
    fwd, bwd = (lt.lt_attn_fwd_strided, lt.lt_attn_bwd_strided) if dtype == "fp16" else (lt.lt_attn_fwd_bf16, lt.lt_attn_bwd_bf16)
    fwd(Qd, Kd, Vd, O, LSE, causal, cfg.scale, lt.alloc_workspace(256))
    for _ in range(2):
        bwd(Qd, Kd, Vd, O, dOd, LSE, dQ, dK, dV, causal, cfg.scale, ws)
    assert lt.lt_attn_check_status(ws) == lt.LT_OK, lt.last_cuda_error()
    ref = oracle.attn_bwd(*(t.double().numpy() for t in (Q, K, V, dO)), causal, cfg.scale)
    check_grads((dQ, dK, dV), ref, f"one tile {dims}", dtype=dtype, absolute=False)
    assert all(torch.isnan(t[:, S]).all() for t in outs)
