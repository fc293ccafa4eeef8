"""Groups of query heads split over work items on small problems: one tile and several, parts of unequal size, as many
parts as heads, both head dimensions, types and masks, against the oracle; and the entry points that run with whole
groups because their scratch has no room for the split groups' fp32 sums."""
import pytest
import torch

from paper_2606_10415_b200 import workloads
from parity_checks import check_grads

pytestmark = pytest.mark.gpu


def _forward(lt, cfg, dt=torch.float16):
    host = [t.float().to(dt) for t in workloads.make_inputs(cfg)]
    Q, K, V, dO = (t.cuda() for t in host)
    O, LSE = torch.empty_like(Q), torch.empty(Q.shape[:3], dtype=torch.float32, device="cuda")
    fwd = lt.lt_attn_fwd if dt == torch.float16 else lt.lt_attn_fwd_bf16
    fwd(Q, K, V, O, LSE, cfg.causal, cfg.scale, lt.alloc_workspace(256))
    return host, (Q, K, V, O, dO, LSE), [torch.full_like(t, float("nan")) for t in (Q, K, V)]


@pytest.mark.parametrize("B,Hq,Hkv,S,D,causal,launches", [
    (1, 8, 1, 64, 64, True, 4), (1, 64, 8, 128, 128, True, 4), (2, 8, 1, 200, 64, False, 4), (1, 10, 2, 500, 128, False, 4),
    (1, 5, 1, 129, 128, True, 4), (1, 20, 4, 640, 128, True, 4),   # five heads: parts of unequal size
    (4, 8, 1, 300, 64, True, 4),
    (1, 4, 2, 256, 64, True, 3), (2, 8, 4, 256, 128, False, 3),    # short groups stay whole
])
@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
def test_split_on_small_problems(oracle, B, Hq, Hkv, S, D, causal, launches, dtype):
    from paper_2606_10415_b200 import binding as lt
    assert lt.lt_attn_bwd_num_launches(B, Hq, Hkv, S, D, causal) == launches
    cfg = workloads.custom(B, Hq, Hkv, S, D, causal, seed=S + Hq)
    host, ins, outs = _forward(lt, cfg, torch.float16 if dtype == "fp16" else torch.bfloat16)
    ws = lt.alloc_workspace(lt.lt_attn_bwd_workspace_bytes(B, Hq, Hkv, S, D))
    bwd = lt.lt_attn_bwd if dtype == "fp16" else lt.lt_attn_bwd_bf16
    for _ in range(3):  # back to back on one workspace: the next call's kernels start under the conversions
        ws[:256].fill_(0xFF)
        bwd(*ins, *outs, causal, cfg.scale, ws)
        bwd(*ins, *outs, causal, cfg.scale, ws)
    assert lt.lt_attn_check_status(ws) == lt.LT_OK, lt.last_cuda_error()
    ref = oracle.attn_bwd(*(t.double().numpy() for t in host), causal, cfg.scale)
    check_grads(outs, ref, f"split {cfg}", dtype=dtype, absolute=False)


def test_noalloc_without_room_for_the_sums(oracle):
    from paper_2606_10415_b200 import binding as lt
    cfg = workloads.custom(1, 8, 1, 4096, 128, True, seed=5)
    dims = (cfg.B, cfg.Hq, cfg.Hkv, cfg.S, cfg.D)
    assert lt.lt_attn_bwd_workspace_bytes(*dims) > lt.NOALLOC_MAX_SCRATCH_BYTES
    host, ins, outs = _forward(lt, cfg)
    lt.lt_attn_bwd_noalloc(*ins, *outs, cfg.causal, cfg.scale)
    assert lt.lt_attn_bwd_noalloc_check_status() == lt.LT_OK
    ref = oracle.attn_bwd(*(t.double().numpy() for t in host), cfg.causal, cfg.scale)
    check_grads(outs, ref, "noalloc, whole groups")
