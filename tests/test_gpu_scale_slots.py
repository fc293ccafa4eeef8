"""The power of two that dS carries comes from maxima over the whole call, of which every block of the preprocess
kernel leaves its share in a slot.  A share that went missing would let dS overflow fp16, so one outlying row is placed
where a single block sees it: the last row of dO, of V, or a row in the middle."""
import pytest
import torch

from paper_2606_10415_b200 import workloads
from parity_checks import check_grads

pytestmark = pytest.mark.gpu


# 1 block; 444 blocks of one trip each; more rows than 444 blocks take in one trip; ragged, D = 64
@pytest.mark.parametrize("B,H,S,D", [(1, 1, 3, 64), (2, 111, 128, 128), (3, 75, 128, 128), (1, 3, 200, 64)])
@pytest.mark.parametrize("where", ["dO_last", "V_last", "dO_middle"])
def test_one_outlying_row_sets_the_scale(oracle, B, H, S, D, where):
    from paper_2606_10415_b200 import binding as lt
    cfg = workloads.custom(B, H, H, S, D, False, qkv_std=0.3, do_std=1e-3, seed=H + S)
    Q, K, V, dO = workloads.make_inputs(cfg)
    if where == "dO_last":
        dO[-1, -1, -1] *= 2.0 ** 14
    elif where == "V_last":
        V[-1, -1, -1] *= 2.0 ** 14
    else:
        dO[B // 2, H // 2, S // 2] *= 2.0 ** 14
    Qd, Kd, Vd, dOd = (t.cuda() for t in (Q, K, V, dO))
    O, LSE = torch.empty_like(Qd), torch.empty(Q.shape[:3], dtype=torch.float32, device="cuda")
    dQ, dK, dV = torch.empty_like(Qd), torch.empty_like(Kd), torch.empty_like(Vd)
    dims = (B, H, H, S, D)
    fws = lt.alloc_workspace(lt.lt_attn_fwd_workspace_bytes(*dims))
    ws = lt.alloc_workspace(lt.lt_attn_bwd_workspace_bytes(*dims))
    ws.fill_(0xFF)  # nothing in the workspace may be expected to be clear
    lt.lt_attn_fwd(Qd, Kd, Vd, O, LSE, cfg.causal, cfg.scale, fws)
    lt.lt_attn_bwd(Qd, Kd, Vd, O, dOd, LSE, dQ, dK, dV, cfg.causal, cfg.scale, ws)
    assert lt.lt_attn_check_status(ws) == lt.LT_OK
    # the head that holds the outlier, at the gates of every other test
    b, h = (B - 1, H - 1) if where != "dO_middle" else (B // 2, H // 2)
    ref = oracle.attn_bwd(*(t[b:b + 1, h:h + 1].double().numpy() for t in (Q, K, V, dO)), cfg.causal, cfg.scale)
    check_grads([t[b:b + 1, h:h + 1] for t in (dQ, dK, dV)], ref, f"{where} {dims}", absolute=False)
    assert all(torch.isfinite(t.float()).all() for t in (dQ, dK, dV))
