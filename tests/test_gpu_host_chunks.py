"""The host-buffer call cut into chunks (six of them, or four: 16 heads on 8): every unit of every chunk
against the device entry points on the whole problem, with and without the optional outputs, calls back to back."""
import pytest
import torch

from paper_2606_10415_b200 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,S,D,causal", [(4, 16, 16, 1024, 128, False), (1, 24, 24, 3000, 128, True), (1, 16, 8, 3000, 128, True)])
@pytest.mark.parametrize("with_o", [True, False])
def test_many_chunks(B, Hq, Hkv, S, D, causal, with_o):
    from paper_2606_10415_b200 import binding as lt
    cfg = workloads.custom(B, Hq, Hkv, S, D, causal, seed=S)
    host = [t.pin_memory() for t in workloads.make_inputs(cfg)]
    Q, K, V, dO = (t.cuda() for t in host)
    O, LSE = torch.empty_like(Q), torch.empty(Q.shape[:3], dtype=torch.float32, device="cuda")
    want = [torch.empty_like(t) for t in (Q, K, V)]
    dims = (B, Hq, Hkv, S, D)
    ws = lt.alloc_workspace(lt.lt_attn_bwd_workspace_bytes(*dims))
    lt.lt_attn_fwd(Q, K, V, O, LSE, causal, cfg.scale, ws)
    lt.lt_attn_bwd(Q, K, V, O, dO, LSE, *want, causal, cfg.scale, ws)
    h_O = torch.full(Q.shape, float("nan"), dtype=torch.float16, pin_memory=True) if with_o else None
    h_L = torch.full(Q.shape[:3], float("nan"), dtype=torch.float32, pin_memory=True) if with_o else None
    got = [torch.full(t.shape, float("nan"), dtype=torch.float16, pin_memory=True) for t in (Q, K, V)]
    arena = lt.alloc_workspace(lt.lt_attn_host_arena_bytes(*dims))
    for _ in range(3):  # later calls reuse the arena under the earlier ones' copies
        lt.lt_attn_fwd_bwd_host(*host, h_O, h_L, *got, causal, cfg.scale, arena)
    torch.cuda.synchronize()
    if with_o:
        # a chunk of few heads may take its keys in two chains: probabilities round to fp16 against another running
        # maximum, and so does the result, 2^-11 each; S terms of the fp32 row sums are added in another order
        g, w = h_O.double(), O.cpu().double()
        assert torch.isfinite(g).all() and (g - w).norm() <= 2 * 2.0 ** -11 * w.norm()
        assert (h_L.double() - LSE.cpu().double()).abs().max() <= S * 2.0 ** -24
    for name, g, w in zip(("dQ", "dK", "dV"), got, want):
        g, w = g.double(), w.cpu().double()
        assert torch.isfinite(g).all(), name
        # a chunk picks its own power of two for dS, so roundings to fp16 may fall on the other side: half a unit
        # in the last place of the operands, of the result and of the O that delta is formed from, 2^-11 each
        assert (g - w).norm() <= 3 * 2.0 ** -11 * w.norm(), name


@pytest.mark.parametrize("B,Hq,Hkv,S,D,causal", [(4, 16, 16, 1024, 128, False), (1, 16, 8, 3000, 128, True), (1, 24, 24, 3000, 128, True)])
def test_calls_on_changing_data(B, Hq, Hkv, S, D, causal):
    """Calls in a row on one arena, each with other inputs and into outputs of its own: a copy that overtook the kernels it
    waits for, or a chunk that was overwritten under a copy, would leave another call's values."""
    from paper_2606_10415_b200 import binding as lt
    dims = (B, Hq, Hkv, S, D)
    arena, ws = lt.alloc_workspace(lt.lt_attn_host_arena_bytes(*dims)), lt.alloc_workspace(lt.lt_attn_bwd_workspace_bytes(*dims))
    problems = []
    for seed in (1, 2):
        cfg = workloads.custom(B, Hq, Hkv, S, D, causal, seed=seed)
        host = [t.pin_memory() for t in workloads.make_inputs(cfg)]
        Q, K, V, dO = (t.cuda() for t in host)
        O, LSE = torch.empty_like(Q), torch.empty(Q.shape[:3], dtype=torch.float32, device="cuda")
        want = [torch.empty_like(t) for t in (Q, K, V)]
        lt.lt_attn_fwd(Q, K, V, O, LSE, causal, cfg.scale, ws)
        lt.lt_attn_bwd(Q, K, V, O, dO, LSE, *want, causal, cfg.scale, ws)
        problems.append((host, [t.cpu().double() for t in (O, LSE, *want)]))
    calls = [(k, [torch.full(t.shape, float("nan"), dtype=torch.float32 if i == 1 else torch.float16, pin_memory=True)
                  for i, t in enumerate(problems[k][1])]) for k in (0, 1, 0, 1)]
    arena.fill_(0xFF)
    torch.cuda.synchronize()
    for k, out in calls:
        lt.lt_attn_fwd_bwd_host(*problems[k][0], *out, causal, D ** -0.5, arena)
    torch.cuda.synchronize()
    for n, (k, out) in enumerate(calls):
        for name, g, w in zip(("O", "LSE", "dQ", "dK", "dV"), out, problems[k][1]):
            g = g.double()
            assert torch.isfinite(g).all(), (n, name)
            if name == "LSE":
                assert (g - w).abs().max() <= S * 2.0 ** -24, n
            else:  # (the bounds of test_many_chunks)
                assert (g - w).norm() <= (2 if name == "O" else 3) * 2.0 ** -11 * w.norm(), (n, name)
