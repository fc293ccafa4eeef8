"""Key tiles split over several CTAs: dealt out (one tile and several, one query head per key/value head and many, stretches
of a single pair, tiles of many parts, both head dimensions, types and masks) and in halves, against the oracle; dK and dV
the same from run to run; and the entry points that run with whole key tiles because their scratch has no room for the fp32
shares."""
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
    (1, 5, 1, 129, 128, True, 4), (1, 20, 4, 640, 128, True, 4),   # five heads: tiles cut at unequal places
    (4, 8, 1, 300, 64, True, 4),
    (1, 1, 1, 407, 128, True, 4), (1, 2, 2, 1000, 128, False, 4), (3, 2, 2, 1500, 64, True, 4),  # one head per kv head
    (1, 4, 2, 256, 64, True, 4), (2, 8, 4, 256, 128, False, 4),    # stretches of one or two pairs
    (1, 4, 4, 144, 64, True, 3), (2, 8, 8, 384, 128, False, 3),    # short walks stay whole
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
        again = [t.clone() for t in outs[1:]]
        bwd(*ins, *outs, causal, cfg.scale, ws)
        assert all(torch.equal(x, y) for x, y in zip(again, outs[1:])), "dK, dV differ between runs"
    assert lt.lt_attn_check_status(ws) == lt.LT_OK, lt.last_cuda_error()
    ref = oracle.attn_bwd(*(t.double().numpy() for t in host), causal, cfg.scale)
    check_grads(outs, ref, f"split {cfg}", dtype=dtype, absolute=False)


@pytest.mark.parametrize("B,Hq,Hkv,S,D,causal", [(1, 8, 1, 300, 64, False), (1, 40, 8, 1024, 128, True), (1, 2, 2, 1000, 64, True),
                                                 (1, 2, 1, 3566, 128, True)])
@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
def test_split_calls_on_changing_data(B, Hq, Hkv, S, D, causal, dtype):
    """The kernels of a call start under one another's tails, and two calls share a workspace: what a call adds up and
    converts has to be its own.  Two problems in turn without a synchronisation, each call into outputs of its own, against the
    same calls made alone on a workspace full of NaN."""
    from paper_2606_10415_b200 import binding as lt
    dt = torch.float16 if dtype == "fp16" else torch.bfloat16
    bwd = lt.lt_attn_bwd if dtype == "fp16" else lt.lt_attn_bwd_bf16
    assert lt.lt_attn_bwd_num_launches(B, Hq, Hkv, S, D, causal) == 4
    scale = D ** -0.5
    problems = [_forward(lt, workloads.custom(B, Hq, Hkv, S, D, causal, seed=seed), dt)[1:] for seed in (1, 2)]
    ws = lt.alloc_workspace(lt.lt_attn_bwd_workspace_bytes(B, Hq, Hkv, S, D))
    for ins, outs in problems:
        ws.fill_(0xFF)
        bwd(*ins, *outs, causal, scale, ws)
        torch.cuda.synchronize()
        assert lt.lt_attn_check_status(ws) == lt.LT_OK, lt.last_cuda_error()
        assert all(torch.isfinite(t).all() for t in outs)
    ws.fill_(0xFF)
    calls = [(k, [torch.full_like(t, float("nan")) for t in problems[k][1]]) for k in (0, 1) * 6]
    torch.cuda.synchronize()
    for k, outs in calls:
        bwd(*problems[k][0], *outs, causal, scale, ws)
    assert lt.lt_attn_check_status(ws) == lt.LT_OK, lt.last_cuda_error()
    for k, outs in calls:
        want = problems[k][1]
        assert torch.equal(outs[1], want[1]) and torch.equal(outs[2], want[2])
        # dQ's fp32 partials arrive in any order, so a result may round to the other neighbour: 2^-11 (2^-8) of it
        assert (outs[0].double() - want[0].double()).norm() <= (2.0 ** -11 if dtype == "fp16" else 2.0 ** -8) * want[0].double().norm()


@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
def test_halves(oracle, dtype):
    # 256 key tiles of up to 256 pairs on a working set of 1.1 GB: too few for batches, so each is two items
    from paper_2606_10415_b200 import binding as lt
    B, Hq, Hkv, S, D = 32, 32, 1, 900, 128
    assert lt.lt_attn_bwd_num_launches(B, Hq, Hkv, S, D, True) == 4
    dt, scale = torch.float16 if dtype == "fp16" else torch.bfloat16, D ** -0.5
    gen = torch.Generator(device="cuda").manual_seed(9)
    Q, K, V, dO = (torch.randn((B, h, S, D), generator=gen, device="cuda").to(dt) for h in (Hq, Hkv, Hkv, Hq))
    O, LSE = torch.empty_like(Q), torch.empty((B, Hq, S), dtype=torch.float32, device="cuda")
    fwd, bwd = (lt.lt_attn_fwd, lt.lt_attn_bwd) if dtype == "fp16" else (lt.lt_attn_fwd_bf16, lt.lt_attn_bwd_bf16)
    fwd(Q, K, V, O, LSE, True, scale, lt.alloc_workspace(256))
    outs = [torch.full_like(t, float("nan")) for t in (Q, K, V)]
    ws = lt.alloc_workspace(lt.lt_attn_bwd_workspace_bytes(B, Hq, Hkv, S, D))
    ws.fill_(0xFF)
    bwd(Q, K, V, O, dO, LSE, *outs, True, scale, ws)
    assert lt.lt_attn_check_status(ws) == lt.LT_OK, lt.last_cuda_error()
    assert all(torch.isfinite(t).all() for t in outs)
    for b in (0, 13, 31):
        ref = oracle.attn_bwd(*(t[b:b + 1].cpu().double().numpy() for t in (Q, K, V, dO)), True, scale)
        check_grads([t[b:b + 1] for t in outs], ref, f"halves, batch {b}", dtype=dtype, absolute=False)


def test_noalloc_without_room_for_the_shares(oracle):
    from paper_2606_10415_b200 import binding as lt
    cfg = workloads.custom(1, 8, 1, 4096, 128, True, seed=5)
    dims = (cfg.B, cfg.Hq, cfg.Hkv, cfg.S, cfg.D)
    assert lt.lt_attn_bwd_workspace_bytes(*dims) > lt.NOALLOC_MAX_SCRATCH_BYTES
    host, ins, outs = _forward(lt, cfg)
    lt.lt_attn_bwd_noalloc(*ins, *outs, cfg.causal, cfg.scale)
    assert lt.lt_attn_bwd_noalloc_check_status() == lt.LT_OK
    ref = oracle.attn_bwd(*(t.double().numpy() for t in host), cfg.causal, cfg.scale)
    check_grads(outs, ref, "noalloc, whole key tiles")


@pytest.mark.parametrize("B,Hq,Hkv,S,D,causal", [(1, 4, 4, 938, 128, True), (1, 2, 2, 1000, 64, False), (1, 20, 4, 640, 128, True)])
@pytest.mark.parametrize("room", [0, 3, 40])
def test_workspace_with_room_for_few_shares(oracle, B, Hq, Hkv, S, D, causal, room):
    """`room`: shares that fit behind the accumulator.  Nothing past the size given is touched."""
    from paper_2606_10415_b200 import binding as lt
    cfg = workloads.custom(B, Hq, Hkv, S, D, causal, seed=S)
    host, ins, outs = _forward(lt, cfg)
    rows = B * Hq * -(-S // 128) * 128
    n = 256 + 2 * rows * 16 + rows * D * 4 + room * 2 * 128 * D * 4
    assert n < lt.lt_attn_bwd_workspace_bytes(B, Hq, Hkv, S, D)
    buf = lt.alloc_workspace(lt.lt_attn_bwd_workspace_bytes(B, Hq, Hkv, S, D))
    buf.fill_(0xFF)
    lt.lt_attn_bwd(*ins, *outs, causal, cfg.scale, buf[:n])
    assert lt.lt_attn_check_status(buf) == lt.LT_OK, lt.last_cuda_error()
    assert (buf[n:] == 0xFF).all()
    ref = oracle.attn_bwd(*(t.double().numpy() for t in host), causal, cfg.scale)
    check_grads(outs, ref, f"room for {room} shares {cfg}", absolute=False)
