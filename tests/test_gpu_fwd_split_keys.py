"""Forward whose CTAs take one query tile with its key tiles in two chains (few heads): one key tile (an empty second
chain) to many, odd and even counts, ragged ends, both masks, head dimensions and types, a negative scale, maxima that
rise late in one chain only, against fp64 softmax."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,Hkv,S,D", [(2, 1, 129, 64), (1, 1, 256, 128), (3, 3, 300, 128), (2, 2, 640, 64), (4, 2, 1153, 128),
                                       (1, 1, 2048, 64)])
@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("dtype,scale_sign,ramp", [(torch.float16, 1, False), (torch.bfloat16, 1, False),
                                                   (torch.float16, -1, False), (torch.float16, 1, True)])
def test_split_keys(H, Hkv, S, D, causal, dtype, scale_sign, ramp):
    from paper_2606_10415_b200 import binding as lt
    assert lt.lt_dbg_fwd_plan(1, H, S, D, causal) == (True, True)  # (keys split, walk in one copy)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(S + D)
    Q, K, V = (torch.randn((1, h, S, D), generator=gen, device="cuda") for h in (H, Hkv, Hkv))
    if ramp:  # scores that grow along the keys, by far the most in the odd key tiles
        tile = torch.arange(S, device="cuda") // 128
        K = K * (0.2 + 0.8 * tile * (tile % 2)).view(1, 1, S, 1)
    Q, K, V = (t.to(dtype) for t in (Q, K, V))
    scale = scale_sign * D ** -0.5
    O, LSE = torch.full_like(Q, float("nan")), torch.full((1, H, S), float("nan"), device="cuda")
    ws = lt.alloc_workspace(256)
    ws.fill_(0xFF)
    fn = lt.lt_attn_fwd if dtype == torch.float16 else lt.lt_attn_fwd_bf16
    fn(Q, K, V, O, LSE, causal, scale, ws)
    assert lt.lt_attn_check_status(ws) == lt.LT_OK, lt.last_cuda_error()
    k, v = (t.double().repeat_interleave(H // Hkv, 1) for t in (K, V))
    s = Q.double() @ k.transpose(-1, -2) * scale
    if causal:
        s.masked_fill_(torch.ones(S, S, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
    lse = torch.logsumexp(s, -1)
    ref = torch.exp(s - lse[..., None]) @ v
    # the forward's gates: rounding of P and O, 2^-11 (fp16) or 2^-8 (bf16) each, in the 2-norm
    assert (O.double() - ref).norm() <= (2e-3 if dtype == torch.float16 else 4e-3) * ref.norm()
    # LSE is fp32: one unit of its own size besides the flat gate
    assert ((LSE.double() - lse).abs() <= 1e-3 + 2.0 ** -22 * lse.abs()).all()


@pytest.mark.parametrize("H,Hkv,S,D,hidden", [(1, 1, 256, 128, (1,)), (4, 2, 300, 64, (1,)), (2, 2, 640, 128, (1,)),
                                              (2, 1, 640, 64, (1, 3)), (1, 1, 1100, 128, (1, 2, 3, 5, 7)),
                                              (1, 1, 256, 128, (0,)), (4, 2, 300, 64, (0, 1)), (2, 1, 1153, 128, (0, 2))])
@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
def test_hidden_key_tiles(H, Hkv, S, D, hidden, causal, dtype):
    """Keys hidden by a channel of ones in Q against -inf in K: score -inf, weight zero, also where that is every key of the
    tile a chain starts with, or of all its tiles."""
    from paper_2606_10415_b200 import binding as lt
    assert lt.lt_dbg_fwd_plan(1, H, S, D, causal) == (True, True)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(S + D)
    Q, K, V = (torch.randn((1, h, S, D), generator=gen, device="cuda").to(dtype) for h in (H, Hkv, Hkv))
    Q[..., 0] = 1.0
    gone = torch.isin(torch.arange(S, device="cuda") // 128, torch.tensor(hidden, device="cuda"))
    K[:, :, gone, 0] = float("-inf")
    O, LSE = torch.full_like(Q, float("nan")), torch.full((1, H, S), float("nan"), device="cuda")
    ws = lt.alloc_workspace(256)
    fn = lt.lt_attn_fwd if dtype == torch.float16 else lt.lt_attn_fwd_bf16
    fn(Q, K, V, O, LSE, causal, D ** -0.5, ws)
    assert lt.lt_attn_check_status(ws) == lt.LT_OK, lt.last_cuda_error()
    k, v = (t.double().repeat_interleave(H // Hkv, 1) for t in (K, V))
    s = Q.double() @ k.transpose(-1, -2) * D ** -0.5
    if causal:
        s.masked_fill_(torch.ones(S, S, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
    lse = torch.logsumexp(s, -1)
    sees = torch.isfinite(lse)  # (a row without a visible key has no output)
    ref, lse, O, LSE = (torch.exp(s - lse[..., None]) @ v)[sees], lse[sees], O[sees], LSE[sees]
    assert torch.isfinite(O).all()  # (the gates of test_split_keys)
    assert (O.double() - ref).norm() <= (2e-3 if dtype == torch.float16 else 4e-3) * ref.norm()
    assert ((LSE.double() - lse).abs() <= 1e-3 + 2.0 ** -22 * lse.abs()).all()


@pytest.mark.parametrize("H,S,D,causal", [(32, 1024, 128, True), (8, 700, 64, True), (4, 1500, 64, False)])
@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
def test_no_further_from_64_bits_than_query_pairs(H, S, D, causal, dtype):
    """The same heads alone (their keys in two chains) and many times over (pairs of query tiles): putting two chains
    together costs neither O nor LSE any precision."""
    from paper_2606_10415_b200 import binding as lt
    gen = torch.Generator(device="cuda")
    gen.manual_seed(S)
    Q, K, V = (torch.randn((1, H, S, D), generator=gen, device="cuda").to(dtype) for _ in range(3))
    s = Q.double() @ K.double().transpose(-1, -2) * D ** -0.5
    if causal:
        s.masked_fill_(torch.ones(S, S, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
    lse = torch.logsumexp(s, -1)
    ref = torch.exp(s - lse[..., None]) @ V.double()
    fn = lt.lt_attn_fwd if dtype == torch.float16 else lt.lt_attn_fwd_bf16
    off, last = [], None
    for B in (1, 512 // H):
        q, k, v = (t.expand(B, -1, -1, -1).contiguous() for t in (Q, K, V))
        O, LSE = torch.empty_like(q), torch.empty((B, H, S), device="cuda")
        assert lt.lt_dbg_fwd_plan(B, H, S, D, causal)[0] == (B == 1)
        fn(q, k, v, O, LSE, causal, D ** -0.5, lt.alloc_workspace(256))
        assert last is None or not torch.equal(last, O[0])  # the two forms do differ
        last = O[0]
        off.append(((O[0].double() - ref[0]).norm(), (LSE[0].double() - lse[0]).norm()))
    assert off[0][0] <= off[1][0] and off[0][1] <= off[1][1], off
