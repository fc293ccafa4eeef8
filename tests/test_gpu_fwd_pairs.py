"""Forward whose CTAs take pairs of query tiles (many heads), and the forms of the kernel that fewer or longer walks select: a lone last tile, walks shorter and longer than the ring of
key and value tiles, ragged ends, both masks, maxima that rise late, keys hidden by -inf (the first tile's among them, as
left padding has it), and an output between other columns and rows that must stay as they are; against fp64 softmax."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,D", [(1, 64), (127, 128), (129, 64), (257, 128), (384, 64), (511, 128), (700, 64), (897, 128)])
@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("dtype,kind", [(torch.float16, "plain"), (torch.bfloat16, "plain"), (torch.float16, "ramp"), (torch.float16, "hidden"),
                                        (torch.float16, "hidden first"), (torch.bfloat16, "hidden first")])
def test_query_pairs(S, D, causal, dtype, kind):
    check(3, 64, 16, S, D, causal, dtype, kind, (False, D == 64 or S <= 128))


# D = 128: pairs with the walk in one copy (few CTAs, several tiles), split keys with the unrolled one (many CTAs, long walks)
@pytest.mark.parametrize("H,Hkv,S,causal,form", [(64, 8, 512, True, (False, True)), (64, 16, 500, False, (False, True)), (64, 64, 897, False, (False, True)),
                                                 (44, 4, 897, True, (False, True)), (20, 4, 2048, True, (True, False)),
                                                 (4, 2, 3201, False, (True, False)), (28, 7, 1290, False, (True, False))])
@pytest.mark.parametrize("dtype,kind", [(torch.float16, "plain"), (torch.bfloat16, "plain"), (torch.float16, "ramp"), (torch.float16, "hidden"),
                                        (torch.float16, "hidden first")])
def test_other_forms(H, Hkv, S, causal, form, dtype, kind):
    check(1, H, Hkv, S, 128, causal, dtype, kind, form)


def check(B, H, Hkv, S, D, causal, dtype, kind, form):
    from paper_2606_10415_b200 import binding as lt
    assert lt.lt_dbg_fwd_plan(B, H, S, D, causal) == form  # (keys split, walk in one copy)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(S + D)
    Q, K, V = (torch.randn((B, h, S, D), generator=gen, device="cuda") for h in (H, Hkv, Hkv))
    tile = torch.arange(S, device="cuda") // 128
    if kind == "ramp":  # scores that grow along the keys: the output is rescaled
        K = K * (0.2 + 0.8 * tile).view(1, 1, S, 1)
    Q, K, V = (t.to(dtype) for t in (Q, K, V))
    if kind in ("hidden", "hidden first"):  # every key of the odd key tiles, or of the first one
        Q[..., 0] = 1.0
        K[:, :, tile % 2 == 1 if kind == "hidden" else tile == 0, 0] = float("-inf")
    around = torch.full((B, S + 2, (H + 2) * D), 7.0, dtype=dtype, device="cuda")
    O = around.view(B, S + 2, H + 2, D).permute(0, 2, 1, 3)[:, 1:H + 1, 1:S + 1]
    LSE = torch.full((B, H, S), float("nan"), device="cuda")
    ws = lt.alloc_workspace(256)
    ws.fill_(0xFF)
    fn = lt.lt_attn_fwd_strided if dtype == torch.float16 else lt.lt_attn_fwd_bf16
    fn(Q, K, V, O, LSE, causal, D ** -0.5, ws)
    assert lt.lt_attn_check_status(ws) == lt.LT_OK, lt.last_cuda_error()
    for b in range(B):
        k, v = (t[b].double().repeat_interleave(H // Hkv, 0) for t in (K, V))
        s = Q[b].double() @ k.transpose(-1, -2) * D ** -0.5
        if causal:
            s.masked_fill_(torch.ones(S, S, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
        lse = torch.logsumexp(s, -1)
        sees = torch.isfinite(lse)  # (a row without a visible key has no output)
        ref, lse, got, got_lse = (torch.exp(s - lse[..., None]) @ v)[sees], lse[sees], O[b][sees].double(), LSE[b][sees].double()
        assert torch.isfinite(got).all()
        # the forward's gates: rounding of P and O, 2^-11 (fp16) or 2^-8 (bf16) each, in the 2-norm
        assert (got - ref).norm() <= (2e-3 if dtype == torch.float16 else 4e-3) * ref.norm()
        assert ((got_lse - lse).abs() <= 1e-3 + 2.0 ** -22 * lse.abs()).all()
    O.fill_(7.0)
    assert (around == 7.0).all()  # nothing but O was written
