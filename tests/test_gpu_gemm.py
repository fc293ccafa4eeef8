"""Parity of the FP16 GEMM (C = A W^T) against the fp64 oracle, through the C ABI."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# fp16 output rounding (2^-11 per element) dominates; fp32 accumulation adds far less
GEMM_REL_FRO_TOL = 1e-3


@pytest.fixture(scope="module")
def lt():
    from paper_2606_10415_b200 import binding
    return binding


def rel_fro(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def make_operands(M, N, K, seed):
    gen = torch.Generator(device="cpu")
    gen.manual_seed(seed)
    A = torch.randn((M, K), generator=gen, dtype=torch.float32).half()
    W = (torch.randn((N, K), generator=gen, dtype=torch.float32) * K ** -0.5).half()
    return A, W


def run_gemm(lt, A, W):
    Ad, Wd = A.cuda(), W.cuda()
    C = torch.full((A.shape[0], W.shape[0]), float("nan"), dtype=torch.float16, device="cuda")
    ws = lt.alloc_workspace(lt.lt_gemm_f16_workspace_bytes())
    lt.lt_gemm_f16(Ad, Wd, C, ws)
    assert lt.lt_attn_check_status(ws) == lt.LT_OK, lt.last_cuda_error()
    return C.cpu()


@pytest.mark.parametrize("M,N,K", [
    (128, 256, 64), (128, 256, 256), (256, 512, 512),            # whole tiles
    (1, 8, 8), (100, 200, 72), (129, 257, 136), (300, 1000, 520),  # ragged in every dimension
    (384, 250, 64), (77, 36, 1024),                                # N not a multiple of 8: scalar stores
    (2048, 1024, 768),                                             # more tiles than SMs would need twice
    (128, 40000, 128),   # one tile row: 157 tiles of the 256-wide kernel over 148 CTAs
    (520, 20000, 192),   # 5 x 79 tiles of the 256-wide kernel, ragged M and N
])
def test_gemm_matches_oracle(lt, oracle, M, N, K):
    A, W = make_operands(M, N, K, seed=M + N + K)
    C = run_gemm(lt, A, W)
    ref = oracle.gemm_nt(A.double().numpy(), W.double().numpy())
    got = C.double().numpy()
    assert np.all(np.isfinite(got))
    assert rel_fro(got, ref) <= GEMM_REL_FRO_TOL, f"{(M, N, K)}: {rel_fro(got, ref):.3e}"
    # element-wise: within fp16 rounding of the exact value plus accumulation slack
    assert np.max(np.abs(got - ref) - 2.0 ** -10 * np.abs(ref)) <= 1e-3


@pytest.mark.parametrize("M,N,K", [
    (1, 8, 64), (5, 64, 8), (128, 64, 72),         # one narrow tile; one contraction block, a ragged second one
    (1, 136, 520), (77, 1000, 1000), (129, 65, 4096),  # shares of unequal length; more CTAs of a cluster than rows
    (3, 130, 8192), (128, 128, 4096),              # eight shares
    (424, 265, 5920), (300, 127, 2056),            # several tile rows, N odd (scalar stores) and just below a tile
    (130, 2048, 2048), (16, 5504, 4096), (40, 6000, 2000),  # 128- and 256-wide tiles, two to six shares
    (150, 1408, 152), (404, 1152, 272), (266, 685, 224), (129, 600, 456),  # short contractions on several tile rows
    (1000, 2040, 4096), (600, 600, 600), (8192, 72, 136),   # more tiles than fit at once, short contractions
    (700, 2047, 136), (260, 2046, 136), (129, 2008, 64),    # narrow tiles whose edge is odd, even, in eights
    (2000, 3999, 2048), (2048, 3998, 2048), (1900, 4040, 2048),  # the same on CTA pairs
])
@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
def test_gemm_few_tiles(lt, M, N, K, dtype):
    """Narrow tiles and split contractions against fp64 products of the same operands."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(M + N + K)
    A = torch.randn((M, K), generator=gen, device="cuda").to(dtype)
    W = (torch.randn((N, K), generator=gen, device="cuda") * K ** -0.5).to(dtype)
    C = torch.full((M + 1, N), float("nan"), dtype=dtype, device="cuda")  # the row past the end must stay untouched
    ws = lt.alloc_workspace(lt.lt_gemm_f16_workspace_bytes())
    ws.fill_(0xFF)
    lt.lt_gemm_f16(A, W, C[:M], ws)
    assert lt.lt_attn_check_status(ws) == lt.LT_OK, lt.last_cuda_error()
    ref = A.double() @ W.double().T
    err = (C[:M].double() - ref).abs()
    half_ulp = 2.0 ** -11 if dtype == torch.float16 else 2.0 ** -8  # rounding of the result, relative to it
    # plus fp32 accumulation: K products of order K^-1/2, each addition off by at most 2^-24 of a sum of order one (a
    # factor of eight above that for the largest of up to a million elements), and the smallest subnormal step
    assert (err <= half_ulp * ref.abs() + 8 * K ** 0.5 * 2.0 ** -24 + 2.0 ** -24).all(), float(err.max())
    assert torch.isnan(C[M]).all()


@pytest.mark.parametrize("M,N,K,plan", [
    # the 256-wide kernel on single CTAs: edges that are odd, even, in eights; the last with up to four tiles per CTA
    (570, 2427, 344, (256, 1, False)), (560, 2430, 344, (256, 1, False)), (570, 2424, 344, (256, 1, False)),
    (4000, 4001, 256, (256, 1, False)),
    # on CTA pairs, up to four tiles per pair, so that both accumulators are used again
    (4000, 4001, 1024, (256, 1, True)), (3970, 4002, 1024, (256, 1, True)), (4000, 4008, 1024, (256, 1, True)),
    # narrow tiles, whole and split contractions
    (260, 2046, 136, (64, 1, False)), (700, 2047, 136, (128, 1, False)), (424, 265, 5920, (64, 6, False)),
    (130, 2048, 2048, (128, 4, False)), (40, 6000, 2000, (256, 5, False)), (1000, 2040, 4096, (256, 2, False)),
])
@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
def test_gemm_each_kernel(lt, M, N, K, plan, dtype):
    """Each kernel of the choice, every element of its result, and that the sizes do select it."""
    assert lt.lt_dbg_gemm_plan(M, N, K) == plan
    test_gemm_few_tiles(lt, M, N, K, dtype)


def test_gemm_pairs_on_two_streams(lt):
    """Two products of the CTA-pair kernel on two streams at once: clusters of both launches share the SMs."""
    shapes = [(1024, 4096, 4096), (1900, 4040, 2048)]
    streams, calls = [torch.cuda.Stream() for _ in shapes], []
    for k, (M, N, K) in enumerate(shapes):
        assert lt.lt_dbg_gemm_plan(M, N, K) == (256, 1, True)
        A, W = (t.cuda() for t in make_operands(M, N, K, seed=30 + k))
        calls.append((A, -A, W, [torch.full((M, N), float("nan"), dtype=torch.float16, device="cuda") for _ in range(4)],
                      lt.alloc_workspace(256)))
    torch.cuda.synchronize()
    for i in range(4):
        for stream, (A, minus_A, W, C, ws) in zip(streams, calls):
            lt.lt_gemm_f16(minus_A if i % 2 else A, W, C[i], ws, stream)
    torch.cuda.synchronize()
    for A, _, W, C, ws in calls:
        assert lt.lt_attn_check_status(ws) == lt.LT_OK, lt.last_cuda_error()
        ref = A.double() @ W.double().T
        for i in range(4):
            err = (C[i].double() - (ref if i % 2 == 0 else -ref)).abs()  # (the bound of test_gemm_few_tiles)
            assert (err <= 2.0 ** -11 * ref.abs() + 8 * A.shape[1] ** 0.5 * 2.0 ** -24 + 2.0 ** -24).all()


@pytest.mark.parametrize("M,N,K", [
    (1, 4096, 1024), (7, 512, 4096), (8, 1024, 1024), (9, 72, 72), (33, 2048, 2048), (57, 11008, 512), (64, 4096, 1024),
    (65, 4096, 1024), (5, 40960, 256), (64, 40000, 128),  # the last two: several tiles per CTA
])
@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
def test_gemm_few_rows(lt, M, N, K, dtype):
    """Few rows of A: the rest of a tile's operand rows are whatever shared memory holds, here NaN from the call before."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(M + N + K)
    A = torch.randn((M, K), generator=gen, device="cuda").to(dtype)
    W = (torch.randn((N, K), generator=gen, device="cuda") * K ** -0.5).to(dtype)
    C = torch.full((M + 1, N), float("nan"), dtype=dtype, device="cuda")  # the row past the end must stay untouched
    ws = lt.alloc_workspace(lt.lt_gemm_f16_workspace_bytes())
    full = torch.full((128, K), float("nan"), dtype=dtype, device="cuda")
    lt.lt_gemm_f16(full, W, torch.empty((128, N), dtype=dtype, device="cuda"), ws)
    lt.lt_gemm_f16(A, W, C[:M], ws)
    assert lt.lt_attn_check_status(ws) == lt.LT_OK, lt.last_cuda_error()
    ref = A.double() @ W.double().T
    err = (C[:M].double() - ref).abs()
    half_ulp = 2.0 ** -11 if dtype == torch.float16 else 2.0 ** -8  # (the bound of test_gemm_few_tiles)
    assert (err <= half_ulp * ref.abs() + 8 * K ** 0.5 * 2.0 ** -24 + 2.0 ** -24).all(), float(err.max())
    assert torch.isnan(C[M]).all()


@pytest.mark.parametrize("M,N", [(77, 512), (256, 640), (600, 2048), (40, 24000)])
def test_gemm_back_to_back(lt, M, N):
    """Each product reads what the one before wrote and overwrites what that one read: calls in a row, whose kernels start
    under each other's tails, give what calls with a synchronisation between them give."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(M)
    W = (torch.randn((N, 256), generator=gen, device="cuda") / 16).half()
    Wt = (torch.randn((256, N), generator=gen, device="cuda") * N ** -0.5).half()
    X0 = torch.randn((M, 256), generator=gen, device="cuda").half()
    ws = lt.alloc_workspace(lt.lt_gemm_f16_workspace_bytes())
    results = []
    for sync in (True, False):
        X, Y = X0.clone(), torch.empty((M, N), dtype=torch.float16, device="cuda")
        torch.cuda.synchronize()
        for _ in range(12):
            lt.lt_gemm_f16(X, W, Y, ws)
            if sync:
                torch.cuda.synchronize()
            lt.lt_gemm_f16(Y, Wt, X, ws)
            if sync:
                torch.cuda.synchronize()
        results.append(X)
    assert torch.isfinite(results[0]).all() and torch.equal(*results)


def test_gemm_before_attention(lt):
    """Attention calls behind the products that make their operands, with nothing between them, and a product behind them."""
    S, D = 384, 64
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    X, W = (torch.randn(shape, generator=gen, device="cuda").half() for shape in ((S, 256), (4, D, 256)))
    W /= 16
    ws = lt.alloc_workspace(lt.lt_attn_bwd_workspace_bytes(1, 1, 1, S, D))
    results = []
    for sync in (True, False):
        Q, K, V, dO, O, dQ, dK, dV = (torch.full((1, 1, S, D), float("nan"), dtype=torch.float16, device="cuda") for _ in range(8))
        LSE, Y = torch.empty((1, 1, S), device="cuda"), torch.empty((S, 256), dtype=torch.float16, device="cuda")
        calls = [lambda t=t, w=w: lt.lt_gemm_f16(X, w, t[0, 0], ws) for t, w in zip((Q, K, V, dO), W)]
        calls += [lambda: lt.lt_attn_fwd(Q, K, V, O, LSE, True, 0.125, ws),
                  lambda: lt.lt_attn_bwd(Q, K, V, O, dO, LSE, dQ, dK, dV, True, 0.125, ws),
                  lambda: lt.lt_gemm_f16(dV[0, 0], W[0].T.contiguous(), Y, ws)]
        torch.cuda.synchronize()
        for call in calls:
            call()
            if sync:
                torch.cuda.synchronize()
        results.append((O, LSE, dK, dV, Y))
    assert all(torch.isfinite(a).all() and torch.equal(a, b) for a, b in zip(*results))


def test_gemm_integer_operands_are_exact(lt, oracle):
    """Small integers: every product and partial sum is exact in fp32 and fp16, so the result must
    equal the oracle bit for bit."""
    gen = torch.Generator(device="cpu")
    gen.manual_seed(1)
    A = torch.randint(-3, 4, (200, 136), generator=gen).half()
    W = torch.randint(-2, 3, (300, 136), generator=gen).half()
    C = run_gemm(lt, A, W)
    ref = oracle.gemm_nt(A.double().numpy(), W.double().numpy())
    assert np.array_equal(C.double().numpy(), ref)


@pytest.mark.parametrize("N,K", [(4096, 4096), (11008, 4096), (4096, 11008), (6656, 6656), (8192, 8192)])
def test_gemm_paper_shapes_sampled_rows(lt, oracle, N, K):
    """The five weight shapes of the paper's GEMM profile (Section 6.6) at its sequence length of 2048
    rows; the launch the benchmark times, compared on sampled rows and columns."""
    M = 2048
    A, W = make_operands(M, N, K, seed=N + K)
    C = run_gemm(lt, A, W)
    assert torch.isfinite(C.float()).all()
    rows = [0, 1, 127, 128, 1000, 2047]
    ref = oracle.gemm_nt(A[rows].double().numpy(), W.double().numpy())
    assert rel_fro(C[rows].double().numpy(), ref) <= GEMM_REL_FRO_TOL
    cols = [0, 255, 256, N // 2 + 3, N - 1]
    ref_c = oracle.gemm_nt(A.double().numpy(), W[cols].double().numpy())
    assert rel_fro(C[:, cols].double().numpy(), ref_c) <= GEMM_REL_FRO_TOL


@pytest.mark.parametrize("M,N,K", [(129, 257, 136), (512, 768, 1024)])
def test_gemm_bf16_matches_oracle(lt, oracle, M, N, K):
    A, W = (t.float().bfloat16() for t in make_operands(M, N, K, seed=7 + M))
    C = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda")
    ws = lt.alloc_workspace(lt.lt_gemm_f16_workspace_bytes())
    lt.lt_gemm_f16(A.cuda(), W.cuda(), C, ws)
    assert lt.lt_attn_check_status(ws) == lt.LT_OK, lt.last_cuda_error()
    ref = oracle.gemm_nt(A.double().numpy(), W.double().numpy())
    # bf16 output rounding: 2^-9 per element
    assert rel_fro(C.cpu().double().numpy(), ref) <= 4e-3


@pytest.mark.parametrize("seed", [0, 1])
def test_gemm_random_shapes(lt, oracle, seed):
    """Seeded sweep over ragged shapes of up to 1 100 rows (narrow tiles, whole and split contractions): integer operands, so
    every result is exact and compared bit for bit."""
    rng = np.random.default_rng(1000 + seed)
    for case in range(12):
        M = int(rng.choice([1, 64, 127, 128, 129, 255, 256, 257, 384, 513, 700, 1100]))
        N = int(rng.integers(1, 1400))
        K = 8 * int(rng.integers(1, 90))
        gen = torch.Generator(device="cpu")
        gen.manual_seed(seed * 100 + case)
        A = torch.randint(-3, 4, (M, K), generator=gen).half()
        W = torch.randint(-2, 3, (N, K), generator=gen).half()
        C = run_gemm(lt, A, W)
        ref = oracle.gemm_nt(A.double().numpy(), W.double().numpy())
        assert np.array_equal(C.double().numpy(), ref), f"case {case}: M={M} N={N} K={K}"


def test_gemm_pair_kernel_on_two_streams(lt, oracle):
    """Two products on two streams at once, whose CTAs share the SMs; each has its own status block and result."""
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    A1, W1 = make_operands(1024, 2048, 512, seed=21)
    A2, W2 = make_operands(768, 1536, 1024, seed=22)
    d = [t.cuda() for t in (A1, W1, A2, W2)]
    C1 = torch.full((1024, 2048), float("nan"), dtype=torch.float16, device="cuda")
    C2 = torch.full((768, 1536), float("nan"), dtype=torch.float16, device="cuda")
    w1, w2 = lt.alloc_workspace(256), lt.alloc_workspace(256)
    torch.cuda.synchronize()
    for _ in range(5):
        lt.lt_gemm_f16(d[0], d[1], C1, w1, s1)
        lt.lt_gemm_f16(d[2], d[3], C2, w2, s2)
    torch.cuda.synchronize()
    assert lt.lt_attn_check_status(w1) == lt.LT_OK and lt.lt_attn_check_status(w2) == lt.LT_OK, lt.last_cuda_error()
    for C, A, W in ((C1, A1, W1), (C2, A2, W2)):
        ref = oracle.gemm_nt(A.double().numpy(), W.double().numpy())
        assert rel_fro(C.cpu().double().numpy(), ref) <= GEMM_REL_FRO_TOL
