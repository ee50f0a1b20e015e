"""Sizes at which the kernels' tiles, rings, runs and dispatch rules change, against the
FP64 oracle within the bounds of helpers.py (or bit for bit where two routes must agree)."""
import numpy as np
import pytest
import torch

import oracle
import paper_1411_2860_gb300 as pj
import synth
from helpers import U_BF16, factor, gamma, gemm_abs_product
from test_gpu_batch import _check_conv, _check_gemm, _conv_case, _desc, _gemm_case
from test_gpu_conv import conv_bound
from test_gpu_gemm import _bf16_case
from test_gpu_gemm_e4m3 import _e4m3_case

pytestmark = pytest.mark.gpu

DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def built():
    pj.build()
    assert torch.cuda.is_available()


def _within(Y, ref, bound):
    assert np.all(np.abs(Y - ref) <= bound), np.nanmax(np.abs(Y - ref) / bound)


# ------------------------------------------------------------------ products --

@pytest.mark.parametrize("split", [1, 2])
@pytest.mark.parametrize("K", [8, 64, 72, 192, 200, 1000])
@pytest.mark.parametrize("M,N", [(33, 100), (300, 256), (65, 300), (190, 512)])
def test_chunk_counts(M, N, K, split):
    """One chunk of components, odd and even counts (the hi and lo tiles of a chunk share
    their ring slots), ring slots of several tile heights, one and two CTAs per tile."""
    _within(*_bf16_case(M, N, K, 8, 8, split))


@pytest.mark.parametrize("split", [1, 2])
@pytest.mark.parametrize("M,N,K", [(16, 128, 8), (100, 300, 136), (240, 256, 128), (241, 129, 1000), (496, 256, 264)])
def test_e4m3_tile_heights(M, N, K, split):
    _within(*_e4m3_case(M, N, K, 8, 8, split))


@pytest.mark.parametrize("split,M,N", [(1, 2048, 1152), (1, 2048, 1408), (2, 2304, 1920), (2, 2560, 1920)])
def test_stream_k_limits(split, M, N):
    """An odd number of tile columns, just below and just above half a wave of tiles
    (0.9 waves with lo terms), where products change from cut to whole tiles."""
    _within(*_bf16_case(M, N, 512, 128, 128, split))


@pytest.mark.parametrize("lp1", range(1, 9))
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("M,K,N", [(9, 7, 70), (500, 1001, 33), (3, 4104, 257)])
def test_unaligned_projection(M, K, N, dtype, lp1):
    """Rows and columns of odd pitch, for every l + 1: partial last groups, quads and runs."""
    rng = np.random.default_rng(lp1)
    A = torch.from_numpy(rng.normal(size=(M, K + 1))).to(DEV).to(dtype)[:, :K]
    B = torch.from_numpy(rng.normal(size=(K, N + 1))).to(DEV).to(dtype)[:, :N]
    A64, B64 = A.double().cpu().numpy(), B.double().cpu().numpy()
    Y = pj.proj_gemm(A, B, 8, lp1, split=2).double().cpu().numpy()
    C, D = oracle.basis("dct2", 8)
    absprod, Kp = gemm_abs_product(A64, B64, 8, C, D, lp1)
    _within(Y, oracle.gemm_proj(A64, B64, 8, lp1, "dct2", 8), factor(3 * Kp, 8, 2) * absprod)


@pytest.mark.parametrize("K,lp1", [(168, 3), (163, 3), (1016, 5), (72, 7), (360, 1)])
@pytest.mark.parametrize("N", [256, 259, 512])
def test_last_quad_of_columns(K, lp1, N):
    """Group counts that are no multiple of four: a last quad inside and past the padded pitch."""
    _within(*_bf16_case(40, N, K, 8, lp1, 2))


@pytest.mark.parametrize("M,N", [(1, 1), (7, 9), (8, 8), (17, 8), (65, 33)])
@pytest.mark.parametrize("K", [63, 64, 65, 130])
@pytest.mark.parametrize("kind,L,lp1", [("dct2", 8, 8), ("dct2", 8, 3), ("haar", 8, 5), ("haar", 4, 4)])
def test_f64_tiles(M, N, K, kind, L, lp1):
    rng = np.random.default_rng(K)
    A, B = rng.normal(size=(M, K)), rng.normal(size=(K, N))
    Y = pj.proj_gemm(torch.from_numpy(A).to(DEV), torch.from_numpy(B).to(DEV), L, lp1, kind, L).cpu().numpy()
    C, D = oracle.basis(kind, L)
    absprod, Kp = gemm_abs_product(A, B, L, C, D, lp1)
    # both sides round: two L-term projections (their coefficients to an ulp) and Kp terms
    _within(Y, oracle.gemm_proj(A, B, L, lp1, kind, L), 2 * gamma(Kp + 2 * L + 4, 2.0 ** -53) * absprod)


@pytest.mark.parametrize("M,N,K", [(7, 130, 40), (257, 64, 520), (129, 255, 1001)])
def test_backward_rounds_f32_gradient(M, N, K):
    """An FP32 dY of BF16 operands gives the gradients of dY rounded to BF16."""
    g = torch.Generator(device=DEV).manual_seed(M)
    A = torch.randn(M, K, device=DEV, generator=g).bfloat16()
    B = torch.randn(K, N, device=DEV, generator=g).bfloat16()
    dY = torch.randn(M, N, device=DEV, generator=g)
    got = pj.proj_gemm_backward(A, B, dY, 8, 4)
    want = pj.proj_gemm_backward(A, B, dY.bfloat16(), 8, 4)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


# -------------------------------------------------------------- correlations --

@pytest.mark.parametrize("R", [64, 256, 1024])
@pytest.mark.parametrize("nt", [1, 3, 6, 33, 61, 64])
@pytest.mark.parametrize("lags", [1, 257, 5001])
def test_correlation_chunks(lags, nt, R):
    """Template counts that end inside a chunk of stored columns, short and long reductions."""
    T = 1024
    s, k, _ = synth.audio_workload(lags + T - 1, T, nt, seed=nt)
    got = pj.proj_conv(torch.from_numpy(s).to(DEV), torch.from_numpy(k).to(DEV), R).double().cpu().numpy()
    s64, k64 = s.astype(np.float64), k.astype(np.float64)
    rng = np.random.default_rng(lags)
    mm, tt = rng.integers(0, lags, 800), rng.integers(0, nt, 800)
    mm[:nt], tt[:nt] = lags - 1, np.arange(nt)
    ref = oracle.conv_proj_entries(s64, k64, mm, tt, R, "haar", 64)
    _within(got[mm, tt], ref, conv_bound(s64, k64, R, mm, tt))


# --------------------------------------------------------------------- batch --

@pytest.mark.parametrize("tuning", [None, {"solo": 1}, {"schedule": 1}, {"schedule": 2, "tile_rows": 32}])
def test_batch_pairs_of_columns(tuning):
    """Odd and single tile columns, cut reductions, BF16 outputs between FP32 ones, and
    correlations whose lags end inside a row of 256 and inside a tile of 256 rows."""
    rng = np.random.default_rng(3)
    gemms = [_gemm_case(rng, 300, 100, 700, 8, 8, 2), _gemm_case(rng, 64, 129, 8000, 8, 8, 1),
             _gemm_case(rng, 257, 384, 64, 8, 3, 2), _gemm_case(rng, 1, 513, 200, 8, 8, 1)]
    for M, N in ((130, 264), (40, 100)):
        c = _gemm_case(rng, M, N, 300, 8, 8, 1)
        c["Y"] = c["Y"].bfloat16()
        gemms.append(c)
    convs = [(2, _conv_case(rng, 255 + lags, 256, nt, R, lags))
             for lags, nt, R in ((1, 1, 256), (255, 1, 64), (257, 3, 256), (66000, 1, 128))]
    c = _conv_case(rng, 3001, 256, 1, 256, 9)
    c["s"] = c["s"][1:]                     # a signal off its 16-byte boundary
    c["out"] = c["out"][:-1]
    convs.append((1, c))
    plan = pj.BatchPlan([_desc(c) for c in gemms] +
                        [pj.batch_conv(c["s"], c["k"], c["out"], c["R"], split=sp) for sp, c in convs], tuning=tuning)
    for _ in range(2):
        plan.run()
        plan.check()
    for c in gemms[:4]:
        _check_gemm(c)
    for c in gemms[4:]:   # one more rounding, to BF16
        A, B = c["A"].double().cpu().numpy(), c["B"].double().cpu().numpy()
        C, D = oracle.basis("dct2", 8)
        absprod, Kp = gemm_abs_product(A, B, 8, C, D, 8)
        ref = oracle.gemm_proj(A, B, 8, 8, "dct2", 8)
        bound = factor(Kp, 8, 1) * absprod
        _within(c["Y"].double().cpu().numpy(), ref, bound + U_BF16 * (np.abs(ref) + bound))
    for sp, c in convs:
        _check_conv(c, split=sp)


# ------------------------------------------------------------- call structure --

@pytest.mark.parametrize("compute,dtype,N", [("bf16", torch.float32, 256), ("bf16", torch.bfloat16, 101),
                                             ("e4m3", torch.float32, 256), ("f64", torch.float64, 40)])
def test_first_kernel_clears_the_error_word(compute, dtype, N):
    """A workspace that holds a stale status gives a clean one, whichever kernel comes first."""
    g = torch.Generator(device=DEV).manual_seed(N)
    A = torch.randn(64, 320, device=DEV, generator=g).to(dtype)
    B = torch.randn(320, N, device=DEV, generator=g).to(dtype)
    ws = torch.full((pj.gemm_workspace_size(64, N, 320, 8, 8, compute=compute),), 7, dtype=torch.uint8, device=DEV)
    pj.proj_gemm(A, B, 8, 8, compute=compute, workspace=ws)
    pj.check(ws)


@pytest.mark.parametrize("case", ["bf16", "bf16-odd", "e4m3", "f64", "conv"])
def test_captured_call_replays(case):
    """A captured call (launches that overlap their predecessors included) replays on new
    inputs with the results of a plain call."""
    g = torch.Generator(device=DEV).manual_seed(11)
    if case == "conv":
        x, y = torch.empty(9000, device=DEV), torch.empty(24, 512, device=DEV)
        out = torch.empty(9000 - 511, 24, device=DEV)
        call = lambda o: pj.proj_conv(x, y, 128, out=o)  # noqa: E731
    else:
        dt = torch.float64 if case == "f64" else torch.float32
        x, y = torch.empty(400, 1000, dtype=dt, device=DEV), torch.empty(1000, 301 if case == "bf16-odd" else 512,
                                                                         dtype=dt, device=DEV)
        # (BF16 outputs: no partial products, whose order of addition may differ)
        out = torch.empty(400, y.shape[1], dtype=dt if case == "f64" else torch.bfloat16, device=DEV)
        call = lambda o: pj.proj_gemm(x, y, 8, 4, compute=case.split("-")[0], out_dtype=o.dtype, out=o)  # noqa: E731
    x.normal_(generator=g)
    y.normal_(generator=g)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        call(out)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        call(out)
    for _ in range(3):
        x.normal_(generator=g)
        y.normal_(generator=g)
        out.zero_()
        graph.replay()
        assert torch.equal(out, call(torch.empty_like(out)))
