"""Products on either side of the lines between whole and shared tiles, and a shared product
replayed from a graph, against the FP64 oracle within the bounds of helpers.py."""
import numpy as np
import pytest
import torch

import oracle
import paper_1411_2860_gb300 as pj
from helpers import factor, gemm_abs_product
from test_gpu_gemm import _bf16_case
from test_gpu_gemm_e4m3 import _e4m3_case

pytestmark = pytest.mark.gpu


def _shared(tiles, stages, sms):
    """The rule for products without lo terms (common.hpp, use_stream_k)."""
    if stages < 16 or tiles * stages < 16 * sms:
        return False
    return 2 * tiles < sms or (10 * tiles < 9 * sms and stages * (sms - tiles) >= 32 * sms)


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _within(Y, ref, bound):
    assert np.all(np.abs(Y - ref) <= bound), np.nanmax(np.abs(Y - ref) / bound)


# Tiles of 64 rows, the smallest height, in odd and even numbers of tile columns.
@pytest.mark.parametrize("rows,cols,stages,shared", [
    (25, 3, 40, True), (26, 3, 40, False),       # half a wave
    (27, 3, 68, False), (27, 3, 69, True),       # 32 stages taken off every SM
    (20, 4, 67, False), (20, 4, 68, True),       # the same on tile columns that pair up
    (34, 4, 100, False),
])
def test_bf16_lines(rows, cols, stages, shared):
    if _sms() == 152:
        assert _shared(rows * cols, stages, 152) == shared
    _within(*_bf16_case(64 * rows - 5, 128 * cols - 3, 64 * stages - 9, 8, 8, 1))


@pytest.mark.parametrize("split,stages,shared", [(1, 68, False), (1, 69, True), (2, 66, False), (2, 69, True)])
def test_e4m3_lines(split, stages, shared):
    """81 tiles of 64 rows; a split chunk of 128 components is three stages."""
    if _sms() == 152:
        assert _shared(81, stages, 152) == shared
    chunks = stages // (3 if split == 2 else 1)
    _within(*_e4m3_case(64 * 27 - 5, 381, 128 * chunks - 9, 8, 8, split))


def test_shared_product_replays():
    """The zeroing of the output and the launch that overlaps it, from a graph."""
    M, N, K = 300, 300, 10496      # 15 tiles of 164 stages
    assert _shared(15, 164, _sms())
    g = torch.Generator(device="cuda").manual_seed(3)
    x, y = torch.empty(M, K, device="cuda"), torch.empty(K, N, device="cuda")
    out = torch.empty(M, N, device="cuda")
    ws = torch.empty(pj.gemm_workspace_size(M, N, K, 8, 8), dtype=torch.uint8, device="cuda")
    x.normal_(generator=g)
    y.normal_(generator=g)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        pj.proj_gemm(x, y, 8, 8, out=out, workspace=ws)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        pj.proj_gemm(x, y, 8, 8, out=out, workspace=ws)
    C, D = oracle.basis("dct2", 8)
    for _ in range(3):
        x.normal_(generator=g)
        y.normal_(generator=g)
        out.fill_(float("nan"))
        graph.replay()
        pj.check(ws)
        A, B = x.double().cpu().numpy(), y.double().cpu().numpy()
        absprod, Kp = gemm_abs_product(A, B, 8, C, D, 8)
        _within(out.double().cpu().numpy(), oracle.gemm_proj(A, B, 8, 8, "dct2", 8), factor(Kp, 8, 1) * absprod)
