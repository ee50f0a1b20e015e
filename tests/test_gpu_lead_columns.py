"""Split products with lo terms on the leading projections alone, at the group counts and
columns where the staged runs of an odd l + 1 begin and end."""
import pytest
import torch

from test_gpu_gemm import test_bf16_split_lead_parity as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lead", [1, 2, 3, 4])
@pytest.mark.parametrize("lp1", [3, 5, 6, 7])
@pytest.mark.parametrize("M,N,K", [(40, 256, 160), (33, 300, 168), (70, 512, 1016), (64, 260, 100)])
def test_odd_runs_with_lead_terms(M, N, K, lp1, lead):
    """Whole quads of groups, a last quad of one and of three, a partial last group; columns
    that end inside a warp's 32."""
    check(M, N, K, 8, lp1, lead)
    torch.cuda.synchronize()
