"""FP64 products over the tile sizes and the row counts their launch takes, against the FP64
oracle within the bound of two FP64 evaluations."""
import numpy as np
import pytest
import torch

import oracle
import paper_1411_2860_gb300 as pj
from helpers import gamma, gemm_abs_product

pytestmark = pytest.mark.gpu


def _check(M, N, K, lp1):
    rng = np.random.default_rng(M + N + K)
    A, B = rng.normal(size=(M, K)), rng.normal(size=(K, N))
    Y = pj.proj_gemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), 8, lp1).cpu().numpy()
    C, D = oracle.basis("dct2", 8)
    absprod, Kp = gemm_abs_product(A, B, 8, C, D, lp1)
    # both sides round: two 8-term projections (their coefficients to an ulp) and Kp terms
    bound = 2 * gamma(Kp + 2 * 8 + 4, 2.0 ** -53) * absprod
    err = np.abs(Y - oracle.gemm_proj(A, B, 8, lp1, "dct2", 8))
    assert np.all(err <= bound), np.nanmax(err / bound)


@pytest.mark.parametrize("M,N,K,lp1", [(600000, 1, 8, 8), (600000, 40, 16, 4), (1100000, 8, 8, 8), (1100000, 16, 8, 8)])
def test_tall_product(M, N, K, lp1):
    """More rows of tiles than the second grid dimension takes (65,535), at every tile size
    the rule picks for few columns."""
    _check(M, N, K, lp1)


@pytest.mark.parametrize("M,N", [(304, 128), (303, 127), (305, 129), (608, 256), (607, 255), (609, 257)])
@pytest.mark.parametrize("K", [7, 32, 33, 130])
def test_larger_tiles(M, N, K):
    """Outputs that take 16 x 16 and 32 x 32 tiles (152 and 152 of them), and their neighbours."""
    _check(M, N, K, 8)
