"""Correlations in a batch: every run length of the box projection, and samples that are not
finite, against the FP64 oracle within the bounds of test_gpu_batch.py."""
import numpy as np
import pytest
import torch

import oracle
import paper_1411_2860_gb300 as pj
from helpers import U_BF16, conv_abs_entries, gamma
from test_gpu_batch import _check_conv, _check_gemm, _conv_case, _desc, _gemm_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [1, 2])
@pytest.mark.parametrize("Lb", [1, 2, 4, 8, 16, 32, 64])
def test_run_lengths(Lb, split):
    """Signals that end inside a run, a warp's 256 positions and a block's 2048, and one that
    starts off its 16-byte boundary."""
    rng = np.random.default_rng(Lb)
    convs = []
    for lags, nt, R, skip in ((1, 1, 64, 0), (Lb + 1, 2, 64, 0), (257 * Lb + 3, 1, 128, 1), (5001, 3, 64, 3),
                              (2048 * Lb + 511, 1, 64, 2)):
        T = R * Lb
        c = _conv_case(rng, lags + T - 1 + skip, T, nt, R, lags)
        c["s"] = c["s"][skip:]
        c["out"] = c["out"][skip:]
        convs.append(c)
    plan = pj.BatchPlan([pj.batch_conv(c["s"], c["k"], c["out"], c["R"], split=split) for c in convs])
    plan.run()
    plan.check()
    for i, c in enumerate(convs):
        _check_conv(c, seed=i, split=split)


@pytest.mark.parametrize("split", [1, 2])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("Lb,R,at", [(1, 256, 2600), (1, 64, 1000), (4, 64, 3001)])
def test_sample_that_is_not_finite(Lb, R, at, value, split):
    """It reaches only the rows of 128 lags (of one phase) whose zero-extended window, the
    reduced template and 127 zeros in whole chunks of 64, holds it."""
    T = R * Lb
    c = _conv_case(np.random.default_rng(at), 6000, T, 1, R, at)
    s = c["s"].double().cpu().numpy()
    k = c["k"].double().cpu().numpy()
    s[at] = 0.0
    c["s"][at] = value
    plan = pj.BatchPlan([pj.batch_conv(c["s"], c["k"], c["out"], R, split=split)])
    plan.run()
    plan.check()
    lag = np.arange(6000 - T + 1)
    phi, row = lag % Lb, lag // Lb // 128
    span = -(-(R + 127) // 64) * 64
    clear = (at < phi + 128 * Lb * row) | (at >= phi + Lb * (128 * row + span))
    assert clear.any() and not clear.all()
    mm, tt = lag[clear], np.zeros(clear.sum(), dtype=int)
    ref = oracle.conv_proj_entries(s, k, mm, tt, R, "haar", 64)
    lead = 4 * U_BF16 ** 2 if split == 2 else 2 * U_BF16 + U_BF16 ** 2
    f = lead + (2 * gamma(Lb) + 2 * gamma((3 if split == 2 else 1) * (R + 128))) * (1 + U_BF16) ** 2
    got = c["out"].double().cpu().numpy()[:, 0]
    assert np.all(np.abs(got[clear] - ref) <= f * conv_abs_entries(s, k, R, mm, tt))
    hit = (lag <= at) & (at < lag + T)   # the lags whose window holds the sample
    assert not np.isfinite(got[hit]).any()


@pytest.mark.parametrize("split", [1, 2])
@pytest.mark.parametrize("products,shape,lags", [(2, (200, 300, 500), (60000, 33000, 5)), (6, (1000, 520, 2048), (700,)),
                                                 (1, (64, 64, 64), (1,))])
def test_beside_products(products, shape, lags, split):
    """Few products beside long correlations (one launch on solo CTAs), and the other way
    round (products on CTA pairs, the correlations in a launch of their own)."""
    rng = np.random.default_rng(products)
    gemms = [_gemm_case(rng, *shape, 8, 8, split) for _ in range(products)]
    convs = [_conv_case(rng, n + 255, 256, 1, R, n) for n in lags for R in (256, 64)]
    plan = pj.BatchPlan([_desc(c) for c in gemms] +
                        [pj.batch_conv(c["s"], c["k"], c["out"], c["R"], split=split) for c in convs])
    for _ in range(2):
        plan.run()
        plan.check()
    for c in gemms:
        _check_gemm(c)
    for i, c in enumerate(convs):
        _check_conv(c, seed=i, split=split)
