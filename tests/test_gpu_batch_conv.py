"""Correlations in a batch: every run length of the box projection, against the FP64 oracle
within the bounds of test_gpu_batch.py."""
import numpy as np
import pytest

import paper_1411_2860_gb300 as pj
from test_gpu_batch import _check_conv, _conv_case

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
