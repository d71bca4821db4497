"""The median tiles' CTA sizes: windows on both sides of the line up to which every-tile launches
and contexts that share the GPU take 256 threads, against the oracle (a selection: its doubles,
bit for bit) and against the other sizes."""
import numpy as np
import pytest

import oracle
from paper_2602_18560_gb300 import gbsub, synth

pytestmark = pytest.mark.gpu

T = synth.YEAR


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    gbsub.lib()


@pytest.mark.parametrize("W", [200, 511, 513, 1000, 1024, 1025, 2000])
def test_sizes(W):
    n = 5 * W + 333
    k_lo = int(np.ceil(1e-4 * T))
    rng = np.random.default_rng(W)
    P = np.where(rng.random(n) < 0.7, 1e-41 * rng.exponential(size=n), 0.0)
    ref = oracle.smooth(gbsub.MEDIAN, W, P)
    m = 4000
    A, f, fdot = (10.0 ** rng.uniform(-23, -20, m), (k_lo + rng.uniform(1, n - 2, m)) / T,
                  np.zeros(m))
    runs = []
    with gbsub.Subtraction(T_obs=T, window=W, estimator=gbsub.MEDIAN,
                           f_max=(k_lo + n - 1 + 0.25) / T) as s:
        s.load(A, f, fdot)
        for div in (1, 2, 4):
            gbsub.sub_set_grid_div(s.ctx, div)
            for th in (0, 256, 512):
                gbsub.sub_set_tuning(s.ctx, gbsub.TUNE_MEDIAN_THREADS, th)
                np.testing.assert_array_equal(s.estimate(P), ref)
                s.run()
                runs.append((s.spectrum().copy(), s.resolved().copy()))
    for S, res in runs[1:]:
        np.testing.assert_array_equal(S, runs[0][0])
        np.testing.assert_array_equal(res, runs[0][1])
