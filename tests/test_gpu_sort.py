"""The chunk sort's two orders, through the running median (a selection: the oracle's doubles,
bit for bit): spectra whose values differ in the lowest bits only, which the first order leaves
out, alone and beside ordinary values, with ties; every sort width and number of elements per
thread."""
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


def spectra(n):
    rng = np.random.default_rng(n)
    base = np.float64(3.0e-41).view(np.uint64) & ~np.uint64(0x1FFF)
    low = (base + rng.integers(0, 8192, n).astype(np.uint64)).view(np.float64)
    some = np.where(rng.random(n) < 0.5, low, 1e-41 * rng.exponential(size=n))
    ties = (base + rng.integers(0, 4, n).astype(np.uint64)).view(np.float64)
    down = (base + (np.arange(n)[::-1] % 8192).astype(np.uint64)).view(np.float64)
    return low, some, ties, down


@pytest.mark.parametrize("W", [20, 100, 400, 1000, 2000, 4000, 8000])
def test_values_that_differ_in_the_lowest_bits(W):
    n = 3 * W + 777
    k_lo = int(np.ceil(1e-4 * T))
    f_max = (k_lo + n - 1 + 0.25) / T
    with gbsub.Subtraction(T_obs=T, window=W, estimator=gbsub.MEDIAN, f_max=f_max) as s:
        for P in spectra(n):
            ref = oracle.smooth(gbsub.MEDIAN, W, P)
            for e in (0, 2, 4, 8):
                try:
                    gbsub.sub_set_tuning(s.ctx, gbsub.TUNE_SORT_E, e)
                except gbsub.SubError:
                    continue  # not a width this window allows
                np.testing.assert_array_equal(s.estimate(P), ref)


@pytest.mark.parametrize("W", [100, 200, 500, 1100, 2000])
def test_passes_of_the_second_order_do_not_overlap(W):
    # every chunk of a band of many takes the second order (three sorts on the same two exchange
    # buffers), several CTAs to an SM: 64, 128, 256 and twice 1024 threads, that is 1, 3, 6 and 15
    # exchanges a sort, odd numbers but for the third
    L, reps = 8 * W, 40  # L values over and over, so that the oracle does three times as many
    n = reps * L
    k_lo = int(np.ceil(1e-4 * T))
    f_max = (k_lo + n - 1 + 0.25) / T
    low = spectra(L)[0]
    r = oracle.smooth(gbsub.MEDIAN, W, np.tile(low, 3))
    ref = np.concatenate([r[:L], np.tile(r[L:2 * L], reps - 2), r[2 * L:]])
    with gbsub.Subtraction(T_obs=T, window=W, estimator=gbsub.MEDIAN, f_max=f_max) as s:
        for _ in range(3):
            np.testing.assert_array_equal(s.estimate(np.tile(low, reps)), ref)
