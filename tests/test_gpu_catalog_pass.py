"""The catalog pass over a stored catalog (through the C ABI) against the FP64 oracle, where its
paths change: observation times of few and of many mantissa bits, sources on and beside the
edges of their bins, catalogs on both sides of the size from which the first bins are added up
in shared memory (removals there included), and ragged ends of a step of 64 sources."""
import numpy as np
import pytest

import oracle
from paper_2602_18560_gb300 import gbsub, synth
from test_gpu_parity import compare_run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    gbsub.lib()


def amplitude(T, k_lo, n, j, p):
    """A of a single-bin source of power p S_instr in bin j."""
    S, R = oracle.tables(T, k_lo, n, True)
    return np.sqrt(5.0 * p * S[j] / (T * R[j]))


@pytest.mark.parametrize("T", [2.0**25, synth.YEAR, 1.87654321 * synth.YEAR, 1e8 / 3.0,
                               np.nextafter(2.0**25, 0.0)])
def test_bins_at_their_edges(T):
    f_max = 1.5e-3
    k_lo, n = oracle.grid(T, 1e-4, f_max)
    rng = np.random.default_rng(5)
    j = rng.integers(-3, n + 3, 60_000)
    off = rng.choice([-0.5, 0.0, 0.5], j.size) + rng.choice([0.0, 1e-9, -1e-9, 1e-6, -1e-6, 1e-3],
                                                            j.size)
    f = (k_lo + j + off) / T
    fdot = rng.choice([0.0, 1.0, -1.0, 0.0], j.size) * 10 ** rng.uniform(-12, 0, j.size) / T**2
    # a sweep that leaves its bin by less than the certificate's margin is a matter of 1e-6 of
    # its power; keep the sources that move away from the edge they sit on
    frac = f * T - np.floor(f * T + 0.5)
    fdot = np.where(np.abs(frac) > 0.499, -np.sign(frac) * np.abs(fdot), fdot)
    A = amplitude(T, k_lo, n, np.clip(j, 0, n - 1), rng.gamma(2.0, size=j.size))
    for est in (gbsub.MEAN, gbsub.MEDIAN):
        compare_run(A, f, fdot, T, est, 101, f_max=f_max)


@pytest.mark.parametrize("N", [999_999, 1_000_000, 1_000_063])
def test_first_bins_in_shared_memory(N):
    T, f_max = synth.YEAR, 4e-4
    k_lo, n = oracle.grid(T, 1e-4, f_max)  # 9 468 bins, the first 4 096 of them kept
    rng = np.random.default_rng(6)
    # a third of the sources in 40 bins (their words carry), some loud ones in and beyond the
    # first 4 096 bins
    j = np.where(rng.random(N) < 0.3, rng.integers(0, 40, N), rng.integers(0, n, N))
    p = 1e-3 * rng.gamma(2.0, size=N)
    p[rng.integers(0, N, 400)] = 10 ** rng.uniform(1.5, 4.0, 400)
    A = amplitude(T, k_lo, n, j, p)
    f = (k_lo + j + rng.uniform(-0.4, 0.4, N)) / T
    st, _, res, _ = compare_run(A, f, np.zeros(N), T, gbsub.MEDIAN_MEAN, 200, f_max=f_max)
    assert res[j < 4096].sum() > 20 and res[j >= 4096].sum() > 20
