"""The catalog pass over a stored catalog (through the C ABI) against the FP64 oracle, where its
paths change: observation times of few and of many mantissa bits, sources on and beside the
edges of their bins, catalogs on both sides of the size from which the first bins are added up
in shared memory (removals there included), and ragged ends of a step of 64 sources."""
import numpy as np
import pytest

import oracle
from paper_2602_18560_gb300 import gbsub, synth
from test_gpu_parity import RTOL, compare_run, rel_err

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


@pytest.mark.parametrize("T", [synth.YEAR, 1.87654321 * synth.YEAR, 1e8 / 3.0,
                               np.nextafter(2.0**25, 0.0)])
@pytest.mark.parametrize("est", [gbsub.MEAN, gbsub.MEDIAN])
def test_sweeps_down_from_an_edge_are_removed_whole(T, est):
    # loud sources that start on the upper edge of their bin, or a few doubles beside it, and move
    # down: FP64 gives the bin above a share of the sweep (none, on the edge), whatever a product
    # of fewer bits says.  They are resolved, and what is taken away is what was deposited, in
    # bins that nothing else is in.
    f_max = 1.5e-3
    k_lo, n = oracle.grid(T, 1e-4, f_max)
    rng = np.random.default_rng(12)
    j = np.arange(20, n - 40, 64)
    f = (k_lo + j + 0.5) / T
    ulps = rng.integers(-2, 3, j.size)
    for step in range(2):
        f = np.where(ulps > step, np.nextafter(f, np.inf), f)
        f = np.where(ulps < -step, np.nextafter(f, 0.0), f)
    fdot = -10 ** rng.uniform(-5.0, np.log10(0.5), j.size) / T**2
    A = amplitude(T, k_lo, n, j, np.full(j.size, 1e4))
    jb = np.arange(8, n, 16)  # a faint background beside them
    jb = jb[(jb - 20) % 64 > 1]
    A = np.append(A, amplitude(T, k_lo, n, jb, 0.05 * rng.gamma(2.0, size=jb.size)))
    f, fdot = np.append(f, (k_lo + jb) / T), np.append(fdot, np.zeros(jb.size))
    _, _, res, _ = compare_run(A, f, fdot, T, est, 101, f_max=f_max)
    assert res[:j.size].all() and not res[j.size:].any()
    with gbsub.Subtraction(T_obs=T, window=101, estimator=est, f_max=f_max) as s:
        s.load(A, f, fdot)
        s.run()
        P = s.power()
    S, R = oracle.tables(T, k_lo, n, True)
    keep = ~res
    ref = oracle.power(T, R, oracle.deposit(T, k_lo, n, A[keep], f[keep], fdot[keep]))
    assert rel_err(P, ref) <= RTOL


@pytest.mark.parametrize("turns", [1, 2, 5])
def test_bands_beyond_32_bit_bins(turns):
    # a band that begins at bin 2^32 turns + 3000: a source of bin 3500 is far below it
    T = 2.0**33 * turns
    k0, n = 2**32 * turns + 3000, 2000
    f_min, f_max = k0 / T, (k0 + n - 1) / T
    k_lo, nb = oracle.grid(T, f_min, f_max)
    assert (k_lo, nb) == (k0, n)
    j = np.append(np.arange(0, n, 3), [700, 701])
    p = np.append(np.full(j.size - 2, 0.1), [1e4, 1e4])
    A = amplitude(T, k0, n, j, p)
    f = (k0 + j + 0.125) / T
    low = np.array([2900.0, 3500.0, 4000.25, 4999.0])  # bins a 32-bit difference puts in the band
    A, f = np.append(A, np.full(low.size, 30.0 * A.max())), np.append(f, low / T)
    for est in (gbsub.MEAN, gbsub.MEDIAN):
        _, _, res, _ = compare_run(A, f, np.zeros(f.size), T, est, 51, f_max=f_max, f_min=f_min)
        assert res.sum() == 2 and not res[j.size:].any()


@pytest.mark.parametrize("N", [1, 15, 16, 17, 47])
def test_the_mask_is_cleared_to_its_last_byte(N):
    # one context: every source resolved, then none, in a mask that does not end on 16 bytes
    T = synth.YEAR
    k_lo, n = oracle.grid(T, 1e-4, 1e-3)
    j = 100 + 200 * np.arange(N)
    f = (k_lo + j) / T
    with gbsub.Subtraction(T_obs=T, window=101, estimator=gbsub.MEDIAN, f_max=1e-3) as s:
        for p, want in ((1e4, 1), (1e-2, 0), (1e4, 1), (1e-2, 0)):
            s.load(amplitude(T, k_lo, n, j, p), f, np.zeros(N))
            s.run()
            assert np.array_equal(s.resolved(), np.full(N, want, np.uint8))
