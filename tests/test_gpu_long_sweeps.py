"""Sources whose sweeps go through the tree of bins (more than 512 bins), through the C ABI,
against the FP64 oracle: sweeps on both sides of the line, starting and ending on and beside
the nodes' edges (32, 1024 and 32768 bins), running out of the band at either end, covering all
of it, and downward; faint and loud, so that some are removed again.  S_gal within 1e-10 of the
oracle's in every bin, and the resolved set, iterations and counts the oracle's, as for every
other run."""
import numpy as np
import pytest

import oracle
from paper_2602_18560_gb300 import gbsub, synth
from test_gpu_parity import RTOL, compare_run, rel_err

pytestmark = pytest.mark.gpu

T = 4 * synth.YEAR
F_MAX = 7e-4                      # 75 738 bins: two nodes of level 3, an incomplete last one


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    gbsub.lib()


def sweeps(n):
    """(first, length) of every sweep in bins relative to the band."""
    out = [(-0.3, n + 5.0), (0.2, n - 1.4), (-700.0, 1300.25), (-40000.0, 90000.0),
           (n - 600.0, 5000.0), (n - 513.0, 600.0), (n + 300.0, -2000.5), (n - 1.0, -n + 2.0)]
    for length in (500.0, 510.6, 511.0, 511.4, 512.0, 512.6, 513.0, 514.2, 600.0, 1023.7, 2100.3,
                   33000.5, 66000.0):
        for first in (31.5, 32.0, 32.5, 1023.4, 1024.0, 1056.5, 32767.5, 32768.0, 4321.123):
            if first + length < n + 400:
                out.append((first, length))
                out.append((first + length, -length))
    return np.array(out)


def catalog(est_seed):
    k_lo, n = oracle.grid(T, 1e-4, F_MAX)
    S, R = oracle.tables(T, k_lo, n, True)
    ratio = R / S
    sw = sweeps(n)
    f = (k_lo + sw[:, 0]) / T
    fdot = sw[:, 1] / T**2
    rng = np.random.default_rng(est_seed)
    # rho_0 from 2 to 60, from the mean response over the sweep's bins inside the band
    rho0 = 2.0 * 30.0 ** rng.random(len(sw))
    A = np.empty(len(sw))
    for i, (a, d) in enumerate(sw):
        lo, hi = max(0, int(min(a, a + d))), min(n, int(max(a, a + d)) + 1)
        A[i] = rho0[i] / np.sqrt(0.8 * T * ratio[lo:hi].sum() / abs(d))
    # a dense background, some of it resolvable
    j = np.repeat(np.arange(n), 2)
    bg = np.sqrt(5.0 * 0.05 * rng.gamma(2.0, size=2 * n) * S[j] / (T * R[j]))
    bg[::997] *= 30.0
    return (np.concatenate([A, bg]), np.concatenate([f, (k_lo + j + 0.1) / T]),
            np.concatenate([fdot, np.zeros(2 * n)]))


@pytest.mark.parametrize("est, W", [(gbsub.MEAN, 400), (gbsub.MEDIAN, 101), (gbsub.MEDIAN, 1024),
                                    (gbsub.MEDIAN_MEAN, 257)])
def test_long_sweeps_against_the_oracle(est, W):
    A, f, fdot = catalog(41 + W)
    st, _, res, _ = compare_run(A, f, fdot, T, est, W, f_max=F_MAX)
    n_sweeps = len(sweeps(st.n_bins))
    assert 5 < res[:n_sweeps].sum() < n_sweeps  # some removed, some not
    assert st.iterations >= 2


def test_long_sweeps_other_precisions():
    A, f, fdot = catalog(7)
    prm = oracle.make_params(T_obs=T, estimator=gbsub.MEDIAN_MEAN, window=257, f_max=F_MAX)
    ref = oracle.run(prm, A, f, fdot)
    for precision, tol in ((gbsub.FP64_STRICT, RTOL), (gbsub.MIXED, 1e-5)):
        with gbsub.Subtraction(T_obs=T, estimator=gbsub.MEDIAN_MEAN, window=257, f_max=F_MAX,
                               precision=precision) as s:
            s.load(A, f, fdot)
            st = s.run()
            assert np.sum(s.resolved().astype(bool) != ref["resolved"]) <= st.n_uncertain
            if st.n_uncertain == 0:
                assert rel_err(s.spectrum(), ref["S_gal"]) <= tol
            # the residual power is the tree's and the bins' together
            P = s.power()
            assert np.all(P > 0)


def test_power_beyond_the_range_is_still_refused():
    # one sweep of 2000 bins whose power passes 2^63 S_instr in every bin: as bin by bin
    k_lo, n = oracle.grid(T, 1e-4, F_MAX)
    S, R = oracle.tables(T, k_lo, n, True)
    A = np.array([np.sqrt(5.0 * 2.0**66 * 2000.0 * np.max(S / R) / T)])
    with gbsub.Subtraction(T_obs=T, window=100, estimator=gbsub.MEAN, f_max=F_MAX) as s:
        s.load(A, np.array([(k_lo + 3000.0) / T]), np.array([2000.0 / T**2]))
        with pytest.raises(gbsub.SubError) as ei:
            s.run()
        assert ei.value.code == gbsub.ERANGE


@pytest.mark.parametrize("first, length", [(-20.3, 75_838.7), (3000.2, 5000.4), (40000.4, -5100.1)])
@pytest.mark.parametrize("delta", [1e-6, -1e-6, 3e-8, -3e-8])
def test_decisions_left_open_by_the_screen(first, length, delta):
    # one long sweep at rho = rho_th (1 + delta) on a faint background: its FP32 screen cannot
    # tell, the FP64 sum of the whole CTA does
    k_lo, n = oracle.grid(T, 1e-4, F_MAX)
    S, R = oracle.tables(T, k_lo, n, True)
    j = np.arange(n)
    f = np.append((k_lo + j + 0.1) / T, (k_lo + first) / T)
    fdot = np.append(np.zeros(n), length / T**2)
    A = np.append(np.sqrt(5.0 * 0.1 * S / (T * R)), 1e-23)
    for _ in range(8):  # the sweep's own power moves S_gal a little
        P = oracle.power(T, R, oracle.deposit(T, k_lo, n, A, f, fdot))
        rho2 = oracle.snr2(T, k_lo, n, S, R, oracle.smooth(gbsub.MEAN, 1001, P), A[-1:], f[-1:],
                           fdot[-1:])[0]
        A[-1] *= 7.0 * (1.0 + delta) / np.sqrt(rho2)
    kw = dict(T_obs=T, estimator=gbsub.MEAN, window=1001, f_max=F_MAX)
    ref = oracle.run(oracle.make_params(**kw), A, f, fdot)
    assert bool(ref["resolved"][-1]) == (delta > 0)
    with gbsub.Subtraction(**kw) as s:
        s.load(A, f, fdot)
        st = s.run()
        res = s.resolved().astype(bool)
    assert st.n_exact > 0
    assert np.array_equal(res, ref["resolved"])


@pytest.mark.parametrize("first, length", [(-20.3, 75_838.7), (3000.2, 5000.4), (70_000.4, -66_000.1)])
@pytest.mark.parametrize("side", [-1.0, 1.0])
def test_open_decisions_have_the_precision_of_fp64(first, length, side):
    # rho_th^2 at 1.5e-15 on either side of the rho^2 that the run's own tables and S_gal give in
    # more than 64 bits.  A sum of correctly rounded quotients in 256 parts of at most 300 is off by
    # some 3e-16 (one rounding of the mean of the parts' errors, the last sums and products, and
    # rho_th^2); quotients of 43 bits, always too small, by 3e-15.
    k_lo, n = oracle.grid(T, 1e-4, F_MAX)
    S, R = oracle.tables(T, k_lo, n, True)
    j = np.arange(n)
    f = np.append((k_lo + j + 0.1) / T, (k_lo + first) / T)
    fdot = np.append(np.zeros(n), length / T**2)
    lo, hi = sorted((first, first + length))
    A = np.append(np.sqrt(5.0 * 0.1 * S / (T * R)),
                  10.0 / np.sqrt(0.8 * T * (R / S)[max(0, int(lo)):int(hi)].sum() / (hi - lo)))
    kw = dict(T_obs=T, estimator=gbsub.MEAN, window=1001, f_max=F_MAX)
    with gbsub.Subtraction(rho_th=9.99, **kw) as s:  # rho is below rho_0 = 10: not resolved
        s.load(A, f, fdot)
        s.run()
        assert not s.resolved().any()
        Sg = s.spectrum()
        S, R = s.tables()
    # the oracle's sweep and weights, the sum in long doubles
    u0 = f[-1] * T
    u1 = u0 + fdot[-1] * (T * T)
    lo, hi = min(u0, u1), max(u0, u1)
    k = np.arange(max(k_lo, int(np.floor(lo + 0.5))),
                  min(k_lo + n - 1, int(np.floor(hi + 0.5))) + 1)
    w = ((np.minimum(hi, k + 0.5) - np.maximum(lo, k - 0.5)) / (hi - lo)).clip(0.0)
    X = np.longdouble
    terms = R[k - k_lo].astype(X) * w.astype(X) / (S[k - k_lo] + Sg[k - k_lo]).astype(X)
    rho2 = X(4.0) * X(T / 5.0) * X(A[-1]) * X(A[-1]) * terms.sum()
    rho_th = float(np.sqrt(rho2 * (X(1.0) + X(side * 1.5e-15))))
    with gbsub.Subtraction(rho_th=rho_th, **kw) as s:
        s.load(A, f, fdot)
        st = s.run()
        res = s.resolved().astype(bool)
    assert st.n_exact > 0 and st.n_near > 0
    assert res[-1] == (side < 0) and not res[:-1].any()


@pytest.mark.parametrize("precision", [gbsub.FP64, gbsub.MIXED])
def test_the_check_measures_the_screen_that_decides(precision):
    # sweeps of 4 to 240 000 bins about the threshold (rho from 6.9999 to 7.0001 on the first
    # estimate).  The check's FP32 value is the one the run decides on, within the bound of its own
    # roundings of the FP64 one: a lane's chain and five levels for a sweep summed by a warp, 26
    # (and one for every 32 nodes of the highest level) for one of more than 512 bins
    f_max = 2e-3
    k_lo, n = oracle.grid(T, 1e-4, f_max)
    S, R = oracle.tables(T, k_lo, n, True)
    rng = np.random.default_rng(3)
    ln = np.append(10 ** rng.uniform(0.6, 5.2, 300), [n + 50.0, n - 3.0])
    first = np.append(rng.uniform(0, 1, 300) * np.maximum(n - ln[:300] - 2, 1.0), [-20.0, 1.2])
    A = np.empty(ln.size)
    for i in range(ln.size):
        lo, hi = max(0, int(first[i])), min(n, int(first[i] + ln[i]) + 1)
        A[i] = 1e-3 / np.sqrt(0.8 * T * (R / S)[lo:hi].sum() / ln[i])
    j = np.arange(n)
    bg = np.sqrt(5.0 * 0.3 * rng.gamma(2.0, size=n) * S / (T * R))
    f = np.append((k_lo + first) / T, (k_lo + j + 0.1) / T)
    fdot = np.append(ln / T**2, np.zeros(n))
    kw = dict(T_obs=T, estimator=gbsub.MEAN, window=400, f_max=f_max)
    m = ln.size
    for _ in range(4):
        P = oracle.power(T, R, oracle.deposit(T, k_lo, n, np.append(A, bg), f, fdot))
        rho2 = oracle.snr2(T, k_lo, n, S, R, oracle.smooth(gbsub.MEAN, 400, P), A, f[:m], fdot[:m])
        A *= 7.0 * (1.0 + rng.uniform(-1e-5, 1e-5, m)) / np.sqrt(rho2)
    with gbsub.Subtraction(precision=precision, **kw) as s:
        s.load(np.append(A, bg), f, fdot)
        s.run()
        chk, res = s.snr_check(), s.resolved().astype(bool)
    src = chk["src"]
    assert src.size >= m // 2
    ex, sc, nb = chk["exact"], chk["screen"].astype(np.float64), chk["nbins"]
    steps = np.where(nb > 512, 26 + (n >> 15) // 32,
                     np.where(nb > 4, np.ceil(nb / 32.0) + 5, nb))
    assert np.all(np.abs(sc / ex - 1.0) <= 2.2e-6 + 2e-7 * steps)
    assert res[:m].any() and not res[:m].all()  # (a removal lifts the others over the threshold)
    if precision == gbsub.MIXED:
        assert np.all(sc[~res[src]] <= np.float64(np.float32(49.0)))
