"""Coarse graining by one CTA or a cluster of CTAs per output bin: numbers of bins on both sides of
the line between them, against exactly rounded sums.  A thread adds at most n / 256 terms in
turn (one CTA for a whole bin) or an eighth of that, then fifteen more roundings: rel 1e-13 for positive
values is some ten times that at the sizes here."""
import math

import numpy as np
import pytest

import oracle
from paper_2602_18560_gb300 import gbsub, synth

pytestmark = pytest.mark.gpu

T = synth.YEAR


@pytest.mark.parametrize("nbins", [1, 3, 100, 101, 102, 400, 5000])
def test_both_forms(nbins):
    import torch
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    k_lo, n = oracle.grid(T)
    x = np.random.default_rng(nbins).exponential(size=n) * 1e-41
    with gbsub.Subtraction(T_obs=T) as s:
        S, f, cnt = s.coarse_grain(x, nbins)
        S2, _, _ = s.coarse_grain(torch.from_numpy(x).cuda(), nbins)
    np.testing.assert_array_equal(S, S2.cpu().numpy())
    assert int(cnt.sum()) == n
    a = np.concatenate([[0], np.cumsum(cnt)])
    for k in range(nbins):
        if cnt[k] == 0:
            assert np.isnan(S[k]) and np.isnan(f[k])
            continue
        ref = math.fsum(x[a[k]:a[k + 1]]) / int(cnt[k])
        assert abs(S[k] - ref) <= 1e-13 * ref
        assert abs(f[k] - (2 * k_lo + a[k] + a[k + 1] - 1) / (2 * T)) <= 1e-14 * f[k]
