"""The running mean's kernels at the sizes where they change shape, against the FP64 oracle:
windows on both sides of the chunk lengths that take four or eight values per thread, of one
bin, of less than a warp and of one part of a CTA's outputs; ragged last chunks; spectra that
start beside a 16-byte boundary.  Tolerance 1e-12 relative per bin, as for every estimator."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2602_18560_gb300 import gbsub, synth

pytestmark = pytest.mark.gpu

CASES = [(1, 40), (31, 1000), (32, 1024), (255, 5001), (257, 4097), (1024, 9999), (1025, 9999),
         (4096, 20_003), (4097, 20_003), (8192, 30_001)]


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    gbsub.lib()


def spectrum(n, seed):
    rng = np.random.default_rng(seed)
    P = 1e-40 * rng.exponential(size=n) * 10 ** rng.uniform(-8, 8, n)
    P[rng.random(n) < 0.2] = 0.0
    return P


def rel_err(got, ref):
    assert np.all(got[ref == 0] == 0)
    nz = ref != 0
    return float(np.max(np.abs(got[nz] - ref[nz]) / ref[nz])) if nz.any() else 0.0


@pytest.mark.parametrize("W, n", CASES)
@pytest.mark.parametrize("offset", [0, 1])
def test_no_alloc_mean_of_any_alignment(W, n, offset):
    import torch
    P = spectrum(n, W)
    x = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
    x[offset:offset + n] = torch.from_numpy(P)
    out = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
    rc = gbsub.lib().sub_running_mean_noalloc(
        ctypes.c_void_p(x.data_ptr() + 8 * offset), ctypes.c_void_p(out.data_ptr() + 8 * offset),
        n, W, torch.cuda.current_stream().cuda_stream)
    assert rc == gbsub.OK
    got = out.cpu().numpy()[offset:offset + n]
    assert rel_err(got, oracle.smooth(gbsub.MEAN, W, P)) <= 1e-12
    assert out.cpu().numpy()[n if offset == 0 else 0] == 0.0  # nothing beside the output


@pytest.mark.parametrize("W", [31, 1025, 4096, 4097])
def test_mean_of_a_runs_spectrum(W):
    # the run's own spectrum as the input: its power and its S_gal belong together
    T, f_max = synth.YEAR, 1e-3
    A, f, fdot = synth.catalog(40_000, 3, synth.Population(2.5, 2.0))
    with gbsub.Subtraction(T_obs=T, window=W, estimator=gbsub.MEAN, f_max=f_max) as s:
        s.load(A * 2.0, f, fdot)
        s.run()
        P, sg = s.power(), s.spectrum()
    assert rel_err(sg, oracle.smooth(gbsub.MEAN, W, P)) <= 1e-12
