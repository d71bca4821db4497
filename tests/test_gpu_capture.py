"""The running mean of a caller's buffers inside a stream capture (its second kernel is launched as
a dependent of the first): replays give the plain call's bits, on the values captured and on new
ones, alone and several in a row."""
import ctypes

import pytest

from paper_2602_18560_gb300 import gbsub

pytestmark = pytest.mark.gpu


def _call(L, x, out, W, stream):
    rc = L.sub_running_mean_noalloc(ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(out.data_ptr()),
                                    x.numel(), W, ctypes.c_void_p(stream))
    assert rc == gbsub.OK, L.sub_last_error(None).decode()


@pytest.mark.parametrize("n,W", [(333, 16), (70001, 8192), (1249681, 1000)])
def test_replays_equal_the_plain_call(n, W):
    import torch
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    L = gbsub.lib()
    gen = torch.Generator(device="cuda").manual_seed(n)
    a = torch.rand(n, dtype=torch.float64, device="cuda", generator=gen)
    b = torch.rand(n, dtype=torch.float64, device="cuda", generator=gen)
    st = torch.cuda.Stream()
    x, y, mid = a.clone(), torch.empty_like(a), torch.empty_like(a)
    want = []
    for v in (a, b):
        once, twice = torch.empty_like(v), torch.empty_like(v)
        torch.cuda.synchronize()
        _call(L, v, once, W, st.cuda_stream)
        _call(L, once, twice, W, st.cuda_stream)
        st.synchronize()
        want.append(twice)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        _call(L, x, mid, W, st.cuda_stream)
        _call(L, mid, y, W, st.cuda_stream)
    for v, ref in ((a, want[0]), (b, want[1]), (a, want[0])):
        x.copy_(v)
        y.zero_()
        torch.cuda.synchronize()
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, ref)
