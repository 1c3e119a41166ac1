"""The gradient of large balls among many small ones (rows of hundreds of edges that start with one atom), the large
ball first or last in the input. Either way it must equal the gradient taken with atomics (ac_backward_noalloc, another
order of summation: 1e-12 of the largest component, as in that entry point's own test), twice bit for bit the same, and
the order must not decide the time: ac_backward with the large ball first took up to 70 times as long when eight lanes went
over all its rows for each of its edges; ten times is allowed here.
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _hub(k, first, seed):
    rng = np.random.default_rng(seed)
    i = np.arange(k) + 0.5
    ph, th = np.arccos(1 - 2 * i / k), np.pi * (1 + 5**0.5) * i
    small = 3.9 * np.stack([np.cos(th) * np.sin(ph), np.sin(th) * np.sin(ph), np.cos(ph)], -1) + rng.normal(0, 0.03, (k, 3))
    big = np.zeros((1, 3))
    c = np.concatenate([big, small] if first else [small, big])
    r = np.concatenate([[3.6], np.full(k, 0.45)] if first else [np.full(k, 0.45), [3.6]])
    return c, r


def _gradients(ac, cx, w):
    import torch

    ptrs = (ctypes.c_void_p * 4)(*[x.data_ptr() if x.numel() else None for x in w])
    dc = torch.empty((cx.n, 3), dtype=torch.float64, device="cuda")
    dr = torch.empty((cx.n,), dtype=torch.float64, device="cuda")
    assert ac.lib().ac_backward_noalloc(cx._h, ctypes.cast(ptrs, ctypes.c_void_p), dc.data_ptr(), dr.data_ptr(), None) == 0
    return dc, dr


def _ms(f):
    import torch

    t = []
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        b.synchronize()
        t.append(a.elapsed_time(b))
    return sorted(t)[2]


@pytest.mark.parametrize("k", [40, 300, 700])
def test_hub(k):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_05944_gb300 as ac

    ms = {}
    for first in (True, False):
        c, r = _hub(k, first, k)
        cx = ac.AlphaComplex(torch.from_numpy(c).cuda(), torch.from_numpy(r).cuda(), 0.0).build()
        g = torch.Generator(device="cuda").manual_seed(k)
        w = [torch.randn(cx.count(d), dtype=torch.float64, device="cuda", generator=g) for d in range(4)]
        dc, dr = cx.backward(w)
        again = cx.backward(w)
        assert torch.equal(dc, again[0]) and torch.equal(dr, again[1])
        nc, nr = _gradients(ac, cx, w)
        assert (dc - nc).abs().max() <= 1e-12 * nc.abs().max()
        assert (dr - nr).abs().max() <= 1e-12 * nr.abs().max()
        ms[first] = _ms(lambda: cx.backward(w))
        cx.close()
    assert ms[True] <= 10 * ms[False], ms
