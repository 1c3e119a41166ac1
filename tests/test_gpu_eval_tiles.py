"""Values and gradients at moved atoms at the edges of the evaluation tiles (128 rows in short lists, 512 in lists of
at least 155,648 rows) and with some of the lists left out.

Isolated pairs of overlapping balls on a lattice: K^0 and K^1 have one row per ball and per pair, every row is its own
source, and values and gradients have closed forms, taken here in extended precision. With u = 2^-53, distances in
[1.5, 1.9] and radii in [1, 1.4], every intermediate of an edge is below 8 in magnitude and a value is a double-double
result rounded once (8u allowed); a gradient component is about 30 FP64 operations on them (at most 512u), plus the
rounding of a centre's coordinate if the orthocentre is formed in absolute coordinates (3.5 times u * |coordinate|).
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0**-53


def _pairs(m):
    rng = np.random.default_rng(m)
    site = np.arange(m)
    k = int(np.ceil(m ** (1 / 3)))
    base = np.stack([site % k, site // k % k, site // (k * k)], 1) * 8.0
    v = rng.normal(size=(m, 3))
    v *= (rng.uniform(1.5, 1.9, m) / np.linalg.norm(v, axis=1))[:, None]
    c = np.empty((2 * m, 3))
    c[0::2] = base
    c[1::2] = base + v
    return c, rng.uniform(1.0, 1.4, 2 * m)


def _closed_form(c, r, w):
    p, q = c[0::2].astype(np.longdouble), c[1::2].astype(np.longdouble)
    R, S = r[0::2].astype(np.longdouble), r[1::2].astype(np.longdouble)
    v = q - p
    D = (v * v).sum(1)
    mu = (D + R * R - S * S) / (2 * D)
    f = [-r.astype(np.longdouble) ** 2, mu * mu * D - R * R]
    dr = -2 * w[0] * r.astype(np.longdouble)
    dc = np.zeros((len(r), 3), np.longdouble)
    o = p + mu[:, None] * v
    for at, x, rad, lam in ((0, p, R, 1 - mu), (1, q, S, mu)):
        dc[at::2] = 2 * (w[1] * lam)[:, None] * (x - o)
        dr[at::2] += -2 * w[1] * lam * rad
    return f, dc, dr


@pytest.mark.parametrize("m", [1, 127, 128, 129, 511, 513, 77823, 77824, 77825, 155647, 155648, 155649])
def test_pairs_at_tile_edges(m):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_05944_gb300 as ac

    c, r = _pairs(m)
    ct, rt = torch.from_numpy(c).cuda(), torch.from_numpy(r).cuda()
    cx = ac.AlphaComplex(ct, rt, 0.0).build()
    assert [cx.count(d) for d in range(4)] == [2 * m, m, 0, 0]
    assert np.array_equal(cx.simplices(1).cpu().numpy(), np.arange(2 * m).reshape(m, 2))
    rng = np.random.default_rng(m + 1)
    w = [rng.uniform(-1, 1, 2 * m), rng.uniform(-1, 1, m)]
    f, dc, dr = _closed_form(c, r, w)
    got = cx.eval_filtration(ct, rt)
    for d in (0, 1):
        assert np.max(np.abs(got[d].cpu().numpy() - f[d])) <= 8 * U
    gc, gr = cx.backward([torch.from_numpy(w[0]).cuda(), torch.from_numpy(w[1]).cuda(), None, None])
    assert np.max(np.abs(gc.cpu().numpy() - dc)) <= 512 * U + 3.5 * U * np.abs(c).max()
    assert np.max(np.abs(gr.cpu().numpy() - dr)) <= 512 * U
    # one list at a time: the same numbers, the other's memory untouched
    for d in (0, 1):
        one = torch.full((cx.count(d) + 1,), 7.0, dtype=torch.float64, device="cuda")
        ptrs = (ctypes.c_void_p * 4)(*[one.data_ptr() if e == d else None for e in range(4)])
        assert ac.lib().ac_eval_filtration(cx._h, ct.data_ptr(), rt.data_ptr(), ctypes.cast(ptrs, ctypes.c_void_p), None) == 0
        assert torch.equal(one[:-1], got[d]) and one[-1].item() == 7.0


def test_attached_rows_without_their_sources_list():
    # the values of the attached rows come from lists the caller did not ask for
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_05944_gb300 as ac

    rng = np.random.default_rng(5)
    c, r = rng.uniform(0, 14, (700, 3)), rng.uniform(1.0, 1.9, 700)
    ct, rt = torch.from_numpy(c).cuda(), torch.from_numpy(r).cuda()
    cx = ac.AlphaComplex(ct, rt, 1.0).build()
    assert cx.attached(1).any() and cx.attached(2).any()
    moved = ct + torch.from_numpy(rng.uniform(-1e-3, 1e-3, c.shape)).cuda()
    want = cx.eval_filtration(moved, rt)
    for d in range(4):
        one = torch.empty(cx.count(d), dtype=torch.float64, device="cuda")
        ptrs = (ctypes.c_void_p * 4)(*[one.data_ptr() if e == d else None for e in range(4)])
        assert ac.lib().ac_eval_filtration(cx._h, moved.data_ptr(), rt.data_ptr(), ctypes.cast(ptrs, ctypes.c_void_p), None) == 0
        assert torch.equal(one, want[d])
