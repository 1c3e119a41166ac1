"""The list getters and the rows of a sub-complex against plain indexing.

* ac_copy_list: a list copied out equals the view of it, for every list and molecule, also into host memory; another
  count and unknown lists are refused.
* ac_subcomplex_lists: the flagged rows and values in list order equal boolean indexing, for flags that fill,
  leave empty and end tiles of the compaction (4,096 flags), on lists of lengths below, at and above a few tiles.
"""
import ctypes

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ac():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_05944_gb300 as ac

    return ac


def _built(ac, n, offsets=None):
    import torch

    c, r = synth.globule(41, n, probe=True) if n else (np.zeros((0, 3)), np.zeros(0))
    return ac.AlphaComplex(torch.from_numpy(c).cuda(), torch.from_numpy(r).cuda(), 0.0, offsets=offsets).build()


def test_copies_equal_views(ac):
    import torch

    bx = _built(ac, 700, offsets=[0, 300, 300, 700])
    for m in range(3):
        for d in range(4):
            for get in (bx.simplices, bx.filtration_values, bx.attached):
                a, b = get(d, m), get(d, m, copy=False)
                assert a.dtype == b.dtype and a.shape == b.shape and torch.equal(a, b)
    cx = _built(ac, 500)
    L, n = ac.lib(), cx.count(2)
    host = np.zeros(n)
    assert L.ac_copy_list(cx._h, ac.AC_LIST_VALUES, 2, -1, host.ctypes.data, n, None) == ac.AC_OK
    torch.cuda.synchronize()
    assert np.array_equal(host, cx.filtration_values(2).cpu().numpy())
    assert L.ac_copy_list(cx._h, ac.AC_LIST_VALUES, 2, -1, host.ctypes.data, n - 1, None) == ac.AC_ERR_INVALID_ARG
    assert L.ac_copy_list(cx._h, 3, 2, -1, host.ctypes.data, n, None) == ac.AC_ERR_INVALID_ARG
    assert L.ac_copy_list(cx._h, ac.AC_LIST_ROWS, 2, -1, None, n, None) == ac.AC_ERR_INVALID_ARG


@pytest.mark.parametrize("n", [0, 1, 40, 700, 2500])
@pytest.mark.parametrize("pattern", ["all", "none", "last", "first", "random", "tile"])
def test_subcomplex_lists_equal_indexing(ac, n, pattern):
    import torch

    cx = _built(ac, n)
    for d in range(4):
        m = cx.count(d)
        flags = torch.zeros(max(m, 1), dtype=torch.uint8, device="cuda")
        if m and pattern == "all":
            flags[:] = 1
        elif m and pattern == "last":
            flags[m - 1] = 1
        elif m and pattern == "first":
            flags[0] = 1
        elif pattern == "random":
            flags[:] = (torch.rand(len(flags), device="cuda", generator=torch.Generator("cuda").manual_seed(d)) < 0.4)
        elif pattern == "tile":  # the second tile only
            flags[4096:8192] = 1
        keep = flags[:m].bool()
        k = int(keep.sum())
        rows = torch.full((k + 1, d + 1), -7, dtype=torch.int32, device="cuda")
        f = torch.full((k + 1,), -7.0, dtype=torch.float64, device="cuda")
        rc = ac.lib().ac_subcomplex_lists(cx._h, d, -1, flags.data_ptr(), k, rows.data_ptr(), f.data_ptr(),
                                          torch.cuda.current_stream().cuda_stream)
        assert rc == ac.AC_OK
        assert torch.equal(rows[:k], cx.simplices(d)[keep]) and torch.equal(f[:k], cx.filtration_values(d)[keep])
        assert bool((rows[k] == -7).all()) and float(f[k]) == -7.0  # nothing past the count


def test_subcomplex_lists_arguments(ac):
    cx = _built(ac, 40)
    L = ac.lib()
    assert L.ac_subcomplex_lists(cx._h, 4, -1, None, 0, None, None, None) == ac.AC_ERR_INVALID_ARG
    assert L.ac_subcomplex_lists(cx._h, 1, -1, None, 1, None, None, None) == ac.AC_ERR_INVALID_ARG
    assert L.ac_subcomplex_lists(None, 1, -1, None, 1, None, None, ctypes.c_void_p()) == ac.AC_ERR_INVALID_ARG
