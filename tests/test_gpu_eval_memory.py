"""ac_eval_filtration with lists left out takes no device memory: the rows that were asked for evaluate what they take
from the others themselves. (A buffer for the lists left out would be shared by calls on several streams, and its
length is theirs, however few rows were asked for.) Checked on a context that has not evaluated anything yet, for every
choice of lists; the values equal those of the call that asks for all lists, bit for bit."""
import ctypes
import gc
import itertools

import pytest

import synth
from test_zz_no_alloc import _pool_used_bytes

pytestmark = pytest.mark.gpu


def test_lists_left_out():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_05944_gb300 as ac

    c, r = synth.globule(71, 30000, probe=True)
    ct, rt = torch.from_numpy(c).cuda(), torch.from_numpy(r).cuda()
    cx = ac.AlphaComplex(ct, rt, 0.0).build()
    moved = ct + 1e-3 * torch.sin(37.0 * ct)
    got = {}
    gc.collect()  # contexts of earlier tests
    torch.cuda.synchronize()
    before = _pool_used_bytes()
    for k in range(5):
        for dims in itertools.combinations(range(4), k):
            out = [torch.full((cx.count(d),), 7.0, dtype=torch.float64, device="cuda") for d in range(4)]
            ptrs = (ctypes.c_void_p * 4)(*[out[d].data_ptr() if d in dims else None for d in range(4)])
            rc = ac.lib().ac_eval_filtration(cx._h, moved.data_ptr(), rt.data_ptr(), ctypes.cast(ptrs, ctypes.c_void_p), None)
            assert rc == ac.AC_OK
            got[dims] = out
    assert _pool_used_bytes() <= before
    want = got[(0, 1, 2, 3)]
    for dims, out in got.items():
        for d in range(4):
            if d in dims:
                assert torch.equal(out[d], want[d]), (dims, d)
            else:
                assert bool((out[d] == 7.0).all()), (dims, d)
