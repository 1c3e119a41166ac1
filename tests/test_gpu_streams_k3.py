"""K^3 canonicalised beside K^2 (up to 2^20 atoms) and before it (above): batches of copies of one molecule on either
side of the line and well below it. Every copy's lists are the single molecule's, which equal the oracle's; tolerance
none (the values are the same rationals rounded the same way)."""
import gc

import numpy as np
import pytest

import oracle
import synth
from gpu_util import assert_same_complex, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    # contexts that earlier tests left in reference cycles (an expected exception keeps its frame) hold up to 90 GB
    # of the device until Python collects them
    gc.collect()
    yield
    gc.collect()


@pytest.mark.parametrize("copies,extra", [(3, 0), (1024, 0), (1024, 1)])
@pytest.mark.parametrize("host", [False, True])
def test_copies_of_a_molecule(copies, extra, host):
    import torch

    import paper_1908_05944_gb300 as ac

    m = 1024
    c, r = synth.globule(23, m, probe=True)
    one = run_gpu(c, r, 0.0)
    assert_same_complex(one, oracle.alpha_complex(c, r, 0.0))
    want = [(one.simplices(d).cpu().numpy(), one.filtration_values(d).cpu().numpy(), one.attached(d).cpu().numpy())
            for d in range(4)]
    cc = np.concatenate([np.tile(c, (copies, 1)), np.zeros((extra, 3))])
    rr = np.concatenate([np.tile(r, copies), np.ones(extra)])
    off = list(range(0, copies * m + 1, m)) + [copies * m + 1] * extra
    cx = ac.AlphaComplex(torch.from_numpy(cc).cuda(), torch.from_numpy(rr).cuda(), 0.0,
                         ac.options(host_results=True) if host else None, offsets=np.array(off, np.int64))
    for _ in range(2):  # the first build and a replay
        cx.build()
        for d in range(4):
            for k in range(copies):
                if host:
                    got = cx.host_lists(d, k, copy=False)
                else:
                    got = [x.cpu().numpy() for x in (cx.simplices(d, k, copy=False), cx.filtration_values(d, k, copy=False),
                                                     cx.attached(d, k, copy=False))]
                assert all(np.array_equal(a, b) for a, b in zip(got, want[d])), (d, k)
            if extra:
                assert cx.count(d, copies) == (1 if d == 0 else 0)
