"""The memory of builds that do not wait for their row counts (up to 65,536 atoms): their lists are sized by upper bounds.

* A build has room wherever it had with lists of the rows' sizes: in a memory pool of what a context that waits
  (host_results) took, 64 MB for the pool's granularity added, it builds the same lists.
* Contexts kept side by side hold at most 16 GB beyond what they hold with lists of the rows' sizes, however many there
  are (64 MB more allowed for the granularity).

Runs in a process of its own, whose library holds no idle blocks of other contexts.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

MB = 1 << 20
N = 60000
KEPT = 130  # by upper bounds they would hold 22 GB beyond


def child():
    import numpy as np
    import torch

    import paper_1908_05944_gb300 as ac
    import synth
    from test_gpu_failed_builds import LimitedPool

    c, r = (torch.from_numpy(x).cuda() for x in synth.globule(29, N, probe=True))

    def build(limit, count, **opt):
        """`count` contexts and the pool's largest use."""
        pool = LimitedPool(limit)
        with pool:
            made = [ac.AlphaComplex(c, r, 0.0, ac.options(**opt)).build() for _ in range(count)]
            torch.cuda.synchronize()
            return made, pool.used_high()

    (waits,), exact = build(0, 1, host_results=True)
    (free,), bound = build(0, 1)
    print("waits", exact // MB, "upper bounds", bound // MB)
    assert waits.stats()["host_syncs"] > free.stats()["host_syncs"]  # the two kinds
    (tight,), high = build(exact + 64 * MB, 1)
    assert high < bound  # the pool rounds its limit up
    for d in range(4):
        for a, b, h in zip((tight.simplices(d), tight.filtration_values(d), tight.attached(d)),
                           (free.simplices(d), free.filtration_values(d), free.attached(d)), waits.host_lists(d)):
            assert torch.equal(a, b) and np.array_equal(a.cpu().numpy(), h)
    assert tight.build().stats()["replayed"] == 1
    kept, all_ = build(0, KEPT)
    print("kept", all_ // MB)
    assert all_ <= KEPT * exact + (16384 + 64) * MB


def test_memory():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    here = os.path.dirname(os.path.abspath(__file__))
    root = os.path.dirname(here)
    p = subprocess.run([sys.executable, os.path.abspath(__file__)], cwd=root, capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, PYTHONPATH=root + os.pathsep + here))
    assert p.returncode == 0, p.stdout[-2000:] + p.stderr[-4000:]


if __name__ == "__main__":
    child()
