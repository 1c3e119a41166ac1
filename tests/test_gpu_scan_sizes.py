"""The one-launch scan at the edges of its ranges (one block, a cluster with 4, 8 or 16 elements per thread, the
two-launch scan above): atom counts around 2^12, 2^15, 2^16 and 2^17.

Isolated balls on a lattice, some with a small ball inside that has no cell of its own: K^0 is known without an
oracle (the hidden balls are missing, all others are there), and its rows come from a scan over the atoms.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _balls(n):
    rng = np.random.default_rng(n)
    hidden = np.zeros(n, bool)
    hidden[1:] = rng.random(n - 1) < 0.3
    hidden[1:] &= ~hidden[:-1]  # its big ball comes right before
    site = np.cumsum(~hidden) - 1
    m = int(np.ceil((site[-1] + 1) ** (1 / 3)))
    c = np.stack([site % m, site // m % m, site // (m * m)], 1) * 8.0
    c[hidden] += 0.125
    return c, np.where(hidden, 0.5, 2.0), hidden


@pytest.mark.parametrize("n", [1, 2, 31, 4094, 4095, 4096, 32766, 32767, 32768, 65535, 65536, 65537, 131070, 131071, 131072,
                               140000])
def test_vertices_at_scan_edges(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_05944_gb300 as ac

    c, r, hidden = _balls(n)
    cx = ac.AlphaComplex(torch.from_numpy(c).cuda(), torch.from_numpy(r).cuda(), 0.0).build()
    want = np.flatnonzero(~hidden)
    for _ in range(2):  # the first build and a replay
        assert np.array_equal(cx.simplices(0).cpu().numpy()[:, 0], want)
        assert [cx.count(d) for d in (1, 2, 3)] == [0, 0, 0]
        assert not cx.attached(0).any()
        cx.build()
