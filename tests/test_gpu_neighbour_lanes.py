"""The two forms of the neighbour search around the atom count where one takes over from the other (32,768), and
molecules too small to fill a block of either: lists, flags and values equal the oracle's."""
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


@pytest.mark.parametrize("n,kind", [(1, "probe"), (3, "probe"), (33, "probe"), (32768, "vdw"), (32769, "vdw"),
                                    (32768, "probe"), (32769, "probe"), (3001, "particles")])
@pytest.mark.parametrize("cell_factor", [1.0, 0.5, 3.0])
def test_neighbours_around_the_switch(n, kind, cell_factor):
    if n > 30000 and cell_factor != 1.0 and kind == "probe":
        pytest.skip("one cell size is enough for the large dense case")
    c, r = synth.particles(17, n) if kind == "particles" else synth.globule(17, n, probe=kind == "probe")
    gpu = run_gpu(c, r, 0.0, cell_factor=cell_factor)
    ref = oracle.alpha_complex(c, r, 0.0)
    assert_same_complex(gpu, ref)
    # the neighbour counts themselves: pairs of atoms whose grown balls meet (exact integers)
    if n <= 3001:
        P, W = np.rint(c * 1024).astype(np.int64), np.rint(r * 1024).astype(np.int64) ** 2
        D = ((P[:, None] - P[None]) ** 2).sum(2)
        t = D - W[:, None] - W[None]
        meet = (t <= 0) | (t * t <= 4 * W[:, None] * W[None])
        np.fill_diagonal(meet, False)
        st = gpu.stats()
        assert st["neighbour_pairs"] == int(meet.sum()) and st["max_degree"] == int(meet.sum(1).max())
