"""Tetrahedra over triangles whose AC3 the FP32 bounds leave open (csrc/ac_reach.h).

Each input is four balls in quanta of 1/1024 A: four radii, then the places of
the second to fourth ball from the first, at alpha = 0. The first three (the
first ball and the two nearest to it) are a triangle whose orthoradius is within
FP32's resolution of the limit: its AC3 stays open in FP32, and the whole numbers
near T = W_0 + alpha > 2^23 are too coarse to tell S + e_S from T, while
(T - S) - e_S is positive. The fourth ball lies about that triangle's orthocentre.
Found by a host search over the kernel's FP32 operations (rcp.approx taken within
one place of 1/x). The oracle has one tetrahedron for each. Tolerance: lists
none, values that of gpu_util.
"""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same_complex

pytestmark = pytest.mark.gpu

INPUTS = [
    (2990, 2990, 3174, 3277, 1048, -2036, 4217, 5342, 72, 1728, 3131, -3189, 3671),
    (3174, 3277, 2990, 2990, -3825, -3133, -100, -674, -1603, -4925, -2028, -4612, -2889),
    (3174, 3277, 3174, 3277, -5611, 2679, 438, -3936, -2272, -1083, -6174, 1168, 983),
    (3021, 3277, 3021, 3174, -975, -3030, 1702, 2247, -5454, -1284, 3168, -5139, -387),
    (3174, 3174, 3174, 3277, -4415, 271, 856, -1450, -4256, 3474, -3879, -4378, 1320),
    (2990, 3277, 3174, 3174, -1239, 2090, 5410, -4749, 831, 2289, -2863, 2672, 4675),
    (3021, 3021, 3277, 3174, -341, -2870, -4863, -2994, -4541, -1474, -1267, -5241, -1764),
    (2990, 2990, 3021, 3277, 2034, -2205, 502, 4273, -504, 4050, 2707, -489, 5336),
    (2990, 3277, 3021, 2990, -2789, 473, -4982, -1544, 4419, -1510, -3863, 2613, -3480),
    (3174, 3277, 3021, 3277, 5253, 570, -3028, 1105, 2498, -4571, 4055, 3162, -3469),
    (3277, 3277, 2990, 3174, -2936, 2876, 4400, -4116, 3003, -781, -5355, 2305, 2060),
    (3174, 3021, 2990, 3277, -1668, 2531, -2379, -1514, 624, -5836, -1578, -2295, -5412),
    (3174, 2990, 3021, 3277, 1998, 2668, -3950, 5378, -323, -1564, 3721, -477, -4590),
    (3277, 2990, 3277, 3174, -1477, 2562, -4628, 3827, 1655, -1882, 3394, 1096, -4200),
    (3174, 3021, 3021, 3277, -672, 3461, -3576, 125, 5488, 1220, 1563, 4621, -2965),
    (3277, 2990, 3021, 3277, 1926, -2196, 2235, 5625, -2197, 992, 5083, -3278, -974),
    (3021, 3277, 3174, 2990, -3930, 2371, 3427, -4119, 549, -2152, -5161, 1000, 2422),
    (2990, 3174, 3021, 3277, -754, -54, -3018, 4518, 1943, -3397, 3590, 3035, -3940),
    (2990, 3174, 3277, 3277, -1414, -1686, -2686, -3467, 3740, 131, -5360, 335, 74),
    (3021, 2990, 3174, 3277, 1016, -3635, -3168, 1142, -5320, 1755, -406, -5825, -1340),
    (3174, 3174, 3277, 2990, -3758, 2061, 1700, 1993, 4212, 2851, -1868, 5102, 2677),
    (3277, 3021, 2990, 3174, -3211, -2526, 2935, -954, 1464, 5471, -3986, 891, 4344),
    (3277, 3021, 3021, 3277, 2762, -734, -383, 2790, -5089, 2406, 2442, -4318, 3946),
    (3277, 2990, 3174, 3021, -2624, 3265, 2969, -5329, -1025, 373, -5179, 2666, 2059),
    (3174, 2990, 3277, 3174, -238, 2099, -2631, 576, 3836, 3314, 2661, 4858, 1092),
    (3277, 3174, 3277, 3277, 1532, 1405, 3695, 5940, 1863, -257, 5473, 899, 2922),
    (3021, 3174, 3277, 3277, 852, 5884, 667, 1903, 2555, 4108, -321, 5693, 2051),
    (3277, 2990, 3277, 2990, 3108, -1035, 3753, -661, 3559, 4031, 1565, -1081, 5130),
    (3277, 3277, 2990, 3021, -92, 4424, -3315, -4318, 660, -1035, -4144, 1436, -3569),
    (3021, 3174, 2990, 3277, -6067, 952, 201, -5021, -1919, 1144, -5899, 434, 1745),
    (3174, 3277, 3277, 3174, -1088, -5712, -289, 587, -951, -4085, -1551, -5485, -2565),
    (3174, 3277, 2990, 3277, -11, -2943, 3671, 513, -5741, -1037, -1568, -5824, -181),
    (3277, 3277, 2990, 3021, -3767, -44, -4076, 378, 223, -6039, -1712, 1337, -5734),
    (3021, 3174, 3277, 3174, 1447, 1692, -5381, -1264, 4211, -879, -1116, 2689, -5136),
    (3021, 3021, 3277, 3174, 2894, 2125, -3855, 3484, 4048, 1164, 5010, 2259, -2116),
    (2990, 3174, 2990, 3277, -1374, -4254, -2794, -4811, -133, -1229, -3610, -4380, -2068),
    (2990, 3021, 2990, 3277, 542, 1626, 5551, -1722, 1759, 3059, 2128, 2851, 4764),
    (3277, 2990, 3277, 3021, -1103, 1259, 5754, -115, -3268, 4393, -1378, -189, 6115),
    (3021, 3174, 3277, 3277, -795, -4234, 2550, -518, 677, 5543, 1237, -2909, 4936),
    (3021, 2990, 3277, 3277, 3841, 2650, -547, 3779, 80, 4364, 5691, -25, 1233),
    (3277, 3174, 3277, 3277, 5794, 539, 505, 1293, -2576, 3338, 4942, -3027, 2242),
    (2990, 3277, 2990, 3174, 2428, 4044, -1827, 5314, -540, -965, 5431, 1002, 748),
    (3174, 3021, 3277, 2990, -2952, -793, 3921, -795, 4594, 2384, -1573, 1975, 5376),
]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _balls():
    t = np.array(INPUTS, dtype=np.int64)
    r = t[:, :4] / 1024.0
    c = np.concatenate([np.zeros((len(t), 1, 3)), t[:, 4:].reshape(-1, 3, 3) / 1024.0], axis=1)
    return c, r


@pytest.mark.parametrize("precision", [0, 1])
def test_every_tetrahedron_is_there(precision):
    import torch

    import paper_1908_05944_gb300 as ac

    c, r = _balls()
    k = len(c)
    # cells larger than a molecule: sorted positions follow the input, so the first ball owns the tetrahedron
    opt = ac.options(precision=precision, cell_factor=5.0)
    cx = ac.AlphaComplex(torch.from_numpy(c.reshape(-1, 3)).cuda(), torch.from_numpy(r.reshape(-1)).cuda(), 0.0, opt,
                         offsets=np.arange(0, 4 * k + 1, 4))
    for _ in range(2):  # the first build and a replay
        cx.build()
        missing = [m for m in range(k) if cx.count(3, m) != 1]
        assert not missing, f"{len(missing)} of {k} tetrahedra are missing: inputs {missing}"
        for m in range(k):
            assert_same_complex(cx, oracle.alpha_complex(c[m], r[m], 0.0), mol=m)
    st = cx.stats()
    assert st["candidates"][3] == k and st["simplices"] == [4 * k, 6 * k, 4 * k, k]


def test_candidates_of_one_input():
    """One molecule, its candidate lists kept: the tetrahedron is a candidate once and a row of K^3."""
    import torch

    import paper_1908_05944_gb300 as ac

    c, r = _balls()
    used = 0
    for m in range(len(c)):
        if r[m].max() != 3277 / 1024.0:  # the bounds are those of the largest radius
            continue
        cx = ac.AlphaComplex(torch.from_numpy(c[m]).cuda(), torch.from_numpy(r[m]).cuda(), 0.0,
                             ac.options(keep_candidates=True, cell_factor=5.0)).build()
        assert cx.candidates(3).cpu().tolist() == [[0, 1, 2, 3]]
        assert cx.simplices(3).cpu().tolist() == [[0, 1, 2, 3]]
        cx.close()
        used += 1
    assert used > 0
