"""Builds that run out of device memory half way, and the builds after them.

A memory pool of a limited size, made the device's current pool for one build, lets the build fail with AC_ERR_OOM at
one reservation after another: before and after the per-atom pass forks its wide tiers, K^3 and the filtration to the
side stream and the copies of host lists to the copy stream. After each failure the same context, with the device's own
pool again, builds the complex of an undisturbed context, twice (a synchronised build and a replay), lists on the
device and on the host alike. Runs in a process of its own, whose library holds no idle blocks of other contexts.
"""
import ctypes
import glob
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

MB = 1 << 20


class _Props(ctypes.Structure):  # cudaMemPoolProps
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int), ("loc_type", ctypes.c_int),
                ("loc_id", ctypes.c_int), ("security", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


class LimitedPool:
    """The device's current memory pool, while entered: a pool of at most `limit` bytes (0: as the device allows)."""

    def __init__(self, limit):
        names = ["libcudart.so"] + sorted(glob.glob("/usr/local/cuda/lib64/libcudart.so*"))
        for name in names:
            try:
                self.rt = ctypes.CDLL(name)
                break
            except OSError:
                continue
        else:
            pytest.skip("libcudart not found")
        self.old, self.pool = ctypes.c_void_p(), ctypes.c_void_p()
        props = _Props(alloc_type=1, handle_types=0, loc_type=1, loc_id=0, max_size=limit)  # pinned, on device 0
        assert self.rt.cudaMemPoolCreate(ctypes.byref(self.pool), ctypes.byref(props)) == 0
        assert self.rt.cudaDeviceGetMemPool(ctypes.byref(self.old), 0) == 0

    def __enter__(self):
        assert self.rt.cudaDeviceSetMemPool(0, self.pool) == 0
        return self

    def __exit__(self, *exc):
        assert self.rt.cudaDeviceSetMemPool(0, self.old) == 0

    def attribute(self, which):
        v = ctypes.c_uint64()
        assert self.rt.cudaMemPoolGetAttribute(self.pool, which, ctypes.byref(v)) == 0
        return v.value

    def used_high(self):
        return self.attribute(8)  # cudaMemPoolAttrUsedMemHigh


def _inputs(kind):
    import numpy as np

    import synth

    if kind == "wide":  # radii over a factor of 16: every tier of the per-atom pass
        rng = np.random.default_rng(3)
        n = 100000
        return rng.random((n, 3)) * (n / 0.6) ** (1 / 3), 3.9 * np.exp(-rng.random(n) ** 0.5 * np.log(16.0))
    return synth.globule(29, 60000, probe=True)


def _lists(cx, host):
    if host:
        return [x.copy() for d in range(4) for x in cx.host_lists(d, copy=False)]
    return [x.cpu().numpy() for d in range(4) for x in (cx.simplices(d), cx.filtration_values(d), cx.attached(d))]


def child(kind):
    import numpy as np
    import torch

    import paper_1908_05944_gb300 as ac

    c, r = (torch.from_numpy(x).cuda() for x in _inputs(kind))
    host = kind == "host"

    def context():
        return ac.AlphaComplex(c, r, 0.0, ac.options(host_results=host))

    kept, failed, limit = [context()], 0, 32 * MB  # closed contexts would leave idle blocks to the next ones
    want = _lists(kept[0].build(), host)
    while True:
        cx = context()
        kept.append(cx)
        with LimitedPool(limit):
            rc = ac.lib().ac_build(cx._h, None)
        if rc == ac.AC_OK:
            break
        assert rc == ac.AC_ERR_OOM, (rc, ac.lib().ac_last_error_detail())
        failed += 1
        for _ in range(2):
            cx.build()
            got = _lists(cx, host)
            assert all(np.array_equal(a, b) for a, b in zip(got, want)), (kind, limit)
        assert cx.stats()["replayed"] == 1
        limit = limit + 32 * MB if limit < 512 * MB else limit * 5 // 4
        assert limit < 16384 * MB
    got = _lists(cx, host)
    assert all(np.array_equal(a, b) for a, b in zip(got, want)), (kind, limit)
    assert failed >= 4, failed
    print("failed", failed, "limit", limit // MB)


@pytest.mark.parametrize("kind", ["plain", "host", "wide"])
def test_build_after_a_failed_build(kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    p = subprocess.run([sys.executable, os.path.abspath(__file__), kind], cwd=root, capture_output=True, text=True,
                       timeout=600, env=dict(os.environ, PYTHONPATH=root))
    assert p.returncode == 0, p.stdout[-2000:] + p.stderr[-4000:]


if __name__ == "__main__":
    child(sys.argv[1])
