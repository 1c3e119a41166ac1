"""AC3 and reach of a triangle's line (csrc/ac_reach.h), compiled for the host with
directed rounding by fesetround and checked against exact fractions: for random
and edge values of T, S and e_S (S + e_S within a few places of T on either
side, T below and above 2^23), in FP32 and FP64,

* ac3 = 1 only if S + e_S < T, -1 only if S - e_S > T;
* lo <= T - S - e_S (or 0), up >= T - S + e_S (or 0), both at least 0;
* an undecided line has lo = 0: nothing over it counts as decided.
"""
import os
import random
import shutil
import subprocess
from fractions import Fraction

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1908_05944_gb300", "csrc")

HARNESS = r"""
#include <fenv.h>
#include <stdio.h>
#include "ac_reach.h"
template <class R>
struct Directed {
    static R op(R a, R b, int mode) {
        volatile R x = a, y = b;
        fesetround(mode);
        volatile R r = x + y;
        fesetround(FE_TONEAREST);
        return r;
    }
    static R sub_dn(R a, R b) { return op(a, -b, FE_DOWNWARD); }
    static R add_up(R a, R b) { return op(a, b, FE_UPWARD); }
    static R max(R a, R b) { return a > b ? a : b; }
};
template <class R>
void one(R T, R S, R e) {
    const ac::Reach<R> r = ac::reach_of<Directed<R>>(T, S, e);
    printf("%d %a %a\n", r.ac3, (double)r.lo, (double)r.up);
}
int main() {
    int wide;
    double T, S, e;
    while (scanf("%d %la %la %la", &wide, &T, &S, &e) == 4) {
        if (wide) one<double>(T, S, e);
        else one<float>((float)T, (float)S, (float)e);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("reach")
    src = d / "h.cpp"
    src.write_text(HARNESS)
    exe = d / "h"
    subprocess.check_call([cxx, "-O1", "-std=c++17", "-frounding-math", "-I", CSRC, str(src), "-o", str(exe)])
    return str(exe)


def _f32(x):
    import struct

    return struct.unpack("f", struct.pack("f", x))[0]


def _cases(wide):
    rng = random.Random(31 + wide)
    out = []
    cut = (lambda x: x) if wide else _f32
    for _ in range(20000):
        T = float(rng.choice([rng.randint(1, 1 << 24), rng.randint(1 << 23, 1 << 24), 8388608, 1 << 24]))
        e = cut(T * 2.0 ** rng.uniform(-40, -10))
        near = rng.choice([0, 1, 2, 3])
        if near == 0:
            S = cut(T * rng.uniform(0.0, 2.0))
        elif near == 1:  # S + e_S just below or above T
            S = cut(T - e + rng.uniform(-2.0, 2.0) * T * 2.0 ** (-52 if wide else -23))
        elif near == 2:  # S - e_S just below or above T
            S = cut(T + e + rng.uniform(-2.0, 2.0) * T * 2.0 ** (-52 if wide else -23))
        else:
            S, e = T, cut(rng.choice([0.0, e]))
        out.append((T, max(S, 0.0), e))
    return out


@pytest.mark.parametrize("wide", [0, 1], ids=["fp32", "fp64"])
def test_one_answer(harness, wide):
    cases = _cases(wide)
    inp = "".join(f"{wide} {T.hex()} {S.hex()} {e.hex()}\n" for T, S, e in cases)
    out = subprocess.run([harness], input=inp, capture_output=True, text=True, check=True).stdout.split("\n")
    seen = {-1: 0, 0: 0, 1: 0}
    for (T, S, e), line in zip(cases, out):
        ac3, lo, up = line.split()
        ac3, lo, up = int(ac3), float.fromhex(lo), float.fromhex(up)
        d, E = Fraction(T) - Fraction(S), Fraction(e)
        assert 0 <= lo <= max(d - E, 0) and up >= max(d + E, 0), (T, S, e)
        if ac3 == 1:
            assert d - E > 0, (T, S, e)
        elif ac3 == -1:
            assert d + E < 0, (T, S, e)
        else:
            assert lo == 0.0, (T, S, e)
        seen[ac3] += 1
    assert min(seen.values()) > 100, seen
