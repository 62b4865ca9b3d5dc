"""The bounds that keep the FP64 interpolation's taps on the spectrum, on the CPU: every window offset by
offset, anchors from the spectrum's ends to the largest accepted (|r| < 4.5e15)."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = """
#include "tap_range.cuh"
extern "C" void taps(long long k0, int m, long long nb, int neg, int jl, int jh, int *out) {
    const fdas::TapRange on = fdas::taps_on_spectrum(k0, m, nb);
    const fdas::TapRange part = fdas::taps_between(on, neg != 0, jl, jh);
    out[0] = on.lo; out[1] = on.hi; out[2] = part.lo; out[3] = part.hi;
}
"""


@pytest.fixture(scope="module")
def taps(tmp_path_factory):
    d = tmp_path_factory.mktemp("taps")
    (d / "taps.cpp").write_text(SRC)
    so = str(d / "taps.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ftrapv", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2206_12205_gb300", "csrc"), str(d / "taps.cpp"), "-o", so], check=True)
    f = ctypes.CDLL(so).taps
    f.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.c_longlong] + [ctypes.c_int] * 3 + [ctypes.c_void_p]

    def call(*a):
        out = (ctypes.c_int * 4)()
        f(*a, out)
        return list(out)
    return call


FAR = [2 ** 24, 2 ** 31 - 1, 2 ** 31, 2 ** 31 + 12, 3 * 10 ** 9, 2 ** 32, 2 ** 32 + 5, 10 ** 12, 4 * 10 ** 15,
       4500000000000000 + 2 ** 24]


@pytest.mark.parametrize("nb,m", [(1024, 2), (1024, 64), (1 << 20, 64), (1 << 26, 4096)])
def test_taps_stay_on_the_spectrum(taps, nb, m):
    half = m // 2
    near = [-half - 1, -half, -1, 0, 1, half - 1, half, half + 1, nb // 2, nb - half - 1, nb - half, nb - half + 1, nb - 1,
            nb, nb + half - 1, nb + half, nb + half + 1]
    for k0 in near + FAR + [-k for k in FAR]:
        want = range(max(-half, -k0), min(m - half - 1, nb - 1 - k0) + 1)
        for neg in (0, 1):
            folded = [-j for j in want][::-1] if neg else want
            flo, fhi = (folded[0], folded[-1]) if len(folded) else (1, 0)
            for jl, jh in ((-12, 12), (-12, 13), (5, 20), (-(1 << 24) - 12, -(1 << 24) + 13), ((1 << 24) - 12, (1 << 24) + 13)):
                lo, hi, plo, phi = taps(k0, m, nb, neg, jl, jh)
                if len(want):
                    assert (lo, hi) == (want[0], want[-1])
                    part = (max(jl, flo), min(jh, fhi))
                    assert (plo, phi) == part if part[0] <= part[1] else plo > phi
                else:
                    assert lo > hi and plo > phi
