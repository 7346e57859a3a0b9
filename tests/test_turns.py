"""The phases and unit phasors of the column and row tables (csrc/turns.cuh), compiled as host code,
against exact rational phases and 64-bit cos and sin."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0907_4027_gb300", "csrc")
SRC = """
#include "turns.cuh"
extern "C" {
void cis(long n, const unsigned long long *ph, float *out) {
  for (long i = 0; i < n; i++) {
    const float2 v = hot::cis_turns(ph[i]);
    out[2 * i] = v.x;
    out[2 * i + 1] = v.y;
  }
}
void phases(double lin, double quad, long n, const int *q, unsigned long long *out) {
  const hot::TrapTurns t = hot::trap_turns(lin, quad);
  for (long i = 0; i < n; i++) out[i] = hot::phase_at(t, q[i]);
}
}
"""


@pytest.fixture(scope="module")
def turns(tmp_path_factory):
    d = tmp_path_factory.mktemp("turns")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(d / "t.cpp"), "-o",
                    str(d / "t.so")], check=True)
    return ctypes.CDLL(str(d / "t.so"))


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def exact_cis(ph):
    """cos and sin in 64 bits of phases in 2^-64 turns, reduced to an eighth of a turn in integers."""
    n = ((ph >> np.uint64(61)) + np.uint64(1)) >> np.uint64(1)
    r = (ph - (n << np.uint64(62))).view(np.int64).astype(np.float64) * (2 * np.pi / 2.0 ** 64)
    c, s = np.cos(r), np.sin(r)
    k = (n & np.uint64(3)).astype(int)
    return np.choose(k, [c, -s, -c, s]), np.choose(k, [s, c, -s, -c])


def ulps(got, ref):
    """Error in units of the last place of ref's binade."""
    ulp = np.ldexp(1.0, np.frexp(np.abs(ref))[1] - 24)
    return np.abs(got.astype(np.float64) - ref) / ulp


@pytest.mark.parametrize("kind", ["uniform", "near zeros", "eighths"])
def test_unit_phasors_are_rounded_correctly_but_for_a_few(turns, kind):
    """0.5 ulp and what the series leaves out: the next terms are below (pi/2)^13/13! 2^-13 of sine and
    (pi/2)^14/14! 2^-14 of cosine, the products after float-float below 2^-22 of their 0.06: 0.002 ulp."""
    rng = np.random.default_rng(1)
    ph = rng.integers(0, 2 ** 64, 400000, dtype=np.uint64)
    if kind == "near zeros":  # quarter turns and small distances of every magnitude
        d = (ph >> rng.integers(4, 62, ph.size).astype(np.uint64)).astype(np.uint64)
        ph = (ph & np.uint64(3 << 62)) + np.where(ph & np.uint64(1), d, np.uint64(0) - d)
    elif kind == "eighths":
        ph = (ph & np.uint64(7 << 61)) + (ph & np.uint64(0xffffffff)) - np.uint64(1 << 31)
    out = np.empty((ph.size, 2), dtype=np.float32)
    turns.cis(ctypes.c_long(ph.size), ptr(ph), ptr(out))
    for got, ref in zip(out.T, exact_cis(ph)):
        some = ref != 0
        assert np.all(got[~some] == 0)
        assert ulps(got[some], ref[some]).max() <= 0.502
        assert np.mean(got != ref.astype(np.float32)) < 1e-3


@pytest.mark.parametrize("lin,quad", [(0.013, -1.7e-6), (-0.4999, 3.3e-4), (-1.0 / 3, 0.0), (17.25, -2.5), (1e-30, 7e-25),
                                      (-123456.789, 4096.125)])
def test_phases_against_rationals(turns, lin, quad):
    """The linear turns are cut at 2^-64 (|q| units at most), the quadratic ones at 2^-96 and the product's unit."""
    q = np.r_[np.arange(-33, 34), [-32768, -1023, 959, 960, 32767]].astype(np.int32)
    out = np.empty(q.size, dtype=np.uint64)
    turns.phases(ctypes.c_double(lin), ctypes.c_double(quad), ctypes.c_long(q.size), ptr(q), ptr(out))
    for qi, got in zip(q.tolist(), out.tolist()):
        exact = (Fraction(lin) * qi + Fraction(quad) * qi * qi) * 2 ** 64
        off = (Fraction(got) - exact) % 2 ** 64
        assert min(off, 2 ** 64 - off) <= abs(qi) + 2, qi
