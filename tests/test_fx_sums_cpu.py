"""The multigrid's integer neighbour sums (tde_fx.cuh, compiled for the host) against exact
rational arithmetic over the exponent range: within their stated truncation, or declined in
favour of FP64 -- at the top of the range in particular, where a sum may overflow."""
import ctypes as C
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2609_37859_gb300", "csrc")
SRC = r"""
#include "tde_fx.cuh"
extern "C" int lap6(double c, const double *n, double *s) {
  bool taken = true;
  *s = tde::fx_lap6(c, n, [&] { taken = false; return 0.0; });
  return taken;
}
extern "C" int group(const double *q, const double *o, double *s) { return tde::fx_lap_group(q, o, *s); }
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    src, so = str(d / "sums.cpp"), str(d / "sums.so")
    open(src, "w").write(SRC)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-w", "-fPIC", "-shared", "-I", CSRC, "-o", so, src])
    lib = C.CDLL(so)
    P = C.POINTER(C.c_double)
    lib.lap6.argtypes, lib.group.argtypes = [C.c_double, P, P], [P, P, P]
    return lib


def check(taken, got, weights, values, guard, e):
    big = max(abs(v) for v in values)
    if not taken:
        assert not 1e-280 < big < 2.0 ** 1017, e   # (declined at the ends of the range only)
        return
    exact = sum(w * Fraction(float(v)) for w, v in zip(weights, values))
    assert np.isfinite(got), e
    # each value truncated below a unit of the largest's exponent, then one rounding
    unit = Fraction(2) ** (int(np.frexp(big)[1]) - 1 - 52 - guard)
    bound = sum(abs(w) for w in weights) * unit + Fraction(float(np.spacing(abs(got)))) / 2
    assert abs(Fraction(float(got)) - exact) <= bound, e


@pytest.mark.parametrize("e", [-1060, -1022, -951, -948, -300, 0, 1, 500, 1015, 1016, 1017, 1018, 1019, 1020, 1021, 1022, 1023])
@pytest.mark.parametrize("spread", [0, 3, 70])
@pytest.mark.parametrize("signs", ["equal", "opposite", "mixed"])
def test_sums_are_exact_or_declined(fx, e, spread, signs):
    rng = np.random.default_rng(e + 2000 + spread)
    out = C.c_double()
    ptr = lambda a: a.ctypes.data_as(C.POINTER(C.c_double))  # noqa: E731
    for trial in range(60):
        v = np.ldexp(1.0 + rng.random(33), np.maximum(e - rng.integers(0, spread + 1, 33), -1074))
        if trial == 0:
            v[:] = np.ldexp(2.0 - 2.0 ** -52, e)     # the largest of the binade throughout
        if trial % 3 == 1:
            v[rng.integers(0, 33, 6)] = 0.0
        s = np.ones(33)
        if signs == "opposite":
            s[:8] = -1.0
        elif signs == "mixed":
            s = rng.choice([-1.0, 1.0], 33)
        v = np.ascontiguousarray(v * s)
        c, n = float(v[0]), np.ascontiguousarray(v[8:14])
        taken = fx.lap6(c, ptr(n), C.byref(out))
        check(taken, out.value, [-6] + [1] * 6, [c] + list(n), 6, e)
        q, o = np.ascontiguousarray(v[:8]), np.ascontiguousarray(v[8:32])
        taken = fx.group(ptr(q), ptr(o), C.byref(out))
        check(taken, out.value, [-3] * 8 + [1] * 24, list(q) + list(o), 4, e)


def test_infinities_are_declined(fx):
    ptr = lambda a: a.ctypes.data_as(C.POINTER(C.c_double))  # noqa: E731
    out = C.c_double()
    for bad in (np.inf, -np.inf, np.nan):
        v = np.ones(24)
        v[3] = bad
        assert not fx.lap6(1.0, ptr(v), C.byref(out))
        assert not fx.group(ptr(np.ones(8)), ptr(v), C.byref(out))
