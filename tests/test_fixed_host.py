"""The fixed-point orbit of csrc/mt_fix.cuh, compiled for the host, against
exact rational arithmetic at the ends of its range: points whose own or whose
orbit's real part lies just below 2^(30 - FB)."""
from __future__ import annotations

import ctypes
import os
import shutil
import subprocess
from decimal import Context, Decimal
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include <cstdint>
#include <cstring>
#include <algorithm>
#include "mt_fix.cuh"
using namespace mt;
template <int FB, bool CAP>
static int newton(int m, int lcap, double x, double y, double* q) {
  if (!(fx_fits<FB>(x) && fx_fits<FB>(y))) return -1;  // the caller's binary64 path
  FxVal o;
  const FxTarget T{0, 0, ff{0.f, 0.f}, ff{0.f, 0.f}, true};
  fx_eval<FB, CAP>(m, lcap, 8, fx_from_f64<FB>(x), fx_from_f64<FB>(y), T, o);
  ff qr, qi;
  fx_cmul(o.nr, o.ni, o.ir, o.ii, o.sc, qr, qi);
  q[0] = (double)qr.hi + qr.lo;
  q[1] = (double)qi.hi + qi.lo;
  return o.over ? 1 : 0;
}
extern "C" int fx_newton(int fb, int m, int lcap, double x, double y, double* q) {
  if (fb == 28) return lcap < 1 ? newton<28, false>(m, lcap, x, y, q) : newton<28, true>(m, lcap, x, y, q);
  if (fb == 27) return lcap < 1 ? newton<27, false>(m, lcap, x, y, q) : newton<27, true>(m, lcap, x, y, q);
  return lcap < 1 ? newton<26, false>(m, lcap, x, y, q) : newton<26, true>(m, lcap, x, y, q);
}
extern "C" float rho2(const float* k) { return series_rho2(k[0], k[1], k[2], k[3], k[4], k[5]); }
extern "C" int fx_value(int m, double x, double y, double* v) {  // FB = 28
  if (!(fx_fits<28>(x) && fx_fits<28>(y))) return -1;
  long long wr, wi;
  float dr, di, kr, ki;
  const bool in = fx_value_d32_k<28>(m, fx_from_f64<28>(x), fx_from_f64<28>(y), wr, wi, dr, di, kr, ki);
  v[0] = (double)wr / 72057594037927936.0;
  v[1] = (double)wi / 72057594037927936.0;
  return in ? 0 : 1;
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    d = tmp_path_factory.mktemp("fix")
    src, lib = str(d / "shim.cpp"), str(d / "shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    # -fwrapv: an integer that leaves its range wraps, as on the GPU
    subprocess.run(["g++", "-std=c++17", "-O1", "-fwrapv", "-ffp-contract=off", "-shared", "-fPIC", "-I", inc, "-I",
                    os.path.join(ROOT, "paper_2402_06083_gb300", "csrc"), src, "-o", lib], check=True)
    L = ctypes.CDLL(lib)
    L.fx_newton.argtypes = [ctypes.c_int] * 3 + [ctypes.c_double] * 2 + [ctypes.c_void_p]
    L.fx_value.argtypes = [ctypes.c_int] + [ctypes.c_double] * 2 + [ctypes.c_void_p]
    L.rho2.argtypes = [ctypes.c_void_p]
    L.rho2.restype = ctypes.c_float
    return L


def _exact(m, lcap, x, y):
    """P and P' of p_m (+ p_lcap) at x + iy, exactly."""
    x, y = Fraction(x), Fraction(y)
    z, d, cap = (x, y), (Fraction(1), Fraction(0)), None
    for k in range(1, m + 1):
        if k == lcap:
            cap = (z, d)
        if k < m:
            d = (2 * (z[0] * d[0] - z[1] * d[1]) + 1, 2 * (z[0] * d[1] + z[1] * d[0]))
            z = (z[0] * z[0] - z[1] * z[1] + x, 2 * z[0] * z[1] + y)
    if cap:
        z = (z[0] + cap[0][0], z[1] + cap[0][1])
        d = (d[0] + cap[1][0], d[1] + cap[1][1])
    return z, d


def _quotient(z, d):
    den = d[0] * d[0] + d[1] * d[1]
    return float((z[0] * d[0] + z[1] * d[1]) / den), float((z[1] * d[0] - z[0] * d[1]) / den)


def _edge_points(end):
    """Real or imaginary parts end - 2^-k (both signs), down to the last
    binary64 below the end."""
    e = [end - 2.0 ** -k for k in range(12, 51)] + [float(np.nextafter(end, 0.0))]
    other = [0.0, 0.4, -1.3, 0.75 * end, -0.75 * end, e[0], -e[0], e[20], -e[20], e[-1], -e[-1]]
    return [p for a in e for s in (a, -a) for b in other for p in ((s, b), (b, s))]


def _landing_points(end, rng):
    """c whose c^2 + c has a real part from just below to just above end."""
    out = []
    for _ in range(200):
        y = rng.uniform(-0.9, 0.9) * end ** 0.5
        t = end - 2.0 ** -rng.uniform(18, 45) * rng.choice([1, 1, 1, -1])
        out.append((float((-1 + rng.choice([-1, 1]) * np.sqrt(1 + 4 * (t + y * y))) / 2), float(y)))
    return out


@pytest.mark.parametrize("fb", [28, 27, 26])
@pytest.mark.parametrize("m,lcap", [(1, 0), (2, 0), (3, 0), (4, 0), (6, 0), (3, 1), (5, 2)])
def test_newton_quotient_next_to_the_end_of_the_range(fx, fb, m, lcap):
    """The quotient is off by what its float-float arithmetic allows: a
    multiplication loses 2^-46 and an orbit past the range takes m of them
    for each of P and P', 2^-40 of 1 + |q| for m <= 8."""
    end = 2.0 ** (30 - fb)
    rng = np.random.default_rng(fb + 100 * m)
    q = (ctypes.c_double * 2)()
    seen = 0
    for x, y in _edge_points(end) + _landing_points(end, rng):
        if fx.fx_newton(fb, m, lcap, x, y, q) != 0:
            continue
        z, d = _exact(m, lcap, x, y)
        if d == (0, 0):
            continue
        er, ei = _quotient(z, d)
        if abs(er) + abs(ei) > 64:  # next to a zero of P'
            continue
        seen += 1
        assert abs(q[0] - er) + abs(q[1] - ei) <= 2.0 ** -40 * (1 + abs(er) + abs(ei)), (x, y, q[0], q[1], er, ei)
    assert seen > 200


@pytest.mark.parametrize("m", [2, 3])
def test_value_next_to_the_end_of_the_range(fx, m):
    """The value alone (the mixed tier's finish): three quarters of 2^-56 a
    step, multiplied by the steps that follow (|2 p_k| < 16 in the range).  A
    p_k next to the end, k <= 2 here, is out of the range one step later."""
    rng = np.random.default_rng(m)
    v = (ctypes.c_double * 2)()
    seen = 0
    for x, y in _edge_points(4.0) + _landing_points(4.0, rng):
        if fx.fx_value(m, x, y, v) != 0:
            continue
        z, _ = _exact(m, 0, x, y)
        tol = 2.0 ** -56 * sum(16.0 ** k for k in range(m)) + 2.0 ** -52 * float(abs(z[0]) + abs(z[1]))
        seen += 1
        assert abs(v[0] - float(z[0])) + abs(v[1] - float(z[1])) <= 2 * tol, (x, y)
    assert seen > 20


def _log2_exact(m, x, y):
    """log2 of the larger component of P and of P' of p_m, past any range."""
    C = Context(prec=40, Emax=10 ** 9, Emin=-10 ** 9)
    add, sub, mul = C.add, C.subtract, C.multiply
    x, y, zero = Decimal(x), Decimal(y), Decimal(0)
    zr, zi, dr, di = x, y, Decimal(1), zero
    for _ in range(2, m + 1):
        tr, ti = sub(mul(zr, dr), mul(zi, di)), add(mul(zr, di), mul(zi, dr))
        dr, di = add(add(tr, tr), 1), add(ti, ti)
        zr, zi = add(sub(mul(zr, zr), mul(zi, zi)), x), add(mul(2, mul(zr, zi)), y)
    big = lambda a, b: float(C.ln(max(abs(a), abs(b)))) / np.log(2.0)
    return big(zr, zi), big(dr, di)


@pytest.mark.parametrize("m", [10, 11])
def test_orbits_past_the_range_of_binary64(fx, m):
    """Reported where P or P' reaches 2^1024, whichever comes first (a component
    of a value of that size may be half a bit smaller: a band of one bit at
    either side is left out)."""
    rng = np.random.default_rng(m)
    q = (ctypes.c_double * 2)()
    seen = [0, 0, 0]
    for _ in range(6000):
        r, a = rng.uniform(2.0, 5.6), rng.uniform(0, 2 * np.pi)
        x, y = float(r * np.cos(a)), float(r * np.sin(a))
        got = fx.fx_newton(28, m, 0, x, y, q)
        if got < 0:
            continue
        lp, ld = _log2_exact(m, x, y)
        if abs(max(lp, ld) - 1024) < 1:
            continue
        assert got == (1 if max(lp, ld) > 1024 else 0), (x, y, lp, ld)
        seen[0 if max(lp, ld) < 1024 else 1 if lp > 1024 else 2] += 1
    assert min(seen) >= 5, seen


def test_series_out_of_range_holds_nowhere(fx):
    """The radius of the mixed descents' series: that of its definition, and
    none at all (the anchor's own d = 0 lies outside) for coefficients that
    binary32 cannot hold."""
    inf, nan = float("inf"), float("nan")
    f = lambda *k: fx.rho2((ctypes.c_float * 6)(*k))
    assert abs(f(2.0 ** 30, 0, 2.0 ** 50, 0, 2.0 ** 80, 0) / (1e-4 * 2.0 ** -50) - 1) < 1e-6
    assert abs(f(0, -2.0 ** 30, 0, 2.0 ** 60, 1.0, 0) / (1e-4 * 2.0 ** -60) - 1) < 1e-6
    for C in ((1e37, 0), (0, -2e37), (inf, 0), (nan, 0), (0, nan), (nan, nan), (-inf, nan)):
        assert not 0.0 <= f(2.0 ** 41, 0, 2.0 ** 80, 0, *C), C
    for AB in ((inf, 0, 1, 0), (nan, nan, 1, 0), (1, 0, inf, 0), (1, 0, nan, nan), (2.0 ** 41, 0, 3e38, 3e38)):
        assert not 0.0 <= f(*AB, 1.0, 0.0), AB
