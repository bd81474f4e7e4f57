"""The FP64 solve for u_tau (csrc/lbm_newton.h) on the host: its exponential and
logarithm against 40 digits, its root against a bisection."""
import ctypes as ct
import math
import shutil
import subprocess
from decimal import Decimal as D, getcontext

import numpy as np
import pytest

from paper_2304_04214_gb300 import build

getcontext().prec = 40


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("newton")
    (d / "n.cpp").write_text('#include "lbm_newton.h"\nextern "C" {\n'
                             'double e(double x) { double p; return lbmk::exp_neg_d(x, p); }\n'
                             'double l(double z) { return lbmk::log1p_d(z); }\n'
                             'float s(float uhat, float y1, float kap, float B, float guess, int *ok) '
                             '{ bool o; const float u = lbmk::solve_utau_d(uhat, y1, kap, B, guess, &o); *ok = o; '
                             'return u; }\n}\n')
    so = str(d / "n.so")
    subprocess.run([cxx, "-std=c++17", "-O2", "-shared", "-fPIC", "-I", build.CSRC, str(d / "n.cpp"), "-o", so],
                   check=True)
    c = ct.CDLL(so)
    c.e.restype = c.l.restype = ct.c_double
    c.e.argtypes = c.l.argtypes = [ct.c_double]
    c.s.restype = ct.c_float
    c.s.argtypes = [ct.c_float] * 5 + [ct.POINTER(ct.c_int)]
    return c


def test_exponential_and_logarithm(lib):
    """Errors far below the 1e-12 at which the iteration stops, at every argument a
    channel has (y+ from 1e-12 to 1e6); the ends of the series and of its halvings
    among them."""
    edges = [0.05, 0.25, 0.5, 1.0, 2.0, 4.0]
    xs = [10.0 ** p for p in np.linspace(-12, 6, 700)]
    xs += [math.nextafter(x, y) for x in edges for y in (0.0, 10.0)] + edges
    for x in xs:
        if x <= 700.0:
            assert abs(D(lib.e(x)) - (-D(x)).exp()) <= D("1e-15")
        ref = (1 + D(x)).ln()
        assert abs(D(lib.l(x)) - ref) <= D("1e-14") * ref, x
    assert lib.e(1e4) == 0.0 and lib.l(0.0) == 0.0 and lib.e(0.0) == 1.0
    assert math.isnan(lib.e(math.nan)) and math.isnan(lib.l(math.nan))


def test_root(lib):
    """The root rounded to FP32, from guesses far above and below it."""
    rng = np.random.Generator(np.random.PCG64(2))

    def residual(u, uhat, y1, kap, B):
        yp = u * y1
        return u * ((1 + kap * yp).ln() / kap + B * (1 - (-yp / 11).exp() - yp / 11 * (-yp / 3).exp())) - uhat

    for _ in range(60):
        uhat = np.float32(10.0 ** rng.uniform(-7, -0.5))
        y1, kap = np.float32(10.0 ** rng.uniform(1, 5)), np.float32(rng.uniform(0.35, 0.45))
        B = np.float32(rng.uniform(5, 9))
        args = [D(float(v)) for v in (uhat, y1, kap, B)]
        lo, hi = D("1e-8"), D(1)
        for _ in range(60):
            mid = (lo * hi).sqrt()
            lo, hi = (lo, mid) if residual(mid, *args) > 0 else (mid, hi)
        for guess in (1e-3, 1e-1):
            ok = ct.c_int()
            u = lib.s(uhat, y1, kap, B, guess, ct.byref(ok))
            assert ok.value == 1
            # 1e-11 besides half an ulp: the stop of the iteration and of the bisection
            ulp = float(np.spacing(np.float32(u)))
            assert abs(u - float(lo)) <= 0.5 * ulp + 1e-11 * u, (uhat, y1, kap, B)
