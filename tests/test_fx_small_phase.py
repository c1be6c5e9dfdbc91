"""The fixed-point kernel value (csrc/lcq_fx.cuh) at small |k| r, compiled for the host, against
50-digit arithmetic, the real and the imaginary part each by itself: the imaginary part of S is
sin(kr) and of the double layer sin(kr) - kr cos(kr) ~ (kr)^3 / 3, far below the real parts."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
U = 2.0 ** -53

SRC = r"""
#include "lcq_fx.cuh"
using namespace lcq;
extern "C" int fx_one(const u64* cs, const u64* dec, int kind, const double* kp, const double* d,
                      const double* n, double W, int ints, double* out) {
  const FxKernel K = fx_kernel(kind, kp[0], kp[1], kp[2], kp[3], kp[4], kp[5]);
  FxS ns[3];
  for (int c = 0; c < 3; ++c) ns[c] = fx_split(fx_fix(n[c], 0));
  int ew;
  const u64 w = (u64)fx_mant(W, &ew);
  const FxTables t = {(const FxCs*)cs, dec};
  return ints ? fx_eval<true>(K, t, d[0], d[1], d[2], ns, w, ew, out, out + 1, nullptr, 0, 0, 0, 0, 0)
              : fx_eval<false>(K, t, d[0], d[1], d[2], ns, w, ew, out, out + 1, nullptr, 0, 0, 0, 0, 0);
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("fx")
    src, lib = d / "fx.cpp", d / "fx.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2006_02545_gb300", "csrc"), str(src), "-o", str(lib)],
                   check=True)
    f = C.CDLL(str(lib)).fx_one
    mp.mp.dps = 50
    cs = np.zeros((1024, 2), np.uint64)
    dec = np.zeros(1024, np.uint64)
    for j in range(1024):
        a = 2 * mp.pi * j / 4096
        cs[j] = [int(mp.nint(mp.cos(a) * 2 ** 62)), int(mp.nint(mp.sin(a) * 2 ** 62))]
        dec[j] = int(mp.nint(mp.mpf(2) ** (-mp.mpf(j) / 1024) * 2 ** 62))

    def one(kind, kp, d, n, W, ints):
        out = np.zeros(2)
        a = [np.ascontiguousarray(v, dtype=np.float64) for v in (kp, d, n)]
        ok = f(cs.ctypes.data_as(C.c_void_p), dec.ctypes.data_as(C.c_void_p), kind,
               *[v.ctypes.data_as(C.c_void_p) for v in a], C.c_double(W), int(ints),
               out.ctypes.data_as(C.c_void_p))
        assert ok
        return out

    one.covers = lambda kind, kp, d, n, W, ints: bool(f(
        cs.ctypes.data_as(C.c_void_p), dec.ctypes.data_as(C.c_void_p), kind,
        *[np.ascontiguousarray(v, dtype=np.float64).ctypes.data_as(C.c_void_p) for v in (kp, d, n)],
        C.c_double(W), int(ints), np.zeros(2).ctypes.data_as(C.c_void_p)))
    return one


def reference(kind, kp, d, n, W):
    """The two parts with 50 digits, and for each the sum of its terms' magnitudes, with |n.d| / r
    and with 1 in its place, and the terms' factors beside sin, cos, f and g."""
    kr, ki = mp.mpf(kp[0]), mp.mpf(kp[1])
    al, be = [mp.mpf(x) for x in kp[2:4]], [mp.mpf(x) for x in kp[4:6]]
    if kind != 2:
        al, be = ([0, 0], [1, 0]) if kind == 0 else ([1, 0], [0, 0])
    r = mp.sqrt(sum(mp.mpf(float(x)) ** 2 for x in d))
    c = sum(mp.mpf(float(x)) * mp.mpf(float(y)) for x, y in zip(n, d)) / r
    t = kr * r
    g0 = mp.mpf(W) * mp.exp(-ki * r) / r ** 2
    co, si = mp.cos(t), mp.sin(t)
    f, g = co + t * si, si - t * co
    re = [c * al[0] * f, -c * al[1] * g, ki * r * c * al[0] * co, -ki * r * c * al[1] * si,
          be[0] * r * co, -be[1] * r * si]
    im = [c * al[0] * g, c * al[1] * f, ki * r * c * al[0] * si, ki * r * c * al[1] * co,
          be[0] * r * si, be[1] * r * co]
    nc = 4   # the first four carry c
    factors = g0 * (abs(c) * (abs(al[0]) + abs(al[1])) * (1 + abs(t) + 2 * ki * r) +
                    r * (abs(be[0]) + abs(be[1])))
    return [(g0 * sum(v), g0 * sum(abs(x) for x in v), g0 * sum(abs(x / c) for x in v[:nc]), factors)
            for v in (re, im)]


KERNELS = [(0, lambda k: (k, 0, 0, 0, 0, 0)), (0, lambda k: (-k, 0.3 * k, 0, 0, 0, 0)),
           (1, lambda k: (k, 0, 0, 0, 0, 0)), (1, lambda k: (-k, 0, 0, 0, 0, 0)),
           (1, lambda k: (k, 0.2 * k, 0, 0, 0, 0)), (2, lambda k: (k, 0, 1, 0, 0, -k)),
           (2, lambda k: (-k, 0, 1, 0, 0.3, 0.1)), (2, lambda k: (k, 0.1 * k, 0.7, 0.2, 0.5, -k)),
           (2, lambda k: (k, 0, 1, 0, 1e-9, 1e-12)), (2, lambda k: (k, 0, 0, 1.0, 0, 0))]


@pytest.mark.parametrize("i", range(len(KERNELS)))
@pytest.mark.parametrize("ints", [True, False])
def test_parts(fx, i, ints):
    """Each part within 4 u of its own terms, c = n.d / r with 2^-55 absolute beside them; from 2 pi /
    256 on, where sine and cosine come from the table with 2^-60 absolute, 2^-58 of the factors."""
    kind, kf = KERNELS[i]
    rng = np.random.default_rng(11)
    for it in range(300):
        r = 10.0 ** rng.uniform(-6, 1)
        th = 10.0 ** rng.uniform(-12, 0) if it % 3 else rng.uniform(0.015, 0.05)
        d, n = rng.standard_normal((2, 3))
        n /= np.linalg.norm(n)
        if it % 2:                            # near the tangent plane
            d -= n * (n @ d) * (1.0 - 10.0 ** rng.uniform(-4, 0))
        d *= r / np.linalg.norm(d)
        W = 10.0 ** rng.uniform(-12, 2)
        kp = kf(th / r)
        got = fx(kind, kp, d, n, W, ints)
        table = 2.0 ** -58 if th > 0.999 * 2 * np.pi / 256 else 0.0
        for part, (want, terms, withc, factors) in zip(got, reference(kind, kp, d, n, W)):
            tol = 4 * U * terms + U / 4 * withc + table * factors
            assert abs(mp.mpf(float(part)) - want) <= tol, (it, th, kp)


def test_zero_wave_number(fx):
    """k = 0: the imaginary part is exactly zero."""
    d, n = np.array([0.3, -0.2, 0.5]), np.array([0.6, 0.0, 0.8])
    for kind in (0, 1):
        assert fx(kind, (0.0, 0, 0, 0, 0, 0), d, n, 1.0, True)[1] == 0.0


@pytest.mark.parametrize("kp", [(1.0, 0, 1, 0, np.inf, 0), (1.0, 0, 1, 0, 0, np.nan),
                                (1.0, 0, np.inf, 0, 0, 0), (1.0, 0, 0, np.nan, 1, 0),
                                (np.nan, 0, 1, 0, 1, 0), (1.0, np.inf, 1, 0, 1, 0)])
def test_constants_not_finite(fx, kp):
    """Constants that are not finite are left to the FP64 kernel, which passes them on."""
    assert not fx.covers(2, kp, np.array([0.3, -0.2, 0.5]), np.array([0.6, 0.0, 0.8]), 1.0, True)
