"""The fixed-point kernel value (csrc/lcq_fx.cuh), compiled for the host, against 50-digit
arithmetic at the same inputs, over all kernels (S, D, CFIE; real and complex k and
coefficients, either sign of k), eight decades of distance and the ends of its range."""
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
#include <vector>
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
        return (out[0] + 1j * out[1]) if ok else None
    return one


def reference(kind, kp, d, n, W):
    """(value, magnitude of its terms) with 50 digits."""
    k, al, be = mp.mpc(kp[0], kp[1]), mp.mpc(kp[2], kp[3]), mp.mpc(kp[4], kp[5])
    if kind != 2:
        al, be = (mp.mpf(0), mp.mpf(1)) if kind == 0 else (mp.mpf(1), mp.mpf(0))
    r = mp.sqrt(sum(mp.mpf(float(x)) ** 2 for x in d))
    nd = sum(mp.mpf(float(x)) * mp.mpf(float(y)) for x, y in zip(n, d))
    e = mp.exp(1j * k * r) / r * mp.mpf(W)
    return (e * (al * (1 - 1j * k * r) * nd / r ** 2 + be),
            abs(e) * (abs(al) * abs(1 - 1j * k * r) / r + abs(be)))


KERNELS = [(0, (1.0, 0, 0, 0, 0, 0)), (0, (0.0, 0, 0, 0, 0, 0)), (0, (20.0, 0.4, 0, 0, 0, 0)),
           (1, (6.28, 0, 0, 0, 0, 0)), (1, (7.3, 0.4, 0, 0, 0, 0)),
           (2, (6.28, 0, 1, 0, 0, -6.28)), (2, (-5.0, 0, 1, 0, 0.3, 0.1)),
           (2, (20.0, 0.3, 0.7, 0.2, 0.5, -20.0)), (2, (3.0, 0, 1e-3, 0, 5.0, 0)),
           (2, (3.0, 0, 0, 0, 0, 2.0))]


@pytest.mark.parametrize("kind,kp", KERNELS)
@pytest.mark.parametrize("ints", [True, False])
def test_value(fx, kind, kp, ints):
    rng = np.random.default_rng(5)
    for i in range(300):
        r = 10.0 ** rng.uniform(-7, 1.5)
        d = rng.standard_normal(3)
        n = rng.standard_normal(3)
        n /= np.linalg.norm(n)
        if i % 4 == 1:                       # tangent plane
            d -= n * (n @ d)
        if i % 4 == 2:                       # axes, where components vanish
            d = np.eye(3)[i % 3] * rng.choice([-1.0, 1.0])
            n = np.eye(3)[(i // 3) % 3] * rng.choice([-1.0, 1.0])
        if i % 4 == 3:
            d[i % 3] *= 1e-9
        d *= r / np.linalg.norm(d)
        W = 10.0 ** rng.uniform(-12, 2)
        got = fx(kind, kp, d, n, W, ints)
        want, mag = reference(kind, kp, d, n, W)
        # 1/r, r and the products carry 2^-55 each, c = n.d/r 2^-55 absolute, the phase and the
        # decay 2^-56 (|k| r); the result is rounded to FP64: within 4 u of the terms, and u / 4
        # per radian of phase or decay
        tol = U * (4.0 + 0.25 * abs(complex(kp[0], kp[1])) * r)
        assert abs(mp.mpc(got) - want) <= tol * mag, (i, r, d, n)


def test_range(fx):
    """Outside its range the evaluation says so instead of answering."""
    n = np.array([0.0, 0.0, 1.0])
    kp = (1.0, 0, 1, 0, 1, 0)
    assert fx(2, kp, [0.0, 0.0, 0.0], n, 1.0, True) is None          # coincident points
    assert fx(2, kp, [1e-95, 0.0, 0.0], n, 1.0, True) is None        # |d| < 2^-300
    assert fx(2, kp, [1e95, 0.0, 0.0], n, 1.0, True) is None
    assert fx(2, kp, [np.nan, 0.0, 1.0], n, 1.0, True) is None
    assert fx(2, kp, [np.inf, 0.0, 1.0], n, 1.0, True) is None
    assert fx(0, (1e9, 0, 0, 0, 0, 0), [1.0, 0.0, 0.0], n, 1.0, True) is None   # phase
    assert fx(0, (1.0, 1e5, 0, 0, 0, 0), [1.0, 0.0, 0.0], n, 1.0, True) is None  # decay
    assert fx(2, (1e200, 0, 1e200, 0, 0, 0), [1.0, 0.0, 0.0], n, 1.0, True) is None  # alpha k
    for r in (1e-90, 1e-30, 1e30, 1e89):                             # inside: S, k = 0
        got = fx(0, (0.0, 0, 0, 0, 0, 0), [0.0, r, 0.0], n, 1.0, True)
        assert abs(got - 1.0 / r) <= 4 * U / r
    assert fx(0, (0.0, 0, 0, 0, 0, 0), [0.0, 1.0, 0.0], n, 0.0, True) == 0.0
