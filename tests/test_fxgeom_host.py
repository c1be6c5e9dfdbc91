"""The fixed-point chart (csrc/lcq_fxgeom.cuh), compiled for the host, against the same polynomials in
80-bit arithmetic, beside the FP64 recurrences that it replaces: point, normal and basis values at
random points of patches that resolve their surface and of patches too coarse for their degree."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2006_02545_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
U = 2.0 ** -53

SRC = r"""
#include <cuda_runtime.h>
#include <algorithm>
#include <cmath>
#include <cstring>
using std::max; using std::min;
// what the headers take from the device compiler, for one thread
#define __noinline__
struct Idx { int x, y, z; };
static Idx threadIdx{0, 0, 0}, blockDim{1, 1, 1};
inline void __syncthreads() {}
inline void __syncwarp() {}
inline double __longlong_as_double(long long b) { double x; memcpy(&x, &b, 8); return x; }
inline double rsqrt(double x) { return 1.0 / sqrt(x); }
inline float rsqrtf(float x) { return 1.0f / sqrtf(x); }
inline double __shfl_xor_sync(unsigned, double v, int) { return v; }
template <class T>
inline cudaError_t cudaMemcpyToSymbolAsync(T&, const void*, size_t, size_t, cudaMemcpyKind, cudaStream_t) {
  return cudaSuccess;
}
#include "lcq_device.cuh"
using namespace lcq;
typedef long double LD;

template <int D>
struct Probe {
  static constexpr int n = (D + 1) * (D + 2) / 2, nd = D * (D + 1) / 2;
  double cf[3 * n], cd[6 * nd + 1], R = 0.0;
  FxChart<D> ch;

  static void tables() {
    for (int nn = 0; nn <= kMaxDeg; ++nn)
      for (int m = 0; m <= nn; ++m) {
        const int i = nn * (nn + 1) / 2 + m;
        double b = 1.0;
        for (int k = 1; k <= nn - m; ++k) b = b * (2 * m + 1 + k) / k;
        c_kw[i] = sqrt(2.0 * (2 * m + 1) * (nn + 1));
        frexp(c_kw[i] * b * (1.0 + 1e-12), &c_kwexp[i]);
      }
    const FxBasisTables t = fx_basis_tables(c_kwexp);
    memcpy(c_fxj, t.j, sizeof(t.j));
    memcpy(c_fxj0, t.j0, sizeof(t.j0));
    memcpy(c_fxq, t.q, sizeof(t.q));
    for (int m = 0; m <= kMaxDeg; ++m)
      for (int a = 0; m + a < kMaxDeg; ++a) {
        double* j = c_jac + (m * (kMaxDeg + 1) + a) * 3;
        jacobi_coef(a, 2 * m + 1, j, j + 1, j + 2);
      }
  }

  // the chart of the patch with nodes xyz [3][n], about their mean
  explicit Probe(const double* xyz) {
    tables();
    DegTables dt;
    build_deg_tables(D, &dt);
    for (int c = 0; c < 3; ++c) {
      double mean = 0.0;
      for (int l = 0; l < n; ++l) mean += xyz[c * n + l] / n;
      for (int i = 0; i < n; ++i) {
        LD a = 0;
        for (int l = 0; l < n; ++l) a += (LD)dt.V[i * n + l] * (xyz[c * n + l] - mean);
        cf[3 * i + c] = (double)a;
      }
    }
    std::vector<double> duv(dt.Du);
    duv.insert(duv.end(), dt.Dv.begin(), dt.Dv.end());
    load_coef_derivs<D>(cf, duv.data(), cd);
    double s[12] = {0};
    fx_chart_sums<D>(cf, cd, 0, 1, s);
    R = sqrt(2.0 * s[9]);
    fx_chart_scales<D>(s, &ch);
    memcpy(ch.d, cd, sizeof(ch.d));
    fx_chart_store<D>(cf, 0, 1, &ch);
  }

  // X, X_u, X_v and the basis in 80 bits, from the arguments of the recurrences as every form takes
  // them, in FP64
  void exact(double u, double v, LD (*X)[3], LD* K) const {
    const double sd = 2.0 * u + v - 1.0, qd = 1.0 - v, yd = 1.0 - 2.0 * v;
    const LD s = sd, q2 = (LD)qd * qd, y = yd;
    LD Lp = 0, L = 1;
    for (int m = 0; m <= D; ++m) {
      if (m > 0) {
        const LD Ln = ((2 * m - 1) * s * L - (m - 1) * q2 * Lp) / m;
        Lp = L;
        L = Ln;
      }
      LD Pp = 0, P = 1;
      for (int a = 0; a <= D - m; ++a) {
        const int nn = m + a, b = 2 * m + 1;
        K[nn * (nn + 1) / 2 + m] = sqrtl((LD)(2 * b * (nn + 1))) * L * P;
        const LD den = 2.0L * (a + 1) * (a + b + 1) * (2 * a + b);
        const LD Pn = (((LD)(2 * a + b + 1) * (2 * a + b + 2) * (2 * a + b)) * y -
                       (LD)(2 * a + b + 1) * b * b) / den * P -
                      (LD)(2 * a) * (a + b) * (2 * a + b + 2) / den * Pp;
        Pp = P;
        P = Pn;
      }
    }
    for (int k = 0; k < 3; ++k)
      for (int c = 0; c < 3; ++c) {
        const double* x = k == 0 ? cf : cd + (k - 1) * 3 * nd;
        X[k][c] = 0;
        for (int i = 0; i < (k == 0 ? n : nd); ++i) X[k][c] += x[3 * i + c] * K[i];
      }
  }

  // out: largest errors of X / R, N / (|X_u| |X_v|), K 2^-E in fixed point (rows), N and K without
  // rows, then X and N by the FP64 recurrences; fp64
  void run(int points, unsigned seed, double* out) {
    for (int i = 0; i < 8; ++i) out[i] = 0.0;
    out[7] = ch.fp64;
    if (ch.fp64) return;
    auto worst = [&](int i, LD e) { out[i] = fmax(out[i], (double)e); };
    srand48(seed);
    for (int it = 0; it < points; ++it) {
      double u = drand48(), v = drand48();
      if (u + v > 1.0) u = 1.0 - u, v = 1.0 - v;
      LD X[3][3], K[n], N[3];
      exact(u, v, X, K);
      LD lu = 0, lv = 0;
      for (int c = 0; c < 3; ++c) {
        N[c] = X[1][(c + 1) % 3] * X[2][(c + 2) % 3] - X[1][(c + 2) % 3] * X[2][(c + 1) % 3];
        lu += X[1][c] * X[1][c];
        lv += X[2][c] * X[2][c];
      }
      const LD l = sqrtl(lu * lv);
      u64 row[FxRow<D>::size];
      double kr[KwRow<D>::size], x[3], xu[3], xv[3], kk[n], nn[3];
      for (int m = 0; m <= D; ++m) {
        fx_row_factors<D>(v, m, ch, row);
        kw_row_factors<D>(v, m, cf, cd, kr);
      }
      const FxS s = fx_split(fx_fix(2.0 * u + v - 1.0, 0));
      i64 Xi[3], Ni[3], Mi[3];
      int sn, sm;
      fx_chart_point<D>(s, row, ch.su, ch.sv, Xi, Ni, &sn);
      fx_basis_point<D>(s, row, 0, 1, [&](int i, i64 k) {
        worst(2, fabsl(ldexpl(k, -59) - ldexpl(K[i], -c_kwexp[i])));
      });
      fx_basis_normal<D>(u, v, ch, Mi, &sm, [&](int i, i64 k) {
        worst(4, fabsl(ldexpl(k, -62) - ldexpl(K[i], -c_kwexp[i])));
      });
      kw_geometry_row<D>(u, kr, x, xu, xv, kk);
      cross3(xu, xv, nn);
      LD e[5] = {0, 0, 0, 0, 0};
      for (int c = 0; c < 3; ++c) {
        e[0] += powl(ldexpl(Xi[c], ch.sx - 59) - X[0][c], 2);
        e[1] += powl(ldexpl(Ni[c], sn - 61) - N[c], 2);
        e[2] += powl(ldexpl(Mi[c], sm - 61) - N[c], 2);
        e[3] += powl(x[c] - X[0][c], 2);
        e[4] += powl(nn[c] - N[c], 2);
      }
      worst(0, sqrtl(e[0]) / R);
      worst(1, sqrtl(e[1]) / l);
      worst(3, sqrtl(e[2]) / l);
      worst(5, sqrtl(e[3]) / R);
      worst(6, sqrtl(e[4]) / l);
    }
  }
};

// Largest error of the chord of random Taylor coefficients (order g: up to rho^g) against |d| times the
// smallest singular value of the linear part, over cases up to kFxChordMax; their number.
template <int D>
void chord(int cases, double rho, unsigned seed, double* out) {
  constexpr int n = (D + 1) * (D + 2) / 2;
  srand48(seed);
  for (int it = 0; it < cases; ++it) {
    double t[3 * n], mx = 0.0, a = 0.0, b = 0.0, c = 0.0;
    for (int k = 0; k < 3; ++k) {
      double sum = 0.0;
      for (int g = 0; g <= D; ++g)
        for (int j = 0; j <= g; ++j)
          t[k * n + g * (g + 1) / 2 + j] = g == 0 ? 0.0 : (2.0 * drand48() - 1.0) * pow(rho, g);
      for (int e = 1; e < n; ++e) sum += fabs(t[k * n + e]);
      mx = fmax(mx, sum);
      a += t[k * n + 1] * t[k * n + 1];
      b += t[k * n + 1] * t[k * n + 2];
      c += t[k * n + 2] * t[k * n + 2];
    }
    const double smin = sqrt((a + c - sqrt((a - c) * (a - c) + 4.0 * b * b)) / 2.0);
    int st;
    fx_mant(mx, &st);
    if (!(ldexp(1.0, st) <= kFxChordMax * smin)) continue;
    u64 x[3 * n];
    for (int e = 0; e < 3 * n; ++e) x[e] = fx_join28(fx_fix(t[e], st));
    const double r = pow(10.0, -9.0 * drand48()), du = (2.0 * drand48() - 1.0) * r,
                 dv = (2.0 * drand48() - 1.0) * r;
    i64 o[3];
    int e;
    fx_chord<D>(x, du, dv, o, &e);
    LD err = 0;
    for (int k = 0; k < 3; ++k) {
      LD w = 0;
      for (int g = 1; g <= D; ++g)
        for (int j = 0; j <= g; ++j)
          w += (LD)t[k * n + g * (g + 1) / 2 + j] * powl(du, g - j) * powl(dv, j);
      err += powl(ldexpl(o[k], e + st - 61) - w, 2);
    }
    out[0] = fmax(out[0], (double)(sqrtl(err) / (sqrtl((LD)du * du + (LD)dv * dv) * smin)));
    out[1] += 1.0;
  }
}
extern "C" void chords(int d, int cases, double rho, unsigned seed, double* out) {
  out[0] = out[1] = 0.0;
  switch (d) {
#define CHORD(D) case D: chord<D>(cases, rho, seed, out); break;
    CHORD(1) CHORD(2) CHORD(3) CHORD(4) CHORD(5) CHORD(6) CHORD(7) CHORD(8) CHORD(9) CHORD(10)
  }
}

extern "C" void probe(int d, const double* xyz, int points, unsigned seed, double* out) {
  switch (d) {
#define CASE(D) case D: { Probe<D> p(xyz); p.run(points, seed, out); break; }
    CASE(1) CASE(2) CASE(3) CASE(4) CASE(5) CASE(6) CASE(7) CASE(8) CASE(9) CASE(10)
  }
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not shutil.which("g++") or not os.path.exists(nvcc):
        pytest.skip("needs g++ and the CUDA headers")
    if np.finfo(np.longdouble).nmant < 60:
        pytest.skip("needs a long double of 64 bits")
    d = tmp_path_factory.mktemp("fxgeom")
    csrc = os.path.join(ROOT, "paper_2006_02545_gb300", "csrc")
    (d / "p.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", csrc, "-I",
                    os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include"),
                    str(d / "p.cpp"), os.path.join(csrc, "lcq_tables.cpp"), "-o", str(d / "p.so")],
                   check=True)
    lib = C.CDLL(str(d / "p.so"))
    f = lib.probe

    def surface(s, patches=24, points=40):
        """Worst errors over some patches that the fixed point takes, and the share that it does not."""
        rows = []
        for j in np.unique(np.linspace(0, s.n_patches - 1, patches).astype(int)):
            x = np.ascontiguousarray(s.xyz[:, s.node_off[j]:s.node_off[j + 1]])
            o = np.zeros(8)
            f(int(s.deg[j]), x.ctypes.data_as(C.c_void_p), points, int(j), o.ctypes.data_as(C.c_void_p))
            rows.append(o)
        rows = np.array(rows)
        return rows[:, :7].max(axis=0), rows[:, 7].mean()

    def chords(deg, rho):
        o = np.zeros(2)
        lib.chords(deg, 2000, C.c_double(rho), deg, o.ctypes.data_as(C.c_void_p))
        return o
    surface.chords = chords
    return surface


RESOLVED = [W.ellipsoid(1, d, axes=(1.0, 1.2, 0.9)) for d in range(1, 6)] + [
    W.ellipsoid(4, 6, axes=(1.0, 2.0, 3.0)), W.ellipsoid(2, 10), W.torus(27, 54, 6),
    W.torus(11, 11, 8), W.stellarator(20, 60, 3), W.stellarator(10, 10, 5)]
COARSE = [W.torus(3, 3, 8), W.torus(3, 5, 8), W.torus(3, 9, 6), W.torus(3, 3, 10)]


@pytest.mark.parametrize("i", range(len(RESOLVED) + len(COARSE)))
def test_errors(probe, i):
    """Where the fixed point is taken it is as near to the exact chart as the FP64 recurrences.
    Its roundings are half units 2^-59 of the scale, n + 3 (D + 1) of them in X (the products of the
    sums and of the stored factors): with the scale at most 48 times the root mean square and the
    roundings adding in quadrature 2.5 (3 (n + 3 D + 3))^(1/2) 2^-60 48 < 8 u at the largest degree;
    twice that for the normal, which takes both derivatives.  The basis carries 2^-57."""
    s = (RESOLVED + COARSE)[i]
    e, flagged = probe(s)
    if i < len(RESOLVED):
        assert flagged == 0.0
    else:
        assert flagged > 0.5
    assert e[0] <= 8 * U and e[1] <= 16 * U and e[3] <= 16 * U, e / U
    assert e[2] <= 2.0 ** -56 and e[4] <= 2.0 ** -56, e * 2.0 ** 56
    assert e[0] <= 2 * e[5] and e[1] <= 2 * e[6], e / U


@pytest.mark.parametrize("deg", range(1, 11))
@pytest.mark.parametrize("rho", [0.2, 0.4])
def test_chord(probe, deg, rho):
    """The self rules' chord: n coefficients rounded to 2^-59 of the scale and as many powers of d, in
    quadrature below 2^-56 |d| times the scale, which is at most 32 times the smallest singular
    value of the tangents: 8 u, near the node as away from it."""
    err, cases = probe.chords(deg, rho)
    assert cases > 200 and err <= 8 * U, (err / U, cases)
