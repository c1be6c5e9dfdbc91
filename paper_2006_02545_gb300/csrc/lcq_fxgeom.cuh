// The chart and the Koornwinder basis at the leaf nodes in 64-bit fixed point.
//
// The moment engine needs, at every node of every subtriangle of the refinement trees, the
// basis values as 7-bit slices of a 56-bit integer (block_moments_tc), the point X and the
// normal X_u x X_v.  In FP64 that is about 170 instructions of 64 cycles a node and 250 a rule
// row.  The basis is bounded on the triangle by construction (|L_m| <= 1, |K_nm| < 2^E_nm) and the
// chart by the sum of its coefficients, so the same recurrences run on 62-bit integers: a
// product is three 32 x 32 multiply-adds of 4 cycles, and the basis slices come out of the
// integers directly.  A basis value carries 2^-57 of its bound 2^E_nm, X 2^-57 of the sum of its
// coefficients times these bounds and the normal 2^-57 of such sums of the derivatives, below FP64's
// rounding of the same recurrences as long as the sums are not far above the chart itself; a chart
// where they are takes the FP64 recurrences (FxChart::fp64).
#pragma once

#include "lcq_device.cuh"

namespace lcq {

// A value as a high word and 28 bits of the low one, v = h 2^32 + 16 l, rounded.  A stored one has l
// of either sign (fx_join28), the other factor l >= 0 (fx_28): of their product h h' + (h l' + l h') /
// 2^28 the part l l' is left out, which has no one sign that a sum would add up.  Sums of up to
// 63 cross products h l', |v| < 2^62, stay below 2^63.
__device__ __forceinline__ u64 fx_join28(i64 v) {
  v += 8;
  const u64 h = (u64)(v >> 32) + ((uint32_t)v >> 31);
  return (h << 32) | (uint32_t)((int)(uint32_t)v >> 4);
}
__device__ __forceinline__ FxS fx_28(FxS a) { return {a.h, (int)(((uint32_t)a.l + 4u) >> 3)}; }

// Jacobi recurrences of the scaled basis factors (fx_row_factors), filled by upload_kw_tables:
// [m][a]: g1, g0, g2 2^61 (|g1| + |g0| < 2.4, g2 < 1), and the first factor 2^62 of each m.
static __constant__ i64 c_fxj[(kMaxDeg + 1) * (kMaxDeg + 1) * 3];
static __constant__ i64 c_fxj0[kMaxDeg + 1];
// (m - 1) / m (2 / a_m) (2 / a_{m-1}), a_j = (2j - 1) / j: coefficient of (1 - v)^2 in the
// recurrence of the scaled L_m, 2^62 (below 1.07)
static __constant__ i64 c_fxq[kMaxDeg + 1];

// Host values of the three tables.  kwexp: E_nm.
struct FxBasisTables {
  i64 j[(kMaxDeg + 1) * (kMaxDeg + 1) * 3];
  i64 j0[kMaxDeg + 1];
  i64 q[kMaxDeg + 1];
};
inline FxBasisTables fx_basis_tables(const int* kwexp) {
  FxBasisTables t{};
  auto idx = [](int n, int m) { return n * (n + 1) / 2 + m; };
  auto root = [](double p, double q) {  // sqrt(p / q)
    const HostDD x = dd_div({p, 0.0}, q);
    const double h = sqrt(x.h);
    return HostDD{h, (fma(-h, h, x.h) + x.l) / (2.0 * h)};
  };
  auto fix = [](HostDD a, int e) {  // a 2^e rounded
    const double f = ldexp(1.0, e), x = a.h * f;
    const i64 i = (i64)x;
    return i + llrint((x - (double)i) + a.l * f);
  };
  auto rat = [&](double p, double q, HostDD r) { return dd_div(dd_mul({p, 0.0}, r), q); };
  HostDD kappa = {1.0, 0.0};
  for (int m = 0; m <= kMaxDeg; ++m) {
    if (m >= 2) kappa = rat(2.0 * m - 1.0, 2.0 * m, kappa);
    t.q[m] = m < 2 ? 0 : m == 2 ? fix(dd_div({2.0, 0.0}, 3.0), 62)
                                : fix(dd_div({4.0 * (m - 1) * (m - 1), 0.0}, (2.0 * m - 1.0) * (2 * m - 3)), 62);
    auto E = [&](int a) { return kwexp[idx(m + a, m)]; };
    t.j0[m] = fix(dd_mul(kappa, root(2.0 * (2 * m + 1) * (m + 1), 1.0)), 62 - E(0));
    const int b = 2 * m + 1;
    for (int a = 0; m + a < kMaxDeg; ++a) {
      // jacobi_coef times the ratios of c_nm 2^-E_nm
      const double den = 2.0 * (a + 1) * (a + b + 1) * (2 * a + b);
      const HostDD r1 = root(m + a + 2, m + a + 1), r2 = root(m + a + 2, a > 0 ? m + a : 1);
      i64* g = t.j + (m * (kMaxDeg + 1) + a) * 3;
      g[0] = fix(rat((2.0 * a + b + 1) * (2 * a + b + 2) * (2 * a + b), den, r1), 61 + E(a) - E(a + 1));
      g[1] = -fix(rat((2.0 * a + b + 1) * b * b, den, r1), 61 + E(a) - E(a + 1));
      g[2] = a == 0 ? 0 : fix(rat(2.0 * a * (a + b) * (2 * a + b + 2), den, r2),
                              61 + E(a - 1) - E(a + 1));
    }
  }
  return t;
}

static inline cudaError_t upload_fx_basis(const int* kwexp, cudaStream_t st) {
  const FxBasisTables t = fx_basis_tables(kwexp);
  cudaError_t e = cudaMemcpyToSymbolAsync(c_fxj, t.j, sizeof(t.j), 0, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess)
    e = cudaMemcpyToSymbolAsync(c_fxj0, t.j0, sizeof(t.j0), 0, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess)
    e = cudaMemcpyToSymbolAsync(c_fxq, t.q, sizeof(t.q), 0, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);  // t lives on this stack
  return e;
}

// A patch's chart in fixed point: coefficients x_nm 2^(E_nm + 62 - sx) and the derivative
// series' with their own scales su and sv, each scale above the sum of the magnitudes |x_nm| 2^E_nm,
// so that every partial sum stays below 1.  fp64: the chart is far below its scales or not finite;
// x and d then hold the FP64 coefficients and the nodes take the FP64 recurrences.
template <int D>
struct FxChart {
  static constexpr int n = (D + 1) * (D + 2) / 2, nd = D * (D + 1) / 2;
  u64 x[3 * n];
  u64 d[6 * nd];   // X_u then X_v
  int sx, su, sv, fp64;
};

// The fixed-point errors are fractions of the scales, the FP64 recurrences' of the chart itself, and
// the bounds 2^E_nm are reached at a corner only: where the high coefficients are not small
// beside the low ones (patches too coarse for their degree), the scales are far above the chart.
// Largest errors of 120 points, X against R and the normal against its length, fixed and
// FP64: scale / root mean square of up to 3 (1280-patch ellipsoid, degree 6) 4.5e-17 and 4.5e-16,
// 6e-17 and 1e-15; up to 20 (242-patch torus, degree 8) 1e-16 and 4.8e-16, 4e-16 and 2e-15; up to 50
// (110-patch torus, degree 8; 128 patches) 1.2e-16 and 4.1e-16, 5e-16 to 9e-16 and 1.6e-15; 60 to 90
// (54-patch torus, degree 6) 3e-16 and 5e-16, 1.7e-15 and 1.7e-15; 220 to 760 (30 patches, degree 8)
// 1e-15 and 5e-16, 1.2e-14 and 1.7e-15; 900 to 2800 (18 patches, degree 8) 5e-15 and 4e-16, 1e-13 and
// 5e-15.
constexpr double kFxChartMax = 48.0;

// Sums over the coefficients i0, i0 + step, ...: s[k][c] of |coefficient| 2^E_nm of component c of
// (X, X_u, X_v)[k], s[9 + k] of the squared coefficients.
template <int D>
__device__ __forceinline__ void fx_chart_sums(const double* cf, const double* d, int i0, int step,
                                              double* s) {
  constexpr int n = FxChart<D>::n, nd = FxChart<D>::nd;
  for (int i = i0; i < n; i += step) {
    const double p2 = __longlong_as_double((long long)(c_kwexp[i] + 1023) << 52);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double a = cf[3 * i + c];
      s[c] += fabs(a) * p2;
      s[9] = fma(a, a, s[9]);
      if (i < nd) {
        const double u = d[3 * i + c], v = d[3 * (nd + i) + c];
        s[3 + c] += fabs(u) * p2;
        s[6 + c] += fabs(v) * p2;
        s[10] = fma(u, u, s[10]);
        s[11] = fma(v, v, s[11]);
      }
    }
  }
}
// The scales from the whole sums: the area of T0 is 1/2, so the root mean square of a series is
// (2 sum of squares)^(1/2).
template <int D>
__device__ __forceinline__ void fx_chart_scales(const double* s, FxChart<D>* ch) {
  int e[3];
  ch->fp64 = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double m = fmax(s[3 * k], fmax(s[3 * k + 1], s[3 * k + 2]));
    fx_mant(m, &e[k]);
    e[k] = max(e[k], -1000);
    const double rms = sqrt(2.0 * s[9 + k]);
    // (a sum that is not finite makes the squares' sum so too)
    if (!(s[9 + k] < 1e300) || !(m < 1e150) || (m > 0.0 && !(ldexp(1.0, e[k]) <= kFxChartMax * rms)))
      ch->fp64 = 1;
  }
  ch->sx = e[0];
  ch->su = e[1];
  ch->sv = e[2];
}
// Entries i0, i0 + step, ... of the coefficients; d holds the FP64 derivative series before.
template <int D>
__device__ __forceinline__ void fx_chart_store(const double* cf, int i0, int step, FxChart<D>* ch) {
  constexpr int n = FxChart<D>::n, nd = FxChart<D>::nd;
  for (int i = i0; i < 3 * n; i += step)
    ch->x[i] = ch->fp64 ? fx_bits(cf[i]) : fx_join28(fx_fix(cf[i], ch->sx - c_kwexp[i / 3]));
  if (ch->fp64) return;
  for (int i = i0; i < 6 * nd; i += step) {
    const int k = i / 3;
    const double v = fx_double(ch->d[i]);
    ch->d[i] = k < nd ? fx_join28(fx_fix(v, ch->su - c_kwexp[k]))
                      : fx_join28(fx_fix(v, ch->sv - c_kwexp[k - nd]));
  }
}

// By the block's threads, from the coefficients cf and the projections duv (load_coef_derivs);
// begins and ends with a barrier.  FP64: the chart stays in FP64 whatever its scales.
template <int D, bool FP64 = false>
__device__ void load_fx_chart(const double* cf, const double* __restrict__ duv, FxChart<D>* ch) {
  __syncthreads();
  load_coef_derivs<D>(cf, duv, reinterpret_cast<double*>(ch->d));
  __syncthreads();
  if (threadIdx.x < 32) {
    double s[12] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    fx_chart_sums<D>(cf, reinterpret_cast<const double*>(ch->d), threadIdx.x, 32, s);
#pragma unroll
    for (int k = 0; k < 12; ++k)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
    if (threadIdx.x == 0) {
      fx_chart_scales<D>(s, ch);
      if (FP64) ch->fp64 = 1;
    }
  }
  __syncthreads();
  fx_chart_store<D>(cf, threadIdx.x, blockDim.x, ch);
  __syncthreads();
}

__device__ __forceinline__ void fx_mac28(i64& hh, i64& t, FxS a, FxS b) {
  hh += fx_swide(a.h, b.h);
  t += fx_swide(a.h, b.l) + fx_swide(a.l, b.h);
}

// A rule row (nodes of one v): [Q (D+1), J (n), BX (3 (D+1)), BU (3 D), BV (3 D)], 62-bit values:
// Q[m] the (1 - v)^2 term of the L recurrence, J_nm 2^-E_nm times the scale of L_m (split with 31
// bits), BX, BU, BV the chart's sums over n at fixed m (28 bits).
template <int D>
struct FxRow {
  static constexpr int n = (D + 1) * (D + 2) / 2;
  static constexpr int Q = 0, J = Q + D + 1, BX = J + n, BU = BX + 3 * (D + 1), BV = BU + 3 * D;
  static constexpr int size = BV + 3 * D;
};

// (1 - v)^2 2^62, and the coefficient of L_{m-2} in the recurrence of the scaled L_m (2^62).
__device__ __forceinline__ FxS fx_q2(double v) {
  const FxS q = fx_split(fx_fix(1.0 - v, 0));
  return fx_split(fx_smul_sl<2>(q, q) + 1);  // (the products truncate)
}
__device__ __forceinline__ FxS fx_Q(int m, FxS q2) {
  return fx_split(fx_smul_sl<2>(fx_split(c_fxq[m]), q2) + 1);
}

// The part of the row factors that belongs to one m (Q too when m = 0), so that a block
// spreads a row over D + 1 threads.
template <int D>
__device__ __forceinline__ void fx_row_factors(double v, int m, const FxChart<D>& ch, u64* row) {
  using RW = FxRow<D>;
  constexpr int nd = FxChart<D>::nd;
  if (m == 0) {
    const FxS q2 = fx_q2(v);
#pragma unroll 1
    for (int mm = 2; mm <= D; ++mm) row[RW::Q + mm] = fx_join(fx_Q(mm, q2));
  }
  const FxS y = fx_split(fx_fix(1.0 - 2.0 * v, 0));
  const i64* g = c_fxj + m * (kMaxDeg + 1) * 3;
  i64 J = c_fxj0[m], Jp = 0;
  i64 h[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0}, t[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll 1
  for (int a = 0; a <= D - m; ++a) {
    const int nn = m + a, idx = nn * (nn + 1) / 2 + m;
    const FxS Js = fx_split(J), J8 = fx_28(Js);
    row[RW::J + idx] = fx_join(Js);
#pragma unroll
    for (int c = 0; c < 3; ++c) fx_mac28(h[c], t[c], J8, fx_unjoin(ch.x[idx * 3 + c]));
    if (nn < D) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        fx_mac28(h[3 + c], t[3 + c], J8, fx_unjoin(ch.d[idx * 3 + c]));
        fx_mac28(h[6 + c], t[6 + c], J8, fx_unjoin(ch.d[(nd + idx) * 3 + c]));
      }
      // J_{a+1} = (g1 y + g0) J_a - g2 J_{a-1}
      const FxS f = fx_split(fx_smul_sl<2>(fx_split(g[3 * a]), y) + g[3 * a + 1]);
      const FxS g2 = fx_split(g[3 * a + 2]), Jq = fx_split(Jp);
      const i64 tt = fx_swide(f.h, Js.l) + fx_swide(f.l, Js.h) - fx_swide(g2.h, Jq.l) -
                     fx_swide(g2.l, Jq.h);
      Jp = J;
      J = (i64)((u64)(fx_swide(f.h, Js.h) - fx_swide(g2.h, Jq.h)) << 3) + ((tt + (1 << 28)) >> 28);
    }
  }
  auto out = [&](int o, int k) { row[o] = fx_join28((h[k] << 2) + (t[k] >> 26)); };
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    out(RW::BX + 3 * m + c, c);
    if (m < D) {
      out(RW::BU + 3 * m + c, 3 + c);
      out(RW::BV + 3 * m + c, 6 + c);
    }
  }
}

// Next of the scaled L_m (|L| < 2.84, unit 2^-61): 2 s L - Q Lp, s 2^62 and Q 2^62.  Rounded up by
// the half unit that fx_split then drops on average: a recurrence adds up such biases (K too).
__device__ __forceinline__ i64 fx_next_L(FxS s, FxS L, FxS Q, FxS Lp) {
  const i64 ta = fx_swide(s.h, L.l) + fx_swide(s.l, L.h);
  const i64 tb = fx_swide(Q.h, Lp.l) + fx_swide(Q.l, Lp.h);
  return (i64)(((u64)fx_swide(s.h, L.h) << 3) - ((u64)fx_swide(Q.h, Lp.h) << 2) +
               (u64)(((ta + (1 << 28)) >> 28) - ((tb + (1 << 28)) >> 29)));
}

// X_u x X_v = N 2^(sn - 61) of the integers v = (X_u 2^(62 - su), X_v 2^(62 - sv)).  Both vectors
// are brought to full length first: on a coarse patch they are far below their scales, and the
// product would lose the square of that.
__device__ __forceinline__ void fx_cross(const i64* v, int su, int sv, i64* N, int* sn) {
  FxS d[6];
  int sh[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    u64 m = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) m |= (u64)(v[3 * k + c] ^ (v[3 * k + c] >> 63));
    sh[k] = fx_min(fx_clz(m) - 2, 61);
#pragma unroll
    for (int c = 0; c < 3; ++c) d[3 * k + c] = fx_split(v[3 * k + c] << sh[k]);
  }
  *sn = su + sv - sh[0] - sh[1];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const FxS a = d[(c + 1) % 3], b = d[3 + (c + 2) % 3], e = d[(c + 2) % 3], f = d[3 + (c + 1) % 3];
    const i64 tt = fx_swide(a.h, b.l) + fx_swide(a.l, b.h) - fx_swide(e.h, f.l) - fx_swide(e.l, f.h);
    N[c] = (i64)((u64)(fx_swide(a.h, b.h) - fx_swide(e.h, f.h)) << 1) + (tt >> 30);
  }
}

// X (2^(59 - sx)), and the normal X_u x X_v = N 2^(sn - 61) of the node at s = 2u + v - 1 of a row.
template <int D>
__device__ __forceinline__ void fx_chart_point(FxS s, const u64* row, int su, int sv, i64* X, i64* N,
                                               int* sn) {
  using RW = FxRow<D>;
  i64 h[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0}, t[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  FxS L = {1 << 29, 0}, Lp = {0, 0};
#pragma unroll
  for (int m = 0; m <= D; ++m) {
    if (m == 1) {
      Lp = L;
      L = {s.h >> 1, (int)(((uint32_t)(s.h & 1) << 30) | ((uint32_t)s.l >> 1))};
    } else if (m > 1) {
      const FxS Ln = fx_split(fx_next_L(s, L, fx_unjoin(row[RW::Q + m]), Lp));
      Lp = L;
      L = Ln;
    }
    const FxS L8 = fx_28(L);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      fx_mac28(h[c], t[c], L8, fx_unjoin(row[RW::BX + 3 * m + c]));
      if (m < D) {
        fx_mac28(h[3 + c], t[3 + c], L8, fx_unjoin(row[RW::BU + 3 * m + c]));
        fx_mac28(h[6 + c], t[6 + c], L8, fx_unjoin(row[RW::BV + 3 * m + c]));
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) X[c] = h[c] + ((t[c] + (1 << 27)) >> 28);
  i64 d[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) d[c] = (h[3 + c] << 3) + (t[3 + c] >> 25);
  fx_cross(d, su, sv, N, sn);
}

// Basis values of the node: emit(idx, K_nm 2^(59 - E_nm)) for the m of one part of `parts`.
template <int D, class F>
__device__ __forceinline__ void fx_basis_point(FxS s, const u64* row, int part, int parts, F&& emit) {
  using RW = FxRow<D>;
  FxS L = {1 << 29, 0}, Lp = {0, 0};
#pragma unroll
  for (int m = 0; m <= D; ++m) {
    if (m == 1) {
      Lp = L;
      L = {s.h >> 1, (int)(((uint32_t)(s.h & 1) << 30) | ((uint32_t)s.l >> 1))};
    } else if (m > 1) {
      const FxS Ln = fx_split(fx_next_L(s, L, fx_unjoin(row[RW::Q + m]), Lp));
      Lp = L;
      L = Ln;
    }
    if (parts > 1 && m % parts != part) continue;
#pragma unroll
    for (int a = 0; a <= D - m; ++a) {
      const int nn = m + a, idx = nn * (nn + 1) / 2 + m;
      emit(idx, fx_smul(L, fx_unjoin(row[RW::J + idx])));
    }
  }
}

// The node for fx_eval from the integer normal N 2^(sn - 62) and the rule weight wt (area of the
// subtriangle included): unit normal 2^62, W = |N| wt / (4 pi) = wm 2^(ew - 62).
__device__ __forceinline__ void fx_node_from_normal(const i64* N, int sn, double wt, FxS* n, u64* wm,
                                                    int* ew) {
  const int sh =
      fx_clz((u64)((N[0] ^ (N[0] >> 63)) | (N[1] ^ (N[1] >> 63)) | (N[2] ^ (N[2] >> 63)))) - 2;
  if (sh > 60) {  // no area
    n[0] = n[1] = n[2] = {0, 0};
    *wm = 0;
    *ew = 0;
    return;
  }
  const FxS a = fx_split(N[0] << sh), b = fx_split(N[1] << sh), c = fx_split(N[2] << sh);
  const FxRoot rt = fx_root(a, b, c);
  const FxS ri = fx_split((i64)rt.RI);
  n[0] = fx_split(fx_smul_sl<3>(a, ri));
  n[1] = fx_split(fx_smul_sl<3>(b, ri));
  n[2] = fx_split(fx_smul_sl<3>(c, ri));
  int e;
  const u64 m = (u64)fx_mant(wt * 0.07957747154594767, &e);
  const u64 p = fx_umul(rt.R, m);  // |N| W = p 2^(sn - sh + e - 60)
  const int z = fx_clz(p) - 2;
  *wm = z >= 0 && p != 0 ? p << z : p;
  *ew = sn - sh + e + 2 - (p != 0 ? z : 0);
}

// The basis at a point that shares no row with others: emit(idx, K_nm 2^(62 - E_nm)), and the normal
// X_u x X_v = N 2^(sn - 61) from the chart's derivative series.  The recurrence in n runs on
// K_nm itself, started at L_m.
template <int D, class F>
__device__ __forceinline__ void fx_basis_normal(double u, double v, const FxChart<D>& ch, i64* N,
                                                int* sn, F&& emit) {
  constexpr int nd = FxChart<D>::nd;
  const FxS s = fx_split(fx_fix(2.0 * u + v - 1.0, 0)), y = fx_split(fx_fix(1.0 - 2.0 * v, 0));
  const FxS q2 = fx_q2(v);
  i64 h[6] = {0, 0, 0, 0, 0, 0}, t[6] = {0, 0, 0, 0, 0, 0};
  FxS L = {1 << 29, 0}, Lp = {0, 0};
#pragma unroll 1
  for (int m = 0; m <= D; ++m) {
    if (m == 1) {
      Lp = L;
      L = {s.h >> 1, (int)(((uint32_t)(s.h & 1) << 30) | ((uint32_t)s.l >> 1))};
    } else if (m > 1) {
      const FxS Ln = fx_split(fx_next_L(s, L, fx_Q(m, q2), Lp));
      Lp = L;
      L = Ln;
    }
    const i64* g = c_fxj + m * (kMaxDeg + 1) * 3;
    i64 K = fx_smul_sl<3>(L, fx_split(c_fxj0[m])), Kp = 0;
#pragma unroll 1
    for (int a = 0; a <= D - m; ++a) {
      const int nn = m + a, idx = nn * (nn + 1) / 2 + m;
      emit(idx, K);
      if (nn < D) {
        const FxS Ks = fx_split(K), K8 = fx_28(Ks);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          fx_mac28(h[c], t[c], K8, fx_unjoin(ch.d[idx * 3 + c]));
          fx_mac28(h[3 + c], t[3 + c], K8, fx_unjoin(ch.d[(nd + idx) * 3 + c]));
        }
        const FxS f = fx_split(fx_smul_sl<2>(fx_split(g[3 * a]), y) + g[3 * a + 1]);
        const FxS g2 = fx_split(g[3 * a + 2]), Kq = fx_split(Kp);
        const i64 tt = fx_swide(f.h, Ks.l) + fx_swide(f.l, Ks.h) - fx_swide(g2.h, Kq.l) -
                       fx_swide(g2.l, Kq.h);
        Kp = K;
        K = (i64)((u64)(fx_swide(f.h, Ks.h) - fx_swide(g2.h, Kq.h)) << 3) + ((tt + (1 << 28)) >> 28);
      }
    }
  }
  i64 d[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) d[c] = (h[c] << 2) + (t[c] >> 26);
  fx_cross(d, ch.su, ch.sv, N, sn);
}

constexpr double kFxChordMax = 32.0;
// The chord of chart_taylor's coefficients tX 2^(62 - st) (28 bits of the low word; st above the
// sum of their magnitudes) at (du, dv) = (da, db) 2^e: dX = du A + dv B with A and B polynomials,
// so that its error stays a fraction of |d| as the point approaches the node: 2^-58 |d| 2^st, where the
// FP64 Horner form has 2^-53 of the first terms.  2^st is above the sum of all the coefficients, |dX|
// near the node at least |d| times the smallest singular value s of DX; largest relative errors
// over 60 points of a few nodes of 10 patches, fixed and FP64, by 2^st / s: below 6 (320-patch
// sphere, degree 6) 5e-17 and 3e-16; 13 (1458-patch torus, degree 6) 1e-16 and 6e-16; 8 to 47 (50-patch
// twisted torus, degree 8) 2.3e-16 and 2.4e-16; 30 to 176 (20-patch ellipsoid, degree 6) 1.6e-15 and
// 3e-16; 10^3 to 10^4 (the same, degree 10) 2.5e-13 and 6e-16.  So it serves up to kFxChordMax.
// dX = out 2^(e + st - 61).
template <int D>
__device__ __forceinline__ void fx_chord(const u64* tX, double du, double dv, i64* out, int* eout) {
  constexpr int n = (D + 1) * (D + 2) / 2;
  const FxS u = fx_split(fx_fix(du, 0)), v = fx_split(fx_fix(dv, 0));
  i64 h[6] = {0, 0, 0, 0, 0, 0}, t[6] = {0, 0, 0, 0, 0, 0};  // A, then B
  FxS pj = {1 << 30, 0};  // dv^j
#pragma unroll
  for (int j = 0; j <= D; ++j) {
    FxS q = pj;           // du^(i-1) dv^j
#pragma unroll
    for (int i = 1; i <= D - j; ++i) {
      const int gg = i + j, e = gg * (gg + 1) / 2 + j;
      const FxS q8 = fx_28(q);
#pragma unroll
      for (int c = 0; c < 3; ++c) fx_mac28(h[c], t[c], q8, fx_unjoin(tX[c * n + e]));
      if (i < D - j) q = fx_split(fx_smul_sl<2>(q, u));
    }
    if (j < D) {
      const int gg = j + 1, e = gg * (gg + 1) / 2 + gg;
      const FxS q8 = fx_28(pj);
#pragma unroll
      for (int c = 0; c < 3; ++c) fx_mac28(h[3 + c], t[3 + c], q8, fx_unjoin(tX[c * n + e]));
      pj = fx_split(fx_smul_sl<2>(pj, v));
    }
  }
  int e0, e1;
  fx_mant(du, &e0);
  fx_mant(dv, &e1);
  const int e = max(max(e0, e1), -1000);
  const FxS a = fx_split(fx_fix(du, e)), b = fx_split(fx_fix(dv, e));
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const FxS A = fx_split((h[c] << 2) + (t[c] >> 26)), B = fx_split((h[3 + c] << 2) + (t[3 + c] >> 26));
    const i64 tt = fx_swide(a.h, A.l) + fx_swide(a.l, A.h) + fx_swide(b.h, B.l) + fx_swide(b.l, B.h);
    out[c] = ((fx_swide(a.h, A.h) + fx_swide(b.h, B.h)) << 1) + (tt >> 30);
  }
  *eout = e;
}

}  // namespace lcq
