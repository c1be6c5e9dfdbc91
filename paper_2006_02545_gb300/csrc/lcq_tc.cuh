// Building blocks of the split-precision tensor-core contraction, of the two-float kernel values
// and of the lean FP64 gradients used by the adaptive near integration (Sec. 4.3).
//
// On GB300 the FP64 pipe retires 2 FMA per clock per SM (measured 1.26 TFLOP/s), the FP32
// pipe 128 and the warp-level f16 tensor-core MMA about 0.47 m16n8k16 per clock per SM
// (measured 602 TFLOP/s).  The dense part of the adaptive integration, the contraction of
// kernel values (targets x leaf nodes) with basis values (leaf nodes x n), is therefore
// done exactly on the tensor cores: each operand is written as a sum of NS slices of
// 7 bits on a common power-of-two scale (the row's for the kernel values, a fixed per-column
// bound for the basis values; the Ozaki splitting of Ozaki, Ogita, Oishi and Rump,
// Numer. Algorithms 59, 2012), every product of two slices (< 2^14) and every sum of them
// over a piece of at most 128 nodes and over the at most 8 slice pairs of one diagonal stays
// below 2^24, so the f16 MMA with FP32 accumulators computes each diagonal exactly; the
// diagonals are combined in 64-bit integers and converted to FP64 once per piece.  With
// NS = 8 (56 bits per operand) and the diagonals i + j <= 8 (43 MMAs per 16-node step; the
// dropped products are below 2^-60 of the operands' scales) the result matches an FP64
// contraction to the FP64 rounding level of the sum of |products|.  In shared memory an operand
// is 8 bytes, one slice each, and becomes f16 pairs in registers (half2_slice).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lcq_device.cuh"
#include "lcq_ff.cuh"

namespace lcq {

constexpr int kSliceBits = 7;
constexpr int kPoisonExp = 0x40000000;  // row exponent marking a non-finite kernel value

// Shared-memory layout of the tensor-core moment engine for degree D (byte offsets).  An operand
// value is eight bytes, one 7-bit slice each (slice_bytes): basis values B[n][BST], kernel values
// G[TT][GST] (two operands, Re and Im; the FP64 or FP32 values before they are sliced).  The row
// strides keep the fragment loads of the MMA (128 bits a lane) free of bank conflicts.
template <int D>
struct TcCfg {
  static constexpr int n = (D + 1) * (D + 2) / 2;
  static constexpr int NTILE = (n + 7) / 8;        // MMA n-tiles of 8 basis columns
  static constexpr int CH = D <= 6 ? 256 : 128;    // padded nodes per chunk (two blocks fit an SM)
  static constexpr int CHG = CH / 2;               // columns that share a row scale in the FP32 tier
  static constexpr int PARTS = 256 / CH;           // threads per node
  static constexpr int TT = 8;                     // targets per tile: 16 MMA rows (Re, then Im)
  static constexpr int MAXP = CH / 16;             // pieces (segment parts) per chunk at most
  static constexpr int BST = CH + 8;               // B row stride (8-byte values)
  static constexpr int GST = CH + 1;               // G row stride (16-byte values)
  static constexpr int OFF_G = 0;                              // G; before it the row factors
  static constexpr int G_BYTES = TT * GST * 16;
  static constexpr int OFF_B = (OFF_G + G_BYTES + 15) / 16 * 16;
  static constexpr int OFF_TX = OFF_B + n * BST * 8;           // tx[3 TT], tn[3 TT]
  static constexpr int OFF_EP = OFF_TX + 6 * TT * 8;           // Ep[TT][MAXP] float
  static constexpr int OFF_RE = OFF_EP + TT * MAXP * 4;        // rowE[MAXP][TT][2] int
  static constexpr int OFF_PC = OFF_RE + MAXP * TT * 2 * 4;    // pieces[MAXP][8] int
  static constexpr int OFF_TE = OFF_PC + MAXP * 8 * 4;         // te[TT] int: target far off
  static constexpr int BYTES = OFF_TE + TT * 4;
};

// |x| 2^(7 NS - E) rounded to the nearest integer, for |x| < 2^E: below 2^(7 NS).  Zero,
// subnormal and non-finite x give 0 (non-finite values are flagged by the caller).
template <int NS>
__device__ __forceinline__ unsigned long long fix_mag(double x, int E) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  if (ex == 0 || ex == 0x7ff) return 0ull;
  const unsigned long long m = (b & 0xfffffffffffffull) | 0x10000000000000ull;  // 53 bits
  const int sh = 1075 + E - ex - kSliceBits * NS;
  unsigned long long M;
  if (sh <= 0) {
    M = m << (-sh);
  } else {
    if (sh >= 54) return 0ull;
    M = (m + (1ull << (sh - 1))) >> sh;
  }
  const unsigned long long top = (1ull << (kSliceBits * NS)) - 1ull;
  return M < top ? M : top;
}
template <int NS>
__device__ __forceinline__ unsigned long long fix_mag(float x, int E) {
  const unsigned b = __float_as_uint(x);
  const int ex = (int)((b >> 23) & 0xff);
  if (ex == 0 || ex == 0xff) return 0ull;
  const unsigned long long m = (b & 0x7fffffu) | 0x800000u;  // 24 bits
  const int sh = 150 + E - ex - kSliceBits * NS;
  unsigned long long M;
  if (sh <= 0) {
    M = m << (-sh);
  } else {
    if (sh >= 25) return 0ull;
    M = (m + (1ull << (sh - 1))) >> sh;
  }
  const unsigned long long top = (1ull << (kSliceBits * NS)) - 1ull;
  return M < top ? M : top;
}

// Biased exponent field and the exponent E with |x| < 2^E for a normal number.
__device__ __forceinline__ int exp_field(double x) {
  return (int)((((unsigned long long)__double_as_longlong(x)) >> 52) & 0x7ff);
}
__device__ __forceinline__ int exp_field(float x) { return (int)((__float_as_uint(x) >> 23) & 0xff); }
__device__ __forceinline__ int exp_bound(int field, double) { return field - 1022; }
__device__ __forceinline__ int exp_bound(int field, float) { return field - 126; }
__device__ __forceinline__ bool exp_nonfinite(int field, double) { return field == 0x7ff; }
__device__ __forceinline__ bool exp_nonfinite(int field, float) { return field == 0xff; }

// The eight 7-bit slices of a 56-bit magnitude M with a sign, one a byte: slices 0-3 (the most
// significant) in the low word of the pair, slice i in byte 3 - i % 4, as 128 +- c.
__device__ __forceinline__ uint32_t spread_28(uint32_t h) {
  return h + (h & ~0x7fu) + ((h & ~0x3fffu) << 1) + ((h & ~0x1fffffu) << 2);
}
constexpr uint32_t kZeroSlices = 0x80808080u;
__device__ __forceinline__ uint2 slice_bytes(unsigned long long M, bool neg) {
  const uint32_t a = spread_28((uint32_t)(M >> 28)), b = spread_28((uint32_t)M & 0xfffffffu);
  return neg ? make_uint2(kZeroSlices - a, kZeroSlices - b)
             : make_uint2(kZeroSlices + a, kZeroSlices + b);
}
// Slice i of two values as two f16 (the low half: of x0): the f16 with bits 0x6400 | u is 1024 + u,
// and subtracting 1152 leaves u - 128 = +- c exactly.
template <int I>
__device__ __forceinline__ uint32_t half2_slice(uint2 x0, uint2 x1) {
  constexpr uint32_t j = 3 - (I & 3);
  const uint32_t p = __byte_perm(I < 4 ? x0.x : x0.y, I < 4 ? x1.x : x1.y,
                                 j | (j << 4) | ((4 + j) << 8) | ((4 + j) << 12));
  const uint32_t w = (p & 0x00ff00ffu) | 0x64006400u;
  uint32_t r;
  asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(w), "r"(0x64806480u));
  return r;
}

// D += A B for one m16n8k16 tile: A row-major f16 (4 registers), B column-major f16 (2),
// D FP32 (4).
__device__ __forceinline__ void mma_f16_16816(float* d, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// FP64 value of one accumulator element: the diagonals d = 0..ND-1 (exact integers in FP32)
// weighted 2^(-7 d), combined in 64-bit integers (two halves of at most 53 bits, so that each
// converts exactly), times 2^(E - 14 - 7 (ND - 1)), E = Ea + Eb.
template <int ND>
__device__ __forceinline__ double assemble(const float (*acc)[4], int e, int E) {
  if (E >= kPoisonExp / 2) return __longlong_as_double(0x7ff8000000000000ll);  // NaN
  double v;
  if (ND <= 5) {
    long long s = 0;
#pragma unroll
    for (int d = 0; d < ND; ++d)
      s += (long long)__float2int_rn(acc[d][e]) * (1ll << (kSliceBits * (ND - 1 - d)));
    v = (double)s;
  } else {
    constexpr int H = ND / 2;  // diagonals 0..H-1 in hi, H..ND-1 in lo
    long long hi = 0, lo = 0;
#pragma unroll
    for (int d = 0; d < H; ++d)
      hi += (long long)__float2int_rn(acc[d][e]) * (1ll << (kSliceBits * (H - 1 - d)));
#pragma unroll
    for (int d = H; d < ND; ++d)
      lo += (long long)__float2int_rn(acc[d][e]) * (1ll << (kSliceBits * (ND - 1 - d)));
    v = fma((double)hi, (double)(1ll << (kSliceBits * (ND - H))), (double)lo);
  }
  const int ue = E - 2 * kSliceBits - kSliceBits * (ND - 1);
  if (ue < -1022) return 0.0;
  return v * __longlong_as_double((long long)(ue + 1023) << 52);
}

// FP32 value of an FP64 number by its bits (truncating the mantissa; exponents outside the
// FP32 range flush to zero or saturate): no FP64 instruction, for quantities that only set
// a tolerance floor.
__device__ __forceinline__ float f32_bits(double x) {
  const long long b = __double_as_longlong(x);
  const int hi = (int)(b >> 32);
  const int e = ((hi >> 20) & 0x7ff) - 1023 + 127;
  if (e <= 0) return 0.0f;
  const unsigned s = (unsigned)hi & 0x80000000u;
  if (e >= 255) return __uint_as_float(s | 0x7f800000u);
  return __uint_as_float(s | ((unsigned)e << 23) | ((unsigned)(b >> 29) & 0x7fffffu));
}

// FP64 value of a positive normal FP32 number by its bits (exact; no FP64 instruction).
__device__ __forceinline__ double f64_bits(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned long long e = (unsigned long long)(((b >> 23) & 0xffu) + (1023u - 127u));
  return __longlong_as_double((long long)((e << 52) | ((unsigned long long)(b & 0x7fffffu) << 29)));
}

// 1/sqrt(x) for x > 0: the FP32 estimate (special function unit) refined by one third-order
// Newton-Raphson step in FP64, y1 = y0 (1 + e/2 + 3 e^2/8) with e = 1 - x y0^2 (relative
// error O(e^3), e <= 2^-21): five FP64 instructions.  Arguments outside the FP32 range
// take rsqrt().
__device__ __forceinline__ double rsqrt_nr(double x) {
  const int ex = (__double2hiint(x) >> 20) & 0x7ff;
  if (ex < 1023 - 120 || ex > 1023 + 120) return rsqrt(x);
  const double y0 = f64_bits(rsqrtf(f32_bits(x)));
  const double e = fma(-(x * y0), y0, 1.0);
  return fma(y0, e * fma(e, 0.375, 0.5), y0);
}

// sin and cos of th by table lookup and Taylor polynomials (the table method of Gal and
// Bachelis, ACM TOMS 17, 1991): th = j (2 pi / 1024) + t with j = rint(th 1024 / (2 pi))
// (the 1.5 2^52 shifter) and |t| <= pi / 1024; sin t through t^5 and cos t through t^4
// (the next terms are below 2^-59 relative); then the angle-addition formulas with the
// table's (cos, sin)(2 pi j / 1024): 13 FP64 instructions.  Valid for |th| < 2^20 (j times
// the 27-bit leading part of the step stays exact); larger arguments use sincos().
__device__ __forceinline__ void sincos_tab(double th, const double2* __restrict__ tab, double* sn,
                                           double* cs) {
  if (((__double2hiint(th) >> 20) & 0x7ff) >= 1023 + 20) {  // |th| >= 2^20 or not finite
    sincos(th, sn, cs);
    return;
  }
  constexpr double kInvStep = 162.97466172610083;        // 1024 / (2 pi)
  constexpr double kStepHi = 0x1.921fb54p-8;             // 2 pi / 1024 to 27 bits
  constexpr double kStepLo = 3.875365545627111e-12;      // 2 pi / 1024 - kStepHi
  constexpr double kShift = 6755399441055744.0;          // 1.5 2^52
  const double y = fma(th, kInvStep, kShift);
  const int j = __double2loint(y) & (kSinCosTable - 1);
  const double jd = y - kShift;
  double t = fma(-jd, kStepHi, th);
  t = fma(-jd, kStepLo, t);
  const double z = t * t;
  const double s = fma(t * z, fma(z, 1.0 / 120.0, -1.0 / 6.0), t);
  const double c = fma(z, fma(z, 1.0 / 24.0, -0.5), 1.0);
  const double2 e = __ldg(tab + j);
  *cs = fma(e.x, c, -e.y * s);
  *sn = fma(e.y, c, e.x * s);
}

// Kernel value for real k, kinds S, D and CFIE with a real alpha in lean FP64, the constants folded
// into the per-node source data (the arguments that kernel_eval_ff does not cover): N' = N w alpha / (4 pi) (alpha = 1 for D), Js = beta_r Jw /
// (4 pi) (Jw / (4 pi) for S), Ks = beta_i Jw / (4 pi), fJ = FP32 Jw / (4 pi).  Then
//   S: e^{ikr}/r Js,   D and CFIE: e^{ikr}/r ((1 - ikr) N'.d / r^2 + Js + i Ks),
// about 39 FP64 instructions for the CFIE.  r = 0 gives 0.
__device__ __forceinline__ cplx kernel_eval_fold(int kind, double kr, const KernelParamsF& kf,
                                                 const double2* __restrict__ sct, double x0,
                                                 double x1, double x2, double X0, double X1,
                                                 double X2, double N0, double N1, double N2,
                                                 double Js, double Ks, float fJ, float fR,
                                                 float* env) {
  const double d0 = x0 - X0, d1 = x1 - X1, d2 = x2 - X2;
  const double r2 = fma(d0, d0, fma(d1, d1, d2 * d2));
  if ((__double_as_longlong(r2) << 1) == 0) {
    *env = 0.0f;
    return {0.0, 0.0};
  }
  const double rinv = rsqrt_nr(r2);
  const double r = r2 * rinv;
  const double th = kr * r;
  double sn, cs;
  sincos_tab(th, sct, &sn, &cs);
  {
    // |G| Jw (|beta| + |alpha| |1 - ik r| R / r^2) in FP32, k real
    const float fri = f32_bits(rinv), f1 = kf.kr * f32_bits(r);
    const float fa = sqrtf(fmaf(f1, f1, 1.0f));
    *env = fri * fJ * fmaf(kf.ea * fa * fR, fri * fri, kf.eb);
  }
  const double ec = cs * rinv, es = sn * rinv;
  if (kind == 0) return {ec * Js, es * Js};
  const double nd = fma(N0, d0, fma(N1, d1, N2 * d2)) * (rinv * rinv);
  const double mr = kind == 2 ? nd + Js : nd;
  const double mi = kind == 2 ? fma(-th, nd, Ks) : -th * nd;
  return {fma(ec, mr, -es * mi), fma(ec, mi, es * mr)};
}

// kernel_eval_fold in two-float arithmetic (lcq_ff.cuh) on the FP32 pipe: x - X in FP64 (the
// difference stays FP64 near the singularity), then r^2, 1/r, k r, e^{ikr} and the S, D and
// CFIE factors in two-float, the result converted to FP64 exactly; five FP64 instructions.
// Np, Js, Ks: the folded node data (as kernel_eval_fold) as two-float pairs; krf: k.  Each
// value carries a relative error of a few 2^-46 (plus k r 2^-48 in the phase).  Arguments
// outside the two-float range (r^2 outside [1e-30, 1e30], |k r| >= 2^14) take
// kernel_eval_fold.  r = 0 gives 0.
__device__ __forceinline__ cplx kernel_eval_ff(int kind, double kr, ff krf, const KernelParamsF& kf,
                                               const double2* __restrict__ sct,
                                               const float4* __restrict__ sctf, double x0,
                                               double x1, double x2, double X0, double X1,
                                               double X2, const ff* Np, ff Js, ff Ks, float fJ,
                                               float fR, float* env) {
  const double dd0 = x0 - X0, dd1 = x1 - X1, dd2 = x2 - X2;
  if (((__double_as_longlong(dd0) | __double_as_longlong(dd1) | __double_as_longlong(dd2)) << 1) ==
      0) {
    *env = 0.0f;
    return {0.0, 0.0};
  }
  const ff d[3] = {ff_of(dd0), ff_of(dd1), ff_of(dd2)};
  // r^2: exact squares of the leading parts plus 2 d_h d_l (d_l^2 is below 2^-48 of d_h^2)
  ff sq[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    sq[c] = ff_two_prod(d[c].h, d[c].h);
    sq[c].l = __fmaf_rn(2.0f * d[c].h, d[c].l, sq[c].l);
  }
  const ff s1 = ff_two_sum(sq[0].h, sq[1].h), s2 = ff_two_sum(s1.h, sq[2].h);
  const ff r2 = ff_fast_two_sum(
      s2.h, __fadd_rn(__fadd_rn(s1.l, s2.l), __fadd_rn(__fadd_rn(sq[0].l, sq[1].l), sq[2].l)));
  bool ok = r2.h >= 1e-30f && r2.h <= 1e30f;
  ff rinv = {0.0f, 0.0f}, r = rinv, th = rinv, sn = rinv, cs = rinv;
  if (ok) {
    rinv = ff_rsqrt(r2);
    r = ff_mul(r2, rinv);
    th = ff_mul(krf, r);
    ok = ff_sincos(th, sctf, &sn, &cs);
  }
  if (!ok)
    return kernel_eval_fold(kind, kr, kf, sct, x0, x1, x2, X0, X1, X2, dbl_of(Np[0]), dbl_of(Np[1]),
                            dbl_of(Np[2]), dbl_of(Js), dbl_of(Ks), fJ, fR, env);
  {
    // |G| Jw (|beta| + |alpha| |1 - ik r| R / r^2) in FP32, k real
    const float fri = rinv.h, f1 = kf.kr * r.h;
    const float fa = sqrtf(fmaf(f1, f1, 1.0f));
    *env = fri * fJ * fmaf(kf.ea * fa * fR, fri * fri, kf.eb);
  }
  const ff ec = ff_mul(cs, rinv), es = ff_mul(sn, rinv);
  ff re, im;
  if (kind == 0) {
    re = ff_mul(ec, Js);
    im = ff_mul(es, Js);
  } else {
    const ff nd = ff_mul(ff_dot3(Np, d), ff_mul(rinv, rinv));
    const ff tn = ff_mul(th, nd);
    const ff mr = kind == 2 ? ff_add(nd, Js) : nd;
    const ff mi = kind == 2 ? ff_sub(Ks, tn) : ff_neg(tn);
    re = ff_sub(ff_mul(ec, mr), ff_mul(es, mi));
    im = ff_add(ff_mul(ec, mi), ff_mul(es, mr));
  }
  return {dbl_of(re), dbl_of(im)};
}

// Kernel gradients summed over the targets of one source (or the reverse of k_far_sum): with d =
// x - X, r = |d|, G = e^{ikr} / r, h = (1 - ikr) G / r^2 and w the target's weight,
//   dS~/dX = -G (ik - 1/r) |N| d / r,          dS~/dN = G N / |N|,
//   dD~/dX = -h N - (d.N) h'(r) d / r,          dD~/dN = h d,
//   h'(r) = G (k^2 r^2 + 3ikr - 3) / r^3
// (all over 4 pi; CFIE alpha D~ + beta S~; K~ is homogeneous of degree one in N).  N is the
// source's, so sum w G and sum w h are kept as two scalars and multiplied by N once at the end:
// about 55 FP64 instructions a pair for S and 85 for the CFIE, with the table sincos and the
// Newton-refined 1/r, where the pair-by-pair vectors took 190.
struct GradSum {
  cplx sg, sh, vx[3], vn[3];
};
__device__ __forceinline__ void grad_clear(GradSum& s) {
  s.sg = s.sh = {0.0, 0.0};
#pragma unroll
  for (int c = 0; c < 3; ++c) s.vx[c] = s.vn[c] = {0.0, 0.0};
}
// bN: beta |N| (1 and 0 for the coefficients of S and D as grad_coef gives them)
struct GradCoef {
  cplx al, be;
  bool has_s, has_d;
};
__device__ __forceinline__ GradCoef grad_coef(const KernelParams& kp) {
  GradCoef c;
  c.al = kp.kind == 0 ? cplx{0.0, 0.0} : kp.kind == 1 ? cplx{1.0, 0.0} : cplx{kp.ar, kp.ai};
  c.be = kp.kind == 0 ? cplx{1.0, 0.0} : kp.kind == 1 ? cplx{0.0, 0.0} : cplx{kp.br, kp.bi};
  c.has_s = c.be.re != 0.0 || c.be.im != 0.0;
  c.has_d = c.al.re != 0.0 || c.al.im != 0.0;
  return c;
}
__device__ __forceinline__ void grad_add(GradSum& s, const KernelParams& kp, const GradCoef& cf,
                                         cplx bN, const double* x, const double* X,
                                         const double* N, cplx w) {
  const double d[3] = {x[0] - X[0], x[1] - X[1], x[2] - X[2]};
  const double r2 = fma(d[0], d[0], fma(d[1], d[1], d[2] * d[2]));
  if (r2 == 0.0) return;
  const double ir = rsqrt_nr(r2);
  double r = r2 * ir;
  r = fma(0.5 * ir, fma(-r, r, r2), r);  // the phase k r feels its last bit
  double sn, cs;
  sincos_tab(kp.kr * r, g_sct, &sn, &cs);
  double g = ir;
  if (kp.ki != 0.0) g *= exp(-kp.ki * r);
  const cplx wG = cmul(w, {g * cs, g * sn});
  cplx c = {0.0, 0.0};  // coefficient of -d in d/dX
  if (cf.has_s) {
    s.sg.re += wG.re;
    s.sg.im += wG.im;
    const cplx t = cmul({-kp.ki - ir, kp.kr}, wG);
    c = cmul(bN, {t.re * ir, t.im * ir});
  }
  if (cf.has_d) {
    const double ir2 = ir * ir;
    const cplx t = cmul({fma(kp.ki, r, 1.0), -kp.kr * r}, wG);
    const cplx h = {t.re * ir2, t.im * ir2};
    s.sh.re += h.re;
    s.sh.im += h.im;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      s.vn[k].re = fma(h.re, d[k], s.vn[k].re);
      s.vn[k].im = fma(h.im, d[k], s.vn[k].im);
    }
    const double nd = fma(N[0], d[0], fma(N[1], d[1], N[2] * d[2])) * (ir2 * ir2);
    const cplx poly = {fma(kp.kr * kp.kr - kp.ki * kp.ki, r2, -3.0 * kp.ki * r) - 3.0,
                       fma(2.0 * kp.kr * kp.ki, r2, 3.0 * kp.kr * r)};
    const cplx p = cmul(poly, wG);
    const cplx q = cmul(cf.al, {p.re * nd, p.im * nd});
    c.re += q.re;
    c.im += q.im;
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    s.vx[k].re = fma(-c.re, d[k], s.vx[k].re);
    s.vx[k].im = fma(-c.im, d[k], s.vx[k].im);
  }
}
// dX = sum w dK~/dX, dN = sum w dK~/dN for the source's N (nN = |N|).
__device__ __forceinline__ void grad_finish(const GradSum& s, const GradCoef& cf, const double* N,
                                            double nN, cplx* dX, cplx* dN) {
  constexpr double kInv4Pi = 0.07957747154594767;
  const cplx ah = cmul(cf.al, s.sh), bg = cmul(cf.be, s.sg);
  const double in = nN > 0.0 ? 1.0 / nN : 0.0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const cplx av = cmul(cf.al, s.vn[k]);
    dX[k] = {kInv4Pi * (s.vx[k].re - ah.re * N[k]), kInv4Pi * (s.vx[k].im - ah.im * N[k])};
    dN[k] = {kInv4Pi * fma(bg.re, N[k] * in, av.re), kInv4Pi * fma(bg.im, N[k] * in, av.im)};
  }
}

}  // namespace lcq
