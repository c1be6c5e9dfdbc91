// Helmholtz kernel values in 64-bit fixed-point arithmetic on the integer pipe.
//
// On this GPU a warp's FP64 instruction occupies its pipe for 64 cycles, a 32 x 32 + 64 bit integer
// multiply-add for 4, a shift or logic instruction for 2 and a 64-bit addition for 1 (measured).  A
// product of two 62-bit mantissas to 62 bits is three such multiply-adds, so the whole kernel value, some
// 450 (S) to 730 (CFIE) instructions, takes about 770 to 1,200 cycles a pair and warp in the far sum,
// where 41 FP64 instructions took 3,600, and with more bits: every quantity below is a 57- to 63-bit
// mantissa on a scale of its own, where FP64 has 53.
//
// The value is written without the node's area element in it:
//   K~ = W e^{-ki r} e^{i th} (A + iB) / r^2,   W = Jw / (4 pi),  th = kr r,
//   A = T + th U + Re(beta) r + ki r T,  B = U - th T + Im(beta) r + ki r U,
//   T = Re(alpha) c,  U = Im(alpha) c,  c = n.d / r  (n the unit normal, d = x - X),
// which is alpha (1 - ikr) n.d / r^2 + beta times W e^{ikr} / r.  c, T and U are brought to full length
// and A and B summed at the exponent of the largest term.  Below th = 2 pi / 256, where sin th ~ th and
// g = sin th - th cos th ~ th^3 / 3, these come from their series to full length and every term has its
// own exponent (fx_small_value), so that each part keeps its digits down to th = 0.  The single layer
// alone is W e^{ikr} / r.
//
// Host and device code alike: the arithmetic is plain 64-bit integers, so a host program can
// compare it with higher precision; only the start of the reciprocal square root differs.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define LCQ_HD __host__ __device__ __forceinline__
#define LCQ_HD_NOINLINE static __host__ __device__ __noinline__
#else
#define LCQ_HD inline
#define LCQ_HD_NOINLINE static
#endif

namespace lcq {

typedef unsigned long long u64;
typedef long long i64;

LCQ_HD uint32_t fx_hi(u64 x) { return (uint32_t)(x >> 32); }
LCQ_HD uint32_t fx_lo(u64 x) { return (uint32_t)x; }
LCQ_HD u64 fx_wide(uint32_t a, uint32_t b) { return (u64)a * b; }
LCQ_HD i64 fx_swide(int a, int b) { return (i64)a * b; }

// a b / 2^64 for a, b < 2^63 (error below 2 units): three multiply-adds.
LCQ_HD u64 fx_umul(u64 a, u64 b) {
  const u64 t = fx_wide(fx_hi(a), fx_lo(b)) + fx_wide(fx_lo(a), fx_hi(b));
  return fx_wide(fx_hi(a), fx_hi(b)) + (u64)fx_hi(t);
}
// a b / 2^32 for b < 2^32 and a b < 2^96.
LCQ_HD u64 fx_umul32(u64 a, uint32_t b) {
  return fx_wide(fx_hi(a), b) + (u64)fx_hi(fx_wide(fx_lo(a), b));
}

// A signed value as a signed high word and 31 bits of the low one, v = h 2^32 + 2 l (the last
// bit dropped), so that the cross products are products of signed 32-bit numbers.
struct FxS {
  int h, l;
};
LCQ_HD FxS fx_split(i64 v) { return {(int)(v >> 32), (int)((uint32_t)v >> 1)}; }
// a b / 2^64 for |a|, |b| < 2^63 with |a b| < 2^126.
LCQ_HD i64 fx_smul(FxS a, FxS b) {
  const i64 t = fx_swide(a.h, b.l) + fx_swide(a.l, b.h);
  return fx_swide(a.h, b.h) + (t >> 31);
}
// a b / 2^(64 - K), the extra bits kept
template <int K>
LCQ_HD i64 fx_smul_sl(FxS a, FxS b) {
  const i64 t = fx_swide(a.h, b.l) + fx_swide(a.l, b.h);
  return fx_swide(a.h, b.h) * (1ll << K) + (t >> (31 - K));
}
// (a b + c d) / 2^61, |a|, |c| < 2^62.5, b^2 + d^2 <= 2^122, the products of the low words included
LCQ_HD i64 fx_dot2(FxS a, FxS b, FxS c, FxS d) {
  const i64 l = fx_swide(a.l, b.l) + fx_swide(c.l, d.l);
  const i64 t = fx_swide(a.h, b.l) + fx_swide(a.l, b.h) + fx_swide(c.h, d.l) + fx_swide(c.l, d.h) +
                (l >> 31);
  return ((fx_swide(a.h, b.h) + fx_swide(c.h, d.h)) << 3) + ((t + (1 << 27)) >> 28);
}

LCQ_HD u64 fx_bits(double x) {
#ifdef __CUDA_ARCH__
  return (u64)__double_as_longlong(x);
#else
  u64 b;
  memcpy(&b, &x, 8);
  return b;
#endif
}
LCQ_HD double fx_double(u64 b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}
LCQ_HD int fx_max(int a, int b) { return a > b ? a : b; }
LCQ_HD int fx_min(int a, int b) { return a < b ? a : b; }
LCQ_HD i64 fx_sra(i64 v, int s) { return v >> (s < 63 ? s : 63); }

constexpr int kFxBad = 2000;  // exponents above: not a finite number
// x = m 2^(e - 62) with 2^61 <= |m| < 2^62 (m = 0, e = kFxZero for x = 0 and subnormals).
constexpr int kFxZero = -4000;
LCQ_HD i64 fx_mant(double x, int* e) {
  const u64 b = fx_bits(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  if (ex == 0) {
    *e = kFxZero;
    return 0;
  }
  *e = ex - 1022;
  const i64 m = (i64)(((b & 0xfffffffffffffull) | 0x10000000000000ull) << 9);
  return (b >> 63) ? -m : m;
}
// x 2^62 / 2^e for |x| <= 2^e (truncated toward -infinity below the last bit)
LCQ_HD i64 fx_fix(double x, int e) {
  int ex;
  const i64 m = fx_mant(x, &ex);
  if (m == 0) return 0;
  const int s = e - ex;
  return s < 0 ? m * 2 : fx_sra(m, s);
}

// A constant x = m 2^(e - 62), |m| < 2^62 with the leading bit set.
struct FxConst {
  FxS m;
  int e;
};
LCQ_HD FxConst fx_const(double x) {
  FxConst c;
  c.m = fx_split(fx_mant(x, &c.e));
  return c;
}

// Constants of a kernel (one patch's, or one launch's): kind 0: S, else the general form.
struct FxKernel {
  u64 kt;                // |kr| / (2 pi) = kt 2^(ek - 62)
  u64 ku;                // |kr| = ku 2^(eu - 62), 0: none
  u64 kd;                // ki / ln 2 = kd 2^(ed - 62), 0: none
  FxConst ar, ai;        // alpha
  FxConst p, q;          // Re(alpha) ki, Im(alpha) ki
  FxConst br, bi;        // beta
  int ek, eu, ed;
  int neg;               // kr < 0: the phase's sign
  int single;            // the single layer alone (alpha = 0, beta = 1)
  int has;               // bits kFxBr ... below: the terms that are not zero
  int many;              // 1: more than two of T, U, ki T and the beta terms
};
constexpr int kFxBr = 1, kFxBi = 2, kFxAr = 4, kFxAi = 8, kFxP = 16, kFxQ = 32;
constexpr int kFxUnit = 64;  // Re(alpha) = 1

// kind, k, alpha, beta as KernelParams holds them (kind 0: S, 1 and 3: D form, 2: CFIE).
LCQ_HD FxKernel fx_kernel(int kind, double kr, double ki, double ar, double ai, double br,
                          double bi) {
  FxKernel f;
  if (kind != 2) {
    ar = kind == 0 ? 0.0 : 1.0;
    ai = 0.0;
    br = kind == 0 ? 1.0 : 0.0;
    bi = 0.0;
  }
  f.single = kind == 0;
  f.neg = kr < 0.0;
  int e;
  // kr / (2 pi) and ki / ln 2 to 58 bits: 2^64 / (2 pi) and 2^62 / ln 2 times the mantissas
  u64 m = (u64)fx_mant(fabs(kr), &e);
  f.ku = m;
  f.eu = e;
  m = fx_umul(m, 0x28be60db9391054aull);
  for (f.ek = e; m != 0 && m < (1ull << 61); m <<= 1) --f.ek;
  f.kt = m;
  m = (u64)fx_mant(ki, &e);
  m = fx_umul(m, 0x5c551d94ae0bf85eull);
  for (f.ed = e + 2; m != 0 && m < (1ull << 61); m <<= 1) --f.ed;
  f.kd = m;
  const double p = ar * ki, q = ai * ki;
  // constants that are not finite, or whose product overflows: no phase counts as covered, so that
  // every pair takes the FP64 kernel
  if (!(fabs(p) < 1e300 && fabs(q) < 1e300 && fabs(ar) + fabs(ai) <= 1.7e308 &&
        fabs(br) + fabs(bi) <= 1.7e308))
    f.ek = 100000;
  f.ar = fx_const(ar);
  f.ai = fx_const(ai);
  f.p = fx_const(p);
  f.q = fx_const(q);
  f.br = fx_const(br);
  f.bi = fx_const(bi);
  f.has = (br != 0.0 ? kFxBr : 0) | (bi != 0.0 ? kFxBi : 0) | (ar != 0.0 ? kFxAr : 0) |
          (ai != 0.0 ? kFxAi : 0) | (p != 0.0 ? kFxP : 0) | (q != 0.0 ? kFxQ : 0) |
          (ar == 1.0 ? kFxUnit : 0);
  f.many = (ar != 0.0) + (ai != 0.0) + (p != 0.0 || q != 0.0) + (br != 0.0 || bi != 0.0) > 2;
  return f;
}


// Sine table: (cos, sin)(2 pi j / 4096) 2^62 for j = 0..1023 (one quadrant), and the decay
// table 2^(-j / 1024) 2^62.
constexpr int kFxTab = 1024;
struct FxCs {
  u64 c, s;
};
struct FxTables {
  const FxCs* cs;
  const u64* dec;
};

// |cos|, |sin| 2^62 of the phase ph 2^-64 turns, with their
// signs (bit 0: cos negative, bit 1: sin negative).  The top 12 bits choose quadrant and table
// entry, the other 52 (t < 2^-12 turns) a Taylor step: 1 - cos through t^4, sin through t^5 (the
// next terms are below 2^-66 and 2^-73), combined by the addition theorems with positive
// numbers only.  Absolute error below 2^-60.
LCQ_HD void fx_sincos(u64 ph, const FxCs* __restrict__ tab, u64* cs, u64* sn, int* sign) {
  const uint32_t top = fx_hi(ph);
  const int quad = (int)(top >> 30);
#ifdef __CUDA_ARCH__
  const ulonglong2 e = __ldg(reinterpret_cast<const ulonglong2*>(tab) + ((top >> 20) & 1023u));
  const u64 C = e.x, S = e.y;
#else
  const u64 C = tab[(top >> 20) & 1023u].c, S = tab[(top >> 20) & 1023u].s;
#endif
  const u64 t = ph & 0xfffffffffffffull;              // 2^-64 turns, below 2^52
  const uint32_t th = (uint32_t)(t >> 21), tl = (uint32_t)t & 0x1fffffu;
  const u64 t2 = fx_wide(th, th) + (fx_wide(th, tl) >> 20);   // t^2, unit 2^-86
  const uint32_t t2h = fx_hi(t2);                             // unit 2^-54, below 2^30
  // 1 - cos: 2 pi^2 t^2 - (2 pi^4 / 3) t^4, unit 2^-69
  u64 u = fx_umul(t2, 0x9de9e64df22efull);                    // 2 pi^2 2^47
  const uint32_t v = fx_hi(fx_wide(t2h, t2h));                // unit 2^-76
  u -= fx_hi(fx_wide(v, 0x81e0f841u));                        // (2 pi^4 / 3) 2^25
  // sin: t (2 pi - (4 pi^3 / 3) t^2 + (4 pi^5 / 15) t^4), unit 2^-69
  uint32_t c1 = 0xa55de731u;                                  // (4 pi^3 / 3) 2^26
  c1 -= fx_hi(fx_wide(t2h, 0xa335e33cu)) >> 21;               // (4 pi^5 / 15) 2^25
  const u64 P = 0x1921fb54442d1847ull - (fx_wide(t2h, c1) >> 22);  // 2 pi 2^58
  const u64 s = fx_umul(t << 11, P);
  const u64 tc = fx_wide(fx_hi(C), fx_lo(u)) + fx_wide(fx_lo(C), fx_hi(u)) +
                 fx_wide(fx_hi(S), fx_lo(s)) + fx_wide(fx_lo(S), fx_hi(s));
  const u64 dc = fx_wide(fx_hi(C), fx_hi(u)) + fx_wide(fx_hi(S), fx_hi(s)) + (u64)fx_hi(tc);
  const u64 a = C + 1 - (dc >> 5);  // the unit keeps rounding from going below 0
  const u64 b = S + (fx_umul(C, s) >> 5) - (fx_umul(S, u) >> 5);
  const bool odd = quad & 1;
  *cs = odd ? b : a;
  *sn = odd ? a : b;
  *sign = (int)(((quad + 1) >> 1) & 1) | (quad & 2);
}

// 2^(-x) with x = n + f, f = fr 2^-64: the factor 2^-f 2^62 (table and Taylor terms through x^4).
LCQ_HD u64 fx_exp2n(u64 fr, const u64* __restrict__ tab) {
  const uint32_t j = (uint32_t)(fr >> 54);
#ifdef __CUDA_ARCH__
  const u64 T = __ldg(tab + j);
#else
  const u64 T = tab[j];
#endif
  // y = tau ln 2, tau = low 54 bits 2^-64 < 2^-10; unit 2^-72
  const u64 y = fx_umul((fr & 0x3fffffffffffffull) << 9, 0x58b90bfbe8e7bcd6ull);  // ln 2, 2^63
  // 1 - e^-y = y - y^2/2 + y^3/6 - y^4/24, unit 2^-72
  const uint32_t yh = fx_hi(y << 1);                          // unit 2^-41
  const u64 y2 = fx_umul(y << 1, y << 1);                     // y^2, unit 2^-82
  const uint32_t y2h = (uint32_t)(y2 >> 31);                  // unit 2^-51
  const uint32_t y3 = fx_hi(fx_wide(y2h, yh));                // unit 2^-60
  const uint32_t y4 = fx_hi(fx_wide(y2h, y2h));               // unit 2^-70
  u64 w = y - (y2 >> 11) + (fx_wide(y3, 0xaaaaaaabu) >> 22) -
                fx_hi(fx_wide(y4, 0x2aaaaaabu));
  return T - (fx_umul(T, w) >> 8);
}

// An integer v times 2^e as FP64, rounded to nearest (below the normal range zero, overflow
// infinity).  INT: by integer instructions (ties away from zero), where the FP64 pipe is the
// busier one; else by the conversion instruction, which runs on that pipe.
template <bool INT>
LCQ_HD double fx_pack(i64 v, int e) {
  u64 b;
  int ex;
  if (INT) {
    const u64 sg = (u64)(v >> 63);
    const u64 m = ((u64)v ^ sg) - sg;
#ifdef __CUDA_ARCH__
    const int lz = __clzll((long long)m);
#else
    const int lz = m == 0 ? 64 : __builtin_clzll(m);
#endif
    if (lz > 63) return 0.0;
    ex = e + 1086 - lz;                                 // exponent field of the leading bit
    b = ((m << lz) >> 11) + (((m << lz) >> 10) & 1ull);  // 53 bits, the leading one included
    b += ((u64)(uint32_t)(ex - 1) << 52) | (sg & 0x8000000000000000ull);
  } else {
    if (v == 0) return 0.0;
    b = fx_bits((double)v);
    ex = (int)((b >> 52) & 0x7ff) + e;
    b += (u64)(i64)e << 52;
  }
  if ((unsigned)(ex - 1) >= 2045u)
    return fx_double(((u64)v & 0x8000000000000000ull) | (ex <= 0 ? 0ull : 0x7ff0000000000000ull));
  return fx_double(b);
}

LCQ_HD int fx_clz(u64 v) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)v);
#else
  return v == 0 ? 64 : __builtin_clzll(v);
#endif
}

// Length of the vector D 2^(E - 62), 2^61 <= max |D_c| < 2^62: R 2^(E - 62) with its inverse
// RI 2^(-61 - E); 2^61 <= R < 2^62.8, 2^60.2 < RI <= 2^62.  r2 = |D|^2 / 2^64 in [2^58, 3 2^60];
// f = r2 2^-32 and y = f^(-1/2) to 22 bits from the special function unit; then Y = y 2^44,
// the residual e = 1 - r2 Y^2 2^-120 exactly enough, and RI = Y 2^31 (1 + e/2 + 3 e^2 / 8).
struct FxRoot {
  u64 RI, R;
  float f, y;
};
LCQ_HD FxRoot fx_root(FxS D0, FxS D1, FxS D2) {
  const i64 cr = fx_swide(D0.h, D0.l) + fx_swide(D1.h, D1.l) + fx_swide(D2.h, D2.l);
  const u64 r2 = (u64)(fx_swide(D0.h, D0.h) + fx_swide(D1.h, D1.h) + fx_swide(D2.h, D2.h) +
                       (cr >> 30));
  FxRoot o;
  o.f = (float)fx_hi(r2);
#ifdef __CUDA_ARCH__
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(o.y) : "f"(o.f));
  const uint32_t Y = __float2uint_rz(o.y * 17592186044416.0f);
#else
  o.y = 1.0f / sqrtf(o.f);
  const uint32_t Y = (uint32_t)(o.y * 17592186044416.0f);
#endif
  const u64 G = fx_umul32(r2, Y);                        // sqrt(r2) 2^28
  const i64 e1 = (i64)((1ull << 56) - fx_umul32(G, Y));  // unit 2^-56
  const int e2 = (int)(e1 >> 8);
  const i64 c1 = (e1 + (i64)(((int)(fx_swide(e2, e2) >> 32) * 3) >> 10)) >> 1;
  o.RI = ((u64)Y << 31) + (u64)(((i64)(Y >> 4) * c1) >> 21);
  o.R = fx_umul(r2 << 1, o.RI) << 4;
  return o;
}

// Zeros above the leading bit of |v|, by the high word: at most 32 (a shift below 32 bits is two
// instructions, and no value here means anything 2^-32 below its scale).
LCQ_HD int fx_clz_hi(i64 v) {
  const int h = (int)(v >> 32);
#ifdef __CUDA_ARCH__
  return __clz(h ^ (h >> 31));
#else
  return (h ^ (h >> 31)) == 0 ? 32 : __builtin_clz((unsigned)(h ^ (h >> 31)));
#endif
}
// v 2^e brought to full length, 2^62 <= |v| < 2^63, or by 31 bits.
LCQ_HD void fx_full(i64& v, int& e) {
  const int k = fx_clz_hi(v) - 1;
  v = (i64)((u64)v << (k & 31));
  e -= k;
}

// A number m 2^(e - 62) of a sum, and the sum of two.
struct FxTerm {
  i64 m;
  int e;
};
LCQ_HD FxTerm fx_plus(FxTerm a, FxTerm b) {  // |m| below 2^61.9 and 2^60
  const int e = fx_max(a.e, b.e);
  return {fx_sra(a.m, e - a.e) + fx_sra(b.m, e - b.e), e};
}
// a b, the factors' magnitudes below 2^62 (the product's below 2^61)
LCQ_HD FxTerm fx_times(FxS a, int ea, FxS b, int eb) { return {fx_smul_sl<1>(a, b), ea + eb + 1}; }

// sin th and, if g is asked for, g = sin th - th cos th for th = t 2^(et - 62), 2^58 <= t < 2^62, th <
// 2 pi / 256, to full length with relative errors below 2^-56 (the series' next terms are below 2^-61):
// sin = th (1 - z / 6 + z^2 / 120 - z^3 / 5040), g = th z (1 / 3 - z / 30 + z^2 / 840 - z^3 / 45360),
// z = th^2.
LCQ_HD void fx_small(u64 t, int et, FxTerm* sn, FxTerm* g) {
  const int l = fx_clz(t) - 2;
  t <<= l;
  et -= l;
  const u64 zm = fx_umul(t, t);                          // z = zm 2^(2 et - 60), in [2^58, 2^60)
  const u64 z = zm >> fx_min(-(2 * et + 4), 63);         // unit 2^-64, below 2^53.4
  const uint32_t y = (uint32_t)(z >> 22);                // unit 2^-42
  const u64 z9 = z << 9;                                 // unit 2^-73
  uint32_t c = 0x88888889u - (uint32_t)(fx_wide(y, 0xd00d00d0u) >> 48);   // 2^38 / 120, 2^44 / 5040
  u64 a = 0x2aaaaaaaaaaaaaabull - (fx_wide(y, c) >> 16);                  // 2^64 / 6
  u64 m = fx_umul(t, (1ull << 62) - (fx_umul(z9, a) >> 11));              // [2^58.9, 2^60)
  *sn = {(i64)(m << 2), et};
  if (g == nullptr) return;
  c = 0x9c09c09cu - (uint32_t)(fx_wide(y, 0xb8ef1d2bu) >> 48);            // 2^41 / 840, 2^47 / 45360
  a = 0x2222222222222222ull - (fx_wide(y, c) >> 17);                      // 2^66 / 30
  a = 0x2aaaaaaaaaaaaaabull - (fx_umul(z9, a) >> 12);                     // 2^63 / 3
  m = fx_umul(fx_umul(t, zm << 2) << 2, a);              // g = m 2^(3 et - 61), in [2^56.3, 2^59.5)
  const int k = fx_clz(m) - 2;
  *g = {(i64)(m << k), 3 * et + 1 - k};
}

// The value where th = |kr| r < 2 pi / 256, from the cosine cs of th (sg its and the sine's signs), h and
// eg of W e^{-ki r} / r = h 2^(eg) (fx_core), and n.d = nd 2^(E - 60): the sine and g by their series, and
// every term at its own exponent.  Out of line: pairs nearer than a 256th of a wavelength.
template <bool INT>
LCQ_HD_NOINLINE void fx_small_value(const FxKernel& K, u64 RI, u64 R, int E, u64 cs, u64 h, int eg, i64 nd,
                                    double* re, double* im) {
  const u64 th = fx_umul(R, K.ku) << 1;                 // kr r = th 2^(et - 62), [2^59, 2^61.8)
  const int et = E + K.eu + 1;
  const i64 mt = -(i64)K.neg;
  FxTerm sv, g;
  fx_small(th, et, &sv, K.single ? nullptr : &g);
  if (K.single) {
    *re = fx_pack<INT>((i64)fx_umul(cs, h << 2), eg);
    *im = fx_pack<INT>(((i64)fx_umul((u64)sv.m, h << 2) ^ mt) - mt, eg + sv.e);
    return;
  }
  // W / r^2 to full length: G 2^(eG - 63)
  u64 G = fx_umul(RI, h << 2);                          // W / r^2 = G 2^(eg - E + 1)
  const int lG = fx_clz(G) - 1;
  G <<= lG;
  const int eG = eg - E + 64 - lG;
  const int lc = fx_min(fx_clz((u64)(nd ^ (nd >> 63))) - 2, 61);
  const FxS c = fx_split(fx_smul_sl<2>(fx_split(nd << lc), fx_split((i64)RI)));
  const int ec = 3 - lc;                                // c = n.d / r = . 2^(ec - 62)
  sv.m = (sv.m ^ mt) - mt;
  g.m = (g.m ^ mt) - mt;
  const FxS ct = fx_split((i64)cs), st = fx_split(sv.m), gs = fx_split(g.m), Rs = fx_split((i64)R);
  // f = cos + th sin at the exponent 1
  const FxS f = fx_split((i64)(cs >> 1) +
                         fx_sra(fx_smul_sl<1>(fx_split((i64)th), fx_split(sv.m ^ mt)), -et - sv.e));
  const FxTerm none = {0, kFxZero};
  FxTerm A = none, B = none, vr = none, vi = none;
  if (K.has & kFxBr) A = fx_times(K.br.m, K.br.e, Rs, E);
  if (K.has & kFxBi) B = fx_times(K.bi.m, K.bi.e, Rs, E);
  if (K.has & kFxP) {
    const FxTerm v = fx_times(K.p.m, K.p.e, Rs, E);
    A = fx_plus(A, fx_times(fx_split(v.m), v.e, c, ec));
  }
  if (K.has & kFxQ) {
    const FxTerm v = fx_times(K.q.m, K.q.e, Rs, E);
    B = fx_plus(B, fx_times(fx_split(v.m), v.e, c, ec));
  }
  if (K.has & kFxAr) {
    const FxTerm T = fx_times(K.ar.m, K.ar.e, c, ec);
    const FxS m = fx_split(T.m);
    vr = fx_times(m, T.e, f, 1);
    vi = fx_times(m, T.e, gs, g.e);
  }
  if (K.has & kFxAi) {
    const FxTerm U = fx_times(K.ai.m, K.ai.e, c, ec);
    const FxS m = fx_split(U.m), mn = {-m.h, -m.l};
    vr = fx_plus(vr, fx_times(mn, U.e, gs, g.e));
    vi = fx_plus(vi, fx_times(m, U.e, f, 1));
  }
  const FxS Am = fx_split(A.m), Bm = fx_split(B.m), Bn = {-Bm.h, -Bm.l};
  vr = fx_plus(fx_plus(vr, fx_times(Am, A.e, ct, 0)), fx_times(Bn, B.e, st, sv.e));
  vi = fx_plus(fx_plus(vi, fx_times(Am, A.e, st, sv.e)), fx_times(Bm, B.e, ct, 0));
  // . 2^(e - 62) G 2^(eG - 63)
  const FxS Gs = fx_split((i64)G);
  *re = fx_pack<INT>(fx_smul(fx_split(vr.m), Gs), vr.e + eG - 61);
  *im = fx_pack<INT>(fx_smul(fx_split(vi.m), Gs), vi.e + eG - 61);
}

// The kernel value of one pair from d = x - X = D 2^(E - 62), 2^61 <= max |D_c| < 2^62.  False
// (and nothing written) for arguments that it does not cover: a phase above 2^22 turns, a decay
// above 2^9 halvings, a node that is not finite (ew above kFxBad).  With env the rounding
// envelope |G| Jw (eb + ea |1 - ikr| R / r^2) in FP32 (fk: |kr|, fki: ki, feb = eb, feaR = ea R,
// fw = W in FP32); false too where its factors could leave FP32's range (r or W / r beyond 2^+-60
// and 2^+-120: surfaces of a size far from 1).
// Km: K in memory, for a caller that holds K in registers (the call of fx_small_value takes its address).
template <bool INT>
LCQ_HD bool fx_core(const FxKernel& K, const FxTables& tab, FxS D0, FxS D1, FxS D2, int E,
                    const FxS* n, u64 w, int ew, double* re, double* im, float* env, float fk,
                    float fki, float feb, float feaR, float fw, const FxKernel* Km = nullptr) {
  const int sh = E + K.ek + 8;
  if (sh > 30 || ew > kFxBad) return false;
  if (env && ((unsigned)(E + 60) > 120u || (unsigned)(ew + 120) > 240u ||
              (unsigned)(ew - E + 120) > 240u))
    return false;
  const FxRoot rt = fx_root(D0, D1, D2);
  const u64 RI = rt.RI, R = rt.R;
  // the phase in turns 2^-64 and e^{ikr}
  u64 ph = fx_umul(R, K.kt);                            // kr / 2 pi = ph 2^(E + ek - 60)
  ph = sh >= 4 ? ph << (sh - 4) : ph >> fx_min(4 - sh, 63);
  u64 cs, sn;
  int sg;
  fx_sincos(ph, tab.cs, &cs, &sn, &sg);
  if (K.neg) sg ^= 2;
  // g = W e^{-ki r} / r (single) or / r^2
  u64 h = fx_umul(RI, w << 1);                          // W / r = h 2^(ew - E - 60)
  int eg = ew - E - 60;
  if (K.kd != 0) {
    const u64 x = fx_umul(R, K.kd);                     // ki r / ln 2 = x 2^(E + ed - 60)
    const int sx = E + K.ed + 4;                        // to unit 2^-64
    int nn = 0;
    u64 fr;
    if (sx >= 0) {
      if (sx > 13) return false;
      nn = sx == 0 ? 0 : (int)(x >> (64 - sx));
      fr = x << sx;
    } else {
      fr = x >> fx_min(-sx, 63);
    }
    h = fx_umul(h, fx_exp2n(fr, tab.dec) << 1) << 1;
    eg -= nn;
  }
  if (env) {
    // 1/r and r in FP32 from the estimate
#ifdef __CUDA_ARCH__
    const float sc = __int_as_float((127 - E) << 23);
    const float rs = __int_as_float((127 + E) << 23);
#else
    const float sc = ldexpf(1.0f, -E), rs = ldexpf(1.0f, E);
#endif
    const float fri = rt.y * 16384.0f * sc, fr = rt.f * rt.y * rs * 6.103515625e-05f;
    const float fo = fki * fr + 1.0f, f1 = fk * fr;
    const float fab = sqrtf(fo * fo + f1 * f1);
    float g = fri * fw;
    if (fki != 0.0f) g *= expf(-fki * fr);
    *env = g * (feb + feaR * fab * fri * fri);
  }
  const int et = E + K.eu + 1;
  const bool small = et <= -2 && ph < (1ull << 56) && K.ku != 0;
  const i64 ma = -(i64)(sg & 1), mb = -(i64)(sg >> 1);
  i64 nd = 0;
  if (!K.single) {
    const i64 n01 = fx_swide(n[0].h, D0.l) + fx_swide(n[0].l, D0.h) + fx_swide(n[1].h, D1.l) +
                    fx_swide(n[1].l, D1.h);
    const i64 n2 = fx_swide(n[2].h, D2.l) + fx_swide(n[2].l, D2.h);
    nd = fx_swide(n[0].h, D0.h) + fx_swide(n[1].h, D1.h) + fx_swide(n[2].h, D2.h) +
         (n01 >> 31) + (n2 >> 31);                      // n.d 2^(60 - E)
  }
  if (small) {
    fx_small_value<INT>(Km ? *Km : K, RI, R, E, cs, h, eg, nd, re, im);
    return true;
  }
  if (K.single) {
    const u64 a = fx_umul(cs, h << 2), b = fx_umul(sn, h << 2);   // unit 2^eg
    *re = fx_pack<INT>(((i64)a ^ ma) - ma, eg);
    *im = fx_pack<INT>(((i64)b ^ mb) - mb, eg);
    return true;
  }
  u64 g = fx_umul(RI, h << 2);                          // W / r^2 = g 2^(eg - E + 1)
  const int lg = fx_clz_hi((i64)g) - 1;                 // g >= 2^56
  g <<= lg & 31;                                        // [2^62, 2^63)
  const FxS ec = fx_split((i64)fx_umul(cs, g) ^ ma);    // e^{ikr} W / r^2, unit 2^(eg - E + 3 - lg)
  const FxS es = fx_split((i64)fx_umul(sn, g) ^ mb);
  // c = n.d / r to full length, T = Re(alpha) c = . 2^(eT - 63)
  const int lc = fx_clz_hi(nd) - 2;                     // |nd| < 2^61
  i64 Tm = fx_smul_sl<3>(fx_split((i64)((u64)nd << (lc & 31))), fx_split((i64)RI));
  int eT = 3 - lc;
  fx_full(Tm, eT);
  const FxS c = fx_split(Tm);
  const int e0 = eT;
  if (!(K.has & kFxUnit)) {  // (branches on the constants are uniform)
    Tm = fx_smul_sl<2>(K.ar.m, c);
    eT += K.ar.e;
    fx_full(Tm, eT);
  }
  const FxS Rs = fx_split((i64)R);
  const i64 mt = -(i64)K.neg;
  const FxS ts = fx_split(((i64)(fx_umul(R, K.ku) << 1) ^ mt) - mt);   // kr r = . 2^(et - 62)
  // A and B, the sums beside cos and sin, unit 2^(eA - 61) of the largest term
  const int ebr = K.br.e + E, ebi = K.bi.e + E;
  int eA = fx_max(fx_max(eT, eT + et), fx_max(ebr, ebi));
  int eU = kFxZero, ep = kFxZero, eq = kFxZero;
  i64 U = 0;
  if (K.has & (kFxAi | kFxP | kFxQ)) {
    U = fx_smul_sl<2>(K.ai.m, c);
    eU = e0 + K.ai.e;
    fx_full(U, eU);
    ep = K.p.e + E + e0 + 1;
    eq = K.q.e + E + e0 + 1;
    eA = fx_max(fx_max(eA, fx_max(eU, eU + et)), fx_max(ep, eq)) + K.many;
  }
  i64 A = (fx_sra(Tm, eA - eT + 1) + 1) >> 1;
  i64 B = -fx_sra(fx_smul(ts, fx_split(Tm)), eA - eT - et);
  if (K.has & kFxBr) A += fx_sra(fx_smul_sl<1>(K.br.m, Rs), eA - ebr);
  if (K.has & kFxBi) B += fx_sra(fx_smul_sl<1>(K.bi.m, Rs), eA - ebi);
  if (K.has & (kFxAi | kFxP | kFxQ)) {
    A += (fx_sra(fx_smul_sl<1>(ts, fx_split(U)), eA - eU - et) + 1) >> 1;
    B += (fx_sra(U, eA - eU + 1) + 1) >> 1;
    A += fx_sra(fx_smul(fx_split(fx_smul(K.p.m, Rs) << 1), c), eA - ep);
    B += fx_sra(fx_smul(fx_split(fx_smul(K.q.m, Rs) << 1), c), eA - eq);
  }
  const FxS As = fx_split(A), Bs = fx_split(B), Bn = {-Bs.h, -Bs.l};
  const int ev = eA + eg - E + 3 - lg;
  *re = fx_pack<INT>(fx_dot2(As, ec, Bn, es), ev);
  *im = fx_pack<INT>(fx_dot2(As, es, Bs, ec), ev);
  return true;
}

// d = x - X as fx_core takes it, D 2^(E - 62) with 2^61 <= max |D_c| < 2^62, from FP64 coordinates;
// false for |d| outside [2^-300, 2^300], zero among them.
LCQ_HD bool fx_vector(double d0, double d1, double d2, FxS* D, int* E) {
  const u64 b[3] = {fx_bits(d0), fx_bits(d1), fx_bits(d2)};
  int xs[3];
  for (int c = 0; c < 3; ++c) xs[c] = (int)(fx_hi(b[c]) & 0x7fffffffu) >> 20;
  const int ex = fx_max(xs[0], fx_max(xs[1], xs[2]));
  if ((unsigned)(ex - 723) > 600u) return false;
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int c = 0; c < 3; ++c) {
    const u64 m = ((b[c] & 0xfffffffffffffull) | 0x10000000000000ull) << 9;
    D[c] = fx_split((i64)(m >> fx_min(ex - xs[c], 63)) ^ ((i64)b[c] >> 63));
  }
  *E = ex - 1022;
  return true;
}

// The same from d = (d0, d1, d2) 2^(S - 62), |d_c| < 2^62; also false for d = 0.
LCQ_HD bool fx_vector_int(i64 d0, i64 d1, i64 d2, int S, FxS* D, int* E) {
  const int sh = fx_clz((u64)((d0 ^ (d0 >> 63)) | (d1 ^ (d1 >> 63)) | (d2 ^ (d2 >> 63)))) - 2;
  *E = S - sh;
  if (sh > 61 || (unsigned)(*E + 300) > 600u) return false;
  D[0] = fx_split(d0 << sh);
  D[1] = fx_split(d1 << sh);
  D[2] = fx_split(d2 << sh);
  return true;
}

// fx_core from FP64 coordinates of d, and from integers at one exponent.
template <bool INT>
LCQ_HD bool fx_eval(const FxKernel& K, const FxTables& tab, double d0, double d1, double d2,
                    const FxS* n, u64 w, int ew, double* re, double* im, float* env, float fk,
                    float fki, float feb, float feaR, float fw, const FxKernel* Km = nullptr) {
  FxS D[3];
  int E;
  return fx_vector(d0, d1, d2, D, &E) &&
         fx_core<INT>(K, tab, D[0], D[1], D[2], E, n, w, ew, re, im, env, fk, fki, feb, feaR, fw, Km);
}
template <bool INT>
LCQ_HD bool fx_eval_int(const FxKernel& K, const FxTables& tab, i64 d0, i64 d1, i64 d2, int S,
                        const FxS* n, u64 w, int ew, double* re, double* im, float* env, float fk,
                        float fki, float feb, float feaR, float fw) {
  FxS D[3];
  int E;
  return fx_vector_int(d0, d1, d2, S, D, &E) &&
         fx_core<INT>(K, tab, D[0], D[1], D[2], E, n, w, ew, re, im, env, fk, fki, feb, feaR, fw);
}

}  // namespace lcq
