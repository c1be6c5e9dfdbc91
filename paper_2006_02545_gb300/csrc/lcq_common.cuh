// Device code shared by the forward kernels (lcq_kernels.cu) and the adjoint kernels
// (lcq_adjoint.cu): block-level helpers, the moment engine of Sec. 4.2-4.3 and the
// union-tree adaptive kernel, which the adjoint instantiates with gradient accumulation.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "lcq_device.cuh"
#include "lcq_launch.h"
#include "lcq_tc.cuh"

namespace lcq {

constexpr int kThreads = 256;
constexpr double kRoundingFloor = 2e-13;  // multiple of the FP64 rounding envelope never asked below
constexpr double kF32Floor = 2e-6;        // the same for kernel values evaluated in FP32
constexpr double kTwoFloatFloor = 5e-11;  // and in two-float arithmetic (2^8 times the FP64 one)

// ============================================================================ helpers
// Form of the pair evaluations for patch j (block_moments_tc): mode 0, 1 or 2 as given; 3
// chooses per surface of a batch from its tolerance (FP32 for eps >= kMixedMinEps,
// two-float for eps >= kTwoFloatMinEps, FP64 below).
__device__ __forceinline__ int pair_form(const Dev& dv, int j, int mode) {
  if (mode != 3) return mode;
  if (!dv.pgroup) return 0;
  const double e = dv.grp[dv.pgroup[j]].eps;
  return e >= kMixedMinEps ? 1 : (e >= kTwoFloatMinEps ? 2 : 0);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ long long warp_sum_ll(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block-wide exclusive prefix of 0/1 flags for one chunk of blockDim items.
// Returns this thread's position; *total receives the chunk's count.  Uses sm[33].
__device__ __forceinline__ int block_flag_scan(int flag, int* sm, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const unsigned bal = __ballot_sync(0xffffffffu, flag);
  const int inwarp = __popc(bal & ((1u << lane) - 1u));
  __syncthreads();
  if (lane == 0) sm[warp] = __popc(bal);
  __syncthreads();
  if (threadIdx.x == 0) {
    int acc = 0;
    for (int w = 0; w < nw; ++w) {
      const int c = sm[w];
      sm[w] = acc;
      acc += c;
    }
    sm[32] = acc;
  }
  __syncthreads();
  *total = sm[32];
  return sm[warp] + inwarp;
}

// Kernel of patch j: its surface's in a batch of independent surfaces, else the launch's.
// Patch of oversampled source q: the largest j with src_off[j] <= q.
__device__ __forceinline__ int patch_of_source(const int64_t* src_off, int64_t P, int64_t q) {
  int64_t lo = 0, hi = P;  // largest j with src_off[j] <= q
  while (hi - lo > 1) {
    const int64_t mid = (lo + hi) / 2;
    if (src_off[mid] <= q) lo = mid; else hi = mid;
  }
  return (int)lo;
}

__device__ __forceinline__ KernelParams patch_kp(const Dev& dv, int j, const KernelParams& kp) {
  return dv.pgroup ? dv.grp[dv.pgroup[j]].kp : kp;
}

__device__ __forceinline__ double eta_default(int d) {
  const int p = d + 1;
  return p <= 4 ? 2.75 : (p <= 8 ? 2.0 : 1.25);
}

// ============================================================================ moments
template <int D>
struct Cfg {
  static constexpr int n = (D + 1) * (D + 2) / 2;
  static constexpr int CH = 128;  // nodes per chunk (two blocks per SM fit in shared memory)
  static constexpr int BS = n + 1;
  static constexpr int TT = 16;
  // doubles of shared workspace used by block_moments
  static constexpr int WS = CH * BS + 8 * CH + 3 * TT * CH + 6 * TT;
};

// Target accessors of block_moments: pos(i, x) the position of target i; nrm(i, xrel, n)
// its unit normal for S' (the caller's normals tn, SoA [3][NT]; for bare test points the
// radial direction from the centroid, xrel being the position relative to it).
__device__ __forceinline__ void read_nrm(const double* tn, int64_t NT, int64_t t, double* n) {
  n[0] = tn[t];
  n[1] = tn[NT + t];
  n[2] = tn[2 * NT + t];
}
// Output rows of targets: row i at base + i ld, or at base + idx[i] ld.
struct RowsBy {
  cplx* base;
  const int32_t* idx;
  int64_t ld;
  __device__ __forceinline__ cplx* operator()(int i) const {
    return base + (int64_t)(idx ? idx[i] : i) * ld;
  }
  __device__ __forceinline__ RowsBy any() const { return *this; }
};
struct RowsAt {
  cplx* base;
  int64_t ld;
  __device__ __forceinline__ cplx* operator()(int i) const { return base + (int64_t)i * ld; }
  __device__ __forceinline__ RowsBy any() const { return {base, nullptr, ld}; }
};
// Any of the target lists below: ids a[b[c[i]]], lists that are null left out.
struct TgtAny {
  const double* tgt;
  int64_t NT;
  const int32_t *a, *b, *c;
  const double* tn;
  __device__ int64_t id(int i) const {
    if (c) i = c[i];
    if (b) i = b[i];
    return a[i];
  }
  __device__ void pos(int i, double* x) const {
    const int64_t t = id(i);
    x[0] = tgt[t];
    x[1] = tgt[NT + t];
    x[2] = tgt[2 * NT + t];
  }
  __device__ void nrm(int i, const double*, double* n) const { read_nrm(tn, NT, id(i), n); }
};
struct TgtIdx {  // targets by id list
  const double* tgt;
  int64_t NT;
  const int32_t* ids;
  const double* tn;
  __device__ void pos(int i, double* x) const {
    const int64_t t = ids[i];
    x[0] = tgt[t];
    x[1] = tgt[NT + t];
    x[2] = tgt[2 * NT + t];
  }
  __device__ void nrm(int i, const double*, double* n) const { read_nrm(tn, NT, ids[i], n); }
  __device__ TgtAny any() const { return {tgt, NT, ids, nullptr, nullptr, tn}; }
};
struct TgtPairIdx {  // targets of pair ids
  const double* tgt;
  int64_t NT;
  const int32_t* pair_tgt;
  const int32_t* pairs;
  const double* tn;
  __device__ void pos(int i, double* x) const {
    const int64_t t = pair_tgt[pairs[i]];
    x[0] = tgt[t];
    x[1] = tgt[NT + t];
    x[2] = tgt[2 * NT + t];
  }
  __device__ void nrm(int i, const double*, double* n) const {
    read_nrm(tn, NT, pair_tgt[pairs[i]], n);
  }
  __device__ TgtAny any() const { return {tgt, NT, pair_tgt, pairs, nullptr, tn}; }
};
struct TgtAdaptive {  // targets of a union-tree node: local ids -> pairs -> targets
  const double* tgt;
  int64_t NT;
  const int32_t* pair_tgt;
  const int32_t* apairs;
  const int* ST;
  const double* tn;
  __device__ void pos(int i, double* x) const {
    const int64_t t = pair_tgt[apairs[ST[i]]];
    x[0] = tgt[t];
    x[1] = tgt[NT + t];
    x[2] = tgt[2 * NT + t];
  }
  __device__ void nrm(int i, const double*, double* n) const {
    read_nrm(tn, NT, pair_tgt[apairs[ST[i]]], n);
  }
  __device__ TgtAny any() const { return {tgt, NT, pair_tgt, apairs, ST, tn}; }
};

// Unit normal of a target (S') as fx_eval takes a node's, negated: S' is the double-layer
// form with -n_x in the place of the source's normal.  A normal that is not finite (the caller's of
// length zero) has no integers for it: it makes the position xrel a NaN, which every form passes on.
template <class TA>
__device__ __forceinline__ void load_fx_normal(const TA& ta, int i, double* xrel, u64* out) {
  double n[3];
  ta.nrm(i, xrel, n);
  if (!isfinite(n[0] + n[1] + n[2])) xrel[0] = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll
  for (int c = 0; c < 3; ++c) out[c] = fx_join(fx_split(fx_fix(-n[c], 0)));
}

// Kernel value of target x and the node at X (stride sx), normal nn (stride sn), W = w 2^(ew-62);
// env: the rounding envelope (FP32 where its range allows, else FP64) for patch radius R.
__device__ __forceinline__ cplx fx_value(const KernelParams& kp, const FxKernel& fx,
                                         const KernelParamsF& kf, const FxTables& tab,
                                         const double* x, const double* X, int sx, const u64* nn,
                                         int sn, u64 w, int ew, double R, double* env) {
  const double d0 = x[0] - X[0], d1 = x[1] - X[sx], d2 = x[2] - X[2 * sx];
  const FxS n[3] = {fx_unjoin(nn[0]), fx_unjoin(nn[sn]), fx_unjoin(nn[2 * sn])};
  cplx g;
  // W in FP32 for the envelope: its leading 24 bits at its exponent
  float fw = 0.0f, ev = 0.0f;
  if (env) {
    const int e = min(max(ew, -120), 120);
    fw = (float)(uint32_t)(w >> 32) * 9.31322575e-10f * __int_as_float((127 + e) << 23);
  }
  if (fx_eval<false>(fx, tab, d0, d1, d2, n, w, ew, &g.re, &g.im, env ? &ev : nullptr, kf.kr, kf.ki,
                     kf.eb, kf.ea * (float)R, fw)) {
    if (env) *env = (double)ev;
  } else {
    g = fx_fallback(kp, d0, d1, d2, n[0], n[1], n[2], w, ew, R, env);
  }
  return g;
}

struct SegMap {
  double ax, ay, e1x, e1y, e2x, e2y, det;
};

// Moments I[i][seg][nm] = sum_{q in seg} w_q K(x_i, X_q) J_q K_nm(u_q, v_q) for a smooth
// rule (Q nodes) pushed onto nseg affine images of T0, for T targets, geometry and contraction in FP64,
// kernel values in fixed point
// (the far order q_j, whose decisions compare these moments, and the moments of the
// smallest degrees, block_moments_any).  Geometry is evaluated once per chunk of nodes and
// shared by all targets (Sec. 4.3 reuse).
// TA: target accessor (pos(i, x[3])); out row of target i: out + orow(i) * ostride.
// Positions are relative to the patch centroid cen (the coefficients cf describe
// X - cen); cfd holds the derivative series of load_coef_derivs, which replace the
// derivative recurrences.  With ENV, eout[i * nseg + seg] also receives the summed FP64
// rounding envelope (through the basis rows' column of ones).
template <int D, bool ENV = false, class TA, class OR>
__device__ void block_moments(const double* cf, const double* cfd, const double* __restrict__ ru,
                              const double* __restrict__ rv, const double* __restrict__ rw, int Q,
                              const SegMap* segs, int nseg, const TA& ta, int T, OR orow,
                              int64_t ostride, const KernelParams& kp, double* sm,
                              const double* cen, double R = 0.0, double* eout = nullptr) {
  using C = Cfg<D>;
  double* B = sm;
  double* Xs = B + C::CH * C::BS;
  u64* Ns = reinterpret_cast<u64*>(Xs + 3 * C::CH);  // nodes as fx_eval takes them
  u64* Ws = Ns + 3 * C::CH;
  u64* Es = Ws + C::CH;
  cplx* G = reinterpret_cast<cplx*>(Es + C::CH);
  double* Ev = reinterpret_cast<double*>(G + C::TT * C::CH);
  double* tx = Ev + C::TT * C::CH;
  u64* tn = reinterpret_cast<u64*>(tx + 3 * C::TT);  // target normals (S')
  static_assert(C::n < C::BS, "the basis rows need a spare column");
  (void)ostride;
  const KernelParamsF kf = to_f32(kp);
  const FxKernel& fx = kp.fx;  // read at its uses: as a register copy it spills (224 B)
  const FxTables tab = fx_tables();
  const int total = nseg * Q;
  // The rules are conical products, rows of mr nodes sharing v, and every segment map
  // here keeps v a function of the rule's v alone (e1y = 0: T0 and all its midpoint
  // descendants); the v-only factors of the basis and chart sums are then formed once per
  // row (kw_row_factors), into the tile area, which is free during the geometry phase.
  const int mr = (int)lrint(sqrt((double)Q));
  bool by_rows = mr * mr == Q;
  for (int sg = 0; sg < nseg; ++sg) by_rows = by_rows && segs[sg].e1y == 0.0;
  using RW = KwRow<D>;
  constexpr int kRowMax = 3 * C::TT * C::CH / RW::size;
  double* rows = reinterpret_cast<double*>(G);
  for (int c0 = 0; c0 < total; c0 += C::CH) {
    const int nch = min(C::CH, total - c0);
    const int row0 = by_rows ? c0 / mr : 0;
    const bool use_rows = by_rows && (c0 + nch - 1) / mr - row0 + 1 <= kRowMax;
    __syncthreads();
    if (use_rows) {
      // one thread per (row, m): the rows spread over all warps, hence all SM sub-partitions
      const int nrow = (c0 + nch - 1) / mr - row0 + 1;
      for (int e = threadIdx.x; e < nrow * (D + 1); e += blockDim.x) {
        const int m = e / nrow, rr = e - m * nrow;  // m-major: the lanes share m
        const int rg = row0 + rr, sg = rg / mr, l0 = (rg - sg * mr) * mr;
        const SegMap& S = segs[sg];
        kw_row_factors<D>(S.ay + ru[l0] * S.e1y + rv[l0] * S.e2y, m, cf, cfd,
                          rows + rr * RW::size);
      }
      __syncthreads();
    }
    for (int ql = threadIdx.x; ql < nch; ql += blockDim.x) {
      const int q = c0 + ql;
      const int sg = q / Q, l = q - sg * Q;
      const SegMap& S = segs[sg];
      const double r0 = ru[l], r1 = rv[l];
      const double u = S.ax + r0 * S.e1x + r1 * S.e2x;
      const double w = rw[l] * S.det;
      double X[3], Xu[3], Xv[3], Nn[3];
      if (use_rows) {
        kw_geometry_row<D>(u, rows + (q / mr - row0) * RW::size, X, Xu, Xv, B + ql * C::BS);
      } else {
        const double v = S.ay + r0 * S.e1y + r1 * S.e2y;
        kw_geometry_proj<D>(u, v, cf, cfd, X, Xu, Xv, B + ql * C::BS);
      }
      if (ENV) B[ql * C::BS + C::n] = 1.0;  // the envelope's column
      cross3(Xu, Xv, Nn);
      FxS nn[3];
      u64 wm;
      int ew;
      fx_make_node(Nn, w, nn, &wm, &ew);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        Xs[c * C::CH + ql] = X[c];
        Ns[c * C::CH + ql] = fx_join(nn[c]);
      }
      Ws[ql] = wm;
      Es[ql] = (u64)(i64)ew;
    }
    __syncthreads();
    for (int t0 = 0; t0 < T; t0 += C::TT) {
      const int nt = min(C::TT, T - t0);
      if (threadIdx.x < nt) {
        double* xp = tx + 3 * threadIdx.x;
        ta.pos(t0 + threadIdx.x, xp);
        xp[0] -= cen[0];
        xp[1] -= cen[1];
        xp[2] -= cen[2];
        if (kp.kind == 3) load_fx_normal(ta, t0 + threadIdx.x, xp, tn + 3 * threadIdx.x);
      }
      __syncthreads();
      // kernel values in fixed point (lcq_fx.cuh); with ENV also their FP32 rounding envelope
      for (int e = threadIdx.x; e < nt * nch; e += blockDim.x) {
        const int i = e / nch, ql = e - i * nch;
        const u64* nn = kp.kind == 3 ? tn + 3 * i : Ns + ql;
        const int st = kp.kind == 3 ? 1 : C::CH;
        G[i * C::CH + ql] = fx_value(kp, fx, kf, tab, tx + 3 * i, Xs + ql, C::CH, nn, st, Ws[ql],
                                     (int)Es[ql], R, ENV ? Ev + i * C::CH + ql : nullptr);
      }
      __syncthreads();
      // one thread per (target, nm), outputs packed densely; with ENV the extra index nm = n
      // sums the envelope through the basis rows' column of ones.  Node ranges are uniform
      // across the block, so the loops do not diverge.
      constexpr int W = C::n + (ENV ? 1 : 0);
      const int nout = nt * W;
      for (int o = threadIdx.x; o < nout; o += blockDim.x) {
        const int i = o / W, nm = o - i * W;
        const bool env = ENV && nm == C::n;
        for (int sg = 0; sg < nseg; ++sg) {
          const int qa = max(sg * Q - c0, 0), qb = min((sg + 1) * Q - c0, nch);
          if (qa >= qb) continue;
          const bool first = sg * Q >= c0;  // the segment starts in this chunk
          double are = 0.0, aim = 0.0;
          const double* pr = env ? Ev + i * C::CH : &G[i * C::CH].re;
          const int st = env ? 1 : 2;
          const double* pi = env ? pr : pr + 1;
          for (int ql = qa; ql < qb; ++ql) {
            const double bv = B[ql * C::BS + nm];
            are = fma(pr[ql * st], bv, are);
            aim = fma(pi[ql * st], bv, aim);
          }
          if (env) {
            double* ed = eout + (int64_t)(t0 + i) * nseg + sg;
            *ed = first ? are : *ed + are;
          } else {
            cplx* dst = reinterpret_cast<cplx*>(orow(t0 + i)) + (int64_t)sg * C::n + nm;
            if (first) {
              dst->re = are;
              dst->im = aim;
            } else {
              dst->re += are;
              dst->im += aim;
            }
          }
        }
      }
      __syncthreads();
    }
  }
}

// A kernel value of a row as slices on the row's power-of-two scale 2^E (|x| < 2^E).
__device__ __forceinline__ uint2 row_slices(double x, int E) {
  return slice_bytes(fix_mag<8>(x, E), __double2hiint(x) < 0);
}
__device__ __forceinline__ uint2 row_slices(float x, int E) {  // five slices
  return slice_bytes(fix_mag<5>(x, E) << 21, __float_as_int(x) < 0);
}

// One n-tile (basis columns 8 ct .. 8 ct + 7) of one piece of the chunk (columns kbeg ..
// kend - 1, one segment sg): the diagonals d = i + j < ND of the slice products over the
// k-steps, then the assembled complex 8 x 8 block into the outputs (stored when first, else
// added).  A lane's share of the operands is four columns of one target (Re and Im) and of one
// basis function; it turns their slice bytes into f16 pairs as it needs them.
template <int FMAX>
struct RowType {
  using type = double;
};
template <>
struct RowType<0xff> {
  using type = float;
};
// rowE[2 g], [2 g + 1]: exponent fields of the rows' scales; FMAX the field of infinities and NaN.
template <int V>
struct IntC {
  static constexpr int value = V;
};
// BST: row stride of Bs (values).
template <int D, int NS, int ND, int FMAX, int BST = TcCfg<D>::BST, class OR>
__device__ __forceinline__ void tc_tile(const uint2* Bs, const uint4* G, const int* rowE, int ct,
                                        int kbeg, int kend, int nt, int t0, int sg, bool first,
                                        OR orow) {
  using C = TcCfg<D>;
  constexpr int n = C::n;
  const int lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
  const int nb = ct * 8 + g;
  float acc[ND][4];
#pragma unroll
  for (int d = 0; d < ND; ++d) acc[d][0] = acc[d][1] = acc[d][2] = acc[d][3] = 0.0f;
  const uint4 z = make_uint4(kZeroSlices, kZeroSlices, kZeroSlices, kZeroSlices);
  // rows and columns beyond the operands are zero
  const bool ga = g < nt, gb = nb < n;
  const uint4* gp = G + (ga ? g : 0) * C::GST + 2 * c;
  const uint2* bp = Bs + (gb ? nb : 0) * BST + 2 * c;
#pragma unroll 1
  for (int k0 = kbeg; k0 < kend; k0 += 16) {
    const uint4 b0 = gb ? *reinterpret_cast<const uint4*>(bp + k0) : z;
    const uint4 b1 = gb ? *reinterpret_cast<const uint4*>(bp + k0 + 8) : z;
    const uint4 v0 = ga ? gp[k0] : z, v1 = ga ? gp[k0 + 1] : z;
    const uint4 v2 = ga ? gp[k0 + 8] : z, v3 = ga ? gp[k0 + 9] : z;
    uint32_t bf[NS][2];
    auto bslice = [&](auto I) {
      constexpr int i = decltype(I)::value;
      if constexpr (i < NS) {
        bf[i][0] = half2_slice<i>(make_uint2(b0.x, b0.y), make_uint2(b0.z, b0.w));
        bf[i][1] = half2_slice<i>(make_uint2(b1.x, b1.y), make_uint2(b1.z, b1.w));
      }
    };
    bslice(IntC<0>{}); bslice(IntC<1>{}); bslice(IntC<2>{}); bslice(IntC<3>{});
    bslice(IntC<4>{}); bslice(IntC<5>{}); bslice(IntC<6>{}); bslice(IntC<7>{});
    auto aslice = [&](auto I) {
      constexpr int i = decltype(I)::value;
      if constexpr (i < NS) {
        const uint32_t af[4] = {half2_slice<i>(make_uint2(v0.x, v0.y), make_uint2(v1.x, v1.y)),
                                half2_slice<i>(make_uint2(v0.z, v0.w), make_uint2(v1.z, v1.w)),
                                half2_slice<i>(make_uint2(v2.x, v2.y), make_uint2(v3.x, v3.y)),
                                half2_slice<i>(make_uint2(v2.z, v2.w), make_uint2(v3.z, v3.w))};
#pragma unroll
        for (int j = 0; j < NS; ++j)
          if (i + j < ND) mma_f16_16816(acc[i + j < ND ? i + j : 0], af, bf[j]);
      }
    };
    aslice(IntC<0>{}); aslice(IntC<1>{}); aslice(IntC<2>{}); aslice(IntC<3>{});
    aslice(IntC<4>{}); aslice(IntC<5>{}); aslice(IntC<6>{}); aslice(IntC<7>{});
  }
  if (g < nt) {
    using V = typename RowType<FMAX>::type;
    const bool bad = rowE[2 * g] == FMAX || rowE[2 * g + 1] == FMAX;
    const int Er = bad ? kPoisonExp : exp_bound(rowE[2 * g], V());
    const int Ei = bad ? kPoisonExp : exp_bound(rowE[2 * g + 1], V());
#pragma unroll
    for (int cc = 0; cc < 2; ++cc) {
      const int nm = ct * 8 + 2 * c + cc;
      if (nm >= n) continue;
      const int e2 = c_kwexp[nm];
      const double re = assemble<ND>(acc, cc, Er + e2);
      const double im = assemble<ND>(acc, 2 + cc, Ei + e2);
      cplx* dst = reinterpret_cast<cplx*>(orow(t0 + g)) + (int64_t)sg * n + nm;
      if (first) {
        dst->re = re;
        dst->im = im;
      } else {
        dst->re += re;
        dst->im += im;
      }
    }
  }
}

// Moments as block_moments (the adaptive walk, the smooth-rule and annulus moments):
// I[i][seg][nm] = sum_{q in seg} w_q K(x_i, X_q) J_q K_nm(u_q, v_q) and, when eout is not
// null, eout[i * nseg + seg] = sum_q of the kernel's rounding envelope (FP32 sums), with the
// contraction over the nodes on the tensor cores by the exact slice split (lcq_tc.cuh):
// 8 slices per operand and the diagonals i + j <= 8; for the mixed form's FP32 kernel values 5
// slices and the diagonals i + j <= 4.
// A chunk is a run of pieces (segment sg, its nodes l0 .. l0 + nq - 1), each padded to a multiple
// of 16 (the MMA depth), that fill up to CH columns, a thread (degrees 8-10: two) per column: the
// four children of a small rule share one chunk, a large rule is cut where the chunk ends.
// Per chunk: (1) row factors, a thread per (row, m); (2) point, normal and basis values of the
// thread's node in fixed point (lcq_fxgeom.cuh); the point stays in registers, the basis goes to
// shared memory as slices.  Per tile of 8 targets: (3) the thread's kernel values (fx_core:
// fixed point; or two-float, or FP32), with the largest exponent of each target's Re and Im over a
// piece (integer maxima); (4) their slices on that scale; (5) a warp per piece and 8 basis columns:
// mma.sync on fragments built from the slice bytes.  Storing an operand as 8 bytes (not as 8
// f16) lets a chunk hold 256 columns where it held 128, so that every thread has a node and the
// barriers come half as often; they, not the pipes, bounded the kernel (1280-patch CFIE, eps
// 1e-9: adaptive walk 295 ms at 32% of the issue slots before, 180 ms at 47% with it;
// 206 at 48% since the kernel values keep the digits of their small parts).
// Positions in fixed point are relative to the centroid at the exponent S = sx + 3 of the patch's own
// chart (|X_c| < 2^sx, no bit of it dropped); a target beyond 2^(S - 1) in some coordinate, over
// four times the chart's bound away, takes the FP64 difference (nothing cancels there).  So a
// target's values do not depend on the targets it shares the call with.  form: 0 FP64 (fixed point); 1 FP32
// kernel values (the mixed form for eps >= kMixedMinEps); 2 two-float ones (kernel_eval_ff; the
// mixed form below that) where the constants fold, else FP64.  GEO64: a chart that the fixed-point
// scales do not fit (FxChart::fp64), with FP64 nodes (the rows of kw_row_factors) and differences.
template <int D, int FORM, bool GEO64, class TA, class OR>
__device__ __forceinline__ void block_moments_form(
    const FxChart<D>& ch, const double* __restrict__ ru, const double* __restrict__ rv,
    const double* __restrict__ rw, int Q, const SegMap* segs, int nseg, const TA& ta, int T, OR orow,
    const KernelParams& kp, unsigned char* smb, const double* cen, double R, double* eout) {
  using C = TcCfg<D>;
  constexpr int n = C::n;
  constexpr bool mixed = FORM == 1, ffe = FORM == 2, fixed = FORM == 0;
  uint4* G = reinterpret_cast<uint4*>(smb + C::OFF_G);
  u64* rows = reinterpret_cast<u64*>(smb + C::OFF_G);
  uint2* Bs = reinterpret_cast<uint2*>(smb + C::OFF_B);
  double* tx = reinterpret_cast<double*>(smb + C::OFF_TX);
  i64* txi = reinterpret_cast<i64*>(tx);  // fixed-point targets, in the FP64 slots
  u64* tn = reinterpret_cast<u64*>(tx + 3 * C::TT);
  float* Ep = reinterpret_cast<float*>(smb + C::OFF_EP);
  int* rowE = reinterpret_cast<int*>(smb + C::OFF_RE);
  int* pcs = reinterpret_cast<int*>(smb + C::OFF_PC);  // [piece][sg, l0, nq, po, row0, rb, first]
  int* te = reinterpret_cast<int*>(smb + C::OFF_TE);
  const KernelParamsF kf = to_f32(kp);
  const float fR = f32_bits(R);
  const int S = ch.sx + 3;
  const FxKernel& fx = kp.fx;  // read at its uses: as a register copy it spills
  const FxTables tab = fx_tables();
  constexpr double kInv4Pi = 0.07957747154594767;
  const float escale = mixed ? (float)(kF32Floor / kRoundingFloor)
                             : ffe ? (float)(kTwoFloatFloor / kRoundingFloor) : 1.0f;
  const int warp = threadIdx.x >> 5;
  const int col = threadIdx.x % C::CH, part = threadIdx.x / C::CH;
  // conical rules: rows of mr nodes sharing v, which every segment map here (T0 and its
  // midpoint descendants) keeps a function of the rule's v alone
  const int mr = (int)lrintf(sqrtf((float)Q));
  using RW = FxRow<D>;
  constexpr int kRowSize = GEO64 ? KwRow<D>::size : RW::size, kRowMax = C::G_BYTES / 8 / kRowSize;
  // targets of a tile; up to TT targets in all are loaded once, in the shadow of the first rows
  auto load_targets = [&](int t0, int nt) {
    if (threadIdx.x < nt) {
      double xp[3];
      ta.pos(t0 + threadIdx.x, xp);
      bool near = fixed && !GEO64;
#pragma unroll
      for (int c = 0; c < 3; ++c) xp[c] -= cen[c];
      if (kp.kind == 3) load_fx_normal(ta, t0 + threadIdx.x, xp, tn + 3 * threadIdx.x);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        int e;
        fx_mant(xp[c], &e);
        near = near && e < S;
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (near) txi[3 * threadIdx.x + c] = fx_fix(xp[c], S);
        else tx[3 * threadIdx.x + c] = xp[c];
      }
      te[threadIdx.x] = !near;
    }
  };
  if (T <= C::TT) {
    __syncthreads();
    load_targets(0, T);
  }
  int sg_next = 0, l_next = 0;
  while (sg_next < nseg) {
    // plan the chunk (uniform across the block); thread 0 records it for indexed lookups.  A
    // piece is cut at the end of the chunk when at least 64 columns are left, or at the end of
    // the row area.  The FP32 tier cuts a rule into equal parts of at most CHG nodes instead and
    // lets the parts that fit CHG columns share a row scale (a group): with five slices the
    // scale shows in the moments' last digits, and its refinement decisions follow those.
    int np = 0, ncp = 0, nrow = 0, gcp = 0, g0 = 0;
    __syncthreads();
    while (sg_next < nseg && np < C::MAXP && ncp < C::CH) {
      int nq = min(Q - l_next, 128);  // the slice sums of 128 nodes are exact in FP32
      const int room = C::CH - ncp;
      if (mixed) {
        const int nparts = (Q + C::CHG - 1) / C::CHG;
        nq = min(nq, (Q + nparts - 1) / nparts);
        const int pad = (nq + 15) & ~15;
        if (gcp > 0 && gcp + pad > C::CHG) {
          gcp = 0;
          if (room < C::CHG) break;
          g0 = np;
        }
        gcp += pad;
      } else if (((nq + 15) & ~15) > room) {
        if (np > 0 && room < 64) break;
        nq = room;
      }
      const int r0 = l_next / mr;
      int prow = (l_next + nq - 1) / mr - r0 + 1;
      if (nrow + prow > kRowMax) {
        if (np > 0) break;
        nq = ((r0 + kRowMax) * mr - l_next) & ~15;  // rows of a first piece beyond the area
        prow = (l_next + nq - 1) / mr - r0 + 1;
      }
      if (threadIdx.x == 0) {
        int* pc = pcs + 8 * np;
        pc[0] = sg_next;
        pc[1] = l_next;
        pc[2] = nq;
        pc[3] = ncp;
        pc[4] = r0;
        pc[5] = nrow;
        pc[6] = l_next == 0;
        pc[7] = mixed ? g0 : np;  // piece whose row scales it uses
      }
      nrow += prow;
      ncp += (nq + 15) & ~15;
      ++np;
      l_next += nq;
      if (l_next >= Q) {
        l_next = 0;
        ++sg_next;
      }
    }
    __syncthreads();
    // (1) m-major, so that the lanes of a warp share m and with it the loop length
    for (int e = threadIdx.x; e < nrow * (D + 1); e += blockDim.x) {
      const int m = e / nrow, rr = e - m * nrow;
      int k = 0;
      for (int kk = 1; kk < np; ++kk)
        if (pcs[8 * kk + 5] <= rr) k = kk;
      const int* pc = pcs + 8 * k;
      const SegMap& Sg = segs[pc[0]];
      const int l = (pc[4] + rr - pc[5]) * mr;
      const double v = Sg.ay + ru[l] * Sg.e1y + rv[l] * Sg.e2y;
      if constexpr (GEO64)
        kw_row_factors<D>(v, m, reinterpret_cast<const double*>(ch.x),
                          reinterpret_cast<const double*>(ch.d),
                          reinterpret_cast<double*>(rows) + rr * kRowSize);
      else
        fx_row_factors<D>(v, m, ch, rows + rr * kRowSize);
    }
    __syncthreads();
    // (2) this thread's node
    int pk = 0;  // its piece
    for (int kk = 1; kk < np; ++kk)
      if (pcs[8 * kk + 3] <= col) pk = kk;
    const int ql = col - pcs[8 * pk + 3];
    const bool in = col < ncp, real = in && ql < pcs[8 * pk + 2];
    const int pe = pcs[8 * pk + 7];  // the piece that holds its row scales
    i64 Xi[3] = {0, 0, 0};   // fixed: point (2^(62 - S)) and node for fx_core
    FxS nn[3] = {{0, 0}, {0, 0}, {0, 0}};
    u64 wm = 0;
    int ew = 0;
    double Xd[3] = {0, 0, 0};  // point in FP64; two-float and FP32: weighted normal and area
    ff Nff[3] = {{0, 0}, {0, 0}, {0, 0}}, Jff = {0, 0}, Kff = {0, 0};
    float Nf[3] = {0, 0, 0}, Jf = 0.0f;
    if (real) {
      const int* pc = pcs + 8 * pk;
      const SegMap& Sg = segs[pc[0]];
      const int l = pc[1] + ql;
      const double r0 = ru[l], r1 = rv[l];
      const double u = Sg.ax + r0 * Sg.e1x + r1 * Sg.e2x;
      const double v = Sg.ay + r0 * Sg.e1y + r1 * Sg.e2y;
      const u64* row = rows + (pc[5] + l / mr - pc[4]) * kRowSize;
      const double w = rw[l] * Sg.det;
      i64 X[3], N[3];
      int sn = 0;
      double Nn[3];  // of the FP64 nodes, and for the two-float and FP32 values
      if constexpr (GEO64) {
        double Xu[3], Xv[3];
        kw_geometry_row_emit<D>(u, reinterpret_cast<const double*>(row), Xd, Xu, Xv,
                                [&](int idx, double k) {
          if (idx % C::PARTS == part)
            Bs[idx * C::BST + col] = slice_bytes(fix_mag<8>(k, c_kwexp[idx]), __double2hiint(k) < 0);
        });
        cross3(Xu, Xv, Nn);
        if (fixed) fx_make_node(Nn, w, nn, &wm, &ew);
      } else {
        const FxS s = fx_split(fx_fix(2.0 * u + v - 1.0, 0));
        fx_basis_point<D>(s, row, part, C::PARTS, [&](int idx, i64 kv) {
          const u64 sgn = (u64)(kv >> 63);
          // 56 bits, rounded; below 2^56, since |K_nm| (1 + 1e-12) < 2^E_nm
          Bs[idx * C::BST + col] = slice_bytes(((((u64)kv ^ sgn) - sgn) + 4) >> 3, kv < 0);
        });
        fx_chart_point<D>(s, row, ch.su, ch.sv, X, N, &sn);
        if (fixed) {
#pragma unroll
          for (int c = 0; c < 3; ++c) Xi[c] = X[c];  // unit 2^(S - 62)
          fx_node_from_normal(N, sn + 1, w, nn, &wm, &ew);
        }
      }
      if (fixed) {
        const int e = min(max(ew, -120), 120);
        Jf = (float)(uint32_t)(wm >> 32) * 9.31322575e-10f * __int_as_float((127 + e) << 23);
      } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          if (GEO64) continue;
          Xd[c] = fx_pack<false>(X[c], ch.sx - 59);
          Nn[c] = fx_pack<false>(N[c], sn - 61);
        }
        const double N2 = fma(Nn[0], Nn[0], fma(Nn[1], Nn[1], Nn[2] * Nn[2]));
        const double Jw = N2 > 0.0 ? N2 * rsqrt_nr(N2) * w : 0.0;
        if (ffe) {
          const double wn = w * (kp.kind == 1 ? 1.0 : kp.ar) * kInv4Pi;
#pragma unroll
          for (int c = 0; c < 3; ++c) Nff[c] = ff_of(Nn[c] * wn);
          Jff = ff_of(Jw * ((kp.kind == 0 ? 1.0 : kp.br) * kInv4Pi));
          Kff = ff_of(Jw * (kp.bi * kInv4Pi));
          Jf = f32_bits(Jw * kInv4Pi);
        } else {
#pragma unroll
          for (int c = 0; c < 3; ++c) Nf[c] = (float)(Nn[c] * w);
          Jf = (float)Jw;
        }
      }
    } else if (in) {
#pragma unroll 1
      for (int idx = part; idx < n; idx += C::PARTS)
        Bs[idx * C::BST + col] = make_uint2(kZeroSlices, kZeroSlices);
    }
    for (int t0 = 0; t0 < T; t0 += C::TT) {
      const int nt = min(C::TT, T - t0);
      for (int e = threadIdx.x; e < C::MAXP * C::TT * 2; e += blockDim.x) rowE[e] = 0;
      if (T > C::TT) load_targets(t0, nt);
      __syncthreads();
      // (3) the column's kernel values; zeros in padding columns
      if (in) {  // whole half-warps: pieces are multiples of 16 columns
        const unsigned half = 0xffffu << (threadIdx.x & 16);
#pragma unroll 1
        for (int i = part; i < nt; i += C::PARTS) {
          float ev = 0.0f;
          uint32_t ex = 0;  // exponent fields of Re (high half) and Im
          if (mixed) {
            float2 g = make_float2(0.0f, 0.0f);
            const double d0 = tx[3 * i] - Xd[0], d1 = tx[3 * i + 1] - Xd[1],
                         d2 = tx[3 * i + 2] - Xd[2];
            const double r2 = d0 * d0 + d1 * d1 + d2 * d2;
            if (real && r2 > 0.0)
              g = kernel_eval_f32f(kp, kf, d0, d1, d2, r2, Nf[0], Nf[1], Nf[2], Jf, fR, &ev);
            ex = ((uint32_t)exp_field(g.x) << 16) | (uint32_t)exp_field(g.y);
            *reinterpret_cast<float4*>(G + i * C::GST + col) = make_float4(g.x, g.y, ev, 0.0f);
          } else {
            cplx g = {0.0, 0.0};
            if (real) {
              if (ffe) {
                g = kernel_eval_ff(kp.kind, kp.kr, ff_of(kp.kr), kf, g_sct, g_sctf, tx[3 * i],
                                   tx[3 * i + 1], tx[3 * i + 2], Xd[0], Xd[1], Xd[2], Nff, Jff, Kff,
                                   Jf, fR, &ev);
              } else {
                FxS nt3[3] = {nn[0], nn[1], nn[2]};
                if (kp.kind == 3) {
                  nt3[0] = fx_unjoin(tn[3 * i]);
                  nt3[1] = fx_unjoin(tn[3 * i + 1]);
                  nt3[2] = fx_unjoin(tn[3 * i + 2]);
                }
                auto diff = [&](int c) {  // x - X in FP64
                  return GEO64   ? tx[3 * i + c] - Xd[c]
                         : te[i] ? tx[3 * i + c] - fx_pack<false>(Xi[c], S - 62)
                                 : fx_pack<false>(txi[3 * i + c] - Xi[c], S - 62);
                };
                FxS dm[3];
                int de;
                const bool ok =
                    GEO64 || te[i] ? fx_vector(diff(0), diff(1), diff(2), dm, &de)
                          : fx_vector_int(txi[3 * i] - Xi[0], txi[3 * i + 1] - Xi[1],
                                          txi[3 * i + 2] - Xi[2], S, dm, &de);
                if (!ok || !fx_core<false>(fx, tab, dm[0], dm[1], dm[2], de, nt3, wm, ew, &g.re,
                                           &g.im, &ev, kf.kr, kf.ki, kf.eb, kf.ea * fR, Jf)) {
                  double e = 0.0;
                  g = fx_fallback(kp, diff(0), diff(1), diff(2), nt3[0], nt3[1], nt3[2], wm, ew, R, &e);
                  ev = (float)e;
                }
              }
            }
            ex = ((uint32_t)exp_field(g.re) << 16) | (uint32_t)exp_field(g.im);
            *reinterpret_cast<cplx*>(G + i * C::GST + col) = g;
          }
#pragma unroll
          for (int o = 8; o > 0; o >>= 1) {
            ex = __vmaxu2(ex, __shfl_xor_sync(half, ex, o));
            ev += __shfl_xor_sync(half, ev, o);
          }
          if ((threadIdx.x & 15) == 0) {
            atomicMax(rowE + (pe * C::TT + i) * 2, (int)(ex >> 16));
            atomicMax(rowE + (pe * C::TT + i) * 2 + 1, (int)(ex & 0xffffu));
            Ep[i * C::MAXP + (col >> 4)] = ev;
          }
        }
      }
      __syncthreads();
      // envelope sums: a thread per (target, piece) over the half-warps' sums; the FP32 tier, whose
      // floor is 2e-6 of them, a warp per target over the columns
      if (eout && mixed) {
        const int lane = threadIdx.x & 31;
        if (warp < nt)
          for (int k = 0; k < np; ++k) {
            const int* pc = pcs + 8 * k;
            float es = 0.0f;
            for (int q = lane; q < pc[2]; q += 32)
              es += reinterpret_cast<const float4*>(G + warp * C::GST + pc[3] + q)->z;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) es += __shfl_xor_sync(0xffffffffu, es, o);
            if (lane == 0) {
              double* ed = eout + (int64_t)(t0 + warp) * nseg + pc[0];
              const double v = (double)(es * escale);
              *ed = pc[6] ? v : *ed + v;
            }
          }
        __syncthreads();  // the slices overwrite the columns
      } else if (eout) {
        // one thread per target, its pieces in order (two may belong to one segment)
        if (threadIdx.x < nt)
          for (int k = 0; k < np; ++k) {
            const int* pc = pcs + 8 * k;
            float es = 0.0f;
            for (int h = pc[3] >> 4; h < (pc[3] + pc[2] + 15) >> 4; ++h)
              es += Ep[threadIdx.x * C::MAXP + h];
            double* ed = eout + (int64_t)(t0 + threadIdx.x) * nseg + pc[0];
            const double v = (double)(es * escale);
            *ed = pc[6] ? v : *ed + v;
          }
      }
      // (4) slices of the column's values on their rows' scales
      if (in) {
#pragma unroll 1
        for (int i = part; i < nt; i += C::PARTS) {
          const int* E = rowE + (pe * C::TT + i) * 2;
          uint4* gp = G + i * C::GST + col;
          uint2 a, b;
          if (mixed) {
            const float2 g = *reinterpret_cast<const float2*>(gp);  // the envelope beside it is done
            a = row_slices(g.x, exp_bound(E[0], 0.0f));
            b = row_slices(g.y, exp_bound(E[1], 0.0f));
          } else {
            const cplx g = *reinterpret_cast<const cplx*>(gp);
            a = row_slices(g.re, exp_bound(E[0], 0.0));
            b = row_slices(g.im, exp_bound(E[1], 0.0));
          }
          *gp = make_uint4(a.x, a.y, b.x, b.y);
        }
      }
      __syncthreads();
      // (5) tensor-core contraction, a warp per n-tile and piece; pieces of one segment add to the
      // same outputs, so the first one's warp takes them all, in order
      for (int e = warp; e < np * C::NTILE; e += kThreads / 32) {
        const int ct = e % C::NTILE;
        int k = e / C::NTILE;
        if (k > 0 && pcs[8 * (k - 1)] == pcs[8 * k]) continue;
        do {
          const int* pc = pcs + 8 * k;
          const int kb = pc[3], ke = pc[3] + ((pc[2] + 15) & ~15);
          const int* E = rowE + pc[7] * C::TT * 2;
          if (mixed)
            tc_tile<D, 5, 5, 0x00ff>(Bs, G, E, ct, kb, ke, nt, t0, pc[0], pc[6] != 0, orow);
          else
            tc_tile<D, 8, 9, 0x7ff>(Bs, G, E, ct, kb, ke, nt, t0, pc[0], pc[6] != 0, orow);
          ++k;
        } while (k < np && pcs[8 * k] == pcs[8 * (k - 1)]);
      }
      __syncthreads();
    }
  }
}

// two-float kernel values: real k, kinds S, D and CFIE with a real alpha, whose constants are
// folded into the node data
template <int D, bool GEO64, class TA, class OR>
__device__ __forceinline__ void block_moments_forms(
    const FxChart<D>& ch, const double* __restrict__ ru, const double* __restrict__ rv,
    const double* __restrict__ rw, int Q, const SegMap* segs, int nseg, const TA& ta, int T, OR orow,
    const KernelParams& kp, unsigned char* smb, const double* cen, double R, double* eout, int form) {
  if (form == 1)
    block_moments_form<D, 1, GEO64>(ch, ru, rv, rw, Q, segs, nseg, ta, T, orow, kp, smb, cen, R, eout);
  else if (form == 2 && kp.ki == 0.0 && kp.kind <= 2 && kp.ai == 0.0)
    block_moments_form<D, 2, GEO64>(ch, ru, rv, rw, Q, segs, nseg, ta, T, orow, kp, smb, cen, R, eout);
  else
    block_moments_form<D, 0, GEO64>(ch, ru, rv, rw, Q, segs, nseg, ta, T, orow, kp, smb, cen, R, eout);
}

// Out of line and for any accessors: few charts take it, so that it costs the others' kernels no
// registers and is compiled once per degree.
template <int D>
__device__ __noinline__ void block_moments_fp64(
    const FxChart<D>& ch, const double* __restrict__ ru, const double* __restrict__ rv,
    const double* __restrict__ rw, int Q, const SegMap* segs, int nseg, const TgtAny& ta, int T,
    const RowsBy& orow, const KernelParams& kp, unsigned char* smb, const double* cen, double R,
    double* eout, int form) {
  block_moments_forms<D, true>(ch, ru, rv, rw, Q, segs, nseg, ta, T, orow, kp, smb, cen, R, eout, form);
}

template <int D, class TA, class OR>
__device__ void block_moments_tc(const FxChart<D>& ch, const double* __restrict__ ru,
                                 const double* __restrict__ rv, const double* __restrict__ rw,
                                 int Q, const SegMap* segs, int nseg, const TA& ta, int T, OR orow,
                                 const KernelParams& kp, unsigned char* smb, const double* cen,
                                 double R, double* eout, int form) {
  if (ch.fp64)
    block_moments_fp64<D>(ch, ru, rv, rw, Q, segs, nseg, ta.any(), T, orow.any(), kp, smb, cen, R,
                          eout, form);
  else
    block_moments_forms<D, false>(ch, ru, rv, rw, Q, segs, nseg, ta, T, orow, kp, smb, cen, R, eout,
                                  form);
}

// The moments of the smallest degrees in the FP64 form (n <= 10 basis functions) by the
// plain FP64 engine (16-target tiles, one thread per output): there the contraction is too
// small to pay for the tensor-core pipeline's fixed cost per 8-target tile (barriers, the
// slices).  2400 patches, S, generation with this engine and with the tensor one: degree 1 eps
// 5e-3 12.6 and 17.9 ms, degree 2 eps 5e-7 43.3 and 46.4, degree 3 eps 5e-3 22.6 and 26.8, eps 5e-7
// 77.7 and 76.1 (the smooth rules alone: 5.8 and 14.6, the adaptive walk alone 60.3 and 56.6: one
// switch serves both, and the walk gains less than the rules lose, except there).  Every other case:
// block_moments_tc.  smb holds either engine's workspace.
constexpr int kFp64MomentsMaxDeg = 3;
template <int D, class TA, class OR>
__device__ __forceinline__ void block_moments_any(
    const double* cf, const double* cfd, const FxChart<D>& ch, const double* __restrict__ ru,
    const double* __restrict__ rv, const double* __restrict__ rw, int Q, const SegMap* segs,
    int nseg, const TA& ta, int T, OR orow, const KernelParams& kp, unsigned char* smb,
    const double* cen, double R, double* eout, int form) {
  if constexpr (D <= kFp64MomentsMaxDeg) {
    if (form == 0) {
      double* sm = reinterpret_cast<double*>(smb);
      if (eout)
        block_moments<D, true>(cf, cfd, ru, rv, rw, Q, segs, nseg, ta, T, orow, Cfg<D>::n, kp, sm,
                               cen, R, eout);
      else
        block_moments<D, false>(cf, cfd, ru, rv, rw, Q, segs, nseg, ta, T, orow, Cfg<D>::n, kp, sm,
                                cen);
      return;
    }
  }
  block_moments_tc<D>(ch, ru, rv, rw, Q, segs, nseg, ta, T, orow, kp, smb, cen, R, eout, form);
}

// Shared-memory bytes of the moment workspace (either engine's).
template <int D>
constexpr size_t moment_ws_bytes() {
  return D <= kFp64MomentsMaxDeg && sizeof(double) * Cfg<D>::WS > (size_t)TcCfg<D>::BYTES
             ? sizeof(double) * Cfg<D>::WS
             : (size_t)TcCfg<D>::BYTES;
}

template <int D>
__device__ __forceinline__ void load_coef(const double* __restrict__ coef, int64_t off, double* cf) {
  constexpr int n = (D + 1) * (D + 2) / 2;
  for (int e = threadIdx.x; e < 3 * n; e += blockDim.x) cf[e] = coef[off * 3 + e];
}

struct TgtPts {  // explicit points [i][3]
  const double* p;
  __device__ void pos(int i, double* x) const {
    x[0] = p[3 * i];
    x[1] = p[3 * i + 1];
    x[2] = p[3 * i + 2];
  }
  __device__ void nrm(int, const double* xr, double* n) const {
    const double r = sqrt(xr[0] * xr[0] + xr[1] * xr[1] + xr[2] * xr[2]);
    if (r > 0.0) {
      n[0] = xr[0] / r;
      n[1] = xr[1] / r;
      n[2] = xr[2] / r;
    } else {
      n[0] = n[1] = 0.0;
      n[2] = 1.0;
    }
  }
};

__device__ __forceinline__ SegMap seg_T0() { return {0.0, 0.0, 1.0, 0.0, 0.0, 1.0, 1.0}; }

// ============================================================================ adjoint
// Gradient moments (adjoint of Sec. 4.2-4.3 rules with the rule frozen): for the nodes of
// a rule pushed onto nseg sub-triangles and T targets with weights wf(i) = conj(g_t)
// (0: skip), accumulates into the thread-private M[3n]
//   dL/dx_nm += sum_nodes K_nm a_X + dK_nm/du (X_v x a_N) + dK_nm/dv (a_N x X_u),
//   a_X = Re(w sigma(u) sum_i wf(i) dK~/dX),  a_N = Re(w sigma(u) sum_i wf(i) dK~/dN),
// where sigma(u) = sum_nm shat_nm K_nm(u) and N = X_u x X_v (so a_N.dN splits into the
// two cross products).  Thread per node; targets staged through shared memory.
// WARP_ACC: M is instead this warp's row of per-warp sums in shared memory; every lane
// takes part (zeros for lanes without a node) and lane 0 adds the warp's sum.
// scratch: 5 kGradTile doubles of shared memory.
constexpr int kGradTile = 32;
template <int D, bool WARP_ACC = false, class TA, class WF>
__device__ void block_grad(const double* cf, const double* __restrict__ ru,
                           const double* __restrict__ rv, const double* __restrict__ rw, int Q,
                           const SegMap* segs, int nseg, const TA& ta, int T, WF wf,
                           const KernelParams& kp, const cplx* shat, const double* cen,
                           double* M, double* scratch) {
  constexpr int TG = kGradTile;
  double (*gx)[3] = reinterpret_cast<double (*)[3]>(scratch);
  cplx* gwt = reinterpret_cast<cplx*>(scratch + 3 * TG);
  const int total = nseg * Q;
  const GradCoef co = grad_coef(kp);
  for (int c0 = 0; c0 < total; c0 += blockDim.x) {
    const int q = c0 + threadIdx.x;
    const bool on = q < total;
    double u = 0.0, v = 0.0, w = 0.0, X[3] = {0, 0, 0}, Xu[3] = {0, 0, 0}, Xv[3] = {0, 0, 0};
    double Nn[3] = {0, 0, 0};
    cplx sg = {0.0, 0.0};
    if (on) {
      const int s = q / Q, l = q - s * Q;
      const SegMap& S = segs[s];
      u = S.ax + ru[l] * S.e1x + rv[l] * S.e2x;
      v = S.ay + ru[l] * S.e1y + rv[l] * S.e2y;
      w = rw[l] * S.det;
      kw_geometry<D>(u, v, cf, X, Xu, Xv, nullptr, 1);
      cross3(Xu, Xv, Nn);
      kw_for_each<D>(u, v, [&](int idx, double k0, double, double) {
        sg.re = fma(shat[idx].re, k0, sg.re);
        sg.im = fma(shat[idx].im, k0, sg.im);
      });
    }
    const double nN = sqrt(Nn[0] * Nn[0] + Nn[1] * Nn[1] + Nn[2] * Nn[2]);
    const cplx bN = {co.be.re * nN, co.be.im * nN};
    GradSum gs;
    grad_clear(gs);
    for (int t0 = 0; t0 < T; t0 += TG) {
      const int nt = min(TG, T - t0);
      __syncthreads();
      if (threadIdx.x < nt) {
        double xp[3];
        ta.pos(t0 + threadIdx.x, xp);
        gx[threadIdx.x][0] = xp[0] - cen[0];
        gx[threadIdx.x][1] = xp[1] - cen[1];
        gx[threadIdx.x][2] = xp[2] - cen[2];
        gwt[threadIdx.x] = wf(t0 + threadIdx.x);
      }
      __syncthreads();
      if (on)
        for (int i = 0; i < nt; ++i) {
          const cplx c = gwt[i];
          if (c.re == 0.0 && c.im == 0.0) continue;
          grad_add(gs, kp, co, bN, gx[i], X, Nn, c);
        }
    }
    if (WARP_ACC || on) {
      cplx SX[3], SN[3];
      grad_finish(gs, co, Nn, nN, SX, SN);
      double aX[3], aN[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        aX[k] = w * (sg.re * SX[k].re - sg.im * SX[k].im);
        aN[k] = w * (sg.re * SN[k].re - sg.im * SN[k].im);
      }
      double bu[3], bv[3];
      cross3(Xv, aN, bu);
      cross3(aN, Xu, bv);
      if constexpr (WARP_ACC) {
        const bool lead = (threadIdx.x & 31) == 0;
        kw_for_each<D>(u, v, [&](int idx, double k0, double ku, double kv) {
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const double s = warp_sum(k0 * aX[k] + ku * bu[k] + kv * bv[k]);
            if (lead) M[idx * 3 + k] += s;
          }
        });
      } else {
        kw_for_each<D>(u, v, [&](int idx, double k0, double ku, double kv) {
#pragma unroll
          for (int k = 0; k < 3; ++k) M[idx * 3 + k] += k0 * aX[k] + ku * bu[k] + kv * bv[k];
        });
      }
    }
  }
}

// Block sum of the thread-private M[3n] in a fixed order, added to out[3n] (global).
// Uses sm[(blockDim/32) * 3n] doubles of shared memory.
template <int D>
__device__ void block_reduce_M(const double* M, double* sm, double* out) {
  constexpr int n3 = 3 * Cfg<D>::n;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
#pragma unroll 1
  for (int e = 0; e < n3; ++e) {
    const double v = warp_sum(M[e]);
    if (lane == 0) sm[wp * n3 + e] = v;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < n3; e += blockDim.x) {
    double acc = 0.0;
    for (int k = 0; k < nw; ++k) acc += sm[k * n3 + e];
    out[e] += acc;
  }
  __syncthreads();
}

// ============================================================================ adaptive
// Adaptive subdivision (Sec. 4.3) for all eta_1-near targets of a patch at once.
// The refinement trees of the targets are walked as one union tree, depth first:
// a node T carries the set S of targets that refine T; the leaf-rule geometry of T's
// four children is evaluated once and contracted with every target in S (the reuse
// of X, K_nm and J across targets of Fig. multipletargpot).  A target accepts the
// children's sum when ||I_T - sum_c I_c||_2 <= max(tol0 4^-L, 2e-13 E), E the summed
// rounding envelope of the kernel over the children's nodes.
constexpr int kMaxTreeNodes = 1 << 16;  // union-tree nodes walked per patch at most

struct AdaptiveWS {
  int64_t stride;   // bytes per block
  int A_max, levels;
};

// Dynamic shared memory of k_adaptive<D>: chart coefficients, the four child maps, scan
// scratch, the walk's stack, alignment, and the tensor-core moment workspace.
template <int D>
constexpr size_t adaptive_smem_bytes() {
  return sizeof(double) * 3 * Cfg<D>::n + sizeof(SegMap) * 4 + 64 * sizeof(int) +
         4 * 32 * sizeof(unsigned long long) + 128 + moment_ws_bytes<D>();
}

// Work items are taken dynamically through the counter *sched, which the caller zeroes
// before the launch.  gofs == nullptr: item b is the patch plist[b] with all its adaptive
// targets.  Otherwise item i is group g of patch plist[b], gofs[b] <= i < gofs[b + 1]
// (an exclusive scan of the groups per listed patch, gofs[count] their total), the group
// being the adaptive targets g gsz .. g gsz + gsz - 1 of the patch: small groups spread one
// patch's walk over several blocks.  Every target's refinement tree, moments and leaf
// count are the same whichever group it walks with (its tests and sums are its own, and a
// depth-first walk of a union tree visits the nodes of each member tree in that tree's own
// depth-first order), so the grouping changes the schedule, not the results.  plist is
// ordered by decreasing number of adaptive targets (longest items first).
template <int D, bool GRAD = false>
__global__ void __launch_bounds__(kThreads, 2) k_adaptive(const int* __restrict__ plist, int count,
                                                       Dev dv, const KernelParams kp, double eps,
                                                       double normV, int leaf_order, int max_depth,
                                                       const cplx* __restrict__ I_smooth,
                                                       cplx* __restrict__ I_near,
                                                       int32_t* __restrict__ leaves_out,
                                                       unsigned char* __restrict__ work,
                                                       AdaptiveWS wsd, int* __restrict__ status,
                                                       int* __restrict__ sched, int form,
                                                       GradArgs ga,
                                                       const int64_t* __restrict__ gofs, int gsz) {
  using C = Cfg<D>;
  constexpr int n = C::n;
  // gradient mode: dL/dx_nm of the accepted leaves, per thread, reduced per patch
  double Mg[GRAD ? 3 * n : 1];
  __shared__ cplx shat[GRAD ? n : 1];
  extern __shared__ double smem[];
  double* cf = smem;
  SegMap* segs = reinterpret_cast<SegMap*>(cf + n * 3);
  int* ism = reinterpret_cast<int*>(segs + 4);  // [64]: scan scratch + misc
  unsigned long long* stk = reinterpret_cast<unsigned long long*>(ism + 64);  // [4 * 32]
  // tensor-core moment workspace, 128-byte aligned (its 128-bit accesses need 16)
  unsigned char* smb = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(stk + 4 * 32) + 127) & ~static_cast<uintptr_t>(127));
  double* ws = reinterpret_cast<double*>(smb);
  // per-block global workspace
  unsigned char* wb = work + (int64_t)blockIdx.x * wsd.stride;
  const int A_max = wsd.A_max;
  cplx* acc = reinterpret_cast<cplx*>(wb);                          // [A_max][n]
  cplx* tmp = acc + (int64_t)A_max * n;                             // [A_max][4][n]
  cplx* lvlI = tmp + (int64_t)A_max * 4 * n;                        // [levels][A_max][4][n]
  int* lvlT = reinterpret_cast<int*>(lvlI + (int64_t)wsd.levels * A_max * 4 * n);  // [levels][A_max]
  int* flags = lvlT + (int64_t)wsd.levels * A_max;                  // [A_max]
  int* lcnt = flags + A_max;                                        // [A_max]
  int* cnt = lcnt + A_max;                                          // [levels]
  double* tmpE = reinterpret_cast<double*>(                          // [A_max][4], 8-aligned
      (reinterpret_cast<uintptr_t>(cnt + wsd.levels) + 7) & ~static_cast<uintptr_t>(7));
  long long my_tests = 0, my_nodes = 0, my_tree = 0;
  __shared__ int next_b, next_g;
  __shared__ KernelParams kps;
  // derivative series of the chart, for the FP64 engine of the smallest degrees
  __shared__ double cfd[D <= kFp64MomentsMaxDeg ? 2 * 3 * (D * (D + 1) / 2) : 1];
  __shared__ FxChart<D> ch;
  const double* cfdp = cfd;

  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) {
      const int it = atomicAdd(sched, 1);
      int bb = -1, gg = 0;
      if (gofs == nullptr) {
        if (it < count) bb = it;
      } else if (it < gofs[count]) {
        int lo = 0, hi = count;  // gofs[lo] <= it < gofs[hi]
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (gofs[mid] <= it) lo = mid;
          else hi = mid;
        }
        bb = lo;
        gg = it - (int)gofs[lo];
      }
      next_b = bb;
      next_g = gg;
    }
    __syncthreads();
    const int b = next_b;
    if (b < 0) break;
    const int j = plist[b];
    const int64_t ap = dv.ad_ptr[j];
    const int Aall = (int)(dv.ad_ptr[j + 1] - ap);
    const int64_t a0 = gofs ? ap + (int64_t)next_g * gsz : ap;
    const int A = gofs ? min(gsz, Aall - next_g * gsz) : Aall;
    if (A <= 0) continue;
    if (A > A_max) {
      if (threadIdx.x == 0) atomicOr(status, kStCapacity);
      continue;
    }
    const int m = leaf_order > 0 ? leaf_order : dv.q[j];
    const int Q = m * m;
    const double* ru = dv.ru + dv.roff[m];
    const double* rv = dv.rv + dv.roff[m];
    const double* rw = dv.rw + dv.roff[m];
    const double tol0 = (dv.pgroup ? dv.grp[dv.pgroup[j]].eps_ad : eps) * dv.dj[j] / normV;
    const int formj = pair_form(dv, j, form);
    const double Rj = dv.rad[j];
    const int32_t* apairs = dv.ad_pair + a0;
    __syncthreads();
    load_coef<D>(dv.coef, dv.node_off[j], cf);
    if (threadIdx.x == 0) kps = patch_kp(dv, j, kp);  // read after block_moments' barrier
    __syncthreads();
    if constexpr (D <= kFp64MomentsMaxDeg) load_coef_derivs<D>(cf, dv.duv[D], cfd);
    load_fx_chart<D>(cf, dv.duv[D], &ch);
    if constexpr (GRAD) {
#pragma unroll
      for (int e = 0; e < 3 * n; ++e) Mg[e] = 0.0;
      const cplx* sh = reinterpret_cast<const cplx*>(ga.shat) + dv.node_off[j];
      for (int e = threadIdx.x; e < n; e += blockDim.x) shat[e] = sh[e];
    }
    // root: level 0 block holds all targets with I_T0 in slot c = 0
    for (int e = threadIdx.x; e < A * n; e += blockDim.x) {
      const int i = e / n, nm = e - i * n;
      acc[e] = {0.0, 0.0};
      if (leaf_order <= 0) lvlI[(int64_t)i * 4 * n + nm] = I_smooth[(int64_t)apairs[i] * dv.ldI + nm];
    }
    for (int i = threadIdx.x; i < A; i += blockDim.x) {
      lvlT[i] = i;
      lcnt[i] = 0;
    }
    if (threadIdx.x == 0) {
      segs[0] = seg_T0();
      cnt[0] = A;
    }
    __syncthreads();
    if (leaf_order > 0) {
      TgtPairIdx ta{dv.tgt, dv.NT, dv.pair_tgt, apairs, dv.tnrm};
      block_moments_any<D>(cf, cfdp, ch, ru, rv, rw, Q, segs, 1, ta, A,
                           RowsAt{lvlI, 4 * n}, kps, smb,
                           dv.cen + 3 * j, Rj, tmpE, formj);
    }
    // DFS stack entries: level (8 bits) | child (2 bits) | path (2 bits per level) << 16
    int sp = 0;
    if (threadIdx.x == 0) stk[0] = 0ull;  // root: level 0, child 0, empty path
    sp = 1;
    int visited = 0;
    while (sp > 0) {
      if (++visited > kMaxTreeNodes) {  // bounded walk: give up on this patch
        if (threadIdx.x == 0) atomicOr(status, kStCapacity);
        break;
      }
      __syncthreads();
      const unsigned long long top = stk[sp - 1];
      --sp;
      const int L = (int)(top & 0xff);
      const int cidx = (int)((top >> 8) & 3);
      const unsigned long long path = top >> 16;  // child digits of T, level 1 at bits 0-1
      const int S = cnt[L];
      const int* ST = lvlT + (int64_t)L * A_max;
      const cplx* IT = lvlI + (int64_t)L * A_max * 4 * n;
      if ((threadIdx.x & 31) == 0 && threadIdx.x < 128) {
        // Every subtriangle of the midpoint tree is T0 scaled by 2^-L, translated and
        // possibly point-reflected: vertex a at (ia, ja) 2^-L, b = a + o (2^-L, 0),
        // c = a + o (0, 2^-L).  The walk down the path runs in integers; the first lane of
        // warp k writes the map of child k (all exact dyadic values).
        const int k = threadIdx.x >> 5;
        long long ia = 0, ja = 0;
        int o = 1;
        for (int l = 0; l < L; ++l) {
          const int dgt = (int)((path >> (2 * l)) & 3);
          ia = 2 * ia + ((dgt & 1) ? o : 0);
          ja = 2 * ja + ((dgt & 2) ? o : 0);
          if (dgt == 3) o = -o;
        }
        const double h = ldexp(1.0, -(L + 1));
        const int ok = k == 3 ? -o : o;
        SegMap sm;
        sm.ax = (double)(2 * ia + ((k & 1) ? o : 0)) * h;
        sm.ay = (double)(2 * ja + ((k & 2) ? o : 0)) * h;
        sm.e1x = ok * h;
        sm.e1y = 0.0;
        sm.e2x = 0.0;
        sm.e2y = ok * h;
        sm.det = h * h;
        segs[k] = sm;
      }
      __syncthreads();
      // children moments of every target in S
      TgtAdaptive ta{dv.tgt, dv.NT, dv.pair_tgt, apairs, ST, dv.tnrm};
      block_moments_any<D>(cf, cfdp, ch, ru, rv, rw, Q, segs, 4, ta, S,
                           RowsAt{tmp, 4 * n}, kps, smb,
                           dv.cen + 3 * j, Rj, tmpE, formj);
      __syncthreads();
      my_tests += S;
      my_nodes += (long long)S * 4 * Q;
      my_tree += 1;
      // decisions: one warp per target
      const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
      const double tauL = tol0 * ldexp(1.0, -2 * L);
      for (int s = w; s < S; s += nw) {
        double e2 = 0.0;
        for (int nm = lane; nm < n; nm += 32) {
          const cplx* tc = tmp + (int64_t)s * 4 * n + nm;
          const double sr = tc[0].re + tc[n].re + tc[2 * n].re + tc[3 * n].re;
          const double si = tc[0].im + tc[n].im + tc[2 * n].im + tc[3 * n].im;
          const cplx it = IT[(int64_t)s * 4 * n + (int64_t)cidx * n + nm];
          const double dr = it.re - sr, di = it.im - si;
          e2 += dr * dr + di * di;
        }
        e2 = warp_sum(e2);
        const double err = sqrt(e2);
        const double* ee = tmpE + (int64_t)s * 4;
        const double tau = fmax(tauL, kRoundingFloor * (ee[0] + ee[1] + ee[2] + ee[3]));
        const bool finite = isfinite(err) && isfinite(tau);
        const bool accept = !finite || (err <= tau) || (L + 1 >= max_depth);
        if (lane == 0) {
          if (!finite) atomicOr(status, kStNonFinite);
          else if (err > tau && accept) atomicOr(status, kStMaxDepth);
        }
        const int tl = ST[s];
        if (accept) {
          for (int nm = lane; nm < n; nm += 32) {
            const cplx* tc = tmp + (int64_t)s * 4 * n + nm;
            cplx& a = acc[(int64_t)tl * n + nm];
            a.re += tc[0].re + tc[n].re + tc[2 * n].re + tc[3 * n].re;
            a.im += tc[0].im + tc[n].im + tc[2 * n].im + tc[3 * n].im;
          }
          if (lane == 0) lcnt[tl] += 4;
        }
        if (lane == 0) flags[s] = accept ? 0 : 1;
      }
      __syncthreads();
      if constexpr (GRAD) {
        // kernel gradients on the accepted children (the tree itself is recomputed, not
        // stored): weight conj(g_t) for a target that accepts here, else 0
        const cplx* gt = reinterpret_cast<const cplx*>(ga.g);
        block_grad<D>(cf, ru, rv, rw, Q, segs, 4, ta, S,
                      [&](int i) -> cplx {
                        if (flags[i] != 0) return {0.0, 0.0};
                        const cplx c = gt[dv.pair_tgt[apairs[ST[i]]]];
                        return {c.re, -c.im};
                      },
                      kps, shat, dv.cen + 3 * j, Mg, ws);
      }
      // stable compaction of the refining targets into level L+1; up to 32 of them by one warp's
      // ballot (cnt[L + 1] carries the count through the barrier below)
      int base = 0;
      int* DT = lvlT + (int64_t)(L + 1) * A_max;
      cplx* DI = lvlI + (int64_t)(L + 1) * A_max * 4 * n;
      if (S <= 32) {
        if (threadIdx.x < 32) {
          const int f = lane < S ? flags[lane] : 0;
          const unsigned bal = __ballot_sync(0xffffffffu, f);
          if (f) {
            const int pos = __popc(bal & ((1u << lane) - 1u));
            flags[lane] = -pos - 1;  // remember destination
            DT[pos] = ST[lane];
          }
          if (lane == 0) ism[0] = __popc(bal);
        }
      } else {
        for (int s0 = 0; s0 < S; s0 += blockDim.x) {
          const int s = s0 + threadIdx.x;
          const int f = s < S ? flags[s] : 0;
          int tot;
          const int pos = block_flag_scan(f, ism, &tot);
          if (f) {
            flags[s] = -(base + pos) - 1;  // remember destination
            DT[base + pos] = ST[s];
          }
          base += tot;
        }
      }
      __syncthreads();
      if (S <= 32) base = ism[0];
      for (int e = threadIdx.x; e < S * 4 * n; e += blockDim.x) {
        const int s = e / (4 * n);
        const int f = flags[s];
        if (f < 0) DI[(int64_t)(-f - 1) * 4 * n + (e - s * 4 * n)] = tmp[e];
      }
      if (threadIdx.x == 0) cnt[L + 1] = base;
      __syncthreads();
      if (base > 0) {
        if (sp + 4 > 4 * 32) {
          if (threadIdx.x == 0) atomicOr(status, kStCapacity);
        } else {
          const unsigned long long np = (L == 0) ? 0ull : path;
          if (threadIdx.x == 0) {
            for (int c = 3; c >= 0; --c)
              stk[sp + (3 - c)] = (unsigned long long)(L + 1) | ((unsigned long long)c << 8) |
                                  ((np | ((unsigned long long)c << (2 * L))) << 16);
          }
          sp += 4;
        }
      }
      (void)cidx;
    }
    __syncthreads();
    // results of the patch
    for (int e = threadIdx.x; e < A * n; e += blockDim.x) {
      const int i = e / n, nm = e - i * n;
      I_near[(int64_t)apairs[i] * dv.ldI + nm] = acc[e];
    }
    for (int i = threadIdx.x; i < A; i += blockDim.x) leaves_out[apairs[i]] = lcnt[i];
    if constexpr (GRAD) block_reduce_M<D>(Mg, ws, ga.M + dv.node_off[j] * 3);
  }
  if (threadIdx.x == 0) {
    atomicAdd(reinterpret_cast<unsigned long long*>(dv.counters + 0), (unsigned long long)my_tests);
    atomicAdd(reinterpret_cast<unsigned long long*>(dv.counters + 1), (unsigned long long)my_nodes);
    atomicAdd(reinterpret_cast<unsigned long long*>(dv.counters + 4), (unsigned long long)my_tree);
  }
}

}  // namespace lcq
