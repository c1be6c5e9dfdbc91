// Degree-templated CUDA kernels of the correction path (sm_103a) and their launchers,
// instantiated one patch degree per translation unit (lcq_deg.cu built with -DLCQ_DEG=d) so
// that the degrees compile in parallel; lcq_kernels.cu dispatches to them by degree.
//
//   k_geom         chart coefficients, centroid, radius, d_j        (Sec. 3.2, Sec. 4)
//   k_farorder     far order q_j and annulus order                  (Sec. 4.2, Eq. qj)
//   k_rule_moments smooth-rule / annulus moments for many targets    (Sec. 4.2, Remark on eta_1)
//   k_adaptive     adaptive subdivision over a per-patch union tree  (Sec. 4.3; lcq_common.cuh)
//   k_self         singular self rules                              (Sec. 4, Eq. errestself)
//   k_v2c          a - s = V^T (I_near - I_smooth) into the CSR       (Sec. 4.3, 5.3)
//   k_far_src      oversampled far sources of the corrected potential (Sec. 5.3)
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "lcq_common.cuh"
#include "lcq_degree.h"

namespace lcq {

// ============================================================================ geometry
// One block per patch: x_nm = V y, J at the nodes, c_j, R_j, d_j (Sec. 3.2, 4).
template <int D>
__global__ void k_geom(const int* __restrict__ plist, int count, const int64_t* __restrict__ node_off,
                       const double* __restrict__ xyz, int64_t N, const double* __restrict__ Vt,
                       const double* __restrict__ nodes, double eta_p, double eta1_p,
                       double* __restrict__ coef, double* __restrict__ cen, double* __restrict__ rad,
                       double* __restrict__ dj, double* __restrict__ eta, double* __restrict__ eta1,
                       int* __restrict__ status) {
  constexpr int n = (D + 1) * (D + 2) / 2;
  __shared__ double y[3][n];
  __shared__ double cf[n * 3];
  __shared__ double J[n];
  __shared__ double c[3];
  __shared__ double red[kThreads / 32];
  for (int b = blockIdx.x; b < count; b += gridDim.x) {
    const int j = plist[b];
    const int64_t off = node_off[j];
    __syncthreads();
    for (int e = threadIdx.x; e < 3 * n; e += blockDim.x) {
      const int cc = e / n, l = e % n;
      const double val = xyz[cc * N + off + l];
      if (!isfinite(val)) atomicOr(status, kStNonFinite);
      y[cc][l] = val;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 3 * n; e += blockDim.x) {
      const int nm = e / 3, cc = e % 3;
      double acc = 0.0;
      for (int l = 0; l < n; ++l) acc = fma(Vt[nm * n + l], y[cc][l], acc);
      cf[nm * 3 + cc] = acc;
    }
    __syncthreads();
    for (int l = threadIdx.x; l < n; l += blockDim.x) {
      double X[3], Xu[3], Xv[3], Nn[3];
      kw_geometry<D>(nodes[l], nodes[n + l], cf, X, Xu, Xv, nullptr, 1);
      cross3(Xu, Xv, Nn);
      const double jj = sqrt(Nn[0] * Nn[0] + Nn[1] * Nn[1] + Nn[2] * Nn[2]);
      if (!(jj > 0.0)) atomicOr(status, kStDegenerate);
      J[l] = jj;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double sw = 0.0, s0 = 0.0, s1 = 0.0, s2 = 0.0, dmin = 1e300;
      for (int l = 0; l < n; ++l) {
        const double wj = nodes[2 * n + l] * J[l];
        sw += wj;
        s0 += wj * y[0][l];
        s1 += wj * y[1][l];
        s2 += wj * y[2][l];
        dmin = fmin(dmin, sqrt(wj));
      }
      c[0] = s0 / sw;
      c[1] = s1 / sw;
      c[2] = s2 / sw;
      dj[j] = dmin;
      const double e1 = eta_p > 0.0 ? eta_p : eta_default(D);
      eta[j] = e1;
      eta1[j] = fmin(eta1_p, e1);
    }
    __syncthreads();
    // radius: 153 vertices of the level-4 subdivision of T0 plus the nodes
    double rmax = 0.0;
    for (int s = threadIdx.x; s < 153 + n; s += blockDim.x) {
      double p0, p1, p2;
      if (s < 153) {
        int a = 0, r = s;
        while (r >= 17 - a) {
          r -= 17 - a;
          ++a;
        }
        double X[3], Xu[3], Xv[3];
        kw_geometry<D>(a / 16.0, r / 16.0, cf, X, Xu, Xv, nullptr, 1);
        p0 = X[0];
        p1 = X[1];
        p2 = X[2];
      } else {
        p0 = y[0][s - 153];
        p1 = y[1][s - 153];
        p2 = y[2][s - 153];
      }
      const double d0 = p0 - c[0], d1 = p1 - c[1], d2 = p2 - c[2];
      rmax = fmax(rmax, sqrt(d0 * d0 + d1 * d1 + d2 * d2));
    }
    rmax = warp_max(rmax);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = rmax;
    __syncthreads();
    if (threadIdx.x == 0) {
      double r = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r = fmax(r, red[w]);
      rad[j] = r;
      cen[3 * j] = c[0];
      cen[3 * j + 1] = c[1];
      cen[3 * j + 2] = c[2];
    }
    // coefficients of X - c_j (K_00 = sqrt(2) is constant): every local quadrature works
    // with positions relative to the centroid
    for (int e = threadIdx.x; e < 3 * n; e += blockDim.x)
      coef[off * 3 + e] = e < 3 ? cf[e] - c[e] * 0.70710678118654752 : cf[e];
  }
}

// Smooth rule q_j moments for every near pair of the patch (Sec. 4.2): I_smooth (modes
// bit 0, rule qv, out_smooth); and annulus-rule moments for the annulus pairs (Remark on
// eta_1; modes bit 1, rule qn, out_ann).  One block per patch and launch, both passes in it.
template <int D>
__global__ void __launch_bounds__(kThreads, 2) k_rule_moments(
    const int* __restrict__ plist, int count, Dev dv, int modes, const int32_t* __restrict__ qv,
    const int32_t* __restrict__ qn, const KernelParams kp, cplx* __restrict__ out_smooth,
    cplx* __restrict__ out_ann, int form) {
  using C = Cfg<D>;
  extern __shared__ double smem[];
  double* cf = smem;
  SegMap* segs = reinterpret_cast<SegMap*>(cf + C::n * 3);
  // tensor-core moment workspace, 128-byte aligned
  unsigned char* smb = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(segs + 4) + 127) & ~static_cast<uintptr_t>(127));
  __shared__ KernelParams kps;
  // derivative series of the chart, for the FP64 engine of the smallest degrees
  __shared__ double cfd[D <= kFp64MomentsMaxDeg ? 2 * 3 * (D * (D + 1) / 2) : 1];
  __shared__ FxChart<D> ch;
  const double* cfdp = cfd;
  const int64_t ld = dv.ldI;
  for (int b = blockIdx.x; b < count; b += gridDim.x) {
    const int j = plist[b];
    const int formj = pair_form(dv, j, form);  // FP64, FP32 or two-float pair evaluation
    __syncthreads();
    load_coef<D>(dv.coef, dv.node_off[j], cf);
    if (threadIdx.x == 0) {
      segs[0] = seg_T0();
      kps = patch_kp(dv, j, kp);
    }
    __syncthreads();
    if constexpr (D <= kFp64MomentsMaxDeg) load_coef_derivs<D>(cf, dv.duv[D], cfd);
    load_fx_chart<D>(cf, dv.duv[D], &ch);
    long long evals = 0;
    for (int mode = 0; mode < 2; ++mode) {
      if (!(modes & (1 << mode))) continue;
      const int m = mode == 0 ? qv[j] : qn[j];
      if (m <= 0) continue;
      const double* ru = dv.ru + dv.roff[m];
      const double* rv = dv.rv + dv.roff[m];
      const double* rw = dv.rw + dv.roff[m];
      if (mode == 0) {
        const int64_t p0 = dv.pair_ptr[j], np = dv.pair_ptr[j + 1] - p0;
        TgtIdx ta{dv.tgt, dv.NT, dv.pair_tgt + p0, dv.tnrm};
        cplx* base = out_smooth + p0 * ld;
        block_moments_any<D>(cf, cfdp, ch, ru, rv, rw, m * m, segs, 1, ta, (int)np,
                             RowsAt{base, ld}, kps, smb,
                             dv.cen + 3 * j, 0.0, nullptr, formj);
        evals += np * m * m;
      } else {
        const int64_t a0 = dv.an_ptr[j], na = dv.an_ptr[j + 1] - a0;
        const int32_t* pl = dv.an_pair + a0;
        TgtPairIdx ta{dv.tgt, dv.NT, dv.pair_tgt, pl, dv.tnrm};
        block_moments_any<D>(cf, cfdp, ch, ru, rv, rw, m * m, segs, 1, ta, (int)na,
                             RowsBy{out_ann, pl, ld}, kps,
                             smb, dv.cen + 3 * j, 0.0, nullptr, formj);
        evals += na * m * m;
      }
    }
    if (threadIdx.x == 0 && evals > 0)
      atomicAdd(reinterpret_cast<unsigned long long*>(dv.counters + 3), (unsigned long long)evals);
  }
}

// ============================================================================ far order
// The cnt farthest (far) or nearest of N near pairs (pair(i): their ids), ties by the smaller
// target id, their targets' positions into pts, by the whole block: each step takes the next
// pair in the order of (distance, target).  One thread's 10 passes over some 460 pairs in global
// memory held the stage: 12.3 -> 10.7 ms (1280 patches, degree 6), 5.9 -> 2.7 ms (2400, degree
// 3).  Distances are >= 0, so their bit patterns order like the values and the compares run on
// the integer pipe.
template <class G>
__device__ void select_targets(const Dev& dv, int64_t N, int cnt, bool far, G pair, double* pts,
                               long long* rkey, int* rtgt) {
  long long lastk = -1;
  int lastt = -1;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int k = 0; k < cnt; ++k) {
    long long bk = 0x7fffffffffffffffll;
    int bt = 0x7fffffff;
    auto take = [&](long long key, int t) {
      if (key < bk || (key == bk && t < bt)) {
        bk = key;
        bt = t;
      }
    };
    for (int64_t i = threadIdx.x; i < N; i += blockDim.x) {
      const int64_t p = pair(i);
      const long long d = __double_as_longlong(dv.pair_d2[p]);
      const long long key = far ? 0x7ffffffffffffffell - d : d;
      const int t = dv.pair_tgt[p];
      if (key > lastk || (key == lastk && t > lastt)) take(key, t);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const long long ok = __shfl_xor_sync(0xffffffffu, bk, o);
      const int ot = __shfl_xor_sync(0xffffffffu, bt, o);
      take(ok, ot);
    }
    __syncthreads();
    if (lane == 0) {
      rkey[w] = bk;
      rtgt[w] = bt;
    }
    __syncthreads();
    for (int i = 0; i < nw; ++i) take(rkey[i], rtgt[i]);
    lastk = bk;
    lastt = bt;
    if (threadIdx.x < 3) pts[3 * k + threadIdx.x] = dv.tgt[threadIdx.x * dv.NT + bt];
  }
}

// q_j (Eq. qj) and the annulus order: smallest m with
//   max_x ||I_m(x) - I_{m+1}(x)||_2 <= eps d_j / ||V||  over the test points.
template <int D>
__global__ void __launch_bounds__(kThreads, 2) k_farorder(const int* __restrict__ plist, int count,
                                                       Dev dv, const KernelParams kp, double eps,
                                                       int m_max, double normV,
                                                       const double* __restrict__ dirs, int ndirs,
                                                       cplx* __restrict__ scratch,
                                                       int32_t* __restrict__ q_out,
                                                       int32_t* __restrict__ qn_out,
                                                       int* __restrict__ sched) {
  using C = Cfg<D>;
  extern __shared__ double smem[];
  double* cf = smem;
  SegMap* segs = reinterpret_cast<SegMap*>(cf + C::n * 3);
  double* pts = reinterpret_cast<double*>(segs + 4);        // [kMaxTestPts][3]
  double* red = pts + 3 * kMaxTestPts;                      // [kThreads/32]
  int* sel = reinterpret_cast<int*>(red + kThreads / 32);   // [2]
  double* ws = reinterpret_cast<double*>(sel + 4);
  __shared__ KernelParams kps;
  __shared__ double cfd[2 * 3 * (D * (D + 1) / 2)];  // derivative series of the chart
  const double* cfdp = cfd;
  cplx* bufA = scratch + (int64_t)blockIdx.x * 2 * kMaxTestPts * C::n;
  cplx* bufB = bufA + kMaxTestPts * C::n;
  const int m_min = (D + 2) / 2;
  __shared__ int next_b, rtgt[kThreads / 32];
  __shared__ long long rkey[kThreads / 32];
  // patches are taken from the counter *sched (zeroed before the launch), so blocks that
  // drew cheap patches take more of them
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) next_b = atomicAdd(sched, 1);
    __syncthreads();
    const int b = next_b;
    if (b >= count) break;
    const int j = plist[b];
    load_coef<D>(dv.coef, dv.node_off[j], cf);
    if (threadIdx.x == 0) {
      segs[0] = seg_T0();
      kps = patch_kp(dv, j, kp);
    }
    __syncthreads();
    load_coef_derivs<D>(cf, dv.duv[D], cfd);
    const int64_t p0 = dv.pair_ptr[j], np = dv.pair_ptr[j + 1] - p0;
    const double R = dv.rad[j], c0 = dv.cen[3 * j], c1 = dv.cen[3 * j + 1], c2 = dv.cen[3 * j + 2];
    const double tol = (dv.pgroup ? dv.grp[dv.pgroup[j]].eps : eps) * dv.dj[j] / normV;
    for (int pass = 0; pass < 2; ++pass) {
      // test points (Sec. 4.2): pass 0 = far order, pass 1 = annulus order
      __syncthreads();
      int F = 0;
      const int64_t a0 = dv.an_ptr[j], na = dv.an_ptr[j + 1] - a0;
      auto sphere = [&](double rr) {  // c_j + rr dir, at most kMaxTestPts points in all
        const int m = max(min(ndirs, kMaxTestPts - F), 0);
        for (int k = threadIdx.x; k < m; k += blockDim.x) {
          pts[3 * (F + k)] = c0 + rr * dirs[3 * k];
          pts[3 * (F + k) + 1] = c1 + rr * dirs[3 * k + 1];
          pts[3 * (F + k) + 2] = c2 + rr * dirs[3 * k + 2];
        }
        F += m;
      };
      if (pass == 0) {
        const int cnt = np >= 20 ? 10 : (int)(np / 2);
        select_targets(dv, np, cnt, true, [&](int64_t p) { return p0 + p; }, pts, rkey, rtgt);
        F = cnt;
        if (np < 20) sphere(dv.eta[j] * R);
      } else if (na > 0) {
        sphere(dv.eta1[j] * R);
        const int cnt = min(na < 10 ? (int)na : 10, kMaxTestPts - F);
        select_targets(dv, na, cnt, false, [&](int64_t a) { return (int64_t)dv.an_pair[a0 + a]; },
                       pts + 3 * F, rkey, rtgt);
        F += max(cnt, 0);
      }
      __syncthreads();
      if (pass == 1 && F == 0) {
        if (threadIdx.x == 0) qn_out[j] = 0;
        continue;
      }
      TgtPts ta{pts};
      int m = m_min, chosen = m_max;
      {
        const double* ru = dv.ru + dv.roff[m];
        block_moments<D>(cf, cfdp, ru, dv.rv + dv.roff[m], dv.rw + dv.roff[m], m * m, segs, 1, ta, F,
                         [=] __device__(int i) { return bufA + (int64_t)i * C::n; }, C::n, kps, ws,
                         dv.cen + 3 * j);
      }
      cplx* A = bufA;
      cplx* Bf = bufB;
      for (; m < m_max; ++m) {
        const int m1 = m + 1;
        block_moments<D>(cf, cfdp, dv.ru + dv.roff[m1], dv.rv + dv.roff[m1], dv.rw + dv.roff[m1], m1 * m1,
                         segs, 1, ta, F, [=] __device__(int i) { return Bf + (int64_t)i * C::n; },
                         C::n, kps, ws, dv.cen + 3 * j);
        __syncthreads();
        // max over points of the 2-norm of the difference
        double e = 0.0;
        const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
        for (int i = w; i < F; i += blockDim.x >> 5) {
          double s = 0.0;
          for (int nm = lane; nm < C::n; nm += 32) {
            const cplx a = A[i * C::n + nm], bb = Bf[i * C::n + nm];
            const double dr = a.re - bb.re, di = a.im - bb.im;
            s += dr * dr + di * di;
          }
          s = warp_sum(s);
          e = fmax(e, sqrt(s));
        }
        if (lane == 0) red[w] = e;
        __syncthreads();
        if (threadIdx.x == 0) {
          double mx = 0.0;
          for (int k = 0; k < (int)(blockDim.x >> 5); ++k) mx = fmax(mx, red[k]);
          sel[1] = mx <= tol ? 1 : 0;
        }
        __syncthreads();
        if (sel[1]) {
          chosen = m;
          break;
        }
        cplx* tmp = A;
        A = Bf;
        Bf = tmp;
      }
      if (threadIdx.x == 0) {
        if (pass == 0) q_out[j] = chosen; else qn_out[j] = chosen;
      }
    }
  }
}

// ============================================================================ self
// Self rule for the target at node i (Sec. 4, Eq. errestself; stand-in for
// generalized Gaussian rules): affine map M = G^{-1/2} (G the first fundamental
// form at the node) making the chart conformal there, split at the node into three
// Duffy triangles; s: n_s-point Gauss-Legendre; t: split at the foot of the
// perpendicular, sinh substitution t - t0 = mu sinh(xi), [0, xi_max] cut into
// ceil(xi_max / 1.5) panels of n_t-point Gauss-Legendre.
struct SelfSeg {
  double E0x, E0y, Dx, Dy, t0, mu, area2, xi_max, side;
  int npan, off;
};

// Block per self target: the self rule above applied to the chart, contracted with the
// basis into the target's self weights (Sec. 4).  About 2000 nodes a target at eps = 1e-9, none
// sharing a row with another: in FP64 a node took 430 instructions of 64 cycles (basis 130, tangents
// 126, chord 105, parameters 50) and 64 more in the contraction.  Here the rule's radial and angular
// factors are formed once per (panel, angle) instead of per node, basis, tangents and chord are
// fixed-point (lcq_fxgeom.cuh), and the contraction runs on the tensor cores (tc_tile with one
// target: the chunk's 128 kernel values are one row).  1280 patches, generation: 262 -> 244 ms.
// The largest degrees keep FP64 basis values and an FP64 contraction: the fixed-point basis and its
// slices are fractions of the bound 2^E_nm, reached at a corner only, which is 2^16 at degree 10.
// Error of one patch's self weights against 80 bits beyond what the chart's coefficients give all
// forms, of the imaginary part, fixed and FP64: degree 6 5.3e-15 and 5.1e-15, degree 8 1.7e-14 and
// 1.3e-14, degree 9 3.0e-14 and 2.6e-14, degree 10 8.0e-14 and 3.8e-14.
constexpr int kSelfFp64Deg = 9;
constexpr int kSelfThreads = 128;
constexpr int kSelfTab = 384;  // (panel, angle) entries kept; longer rules form them per node
template <int D>
struct SelfCfg {
  static constexpr int n = (D + 1) * (D + 2) / 2;
  static constexpr bool fp64 = D >= kSelfFp64Deg;
  static constexpr int BST = kSelfThreads + (fp64 ? 1 : 8);
  static constexpr size_t taylor = ((D + 1) * n + 2 * n * n) * sizeof(double);
  static constexpr size_t basis = (size_t)n * BST * 8;
  static constexpr size_t OFF_G = ((taylor > basis ? taylor : basis) + 15) / 16 * 16;
  static constexpr size_t OFF_TAB = OFF_G + kSelfThreads * 16;
  static constexpr size_t BYTES = OFF_TAB + kSelfTab * 3 * sizeof(double);
};
// The direction and weight of angle entry e = (segment, panel, angle): (du, dv) = s (out[0],
// out[1]) and node weight w_s s out[2] for the radial node s.
__device__ __forceinline__ void self_entry(const SelfSeg* sg, int nseg, int ns, int nt,
                                           const double* __restrict__ glx, const double* __restrict__ glw,
                                           const double* Mm, int e, double* out) {
  int k = 0;
  while (k + 1 < nseg && e * ns >= sg[k + 1].off) ++k;
  const SelfSeg& g = sg[k];
  const int loc = e - g.off / ns;
  const int p = loc / nt, ti = loc - p * nt;
  const double lo = g.xi_max * p / g.npan, hi = g.xi_max * (p + 1) / g.npan;
  const double xi = lo + (hi - lo) * glx[ti];
  // sinh and cosh from one exponential (xi >= 0: the difference loses at most a few
  // 1e-16 absolute near xi = 0, which moves the node by mu times that)
  const double ex = exp(xi), exi = 1.0 / ex;
  const double tpar = g.t0 + g.side * g.mu * (0.5 * (ex - exi));
  const double zx = g.E0x + tpar * g.Dx, zy = g.E0y + tpar * g.Dy;
  out[0] = Mm[0] * zx + Mm[1] * zy;
  out[1] = Mm[2] * zx + Mm[3] * zy;
  out[2] = glw[ti] * (hi - lo) * g.mu * (0.5 * (ex + exi)) * g.area2 * Mm[4];
}

// Basis slices (column B, stride st; of the largest degrees the FP64 values) and normal X_u x X_v of
// a node in FP64: of a chart that the fixed-point scales do not fit, or of the largest degrees.
template <int D>
__device__ __noinline__ void self_node_fp64(double u, double v, const FxChart<D>& ch, uint2* B, int st,
                                            double* N) {
  double K[(D + 1) * (D + 2) / 2], X[3], Xu[3], Xv[3];
  kw_geometry_proj<D>(u, v, reinterpret_cast<const double*>(ch.x),
                      reinterpret_cast<const double*>(ch.d), X, Xu, Xv, K);
#pragma unroll 1
  for (int k = 0; k < (D + 1) * (D + 2) / 2; ++k)
    B[k * st] = SelfCfg<D>::fp64
                    ? make_uint2((uint32_t)__double2loint(K[k]), (uint32_t)__double2hiint(K[k]))
                    : slice_bytes(fix_mag<8>(K[k], c_kwexp[k]), __double2hiint(K[k]) < 0);
  cross3(Xu, Xv, N);
}

template <int D>
__global__ void __launch_bounds__(kSelfThreads, 4) k_self(Dev dv, const int32_t* __restrict__ deg_of_patch,
                                              const KernelParams kp, int order,
                                              cplx* __restrict__ out_self) {
  using SC = SelfCfg<D>;
  constexpr int n = SC::n;
  __shared__ double cf[3 * n];
  __shared__ SelfSeg sg[6];
  __shared__ double Mm[6];  // M00 M01 M10 M11 detM, smallest singular value of DX at the node
  __shared__ double P[2];
  __shared__ int nseg, total;
  __shared__ KernelParams kps;
  __shared__ int ord;
  __shared__ double nP[3];  // unit chart normal at the target node (S')
  __shared__ FxChart<D> ch;
  __shared__ double tX[3 * n];  // Taylor coefficients of the chord at P, in fixed point unless cfp
  __shared__ int st, cfp;
  __shared__ int rowE[2];
  __shared__ cplx acc[n];
  extern __shared__ __align__(16) unsigned char ssm[];
  uint2* Bs = reinterpret_cast<uint2*>(ssm);
  uint4* G = reinterpret_cast<uint4*>(ssm + SC::OFF_G);
  double* tabl = reinterpret_cast<double*>(ssm + SC::OFF_TAB);
  long long my_nodes = 0;
  for (int64_t s = blockIdx.x; s < dv.n_self; s += gridDim.x) {
    const int t = dv.self_tgt[s];
    const int j = dv.tpatch[t];
    if (deg_of_patch[j] != D) continue;
    const int i = dv.tlnode[t];
    __syncthreads();
    load_coef<D>(dv.coef, dv.node_off[j], cf);
    if (threadIdx.x == 0) {
      kps = patch_kp(dv, j, kp);
      ord = dv.pgroup ? dv.grp[dv.pgroup[j]].self_order : order;
    }
    load_fx_chart<D, SC::fp64>(cf, dv.duv[D], &ch);
    const int ns = ord, nt = ord;
    const double* glx = dv.gl_x + dv.gl_off[ord];
    const double* glw = dv.gl_w + dv.gl_off[ord];
    if (threadIdx.x == 0) {
      const double pu = dv.nodes_uv[D][i], pv = dv.nodes_uv[D][n + i];
      P[0] = pu;
      P[1] = pv;
      double X[3], Xu[3], Xv[3];
      kw_geometry<D>(pu, pv, cf, X, Xu, Xv, nullptr, 1);
      {
        double Np[3];
        cross3(Xu, Xv, Np);
        const double ln = sqrt(Np[0] * Np[0] + Np[1] * Np[1] + Np[2] * Np[2]);
        nP[0] = Np[0] / ln;
        nP[1] = Np[1] / ln;
        nP[2] = Np[2] / ln;
      }
      const double a = Xu[0] * Xu[0] + Xu[1] * Xu[1] + Xu[2] * Xu[2];
      const double bb = Xu[0] * Xv[0] + Xu[1] * Xv[1] + Xu[2] * Xv[2];
      const double c = Xv[0] * Xv[0] + Xv[1] * Xv[1] + Xv[2] * Xv[2];
      const double sq = sqrt(a * c - bb * bb);
      const double tt = sqrt(a + c + 2.0 * sq);
      // R = sqrt(G) = (G + sq I)/tt ; M = R^{-1}
      const double R00 = (a + sq) / tt, R01 = bb / tt, R11 = (c + sq) / tt;
      const double detR = R00 * R11 - R01 * R01;
      Mm[0] = R11 / detR;
      Mm[1] = -R01 / detR;
      Mm[2] = -R01 / detR;
      Mm[3] = R00 / detR;
      Mm[4] = 1.0 / detR;
      const double tr = R00 + R11;
      Mm[5] = 2.0 * detR / (tr + sqrt(fmax(tr * tr - 4.0 * detR, 0.0)));
      double Z[3][2];
      const double VX[3] = {0.0, 1.0, 0.0}, VY[3] = {0.0, 0.0, 1.0};
      for (int k = 0; k < 3; ++k) {
        const double dx = VX[k] - pu, dy = VY[k] - pv;
        Z[k][0] = R00 * dx + R01 * dy;
        Z[k][1] = R01 * dx + R11 * dy;
      }
      int cntg = 0, off = 0;
      for (int e = 0; e < 3; ++e) {
        const double E0x = Z[e][0], E0y = Z[e][1];
        const double Dx = Z[(e + 1) % 3][0] - E0x, Dy = Z[(e + 1) % 3][1] - E0y;
        const double L2 = Dx * Dx + Dy * Dy;
        double t0 = -(E0x * Dx + E0y * Dy) / L2;
        t0 = fmin(fmax(t0, 0.0), 1.0);
        const double area2 = fabs(E0x * Dy - E0y * Dx);
        const double mu = area2 / L2;
        for (int sd = 0; sd < 2; ++sd) {
          const double side = sd == 0 ? 1.0 : -1.0;
          const double len = sd == 0 ? 1.0 - t0 : t0;
          if (len <= 0.0) continue;
          const double xm = asinh(len / mu);
          int npan = 1;
          if (isfinite(xm) && xm > 0.0) npan = (int)fmin(ceil(xm / 1.5), 64.0);
          else atomicOr(dv.status, kStNonFinite);
          SelfSeg g{E0x, E0y, Dx, Dy, t0, mu, area2, xm, side, npan, off};
          sg[cntg++] = g;
          off += npan * nt * ns;
        }
      }
      nseg = cntg;
      total = off;
    }
    __syncthreads();
    const FxTables tab = fx_tables();
    FxS nPx[3];  // S': the source's normal replaced by -n_x
    for (int c = 0; c < 3; ++c) nPx[c] = fx_split(fx_fix(-nP[c], 0));
    const bool nbad = kps.kind == 3 && !isfinite(nP[0] + nP[1] + nP[2]);
    const int nent = total / ns;
    for (int e = threadIdx.x; e < nent && e < kSelfTab; e += blockDim.x)
      self_entry(sg, nseg, ns, nt, glx, glw, Mm, e, tabl + 3 * e);
    // the basis area is free until the first chunk
    chart_taylor<D>(P[0], P[1], cf, reinterpret_cast<double*>(ssm), tX);
    if (threadIdx.x == 0) {
      double mx = 0.0;
      for (int c = 0; c < 3; ++c) {
        double a = 0.0;
        for (int e = 1; e < n; ++e) a += fabs(tX[c * n + e]);
        mx = fmax(mx, a);
      }
      fx_mant(mx, &st);
      st = max(st, -1000);
      cfp = !(mx < 1e150 && ldexp(1.0, st) <= kFxChordMax * Mm[5]);
    }
    __syncthreads();
    u64* tXf = reinterpret_cast<u64*>(tX);
    if (!cfp)
      for (int e = threadIdx.x; e < 3 * n; e += blockDim.x) tXf[e] = fx_join28(fx_fix(tX[e], st));
    for (int e = threadIdx.x; e < n; e += blockDim.x) acc[e] = {0.0, 0.0};
    const int tot = total;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int c0 = 0; c0 < tot; c0 += kSelfThreads) {
      if (threadIdx.x < 2) rowE[threadIdx.x] = 0;
      __syncthreads();
      const int idx = c0 + threadIdx.x;
      cplx gk = {0.0, 0.0};
      if (idx < tot) {
        const int e = idx / ns, si = idx - e * ns;
        double direct[3];
        const double* en = tabl + 3 * e;
        if (e >= kSelfTab) {
          self_entry(sg, nseg, ns, nt, glx, glw, Mm, e, direct);
          en = direct;
        }
        const double sv = glx[si], du = sv * en[0], dvv = sv * en[1];
        const double w = glw[si] * sv * en[2];
        i64 N[3], d[3];
        FxS nn[3];
        u64 wm;
        int ew;
        if (SC::fp64 || ch.fp64) {
          double Nd[3];
          self_node_fp64<D>(P[0] + du, P[1] + dvv, ch, Bs + threadIdx.x, SC::BST, Nd);
          fx_make_node(Nd, w, nn, &wm, &ew);
        } else {
          int sn;
          fx_basis_normal<D>(P[0] + du, P[1] + dvv, ch, N, &sn, [&](int k, i64 kv) {
            const u64 sgn = (u64)(kv >> 63);
            Bs[k * SC::BST + threadIdx.x] = slice_bytes(((((u64)kv ^ sgn) - sgn) + 32) >> 6, kv < 0);
          });
          fx_node_from_normal(N, sn + 1, w, nn, &wm, &ew);
        }
        if (nbad) ew = kFxBad + 1;
        // the target is the chart's value at the node: x - X(P + delta) = -dX
        FxS dm[3];
        int E = 0;
        bool ok;
        double dX[3];
        if (cfp) {
          chart_chord<D>(tX, du, dvv, dX);
          ok = fx_vector(-dX[0], -dX[1], -dX[2], dm, &E);
        } else {
          fx_chord<D>(tXf, du, dvv, d, &E);
          E += st + 1;
          ok = fx_vector_int(-d[0], -d[1], -d[2], E, dm, &E);
        }
        const FxS nu[3] = {kps.kind == 3 ? nPx[0] : nn[0], kps.kind == 3 ? nPx[1] : nn[1],
                           kps.kind == 3 ? nPx[2] : nn[2]};
        if (!ok || !fx_core<false>(kps.fx, tab, dm[0], dm[1], dm[2], E, nu, wm, ew, &gk.re, &gk.im,
                                   nullptr, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f)) {
          if (!cfp) {
            int e2;
            fx_chord<D>(tXf, du, dvv, d, &e2);
#pragma unroll
            for (int c = 0; c < 3; ++c) dX[c] = fx_pack<false>(d[c], e2 + st - 61);
          }
          gk = fx_fallback(kps, -dX[0], -dX[1], -dX[2], nu[0], nu[1], nu[2], wm, ew, 0.0, nullptr);
        }
      } else {
        const uint32_t z = SC::fp64 ? 0u : kZeroSlices;
        for (int k = 0; k < n; ++k) Bs[k * SC::BST + threadIdx.x] = make_uint2(z, z);
      }
      if constexpr (SC::fp64) {
        reinterpret_cast<cplx*>(G)[threadIdx.x] = gk;
        __syncthreads();
        for (int k = threadIdx.x; k < n; k += kSelfThreads) {
          const double* K = reinterpret_cast<const double*>(Bs) + k * SC::BST;
          cplx s = {0.0, 0.0};
          for (int q = 0; q < kSelfThreads; ++q) {
            const cplx gq = reinterpret_cast<const cplx*>(G)[q];
            s.re = fma(gq.re, K[q], s.re);
            s.im = fma(gq.im, K[q], s.im);
          }
          acc[k].re += s.re;
          acc[k].im += s.im;
        }
        __syncthreads();
        continue;
      }
      const int fr = __reduce_max_sync(0xffffffffu, exp_field(gk.re));
      const int fi = __reduce_max_sync(0xffffffffu, exp_field(gk.im));
      if (lane == 0) {
        atomicMax(rowE, fr);
        atomicMax(rowE + 1, fi);
      }
      __syncthreads();
      const uint2 a = row_slices(gk.re, exp_bound(rowE[0], 0.0));
      const uint2 b = row_slices(gk.im, exp_bound(rowE[1], 0.0));
      G[threadIdx.x] = make_uint4(a.x, a.y, b.x, b.y);
      __syncthreads();
      const int kend = (min(kSelfThreads, tot - c0) + 15) & ~15;
      for (int ct = warp; ct < TcCfg<D>::NTILE; ct += kSelfThreads / 32)
        tc_tile<D, 8, 9, 0x7ff, SC::BST>(Bs, G, rowE, ct, 0, kend, 1, 0, 0, false,
                                         [&](int) { return acc; });
      __syncthreads();
    }
    my_nodes += tot;
    for (int k = threadIdx.x; k < n; k += blockDim.x) out_self[s * dv.ldI + k] = acc[k];
  }
  if (threadIdx.x == 0)
    atomicAdd(reinterpret_cast<unsigned long long*>(dv.counters + 2), (unsigned long long)my_nodes);
}

// ============================================================================ target normals
// Unit normals for S': the chart normal X_u x X_v / |.| at the node of an on-surface target
// on a degree-D patch; with do_off, the normalized user normal of an off-surface target.
template <int D>
__global__ void k_tgt_normals(Dev dv, const int32_t* __restrict__ deg, const double* __restrict__ user,
                              bool do_off, double* __restrict__ out) {
  constexpr int n = (D + 1) * (D + 2) / 2;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < dv.NT;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int tp = dv.tpatch[t];
    double v[3];
    if (tp >= 0) {
      if (deg[tp] != D) continue;
      double cf[3 * n], X[3], Xu[3], Xv[3];
      const int64_t off = dv.node_off[tp];
      for (int e = 0; e < 3 * n; ++e) cf[e] = dv.coef[off * 3 + e];
      const int i = dv.tlnode[t];
      kw_geometry<D>(dv.nodes_uv[D][i], dv.nodes_uv[D][n + i], cf, X, Xu, Xv, nullptr, 1);
      cross3(Xu, Xv, v);
    } else {
      if (!do_off) continue;
      v[0] = user[t];
      v[1] = user[dv.NT + t];
      v[2] = user[2 * dv.NT + t];
    }
    const double l = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    if (!(l > 0.0) || !isfinite(l)) atomicOr(dv.status, kStNonFinite);
    for (int c = 0; c < 3; ++c) out[c * dv.NT + t] = v[c] / l;
  }
}

// ============================================================================ V contraction
// c_l = sum_nm V[nm][l] (I_near[nm] - I_smooth[nm]) written to the CSR (Sec. 4.3, 5.3).
template <int D>
__global__ void k_v2c(const int* __restrict__ plist, int count, Dev dv,
                      const double* __restrict__ Vt, const cplx* __restrict__ In,
                      const cplx* __restrict__ Is, const cplx* __restrict__ InS,
                      double* __restrict__ val) {
  constexpr int n = (D + 1) * (D + 2) / 2;
  __shared__ double V[n * n];
  __shared__ cplx diff[kThreads / 32][n];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) V[e] = Vt[e];
  __syncthreads();
  for (int b = blockIdx.x; b < count; b += gridDim.x) {
    const int j = plist[b];
    const int64_t p0 = dv.pair_ptr[j], np = dv.pair_ptr[j + 1] - p0;
    const int64_t s0 = dv.self_ptr[j], nsf = dv.self_ptr[j + 1] - s0;
    for (int64_t k = w; k < np + nsf; k += nw) {
      const bool self = k >= np;
      const int64_t id = self ? (s0 + k - np) : (p0 + k);
      // self pairs store the self weights themselves: the own patch is masked out of the
      // far sum (no spurious smooth-rule contribution to subtract)
      const cplx* a = self ? InS + id * dv.ldI : In + id * dv.ldI;
      const cplx* s = Is + id * dv.ldI;
      for (int nm = lane; nm < n; nm += 32)
        diff[w][nm] = self ? a[nm] : cplx{a[nm].re - s[nm].re, a[nm].im - s[nm].im};
      __syncwarp();
      const int64_t dst = self ? dv.self_csr[id] : dv.pair_csr[id];
      for (int l = lane; l < n; l += 32) {
        double re = 0.0, im = 0.0;
        for (int nm = 0; nm < n; ++nm) {
          const double vv = V[nm * n + l];
          re = fma(vv, diff[w][nm].re, re);
          im = fma(vv, diff[w][nm].im, im);
        }
        val[2 * (dst + l)] = re;
        val[2 * (dst + l) + 1] = im;
      }
      __syncwarp();
    }
  }
}

// ============================================================================ apply
// Oversampled sources of rule q_j: X, (X_u x X_v) w, |.| w and the interpolated density
// sigma~_q = sum_nm K_nm(u_q) s_nm, s = V sigma (Sec. 4.2 Remark, Sec. 5.3).  With fx, rows 3-6
// and 9 hold the node as fx_eval takes it instead (fx_make_node): unit normal, mantissa and
// exponent of J w / (4 pi).
template <int D>
__global__ void k_far_src(const int* __restrict__ plist, int count, Dev dv,
                          const double* __restrict__ Vt, const int32_t* __restrict__ qv,
                          const int64_t* __restrict__ src_off, const cplx* __restrict__ sigma,
                          double* __restrict__ src /*[9 or 10][N_over]*/, int64_t n_over,
                          bool fx) {
  constexpr int n = (D + 1) * (D + 2) / 2;
  __shared__ double cf[3 * n];
  __shared__ double cfd[2 * 3 * (D * (D + 1) / 2)];  // derivative series of the chart
  __shared__ cplx sc[n];
  for (int b = blockIdx.x; b < count; b += gridDim.x) {
    const int j = plist[b];
    const int64_t off = dv.node_off[j];
    __syncthreads();
    load_coef<D>(dv.coef, off, cf);
    __syncthreads();
    load_coef_derivs<D>(cf, dv.duv[D], cfd);
    for (int nm = threadIdx.x; nm < n; nm += blockDim.x) {
      double re = 0.0, im = 0.0;
      if (sigma)  // null: geometry only (the adjoint's sources)
        for (int l = 0; l < n; ++l) {
          re = fma(Vt[nm * n + l], sigma[off + l].re, re);
          im = fma(Vt[nm * n + l], sigma[off + l].im, im);
        }
      sc[nm] = {re, im};
    }
    __syncthreads();
    const int m = qv[j], Q = m * m;
    const double* ru = dv.ru + dv.roff[m];
    const double* rv = dv.rv + dv.roff[m];
    const double* rw = dv.rw + dv.roff[m];
    for (int q = threadIdx.x; q < Q; q += blockDim.x) {
      // chart and tangents by the projected derivative series (rolled sums over the stored
      // basis values keep the register count low), then the interpolated density
      double X[3], Xu[3], Xv[3], Nn[3], K[n];
      kw_geometry_proj<D>(ru[q], rv[q], cf, cfd, X, Xu, Xv, K);
      double re = 0.0, im = 0.0;
#pragma unroll 1
      for (int k = 0; k < n; ++k) {
        re = fma(K[k], sc[k].re, re);
        im = fma(K[k], sc[k].im, im);
      }
      cross3(Xu, Xv, Nn);
      const double w = rw[q];
      const int64_t o = src_off[j] + q;
      src[0 * n_over + o] = X[0] + dv.cen[3 * j];
      src[1 * n_over + o] = X[1] + dv.cen[3 * j + 1];
      src[2 * n_over + o] = X[2] + dv.cen[3 * j + 2];
      src[7 * n_over + o] = re;
      src[8 * n_over + o] = im;
      if (fx) {
        FxS nn[3];
        u64 wm;
        int ew;
        fx_make_node(Nn, w, nn, &wm, &ew);
        for (int c = 0; c < 3; ++c)
          src[(3 + c) * n_over + o] = __longlong_as_double((long long)fx_join(nn[c]));
        src[6 * n_over + o] = __longlong_as_double((long long)wm);
        src[9 * n_over + o] = __longlong_as_double((long long)ew);
      } else {
        const double J = sqrt(Nn[0] * Nn[0] + Nn[1] * Nn[1] + Nn[2] * Nn[2]);
        src[3 * n_over + o] = Nn[0] * w;
        src[4 * n_over + o] = Nn[1] * w;
        src[5 * n_over + o] = Nn[2] * w;
        src[6 * n_over + o] = J * w;
      }
    }
  }
}

// ============================================================================ launchers
template <class K>
void set_smem(K kern, size_t bytes) {
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int D>
void GeomL<D>::run(const LaunchCommon& lc, const int* plist, int count, const int64_t* node_off,
                  const double* xyz, int64_t N, const double* Vt, const double* nodes, double eta_p,
                  double eta1_p, double* coef, double* cen, double* rad, double* dj, double* eta,
                  double* eta1, int* status) {
    const int grid = count < lc.num_sms * 8 ? count : lc.num_sms * 8;
    ++*lc.launches;
    k_geom<D><<<grid, 128, 0, lc.stream>>>(plist, count, node_off, xyz, N, Vt, nodes, eta_p, eta1_p,
                                           coef, cen, rad, dj, eta, eta1, status);
  }


template <int D>
size_t moments_smem_bytes(int extra_doubles) {
  using C = Cfg<D>;
  return sizeof(double) * (C::n * 3 + extra_doubles + C::WS) + sizeof(SegMap) * 4 + 1024;
}

template <int D>
void RuleMomL<D>::run(const LaunchCommon& lc, const int* plist, int count, const Dev& dv, int modes,
                  const int32_t* qv, const int32_t* qn, const KernelParams& kp, void* out_smooth,
                  void* out_ann, int form) {
    const size_t sm = sizeof(double) * 3 * Cfg<D>::n + sizeof(SegMap) * 4 + 128 + moment_ws_bytes<D>();
    set_smem(k_rule_moments<D>, sm);
    ++*lc.launches;
    // one block per patch: the hardware hands the next patch to whichever block slot frees
    k_rule_moments<D><<<count, kThreads, sm, lc.stream>>>(plist, count, dv, modes, qv, qn, kp,
                                                          (cplx*)out_smooth, (cplx*)out_ann, form);
  }

template <int D>
void FarOrderL<D>::run(const LaunchCommon& lc, const int* plist, int count, const Dev& dv,
                  const KernelParams& kp, double eps, int m_max, double normV, const double* dirs,
                  int ndirs, void* scratch, int grid, int32_t* q, int32_t* qn, int* sched) {
    const size_t sm = moments_smem_bytes<D>(3 * kMaxTestPts + kThreads / 32 + 4);
    set_smem(k_farorder<D>, sm);
    ++*lc.launches;
    cudaMemsetAsync(sched, 0, sizeof(int), lc.stream);
    k_farorder<D><<<grid, kThreads, sm, lc.stream>>>(plist, count, dv, kp, eps, m_max, normV, dirs,
                                                     ndirs, (cplx*)scratch, q, qn, sched);
  }

template <int D>
int AdaptiveL<D>::blocks_per_sm() {
    int nb = 1;
    const size_t sm = adaptive_smem_bytes<D>();
    set_smem(k_adaptive<D>, sm);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_adaptive<D>, kThreads, sm);
    cudaGetLastError();
    return nb < 1 ? 1 : nb;
  }

template <int D>
void AdaptiveL<D>::run(const LaunchCommon& lc, const int* plist, int count, const Dev& dv,
                  const KernelParams& kp, double eps, double normV, int leaf_order, int max_depth,
                  const void* I_smooth, void* I_near, int32_t* leaves, void* work,
                  int64_t stride, int A_max, int levels, int grid, int* status, int* sched,
                  int form, const int64_t* gofs, int gsz) {
    const size_t sm = adaptive_smem_bytes<D>();
    set_smem(k_adaptive<D>, sm);
    AdaptiveWS w{stride, A_max, levels};
    ++*lc.launches;
    cudaMemsetAsync(sched, 0, sizeof(int), lc.stream);
    k_adaptive<D><<<grid, kThreads, sm, lc.stream>>>(plist, count, dv, kp, eps, normV, leaf_order,
                                                     max_depth, (const cplx*)I_smooth, (cplx*)I_near,
                                                     leaves, (unsigned char*)work, w, status, sched,
                                                     form, GradArgs{}, gofs, gsz);
  }

template <int D>
void SelfL<D>::run(const LaunchCommon& lc, const Dev& dv, const int32_t* deg, const KernelParams& kp,
                  int order, void* out) {
    // one block per self target: short-lived blocks, so that kernels on higher-priority
    // streams take the SMs they free first
    const int64_t g = dv.n_self < (int64_t)0x7fffffff ? dv.n_self : (int64_t)0x7fffffff;
    if (g <= 0) return;
    ++*lc.launches;
    set_smem(k_self<D>, SelfCfg<D>::BYTES);
    k_self<D><<<(int)g, kSelfThreads, SelfCfg<D>::BYTES, lc.stream>>>(dv, deg, kp, order, (cplx*)out);
  }

template <int D>
void TgtNormalsL<D>::run(const LaunchCommon& lc, const Dev& dv, const int32_t* deg, const double* user,
                  bool do_off, double* out) {
    const int64_t b = (dv.NT + 127) / 128;
    const int g = (int)(b < lc.num_sms * 8 ? (b > 0 ? b : 1) : lc.num_sms * 8);
    ++*lc.launches;
    k_tgt_normals<D><<<g, 128, 0, lc.stream>>>(dv, deg, user, do_off, out);
  }

template <int D>
void V2cL<D>::run(const LaunchCommon& lc, const int* plist, int count, const Dev& dv,
                  const double* Vt, const void* In, const void* Is, const void* InS,
                  double* val) {
    const int grid = count < lc.num_sms * 4 ? count : lc.num_sms * 4;
    ++*lc.launches;
    k_v2c<D><<<grid, kThreads, 0, lc.stream>>>(plist, count, dv, Vt, (const cplx*)In,
                                               (const cplx*)Is, (const cplx*)InS, val);
  }

template <int D>
void FarSrcL<D>::run(const LaunchCommon& lc, const int* plist, int count, const Dev& dv,
                  const double* Vt, const int32_t* qv, const int64_t* src_off, const void* sigma,
                  double* src, int64_t n_over, bool fx) {
    const int grid = count < lc.num_sms * 4 ? count : lc.num_sms * 4;
    ++*lc.launches;
    k_far_src<D><<<grid, 128, 0, lc.stream>>>(plist, count, dv, Vt, qv, src_off,
                                              (const cplx*)sigma, src, n_over, fx);
  }

template <int D>
cudaError_t upload_deg_constants(cudaStream_t st) {
  return upload_kw_tables(st);
}

}  // namespace lcq
