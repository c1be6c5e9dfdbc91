// CUDA kernels of the correction path (sm_103a), FP64 precision throughout (kernel values in
// 64-bit fixed point).
//
//   k_geom         chart coefficients, centroid, radius, d_j        (Sec. 3.2, Sec. 4)
//   (near lists: lcq_nearlist.cu)
//   k_farorder     far order q_j and annulus order                  (Sec. 4.2, Eq. qj)
//   k_rule_moments smooth-rule / annulus moments for many targets    (Sec. 4.2, Remark on eta_1)
//   k_adaptive     adaptive subdivision over a per-patch union tree  (Sec. 4.3)
//   k_self         singular self rules                              (Sec. 4, Eq. errestself)
//   k_v2c          a - s = V^T (I_near - I_smooth) into the CSR       (Sec. 4.3, 5.3)
//   k_far_src / k_far_sum / k_csr_apply   corrected potential      (Sec. 5.3)
//   (the degree-templated kernels are in lcq_kernels.cuh, one object per degree: lcq_deg.cu)
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "lcq_common.cuh"
#include "lcq_degree.h"

namespace lcq {

// ============================================================================ near lists
__global__ void k_tgt_patch(const double* __restrict__ tgt, const int64_t* __restrict__ tnode,
                            int64_t NT, const int64_t* __restrict__ node_off, int64_t P, int64_t N,
                            int32_t* __restrict__ tpatch, int32_t* __restrict__ tlnode,
                            int* __restrict__ status) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < NT;
       t += (int64_t)gridDim.x * blockDim.x) {
    for (int c = 0; c < 3; ++c)
      if (!isfinite(tgt[c * NT + t])) atomicOr(status, kStNonFinite);
    const int64_t nd = tnode[t];
    if (nd < 0 || nd >= N) {
      tpatch[t] = -1;
      tlnode[t] = -1;
      continue;
    }
    int64_t lo = 0, hi = P;  // largest j with node_off[j] <= nd
    while (hi - lo > 1) {
      const int64_t mid = (lo + hi) / 2;
      if (node_off[mid] <= nd) lo = mid; else hi = mid;
    }
    tpatch[t] = (int32_t)lo;
    tlnode[t] = (int32_t)(nd - node_off[lo]);
  }
}

// ============================================================================ scans
// Exclusive scan of int64 in blocks of 1024 (two passes + recursion on block sums).
__global__ void k_scan_block(const int64_t* __restrict__ in, int64_t* __restrict__ out, int64_t n,
                             int64_t* __restrict__ bsum) {
  __shared__ int64_t s[1024];
  const int64_t i = blockIdx.x * 1024ll + threadIdx.x;
  const int64_t x = i < n ? in[i] : 0;
  s[threadIdx.x] = x;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {
    const int64_t add = threadIdx.x >= o ? s[threadIdx.x - o] : 0;
    __syncthreads();
    s[threadIdx.x] += add;
    __syncthreads();
  }
  if (i < n) out[i] = s[threadIdx.x] - x;
  if (threadIdx.x == 1023) bsum[blockIdx.x] = s[1023];
}
// Second pass: adds the scanned block sums to each block's entries.
__global__ void k_scan_add(int64_t* __restrict__ out, int64_t n, const int64_t* __restrict__ boff) {
  const int64_t i = blockIdx.x * 1024ll + threadIdx.x;
  if (i < n) out[i] += boff[blockIdx.x];
}

// Direct far sum over the oversampled sources, one thread per target and range of sources
// (tiles staged through shared memory): block (b, s) sums part s of gridDim.y equal parts of
// the sources of target block b into part[s][t], and k_csr_apply adds the parts in a fixed order.  Few
// targets alone leave the chip idle (1000 targets are 8 blocks on 152 SMs), so the launch cuts
// the sources until there are several waves of blocks (far_sum_parts).
// The kernel values are fixed-point (fx_eval): of FP64 there are only the difference x - X and
// the four multiply-adds of the density (448 cycles of the FP64 pipe a pair and warp, beside
// about 440 integer instructions for the single layer, 720 for the CFIE).  35,840 targets x 127,606 sources, CFIE:
// 407 ms with FP64 kernel values (41 FP64 instructions a pair), 137 ms so; 8,960 x 25,920, S: 15.7
// and 4.6 ms.  More warps per SM (128, 96, 80, 64 registers) and two sources a step: within 3%.
// The sources of an on-surface target's own patch are skipped (their contribution is
// carried entirely by the self correction).  In a batch of independent surfaces a target
// sums only its own surface's sources [gsrc[g], gsrc[g+1]) with that surface's kernel.
constexpr int kFarThreads = 128;
__global__ void __launch_bounds__(kFarThreads) k_far_sum(const double* __restrict__ tgt, int64_t NT,
                                                      const double* __restrict__ src, int64_t n_over,
                                                      const KernelParams kp,
                                                      const int32_t* __restrict__ tpatch,
                                                      const int64_t* __restrict__ src_off,
                                                      const int32_t* __restrict__ tgroup,
                                                      const GroupParams* __restrict__ grp,
                                                      const int64_t* __restrict__ gsrc,
                                                      const double* __restrict__ tnrm,
                                                      cplx* __restrict__ part) {
  __shared__ ulonglong2 s[5][kFarThreads];  // X0 X1 | X2 n0 | n1 n2 | w ew | density
  __shared__ unsigned long long blo, bhi;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  double x0 = 0, x1 = 0, x2 = 0;
  int64_t skip0 = -1, skip1 = -1, lo = 0, hi = 0;
  FxS nx[3] = {{0, 0}, {0, 0}, {0, 0}};
  const KernelParams* kt = &kp;
  if (threadIdx.x == 0) {
    blo = ~0ull;
    bhi = 0ull;
  }
  __syncthreads();
  if (t < NT) {
    x0 = tgt[t];
    x1 = tgt[NT + t];
    x2 = tgt[2 * NT + t];
    if (tnrm) {  // S': the double-layer form with -n_x in the place of the source's normal
      for (int c = 0; c < 3; ++c) {
        const double n = tnrm[c * NT + t];
        nx[c] = fx_split(fx_fix(-n, 0));
        if (!isfinite(n)) x0 = n - n;  // a NaN, passed on by the differences
      }
    }
    const int tp = tpatch[t];
    if (tp >= 0) {
      skip0 = src_off[tp];
      skip1 = src_off[tp + 1];
    }
    hi = n_over;
    if (tgroup) {
      const int g = tgroup[t];
      kt = &grp[g].kp;
      lo = gsrc[g];
      hi = gsrc[g + 1];
    }
    atomicMin(&blo, (unsigned long long)lo);
    atomicMax(&bhi, (unsigned long long)hi);
  }
  __syncthreads();
  const int64_t all = (int64_t)bhi - (int64_t)blo;
  const int64_t b0 = (int64_t)blo + all * blockIdx.y / gridDim.y;
  const int64_t b1 = (int64_t)blo + all * (blockIdx.y + 1) / gridDim.y;
  const FxKernel kf = kt->fx;
  const FxTables tab = fx_tables();
  double re = 0.0, im = 0.0;
  for (int64_t s0 = b0; s0 < b1; s0 += kFarThreads) {
    __syncthreads();
    const int64_t q = s0 + threadIdx.x;
    if (q < b1) {
      auto row = [&](int c) { return (u64)__double_as_longlong(src[c * n_over + q]); };
      s[0][threadIdx.x] = make_ulonglong2(row(0), row(1));
      s[1][threadIdx.x] = make_ulonglong2(row(2), row(3));
      s[2][threadIdx.x] = make_ulonglong2(row(4), row(5));
      s[3][threadIdx.x] = make_ulonglong2(row(6), row(9));
      s[4][threadIdx.x] = make_ulonglong2(row(7), row(8));
    }
    __syncthreads();
    const int cnt = (int)min((int64_t)kFarThreads, b1 - s0);
    // this target's sources of the tile: [ka, kb) without [kc, kd)
    const int ka = (int)max(min(lo - s0, (int64_t)cnt), (int64_t)0), kb = (int)min(hi - s0, (int64_t)cnt);
    const int kc = (int)max(min(skip0 - s0, (int64_t)cnt), (int64_t)0);
    const int kd = (int)max(min(skip1 - s0, (int64_t)cnt), (int64_t)0);
    for (int k = 0; k < cnt; ++k) {
      if (k < ka || k >= kb || (k >= kc && k < kd)) continue;
      const ulonglong2 a = s[0][k], b = s[1][k], c = s[2][k], d = s[3][k];
      FxS n[3] = {fx_unjoin(b.y), fx_unjoin(c.x), fx_unjoin(c.y)};
      if (tnrm) {
        n[0] = nx[0];
        n[1] = nx[1];
        n[2] = nx[2];
      }
      const double d0 = x0 - fx_double(a.x), d1 = x1 - fx_double(a.y), d2 = x2 - fx_double(b.x);
      cplx g;
      if (!fx_eval<true>(kf, tab, d0, d1, d2, n, d.x, (int)d.y, &g.re, &g.im, nullptr, 0.0f, 0.0f,
                         0.0f, 0.0f, 0.0f, &kt->fx))
        g = fx_fallback(*kt, d0, d1, d2, n[0], n[1], n[2], d.x, (int)d.y, 0.0, nullptr);
      const double sr = fx_double(s[4][k].x), si = fx_double(s[4][k].y);
      re = fma(g.re, sr, re);
      re = fma(-g.im, si, re);
      im = fma(g.re, si, im);
      im = fma(g.im, sr, im);
    }
  }
  if (t < NT) part[blockIdx.y * NT + t] = {re, im};
}

// The correction part of the corrected potential (Sec. 5.3): warp per target row,
// out_t = the far sum's parts + sum_row c sigma, plus jump * sigma at an on-surface target's own node.
__global__ void k_csr_apply(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                            const double* __restrict__ val, const cplx* __restrict__ sigma,
                            const int64_t* __restrict__ tnode, int64_t NT, double jump,
                            const cplx* __restrict__ part, int parts, cplx* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t t = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); t < NT; t += warps) {
    double re = 0.0, im = 0.0;
    for (int k = lane; k < parts; k += 32) {
      const cplx p = part[k * NT + t];
      re += p.re;
      im += p.im;
    }
    for (int64_t e = row_ptr[t] + lane; e < row_ptr[t + 1]; e += 32) {
      const double vr = val[2 * e], vi = val[2 * e + 1];
      const cplx sg = sigma[col[e]];
      re += vr * sg.re - vi * sg.im;
      im += vr * sg.im + vi * sg.re;
    }
    re = warp_sum(re);
    im = warp_sum(im);
    if (lane == 0) {
      cplx o = {re, im};
      if (jump != 0.0 && tnode[t] >= 0) {
        o.re += jump * sigma[tnode[t]].re;
        o.im += jump * sigma[tnode[t]].im;
      }
      out[t] = o;
    }
  }
}

// complex64 density -> complex128 (apply of a density stored in single precision)
__global__ void k_widen_c64(const float2* __restrict__ in, int64_t n, cplx* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float2 v = in[i];
    out[i] = {(double)v.x, (double)v.y};
  }
}

// ============================================================================ launchers
namespace {
template <template <int> class F, class... Args>
bool dispatch(int d, Args&&... args) {
  switch (d) {
    case 1: F<1>::run(args...); return true;
    case 2: F<2>::run(args...); return true;
    case 3: F<3>::run(args...); return true;
    case 4: F<4>::run(args...); return true;
    case 5: F<5>::run(args...); return true;
    case 6: F<6>::run(args...); return true;
    case 7: F<7>::run(args...); return true;
    case 8: F<8>::run(args...); return true;
    case 9: F<9>::run(args...); return true;
    case 10: F<10>::run(args...); return true;
    default: return false;
  }
}

template <int D>
struct UploadL {
  static void run(cudaStream_t st, cudaError_t* e) {
    if (*e == cudaSuccess) *e = upload_deg_constants<D>(st);
  }
};
template <int D>
struct BlocksL {
  static void run(int* nb) { *nb = AdaptiveL<D>::blocks_per_sm(); }
};
}  // namespace

cudaError_t upload_constants(cudaStream_t st) {
  cudaError_t e = upload_kw_tables(st);
  for (int d = 1; d <= kMaxDeg && e == cudaSuccess; ++d) dispatch<UploadL>(d, st, &e);
  if (e != cudaSuccess) return e;
  return cudaStreamSynchronize(st);
}

bool launch_geom(int d, const LaunchCommon& lc, const int* plist, int count, const int64_t* node_off,
                 const double* xyz, int64_t N, const double* Vt, const double* nodes, double eta_p,
                 double eta1_p, double* coef, double* cen, double* rad, double* dj, double* eta,
                 double* eta1, int* status) {
  return dispatch<GeomL>(d, lc, plist, count, node_off, xyz, N, Vt, nodes, eta_p, eta1_p, coef, cen,
                         rad, dj, eta, eta1, status);
}

void launch_tgt_patch(const LaunchCommon& lc, const double* tgt, const int64_t* tnode, int64_t NT,
                      const int64_t* node_off, int64_t P, int64_t N, int32_t* tpatch,
                      int32_t* tlnode, int* status) {
  const int64_t blocks = (NT + 255) / 256;
  const int g = (int)(blocks < lc.num_sms * 16 ? (blocks > 0 ? blocks : 1) : lc.num_sms * 16);
  ++*lc.launches;
  k_tgt_patch<<<g, 256, 0, lc.stream>>>(tgt, tnode, NT, node_off, P, N, tpatch, tlnode, status);
}

// On-surface targets follow their nodes (a captured regeneration after the nodes moved):
// tgt[:, t] = xyz[:, tnode[t]] where 0 <= tnode[t] < N; off-surface targets are kept.
__global__ void k_tgt_from_nodes(double* __restrict__ tgt, const int64_t* __restrict__ tnode,
                                 int64_t NT, const double* __restrict__ xyz, int64_t N) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < NT;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t nd = tnode[t];
    if (nd < 0 || nd >= N) continue;
    for (int c = 0; c < 3; ++c) tgt[c * NT + t] = xyz[c * N + nd];
  }
}
void launch_tgt_from_nodes(const LaunchCommon& lc, double* tgt, const int64_t* tnode, int64_t NT,
                           const double* xyz, int64_t N) {
  if (NT <= 0) return;
  const int64_t blocks = (NT + 255) / 256;
  const int g = (int)(blocks < lc.num_sms * 16 ? blocks : lc.num_sms * 16);
  ++*lc.launches;
  k_tgt_from_nodes<<<g, 256, 0, lc.stream>>>(tgt, tnode, NT, xyz, N);
}

// out[i] = sum_{k<i} in[i]; needs scratch of >= 2 * ceil(n/1024) + 2048 int64 elements.
void launch_scan(const LaunchCommon& lc, const int64_t* in, int64_t* out, int64_t n,
                 int64_t* scratch) {
  if (n <= 0) return;
  const int64_t nb = (n + 1023) / 1024;
  ++*lc.launches;
  k_scan_block<<<(unsigned)nb, 1024, 0, lc.stream>>>(in, out, n, scratch);
  if (nb > 1) {
    launch_scan(lc, scratch, scratch + nb, nb, scratch + 2 * nb);
    ++*lc.launches;
    k_scan_add<<<(unsigned)nb, 1024, 0, lc.stream>>>(out, n, scratch + nb);
  }
}

bool launch_rule_moments(int d, const LaunchCommon& lc, const int* plist, int count, const Dev& dv,
                         int modes, const int32_t* qv, const int32_t* qn, const KernelParams& kp,
                         void* out_smooth, void* out_ann, int form) {
  return dispatch<RuleMomL>(d, lc, plist, count, dv, modes, qv, qn, kp, out_smooth, out_ann,
                            form);
}
bool launch_farorder(int d, const LaunchCommon& lc, const int* plist, int count, const Dev& dv,
                     const KernelParams& kp, double eps, int m_max, double normV, const double* dirs,
                     int ndirs, void* scratch, int grid, int32_t* q, int32_t* qn, int* sched) {
  return dispatch<FarOrderL>(d, lc, plist, count, dv, kp, eps, m_max, normV, dirs, ndirs, scratch,
                             grid, q, qn, sched);
}
bool launch_adaptive(int d, const LaunchCommon& lc, const int* plist, int count, const Dev& dv,
                     const KernelParams& kp, double eps, double normV, int leaf_order, int max_depth,
                     const void* I_smooth, void* I_near, int32_t* leaves, void* work, int64_t stride,
                     int A_max, int levels, int grid, int* status, int* sched, int form,
                     const int64_t* gofs, int gsz) {
  return dispatch<AdaptiveL>(d, lc, plist, count, dv, kp, eps, normV, leaf_order, max_depth,
                             I_smooth, I_near, leaves, work, stride, A_max, levels, grid, status,
                             sched, form, gofs, gsz);
}

// Groups of at most gsz adaptive targets per listed patch: ng[b] = ceil(A_b / gsz) for
// b < count and ng[count] = 0, so that the exclusive scan of the count + 1 entries (gofs)
// ends with the number of groups.
__global__ void k_group_counts(const int* __restrict__ plist, int count,
                               const int64_t* __restrict__ ad_ptr, int gsz, int64_t* __restrict__ ng) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b <= count; b += gridDim.x * blockDim.x) {
    int64_t g = 0;
    if (b < count) {
      const int j = plist[b];
      g = (ad_ptr[j + 1] - ad_ptr[j] + gsz - 1) / gsz;
    }
    ng[b] = g;
  }
}

void launch_group_offsets(const LaunchCommon& lc, const int* plist, int count, const int64_t* ad_ptr,
                          int gsz, int64_t* ng, int64_t* gofs, int64_t* scratch) {
  const int blocks = (count + 1 + 255) / 256;
  ++*lc.launches;
  k_group_counts<<<blocks < lc.num_sms * 4 ? blocks : lc.num_sms * 4, 256, 0, lc.stream>>>(
      plist, count, ad_ptr, gsz, ng);
  launch_scan(lc, ng, gofs, count + 1, scratch);
}
bool launch_self(int d, const LaunchCommon& lc, const Dev& dv, const int32_t* deg,
                 const KernelParams& kp, int order, void* out) {
  return dispatch<SelfL>(d, lc, dv, deg, kp, order, out);
}
bool launch_tgt_normals(int d, const LaunchCommon& lc, const Dev& dv, const int32_t* deg,
                        const double* user, bool do_off, double* out) {
  return dispatch<TgtNormalsL>(d, lc, dv, deg, user, do_off, out);
}
bool launch_v2c(int d, const LaunchCommon& lc, const int* plist, int count, const Dev& dv,
                const double* Vt, const void* In, const void* Is, const void* InS,
                double* val) {
  return dispatch<V2cL>(d, lc, plist, count, dv, Vt, In, Is, InS, val);
}
bool launch_far_src(int d, const LaunchCommon& lc, const int* plist, int count, const Dev& dv,
                    const double* Vt, const int32_t* qv, const int64_t* src_off, const void* sigma,
                    double* src, int64_t n_over, bool fx) {
  return dispatch<FarSrcL>(d, lc, plist, count, dv, Vt, qv, src_off, sigma, src, n_over, fx);
}
// Parts that the far sum's sources are cut into: enough blocks for about four waves of eight
// on every SM, at least 32 sources each.
int far_sum_parts(int num_sms, int64_t NT, int64_t n_over) {
  const int64_t tb = (NT + kFarThreads - 1) / kFarThreads;
  if (tb <= 0) return 1;
  const int64_t want = (32ll * num_sms + tb - 1) / tb, most = n_over / 32;
  const int64_t s = want < most ? want : most;
  return (int)(s < 1 ? 1 : s);
}
void launch_far_sum(const LaunchCommon& lc, const double* tgt, int64_t NT, const double* src,
                    int64_t n_over, const KernelParams& kp, const int32_t* tpatch,
                    const int64_t* src_off, const int32_t* tgroup, const GroupParams* grp,
                    const int64_t* gsrc, const double* tnrm, void* part, int parts) {
  const int64_t g = (NT + kFarThreads - 1) / kFarThreads;
  if (g <= 0) return;
  ++*lc.launches;
  k_far_sum<<<dim3((unsigned)g, (unsigned)parts), kFarThreads, 0, lc.stream>>>(
      tgt, NT, src, n_over, kp, tpatch, src_off, tgroup, grp, gsrc, tnrm, (cplx*)part);
}
void launch_widen_c64(const LaunchCommon& lc, const void* in, int64_t n, void* out) {
  if (n <= 0) return;
  const int64_t b = (n + 255) / 256;
  ++*lc.launches;
  k_widen_c64<<<(unsigned)(b < lc.num_sms * 8 ? b : lc.num_sms * 8), 256, 0, lc.stream>>>(
      (const float2*)in, n, (cplx*)out);
}
void launch_csr_apply(const LaunchCommon& lc, const int64_t* row_ptr, const int32_t* col,
                      const double* val, const void* sigma, const int64_t* tnode, int64_t NT,
                      double jump, const void* part, int parts, void* out) {
  const int g = lc.num_sms * 8;
  ++*lc.launches;
  k_csr_apply<<<g, 256, 0, lc.stream>>>(row_ptr, col, val, (const cplx*)sigma, tnode, NT, jump,
                                        (const cplx*)part, parts, (cplx*)out);
}

// Resident blocks per SM of k_adaptive<d> (the persistent grid is this times the SM count).
int adaptive_blocks_per_sm(int d) {
  int nb = 1;
  dispatch<BlocksL>(d, &nb);
  return nb;
}

}  // namespace lcq
