// Kernels and launchers instantiated once per precision by vlb_f32.cu / vlb_f64.cu.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>
#include "vlb_launch.h"
#include "vlb_stage.cuh"
#include "vlb_channel.cuh"

namespace vlb {

// ---------------------------------------------------------------- stage dispatch
// Launch shapes ("variants") of the stage kernel: cells per tile TC and threads
// per CTA NT.  Exact instantiations exist for the node counts of the
// configured models; anything else takes the generic kernel.  The autotuner
// (vlb_autotune) times the variants of a context's shape and keeps the best.
// Tile buffers and resident CTAs per SM of a launch shape: one buffer for a launch
// with one CTA per tile; a persistent launch takes two (staging its next tile while
// it computes one) when that leaves as many CTAs resident as one buffer does.
template <typename real, int TC, int NT, int Q0, int Q1, bool EXACT, bool FT = false>
static cudaError_t stage_buffers(int Vp, int persist, int* nbuf, int* per_sm) {
  using L = StageSmem<real, TC, NT>;
  auto kern = couette_stage_kernel<real, TC, Q0, Q1, NT, EXACT, FT>;
  const size_t limit = 227 * 1024;
  const int top = persist && L::bytes(Vp, 2) <= limit ? 2 : 1;
  // the kernel's shared-memory limit is process-wide and shared by contexts of other row
  // lengths (the generic kernels), so it is only ever raised
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, kern);
  if (e != cudaSuccess) return e;
  if (size_t(fa.maxDynamicSharedSizeBytes) < L::bytes(Vp, top)) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(L::bytes(Vp, top)));
    if (e != cudaSuccess) return e;
  }
  *nbuf = 1, *per_sm = 0;
  for (int nb = 1; nb <= top; ++nb) {
    int occ = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, NT, L::bytes(Vp, nb))) != cudaSuccess) return e;
    if (nb == 1 || (occ > 0 && occ >= *per_sm)) *nbuf = nb, *per_sm = occ;
  }
  return cudaSuccess;
}

template <typename real, int TC, int NT, int Q0, int Q1, bool EXACT, bool FT = false>
static cudaError_t go_stage(const StageArgs<real>& a, const ModelArgs& m, const KArgs<real>& k, int grid,
                            cudaStream_t s) {
  return launch_dependent(couette_stage_kernel<real, TC, Q0, Q1, NT, EXACT, FT>, dim3(grid), NT,
                          StageSmem<real, TC, NT>::bytes(a.Vp, a.nbuf), s, a, m, k);
}

enum Shape { SH_16x20 = 0, SH_16x12 = 1, SH_8x4 = 2, SH_SMALL = 3, SH_GENERIC = 4 };

static int shape_of(int nq0, int nq1) {
  if (nq0 == 16 && nq1 == 20) return SH_16x20;
  if (nq0 == 16 && nq1 == 12) return SH_16x12;
  if (nq0 == 8 && nq1 == 4) return SH_8x4;
  if (nq0 * nq1 <= 64) return SH_SMALL;
  return SH_GENERIC;
}

// variant tables per precision and shape: {TC, NT}
template <typename real>
struct VariantTable;
template <>
struct VariantTable<float> {
  // (the first is the default: a thread per velocity and two CTAs of ten cells a SM; with 256 threads
  // a second pass over 64 of the 320 velocities leaves most of them idle)
  static constexpr StageVariant v16x20[] = {{10, 320, 0}, {8, 256, 0},  {4, 320, 0}, {8, 320, 0},
                                            {16, 320, 0}, {4, 256, 0}, {9, 320, 0}};
  static constexpr StageVariant v16x12[] = {{16, 256, 0}, {8, 256, 0}, {16, 384, 0}};
  static constexpr StageVariant v8x4[] = {{16, 64, 0}, {8, 64, 0}};
  static constexpr StageVariant vsmall[] = {{16, 64, 0}};
  static constexpr StageVariant vgen[] = {{16, 256, 0}};
};
template <>
struct VariantTable<double> {
  static constexpr StageVariant v16x20[] = {{4, 256, 0}, {8, 256, 0}, {4, 128, 0}, {8, 128, 0}};
  static constexpr StageVariant v16x12[] = {{8, 256, 0}, {4, 256, 0}, {8, 384, 0}};
  static constexpr StageVariant v8x4[] = {{8, 64, 0}, {16, 64, 0}};
  static constexpr StageVariant vsmall[] = {{8, 64, 0}};
  static constexpr StageVariant vgen[] = {{8, 256, 0}};
};

template <typename real>
int stage_variants(int nq0, int nq1, StageVariant* out) {
  using T = VariantTable<real>;
  const StageVariant* v;
  int n;
  switch (shape_of(nq0, nq1)) {
    case SH_16x20: v = T::v16x20, n = int(sizeof(T::v16x20) / sizeof(StageVariant)); break;
    case SH_16x12: v = T::v16x12, n = int(sizeof(T::v16x12) / sizeof(StageVariant)); break;
    case SH_8x4: v = T::v8x4, n = int(sizeof(T::v8x4) / sizeof(StageVariant)); break;
    case SH_SMALL: v = T::vsmall, n = 1; break;
    default: v = T::vgen, n = 1; break;
  }
  for (int i = 0; i < n; ++i) out[i] = v[i];
  return n;
}

template <typename real>
bool stage_split_tables(int nq0, int nq1) {
  const int sh = shape_of(nq0, nq1);
  return sh == SH_16x20 || sh == SH_16x12 || sh == SH_8x4;
}

template <typename real>
size_t stage_smem_bytes(StageVariant v, int Vp) {
#define VLB_SMEM_CASE(TC_, NT_) \
  if (v.tc == TC_ && v.nt == NT_) return StageSmem<real, TC_, NT_>::bytes(Vp, 1);
  VLB_SMEM_CASE(16, 256) VLB_SMEM_CASE(8, 256) VLB_SMEM_CASE(16, 512) VLB_SMEM_CASE(8, 128)
  VLB_SMEM_CASE(16, 384) VLB_SMEM_CASE(16, 64) VLB_SMEM_CASE(8, 64) VLB_SMEM_CASE(4, 256)
  VLB_SMEM_CASE(4, 128) VLB_SMEM_CASE(8, 384) VLB_SMEM_CASE(4, 320) VLB_SMEM_CASE(8, 320)
  VLB_SMEM_CASE(16, 320) VLB_SMEM_CASE(10, 320) VLB_SMEM_CASE(9, 320)
#undef VLB_SMEM_CASE
  return 0;
}

template <typename real>
cudaError_t launch_stage(StageVariant v, const StageArgs<real>& a, const ModelArgs& m, const KArgs<real>& k, int grid,
                         cudaStream_t s, bool ft) {
  const int sh = shape_of(m.nq0, m.nq1);
  if (ft) {  // the f~ kernels: the first launch shape of each shape's table
#define VLB_FT(SH, TC_, NT_, q0, q1, ex) \
  if (sh == SH && v.tc == TC_ && v.nt == NT_) return go_stage<real, TC_, NT_, q0, q1, ex, true>(a, m, k, grid, s);
    if constexpr (sizeof(real) == 4) {
      VLB_FT(SH_16x20, 10, 320, 16, 20, true) VLB_FT(SH_16x12, 16, 256, 16, 12, true)
      VLB_FT(SH_8x4, 16, 64, 8, 4, true) VLB_FT(SH_SMALL, 16, 64, MAXQ, MAXQ, false)
      VLB_FT(SH_GENERIC, 16, 256, MAXQ, MAXQ, false)
    } else {
      VLB_FT(SH_16x20, 4, 256, 16, 20, true) VLB_FT(SH_16x12, 8, 256, 16, 12, true)
      VLB_FT(SH_8x4, 8, 64, 8, 4, true) VLB_FT(SH_SMALL, 8, 64, MAXQ, MAXQ, false)
      VLB_FT(SH_GENERIC, 8, 256, MAXQ, MAXQ, false)
    }
#undef VLB_FT
    return cudaErrorInvalidValue;
  }
#define VLB_CASE(SH, TC_, NT_, q0, q1, ex) \
  if (sh == SH && v.tc == TC_ && v.nt == NT_) return go_stage<real, TC_, NT_, q0, q1, ex>(a, m, k, grid, s);
  if constexpr (sizeof(real) == 4) {
    VLB_CASE(SH_16x20, 4, 256, 16, 20, true) VLB_CASE(SH_16x20, 8, 256, 16, 20, true)
    VLB_CASE(SH_16x20, 4, 320, 16, 20, true) VLB_CASE(SH_16x20, 8, 320, 16, 20, true)
    VLB_CASE(SH_16x20, 16, 320, 16, 20, true) VLB_CASE(SH_16x20, 10, 320, 16, 20, true)
    VLB_CASE(SH_16x20, 9, 320, 16, 20, true)
    VLB_CASE(SH_16x12, 16, 256, 16, 12, true) VLB_CASE(SH_16x12, 8, 256, 16, 12, true)
    VLB_CASE(SH_16x12, 16, 384, 16, 12, true)
    VLB_CASE(SH_8x4, 16, 64, 8, 4, true) VLB_CASE(SH_8x4, 8, 64, 8, 4, true)
    VLB_CASE(SH_SMALL, 16, 64, MAXQ, MAXQ, false)
    VLB_CASE(SH_GENERIC, 16, 256, MAXQ, MAXQ, false)
  } else {
    VLB_CASE(SH_16x20, 4, 256, 16, 20, true) VLB_CASE(SH_16x20, 8, 256, 16, 20, true)
    VLB_CASE(SH_16x20, 4, 128, 16, 20, true) VLB_CASE(SH_16x20, 8, 128, 16, 20, true)
    VLB_CASE(SH_16x12, 8, 256, 16, 12, true) VLB_CASE(SH_16x12, 4, 256, 16, 12, true)
    VLB_CASE(SH_16x12, 8, 384, 16, 12, true)
    VLB_CASE(SH_8x4, 8, 64, 8, 4, true) VLB_CASE(SH_8x4, 16, 64, 8, 4, true)
    VLB_CASE(SH_SMALL, 8, 64, MAXQ, MAXQ, false)
    VLB_CASE(SH_GENERIC, 8, 256, MAXQ, MAXQ, false)
  }
#undef VLB_CASE
  return cudaErrorInvalidValue;
}

template <typename real>
cudaError_t stage_config(StageVariant v, const ModelArgs& m, int Vp, int* nbuf, int* per_sm, bool ft) {
  const int sh = shape_of(m.nq0, m.nq1);
  if (ft) {
#define VLB_FT(SH, TC_, NT_, q0, q1, ex) \
  if (sh == SH && v.tc == TC_ && v.nt == NT_) return stage_buffers<real, TC_, NT_, q0, q1, ex, true>(Vp, v.persist, nbuf, per_sm);
    if constexpr (sizeof(real) == 4) {
      VLB_FT(SH_16x20, 10, 320, 16, 20, true) VLB_FT(SH_16x12, 16, 256, 16, 12, true)
      VLB_FT(SH_8x4, 16, 64, 8, 4, true) VLB_FT(SH_SMALL, 16, 64, MAXQ, MAXQ, false)
      VLB_FT(SH_GENERIC, 16, 256, MAXQ, MAXQ, false)
    } else {
      VLB_FT(SH_16x20, 4, 256, 16, 20, true) VLB_FT(SH_16x12, 8, 256, 16, 12, true)
      VLB_FT(SH_8x4, 8, 64, 8, 4, true) VLB_FT(SH_SMALL, 8, 64, MAXQ, MAXQ, false)
      VLB_FT(SH_GENERIC, 8, 256, MAXQ, MAXQ, false)
    }
#undef VLB_FT
    return cudaErrorInvalidValue;
  }
#define VLB_CASE(SH, TC_, NT_, q0, q1, ex) \
  if (sh == SH && v.tc == TC_ && v.nt == NT_)      \
    return stage_buffers<real, TC_, NT_, q0, q1, ex>(Vp, v.persist, nbuf, per_sm);
  if constexpr (sizeof(real) == 4) {
    VLB_CASE(SH_16x20, 4, 256, 16, 20, true) VLB_CASE(SH_16x20, 8, 256, 16, 20, true)
    VLB_CASE(SH_16x20, 4, 320, 16, 20, true) VLB_CASE(SH_16x20, 8, 320, 16, 20, true)
    VLB_CASE(SH_16x20, 16, 320, 16, 20, true) VLB_CASE(SH_16x20, 10, 320, 16, 20, true)
    VLB_CASE(SH_16x20, 9, 320, 16, 20, true)
    VLB_CASE(SH_16x12, 16, 256, 16, 12, true) VLB_CASE(SH_16x12, 8, 256, 16, 12, true)
    VLB_CASE(SH_16x12, 16, 384, 16, 12, true)
    VLB_CASE(SH_8x4, 16, 64, 8, 4, true) VLB_CASE(SH_8x4, 8, 64, 8, 4, true)
    VLB_CASE(SH_SMALL, 16, 64, MAXQ, MAXQ, false)
    VLB_CASE(SH_GENERIC, 16, 256, MAXQ, MAXQ, false)
  } else {
    VLB_CASE(SH_16x20, 4, 256, 16, 20, true) VLB_CASE(SH_16x20, 8, 256, 16, 20, true)
    VLB_CASE(SH_16x20, 4, 128, 16, 20, true) VLB_CASE(SH_16x20, 8, 128, 16, 20, true)
    VLB_CASE(SH_16x12, 8, 256, 16, 12, true) VLB_CASE(SH_16x12, 4, 256, 16, 12, true)
    VLB_CASE(SH_16x12, 8, 384, 16, 12, true)
    VLB_CASE(SH_8x4, 8, 64, 8, 4, true) VLB_CASE(SH_8x4, 16, 64, 8, 4, true)
    VLB_CASE(SH_SMALL, 8, 64, MAXQ, MAXQ, false)
    VLB_CASE(SH_GENERIC, 8, 256, MAXQ, MAXQ, false)
  }
#undef VLB_CASE
  *nbuf = 1, *per_sm = 0;
  return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------- channel dispatch
template <typename real, int Q0, int Q1, int CG, int XW, bool CLB, bool HX>
static cudaError_t go_channel(const ChanArgs<real>& a, const void* kpb, int grid, cudaStream_t s) {
  using L = ChanSmem<real, Q0, Q1, CG, XW>;
  auto kern = channel_stage_kernel<real, Q0, Q1, CG, XW, CLB, HX>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(L::bytes));
  if (e != cudaSuccess) return e;
  ChanKP<real, Q0, Q1> kp;
  memcpy(&kp, kpb, sizeof(kp));
  return launch_dependent(kern, dim3(grid), L::NT, L::bytes, s, a, kp);
}

#ifdef VLB_DEFINE_SHARED
// {rows per segment (0: host's choice, 1 << 20: one segment), columns per strip, threads}
static const ChanVariant kChan16x12[] = {{0, 4, 192}, {128, 4, 192}, {1 << 20, 4, 192}, {64, 4, 192}};
static const ChanVariant kChan8x4[] = {{0, 4, 32}, {64, 4, 32}, {16, 4, 32}, {1 << 20, 4, 32}};

int channel_variants(int nq0, int nq1, ChanVariant* out) {
  const ChanVariant* v = nullptr;
  int n = 0;
  if (nq0 == 16 && nq1 == 12) v = kChan16x12, n = int(sizeof(kChan16x12) / sizeof(ChanVariant));
  if (nq0 == 8 && nq1 == 4) v = kChan8x4, n = int(sizeof(kChan8x4) / sizeof(ChanVariant));
  for (int i = 0; i < n; ++i) out[i] = v[i];
  return n;
}
#endif

static inline void put_coef(float2& c, double x) { c.x = c.y = float(x); }
static inline void put_coef(double& c, double x) { c = x; }

// One axis of the ChanKP block: the split of K and Kt = K diag(p) + z v^T.  False if a matrix
// lacks the reflection symmetry or the rank-1 form the kernel relies on.
template <typename C>
static bool fill_force_axis(const AxisTables& t, C* P, C* M, C* p, C* v, C* z) {
  const int nq = t.nq, H = nq / 2;
  double kmax = 0.0, tmax = 0.0, pmax = 0.0;
  for (int k = 0; k < nq * nq; ++k) kmax = std::max(kmax, std::fabs(t.K[k])), tmax = std::max(tmax, std::fabs(t.Kt[k]));
  for (int k = 0; k < nq; ++k) pmax = std::max(pmax, std::fabs(t.p[k]));
  for (int r = 0; r < nq; ++r) {
    const int rr = refl(t.kind, nq, r);
    if (std::fabs(t.p[rr] + t.p[r]) > 1e-13 * pmax) return false;
    for (int q = 0; q < nq; ++q) {
      const int qq = refl(t.kind, nq, q);
      if (std::fabs(t.K[rr * nq + qq] + t.K[r * nq + q]) > 1e-12 * kmax) return false;
      if (std::fabs(t.Kt[rr * nq + qq] - t.Kt[r * nq + q]) > 1e-12 * tmax) return false;
    }
  }
  // E = Kt - K diag(p) = z v^T from its largest entry, in the symmetric scaling sqrt(w_q / w_r) E
  // whose entries are of one size; the residual has to vanish to rounding
  std::vector<double> E(nq * nq);
  double emax = 0.0, scale = 0.0;
  int rm = 0, qm = 0;
  for (int r = 0; r < nq; ++r)
    for (int q = 0; q < nq; ++q) {
      const double s = std::sqrt(t.w[q] / t.w[r]);
      E[r * nq + q] = s * (t.Kt[r * nq + q] - t.K[r * nq + q] * t.p[q]);
      scale = std::max(scale, s * std::fabs(t.Kt[r * nq + q]));
      if (std::fabs(E[r * nq + q]) > emax) emax = std::fabs(E[r * nq + q]), rm = r, qm = q;
    }
  std::vector<double> zz(nq, 0.0), vv(nq, 0.0);
  if (emax > 1e-11 * scale)
    for (int k = 0; k < nq; ++k) zz[k] = E[k * nq + qm] / E[rm * nq + qm], vv[k] = E[rm * nq + k];
  else if (t.kind == 1) return false;
  for (int r = 0; r < nq; ++r) {
    const int rr = refl(t.kind, nq, r);
    if (std::fabs(zz[rr] + zz[r]) > 1e-11 || std::fabs(vv[rr] + vv[r]) > 1e-11 * scale) return false;
    for (int q = 0; q < nq; ++q)
      if (std::fabs(E[r * nq + q] - zz[r] * vv[q]) > 1e-11 * scale) return false;
  }
  for (int r = 0; r < H; ++r) {
    put_coef(p[r], t.p[r]);
    put_coef(z[r], zz[r] * std::sqrt(t.w[r]));
    put_coef(v[r], vv[r] / std::sqrt(t.w[r]));
    for (int q = 0; q < H; ++q) {
      const double x = t.K[r * nq + q], y = t.K[r * nq + refl(t.kind, nq, q)];
      put_coef(P[r * H + q], 0.5 * (x + y));
      put_coef(M[r * H + q], 0.5 * (x - y));
    }
  }
  return true;
}
template <typename real, int Q0, int Q1>
static bool fill_force_block(const AxisTables* ax, std::vector<unsigned char>* out) {
  using KP = ChanKP<real, Q0, Q1>;
  out->assign(sizeof(KP), 0);
  KP& kp = *reinterpret_cast<KP*>(out->data());
  return ax[0].kind == 1 && fill_force_axis(ax[0], kp.P0, kp.M0, kp.p0, kp.v0, kp.z0) &&
         fill_force_axis(ax[1], kp.P1, kp.M1, kp.p1, kp.v1, kp.z1);
}

template <typename real>
bool channel_force_pairs(int nq0, int nq1, const AxisTables* ax, std::vector<unsigned char>* out) {
  if (nq0 == 16 && nq1 == 12) return fill_force_block<real, 16, 12>(ax, out);
  if (nq0 == 8 && nq1 == 4) return fill_force_block<real, 8, 4>(ax, out);
  return false;
}

template <typename real, int Q0, int Q1, int CG, int XW>
static cudaError_t channel_residency(int kind1, bool clb, int* per_sm) {
  using L = ChanSmem<real, Q0, Q1, CG, XW>;
  auto kern = clb ? channel_stage_kernel<real, Q0, Q1, CG, XW, true, false>
                  : kind1 == 1 ? channel_stage_kernel<real, Q0, Q1, CG, XW, false, true>
                               : channel_stage_kernel<real, Q0, Q1, CG, XW, false, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(L::bytes));
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kern, L::NT, L::bytes);
  return e;
}

// A march step of the one-warp kernel of the 8 x 4 set takes about 1.1 (single precision) and 1.8 (double)
// times that of the kernel with a warp per column, with the CTAs that are resident on a busy SM; times of
// an RK3 step, warp per column / one warp.  Single precision: 16 x 128 cells 39.8 / 52.7 us, 64 x 64 44.7 /
// 52.9, 16 x 604 55.1 / 57.3, 30 x 200 51.7 / 47.5, 16 x 612 71 / 58, 64 x 512 162 / 119.  Double precision:
// 16 x 128 268 / 633, 64 x 64 462 / 652, 30 x 200 559 / 545, 16 x 604 848 / 699, 64 x 512 3171 / 2467.
template <typename real>
cudaError_t channel_kernels(int nq0, int nq1, int kind1, bool clb, ChanKernel* out, int* n) {
  cudaError_t e = cudaSuccess;
  *n = 0;
  if (nq0 == 16 && nq1 == 12) {
    *n = 1;
    out[0].step = 10;
    e = channel_residency<real, 16, 12, 1, 0>(kind1, clb, &out[0].per_sm);
  } else if (nq0 == 8 && nq1 == 4) {
    *n = 2;
    out[0].step = sizeof(real) == 8 ? 18 : 11;
    out[1].step = 10;
    e = channel_residency<real, 8, 4, 1, 0>(kind1, clb, &out[0].per_sm);
    if (e == cudaSuccess) e = channel_residency<real, 8, 4, 4, 3>(kind1, clb, &out[1].per_sm);
  }
  return e;
}

// Axis moment vector of the truncated equilibrium at rest (u = 0), in double.
static void rest_moment_vector(int kind, int N, double T, double* m) {
  if (kind == 0) {
    m[0] = 1.0;
    if (N >= 1) m[1] = 0.0;
    for (int l = 2; l <= N; ++l) m[l] = (T - 1.0) * m[l - 2] / double(l);
    return;
  }
  m[0] = 0.5;
  if (N >= 1) m[1] = T / std::sqrt(2.0 * 3.14159265358979323846 * T);
  for (int s = 2; s <= N; ++s) m[s] = double(s - 1) * T * m[s - 2];
}

template <typename real, int Q0, int Q1>
static void fill_chan_tables(const ModelArgs& m, double T0, std::vector<unsigned char>* out) {
  using Tab = ChanTables<real, Q0, Q1>;
  out->assign(sizeof(Tab), 0);
  Tab& t = *reinterpret_cast<Tab*>(out->data());
  for (int k = 0; k < Q0; ++k) {
    t.p0[k] = real(m.p0[k]);
    t.w0[k] = real(m.w0[k]);
    t.sc0[k] = real(weno_pow2(m.iw0[k]));
    t.isc0[k] = real(1) / t.sc0[k];
    for (int s = 0; s <= m.N0; ++s) t.tab[s * (Q0 + Q1) + k] = real(m.tab0[k * MAXN + s]);
  }
  for (int k = 0; k < Q1; ++k) {
    t.p1[k] = real(m.p1[k]);
    t.w1[k] = real(m.w1[k]);
    t.sc1[k] = real(weno_pow2(m.iw1[k]));
    t.isc1[k] = real(1) / t.sc1[k];
    for (int s = 0; s <= m.N1; ++s) t.tab[s * (Q0 + Q1) + Q0 + k] = real(m.tab1[k * MAXN + s]);
  }
  // f_eq(1, 0, T0): factors and the incoming wall flux (the denominator of Eq. nw)
  double mv0[MAXN], mv1[MAXN], g0[Q0], g1[Q1];
  rest_moment_vector(m.kind0, m.N0, T0, mv0);
  rest_moment_vector(m.kind1, m.N1, T0, mv1);
  double den0 = 0.0, den1 = 0.0;
  for (int k = 0; k < Q0; ++k) {
    g0[k] = 0.0;
    for (int s = 0; s <= m.N0; ++s) g0[k] += m.tab0[k * MAXN + s] * mv0[s];
    t.gw0[k] = real(g0[k]);
    if (m.p0[k] < 0.0) den0 += g0[k] * m.p0[k];
  }
  for (int k = 0; k < Q1; ++k) {
    g1[k] = 0.0;
    for (int s = 0; s <= m.N1; ++s) g1[k] += m.tab1[k * MAXN + s] * mv1[s];
    t.gw1[k] = real(g1[k]);
    den1 += g1[k];
  }
  t.wall_den = den0 * den1;
  t.ref_flux_pos = m.ref_flux_pos;
  const double refs[4] = {m.ref_n, m.ref_r, m.ref_p, m.ref_e};
  for (int k = 0; k < 4; ++k) {
    t.ref_hi[k] = real(refs[k]);
    t.ref_lo[k] = real(refs[k] - double(t.ref_hi[k]));
  }
  t.ref_sum[0] = real(sizeof(real) == 4 ? m.ref_sum_f : m.ref_n);
  t.ref_sum[1] = real(sizeof(real) == 4 ? m.ref_sum_f - double(t.ref_sum[0]) : 0.0);
  t.nmax = std::max(m.N0, m.N1), t.kind1 = m.kind1;
}

template <typename real>
bool channel_tables(int nq0, int nq1, const ModelArgs& m, double T0, std::vector<unsigned char>* out) {
  if (nq0 == 16 && nq1 == 12) return fill_chan_tables<real, 16, 12>(m, T0, out), true;
  if (nq0 == 8 && nq1 == 4) return fill_chan_tables<real, 8, 4>(m, T0, out), true;
  return false;
}

template <typename real>
cudaError_t launch_channel(const ChanArgs<real>& a, const void* kp, int nq0, int nq1, int kind1, int kernel, int grid,
                           cudaStream_t s, bool clb) {
#define VLB_CH(q0, q1, cg, xw)                                                                  \
  return clb ? go_channel<real, q0, q1, cg, xw, true, false>(a, kp, grid, s)                    \
             : kind1 == 1 ? go_channel<real, q0, q1, cg, xw, false, true>(a, kp, grid, s)       \
                          : go_channel<real, q0, q1, cg, xw, false, false>(a, kp, grid, s);
  if (nq0 == 16 && nq1 == 12) VLB_CH(16, 12, 1, 0)
  if (nq0 == 8 && nq1 == 4) {
    if (kernel == 1) VLB_CH(8, 4, 4, 3)
    VLB_CH(8, 4, 1, 0)
  }
#undef VLB_CH
  return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------- equilibrium fill
template <typename real>
__global__ void init_equilibrium_kernel(real* F, long long cells, int Vp, const __grid_constant__ ModelArgs m,
                                        double n0, double u0, double u1, double T0) {
  __shared__ double g0[MAXQ], g1[MAXQ];
  if (threadIdx.x < 2) {
    const int ax = threadIdx.x;
    double mp[MAXN], mm[MAXN];
    const int kind = ax ? m.kind1 : m.kind0, N = ax ? m.N1 : m.N0, nq = ax ? m.nq1 : m.nq0;
    const double u = ax ? u1 : u0;
    eq_moment_vector<double>(kind, N, u, T0, mp);
    eq_moment_vector<double>(kind, N, -u, T0, mm);
    for (int k = 0; k < nq; ++k) {
      const double pk = ax ? m.p1[k] : m.p0[k];
      const double* mv = (kind == 1 && pk < 0.0) ? mm : mp;
      double g = 0;
      for (int s = 0; s <= N; ++s) g += (ax ? m.tab1 : m.tab0)[k * MAXN + s] * mv[s];
      (ax ? g1 : g0)[k] = g;
    }
  }
  __syncthreads();
  const int V = m.nq0 * m.nq1;
  const long long total = cells * 2 * Vp;
  for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < total; x += (long long)gridDim.x * blockDim.x) {
    const int e = int(x % (2 * Vp));  // (velocity, field) pairs interleaved
    const int v = e >> 1, d = e & 1;
    real val = real(0);
    if (v < V) {
      const int i = v / m.nq1, j = v - i * m.nq1;
      val = real(n0 * g0[i] * g1[j] * (d ? T0 : 1.0) - m.w0[i] * m.w1[j]);  // stored as the deviation from R
    }
    F[x] = val;
  }
}

template <typename real>
cudaError_t launch_init_equilibrium(real* F, long long cells, int Vp, const ModelArgs& m, double n0, double u0,
                                    double u1, double T0, cudaStream_t s) {
  const long long total = cells * 2 * Vp;
  long long blocks = (total + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  if (blocks < 1) blocks = 1;
  init_equilibrium_kernel<real><<<int(blocks), 256, 0, s>>>(F, cells, Vp, m, n0, u0, u1, T0);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- seeding from moments, one CTA per cell
// Table input vector of the one-axis function xi^k g(p) (xi = p - u, g the
// unit-mass Gaussian of mean u and variance T) for k <= 3, on the semi-axis of
// sign `side` (half range) or the whole line (full range, side ignored).
// Full range: the table takes E[He_l h] / l!, and (p - u) acts on that sequence
// as a_l -> (l + 1) a_{l+1} + a_{l-1} - u a_l (from p He_l = He_{l+1} + l He_{l-1}).
// Half range: the table takes the raw moments int_0^inf p^s h(side p) dp; with
// h(-p) = (-1)^k (p + u)^k g_{-u}(p) both sides are the binomial expansion of
// (p - v)^k, v = side u, over the raw moments of g_v on [0, inf).
__device__ inline void xi_power_vector(int kind, int N, double u, double T, int k, int side, double* out) {
  double m[MAXN + 3];
  if (kind == 0) {
    eq_moment_vector<double>(0, N + k, u, T, m);
    for (int it = 0; it < k; ++it) {
      const int top = N + k - it - 1;  // entries 0..top stay valid after this application
      double prev = 0.0;                // old m[l - 1]
      for (int l = 0; l <= top; ++l) {
        const double cur = m[l];
        m[l] = double(l + 1) * m[l + 1] + prev - u * cur;
        prev = cur;
      }
    }
    for (int l = 0; l <= N; ++l) out[l] = m[l];
    return;
  }
  const double v = side > 0 ? u : -u;
  eq_moment_vector<double>(1, N + k, v, T, m);
  // binomial coefficients C(k, i) (-v)^(k - i)
  double c[4] = {1, 0, 0, 0};
  for (int it = 0; it < k; ++it)
    for (int i = it + 1; i >= 0; --i) c[i] = (i ? c[i - 1] : 0.0) - v * c[i];
  const double sgn = (side < 0 && (k & 1)) ? -1.0 : 1.0;
  for (int s = 0; s <= N; ++s) {
    double acc = 0;
    for (int i = 0; i <= k; ++i) acc += c[i] * m[s + i];
    out[s] = sgn * acc;
  }
}

// Populations of xi^k g on one axis: pop[j] = sum_s tab[j][s] vec_side(j)[s].
__device__ inline void xi_power_populations(int kind, int N, int nq, const double* p, const double* tab, double u, double T,
                                     int k, double* pop) {
  double vp[MAXN], vm[MAXN];
  xi_power_vector(kind, N, u, T, k, 1, vp);
  if (kind == 1) xi_power_vector(kind, N, u, T, k, -1, vm);
  for (int j = 0; j < nq; ++j) {
    const double* v = (kind == 1 && p[j] < 0.0) ? vm : vp;
    double g = 0;
    for (int s = 0; s <= N; ++s) g += tab[j * MAXN + s] * v[s];
    pop[j] = g;
  }
}

// f' = n g0 g1 + q0/T^2 g0 g1 xi0 [(xi0^2 + xi1^2)/(5T) - 4/5],
// f'' = T n g0 g1 + q0/T^2 g0 g1 xi0 [(xi0^2 + xi1^2)/5 - 2T/5]:
// Grad's distribution with the heat-flux part only (along axis 0), p^z
// integrated out, projected on the model basis axis by axis.
template <typename real>
__global__ void seed_kernel(real* F, long long cells, int Vp, const __grid_constant__ ModelArgs m, const double* n,
                            const double* u0, const double* u1, const double* T, const double* q0, CellMap map) {
  __shared__ double A[3][MAXQ], B[2][MAXQ];  // axis 0: xi^0, xi^1, xi^3; axis 1: xi^0, xi^2
  for (long long c = blockIdx.x; c < cells; c += gridDim.x) {
    const long long cc = caller_cell(map, c);  // the fields are in the caller's cell order
    const double Tc = T[cc], qc = q0 ? q0[cc] : 0.0;
    if (threadIdx.x < 5) {
      const int t = threadIdx.x;
      if (t < 3) {
        const int k = t == 2 ? 3 : t;
        xi_power_populations(m.kind0, m.N0, m.nq0, m.p0, m.tab0, u0[cc], Tc, k, A[t]);
      } else {
        xi_power_populations(m.kind1, m.N1, m.nq1, m.p1, m.tab1, u1[cc], Tc, 2 * (t - 3), B[t - 3]);
      }
    }
    __syncthreads();
    const int V = m.nq0 * m.nq1;
    const double cq = qc / (Tc * Tc);
    for (int x = threadIdx.x; x < 2 * Vp; x += blockDim.x) {
      const int v = x >> 1, d = x & 1;  // (velocity, field) pairs interleaved
      real val = real(0);
      if (v < V) {
        const int i = v / m.nq1, j = v - i * m.nq1;
        const double base = n[cc] * A[0][i] * B[0][j];
        const double t3 = A[2][i] * B[0][j] + A[1][i] * B[1][j];
        const double t1 = A[1][i] * B[0][j];
        const double full = d ? Tc * base + cq * (0.2 * t3 - 0.4 * Tc * t1) : base + cq * (t3 / (5.0 * Tc) - 0.8 * t1);
        val = real(full - m.w0[i] * m.w1[j]);  // stored as the deviation from R
      }
      F[c * 2 * Vp + x] = val;
    }
    __syncthreads();
  }
}

template <typename real>
cudaError_t launch_seed(real* F, long long cells, int Vp, const ModelArgs& m, const double* n, const double* u0,
                        const double* u1, const double* T, const double* q0, cudaStream_t s, CellMap map) {
  const long long blocks = cells < 152 * 16 ? cells : 152 * 16;
  seed_kernel<real><<<int(blocks > 0 ? blocks : 1), 128, 0, s>>>(F, cells, Vp, m, n, u0, u1, T, q0, map);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- Shakhov collision
// The Shakhov collision relaxes towards f_eq + (1 - Pr) G, G the heat-flux part of Grad's
// form for the cell's own q (the seed kernel's term, with both axes):
//   G'  = [q0 (t3_0 / (5T) - 4/5 t1_0) + q1 (t3_1 / (5T) - 4/5 t1_1)] / T^2,
//   G'' = [q0 (t3_0 / 5 - 2T/5 t1_0) + q1 (t3_1 / 5 - 2T/5 t1_1)] / T^2,
//   t3_0 = A3 B0 + A1 B2, t1_0 = A1 B0, t3_1 = A2 B1 + A0 B3, t1_1 = A0 B1,
// A_k, B_k the projections of xi^k g on axes 0 and 1.  Against the BGK stage that the stage
// kernel has written, a stage of weight cc adds cc dt (1 - Pr) G[F_prev] / tau to F_out.
// One warp per cell: the cell's n, u, T and q from F_prev (sums and per-cell scalars in the
// bulk type: they enter a correction term), the projections A_k, B_k by the warp, then G for
// every (velocity, field).
// The model arrays a CTA indexes per thread, staged in shared memory: read from the kernel
// parameters with a different index in every lane they would be serialised.
template <typename real>
struct ModelSmem {
  real p[2][MAXQ], w[2][MAXQ], tab[2][MAXQ * MAXN];
};
template <typename real>
__device__ inline void stage_model(const ModelArgs& m, ModelSmem<real>& ms) {
  for (int k = threadIdx.x; k < MAXQ; k += blockDim.x) {
    if constexpr (sizeof(real) == 4) {
      ms.p[0][k] = m.p0f[k], ms.p[1][k] = m.p1f[k], ms.w[0][k] = m.w0f[k], ms.w[1][k] = m.w1f[k];
    } else {
      ms.p[0][k] = m.p0[k], ms.p[1][k] = m.p1[k], ms.w[0][k] = m.w0[k], ms.w[1][k] = m.w1[k];
    }
  }
  for (int k = threadIdx.x; k < MAXQ * MAXN; k += blockDim.x) {
    if constexpr (sizeof(real) == 4) ms.tab[0][k] = m.tab0f[k], ms.tab[1][k] = m.tab1f[k];
    else ms.tab[0][k] = m.tab0[k], ms.tab[1][k] = m.tab1[k];
  }
  __syncthreads();
}
// The tables A_k = [xi^k g] on axis 0 and B_k on axis 1 (k <= 3, xi_power_populations) for
// the cell's u and T, by one warp: the moment vector of each (axis, semi-axis) once, the
// input vector of each (axis, k, semi-axis), then the rows of the node tables in parallel; in
// the bulk type (the term they build is a correction of the collision).
template <typename R>
__device__ inline void power_tables(const ModelArgs& m, const ModelSmem<R>& ms, R u0, R u1, R T, R (*M)[MAXN + 3],
                                    R (*OV)[MAXN], R (*A)[MAXQ], R (*B)[MAXQ]) {
  const int tid = threadIdx.x & 31;
  if (tid < 4) {  // (axis, side): side 0 the positive semi-axis (or the whole line), side 1 the negative
    const int ax = tid >> 1, side = tid & 1;
    const int kind = ax ? m.kind1 : m.kind0, N = ax ? m.N1 : m.N0;
    const R u = ax ? u1 : u0;
    if (kind == 1 || side == 0) eq_moment_vector<R>(kind, N + 3, (kind == 1 && side) ? -u : u, T, M[tid]);
  }
  __syncwarp();
  if (tid < 16) {  // (axis, k, side), as xi_power_vector
    const int ax = tid >> 3, k = (tid >> 1) & 3, side = tid & 1;
    const int kind = ax ? m.kind1 : m.kind0, N = ax ? m.N1 : m.N0;
    const R u = ax ? u1 : u0;
    R* out = OV[tid];
    if (kind == 0) {
      if (side == 0) {
        R mm[MAXN + 3];
        for (int l = 0; l <= N + 3; ++l) mm[l] = M[2 * ax][l];
        for (int it = 0; it < k; ++it) {
          const int top = N + k - it - 1;
          R prev = R(0);
          for (int l = 0; l <= top; ++l) {
            const R cur = mm[l];
            mm[l] = R(l + 1) * mm[l + 1] + prev - u * cur;
            prev = cur;
          }
        }
        for (int l = 0; l <= N; ++l) out[l] = mm[l];
      }
    } else {
      const R v = side ? -u : u;
      R c[4] = {R(1), R(0), R(0), R(0)};
      for (int it = 0; it < k; ++it)
        for (int i = it + 1; i >= 0; --i) c[i] = (i ? c[i - 1] : R(0)) - v * c[i];
      const R sgn = (side && (k & 1)) ? R(-1) : R(1);
      for (int s2 = 0; s2 <= N; ++s2) {
        R acc = R(0);
        for (int i = 0; i <= k; ++i) acc += c[i] * M[2 * ax + side][s2 + i];
        out[s2] = sgn * acc;
      }
    }
  }
  __syncwarp();
  const int nq = m.nq0 + m.nq1;
  for (int x = tid; x < 4 * nq; x += 32) {
    const int k = x / nq, r = x - k * nq, ax = r >= m.nq0 ? 1 : 0, node = r - ax * m.nq0;
    const int kind = ax ? m.kind1 : m.kind0, N = ax ? m.N1 : m.N0;
    const R* tab = ms.tab[ax];
    const int side = (kind == 1 && ms.p[ax][node] < R(0)) ? 1 : 0;
    const R* v = OV[ax * 8 + k * 2 + side];
    R g = R(0);
    for (int s2 = 0; s2 <= N; ++s2) g += tab[node * MAXN + s2] * v[s2];
    (ax ? B : A)[k][node] = g;
  }
  __syncwarp();
}

// One warp per cell (four per CTA): no CTA barrier on a cell's chain, four times the cells in
// flight of a CTA per cell.
template <typename real>
__global__ void __launch_bounds__(128) shakhov_kernel(real* Fout, const real* Fprev, long long cells, int Vp,
                                                      const __grid_constant__ ModelArgs m, const InstDesc* inst,
                                                      int n_inst, double cc, double omp, double kn_fixed, bool early) {
  __shared__ real A[4][4][MAXQ], B[4][4][MAXQ], M[4][4][MAXN + 3], OV[4][16][MAXN];  // per warp
  __shared__ ModelSmem<real> ms;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int V = m.nq0 * m.nq1;
  if (early) grid_launch_dependents();  // (see launch_shakhov)
  stage_model<real>(m, ms);
  grid_dependency_wait();
  auto wsum = [&](real x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
  };
  for (long long c = (long long)blockIdx.x * 4 + w; c < cells; c += (long long)gridDim.x * 4) {
    const real* f = Fprev + c * 2 * Vp;
    // the instance of the cell (its Kn, tau convention and dt): the last with cell0 <= c
    int ii = 0;
    for (int b0 = 0; b0 < n_inst; b0 += 32) {
      const bool in = b0 + lane < n_inst && inst[b0 + lane].cell0 <= c;
      const unsigned bal = __ballot_sync(0xffffffffu, in);
      if (bal) ii = b0 + 31 - __clz(bal);
      if (bal != 0xffffffffu) break;
    }
    // n and n u (Eq. macro_red), F = D + R; every lane gets the sums
    real a = real(0), b = real(0), g = real(0);
    for (int v = lane; v < V; v += 32) {
      const int i = v / m.nq1, j = v - i * m.nq1;
      const real f1 = f[2 * v] + ms.w[0][i] * ms.w[1][j];
      a += f1;
      b += ms.p[0][i] * f1;
      g += ms.p[1][j] * f1;
    }
    const real n = wsum(a), u0 = wsum(b) / n, u1 = wsum(g) / n;
    // 3 n T = sum (xi0^2 + xi1^2) f' + f'',  q = sum [(xi0^2 + xi1^2) f' + f''] xi / 2
    a = b = g = real(0);
    for (int v = lane; v < V; v += 32) {
      const int i = v / m.nq1, j = v - i * m.nq1;
      const real R = ms.w[0][i] * ms.w[1][j];
      const real x0 = ms.p[0][i] - u0, x1 = ms.p[1][j] - u1;
      const real e = (x0 * x0 + x1 * x1) * (f[2 * v] + R) + (f[2 * v + 1] + R);
      a += e;
      b += e * x0;
      g += e * x1;
    }
    const real T = wsum(a) / (real(3) * n), q0 = real(0.5) * wsum(b), q1 = real(0.5) * wsum(g);
    const InstDesc& d = inst[ii];
    const real tau = kn_fixed > 0.0 ? real(kn_fixed) / (n * T) : relaxation_time<real>(d.tau_mode, real(d.kn), n, T);
    const real coef = real(cc * d.dt * omp) / tau;
    const real iT2 = real(1) / (T * T), a0 = q0 * iT2, a1 = q1 * iT2, i5T = real(1) / (real(5) * T);
    power_tables<real>(m, ms, u0, u1, T, M[w], OV[w], A[w], B[w]);
    const real(*Aw)[MAXQ] = A[w];
    const real(*Bw)[MAXQ] = B[w];
    for (int x = lane; x < 2 * V; x += 32) {
      const int v = x >> 1, fi = x & 1;
      const int i = v / m.nq1, j = v - i * m.nq1;
      const real t3a = Aw[3][i] * Bw[0][j] + Aw[1][i] * Bw[2][j], t1a = Aw[1][i] * Bw[0][j];
      const real t3b = Aw[2][i] * Bw[1][j] + Aw[0][i] * Bw[3][j], t1b = Aw[0][i] * Bw[1][j];
      const real G = fi ? a0 * (real(0.2) * t3a - real(0.4) * T * t1a) + a1 * (real(0.2) * t3b - real(0.4) * T * t1b)
                        : a0 * (t3a * i5T - real(0.8) * t1a) + a1 * (t3b * i5T - real(0.8) * t1b);
      real* y = Fout + c * 2 * Vp + x;
      *y = *y + coef * G;
    }
    __syncwarp();  // A, B, M, OV of this warp are rewritten for its next cell
  }
}

// The same for the velocity sets with fixed node counts.  One warp per cell; a lane owns the
// velocities lane + 32 r, whose pairs it reads once and whose nodes it keeps in registers.  The
// one-axis projections come from
//   int x^s (x - v)^k N = T (s int x^{s-1} (x - v)^{k-1} N + (k - 1) int x^s (x - v)^{k-2} N)
//                         + [s = 0] T (-v)^{k-1} N(0; v, T)
// on a semi-axis (integration by parts with (x - v) N = -T N') and, on the full range, from the same
// without the boundary term on E[He_l xi^k] / l!: one lane per (axis, semi-axis), all k in turn.
// With a0 = q0 / T^2, a1 = q1 / T^2 the term is, per velocity,
//   t = (a0 A3, a0 A1, a1 A2, a1 A0)_i . (B0, B2, B1, B3)_j,  l = a0 A1 B0 + a1 A0 B1,
//   G' = t / (5T) - 4/5 l,  G'' = t / 5 - 2T/5 l.
// What bounds it: the warp's serial chain per cell and L2 (F_prev read, F_out read and written).
// 24 instances of 64 .. 96 cells x 320 velocities, single precision, a launch: 20.8 us for the
// general kernel, 15.8 us.
template <typename real, int Q0, int Q1>
__global__ void __launch_bounds__(128) shakhov_fixed_kernel(real* Fout, const real* Fprev, long long cells,
                                                            const __grid_constant__ ModelArgs m, const InstDesc* inst,
                                                            int n_inst, double cc, double omp, double kn_fixed, bool early) {
  using P = pair_t<real>;
  constexpr int V = Q0 * Q1, R = V / 32, NQ = Q0 + Q1;
  static_assert(V % 32 == 0, "whole warps of velocities");
  __shared__ real tab[MAXN * NQ];          // equilibrium tables of both axes, [s][k]
  __shared__ real OV[4][4][4][MAXN];       // per warp: [axis * 2 + side][k][s]
  __shared__ alignas(16) real PA[4][Q0][4], PB[4][Q1][4];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  constexpr bool F32 = sizeof(real) == 4;
  if (early) grid_launch_dependents();  // (see launch_shakhov)
  const int nmax = m.N0 > m.N1 ? m.N0 : m.N1;
  for (int x = threadIdx.x; x < MAXN * NQ; x += 128) {
    const int s = x / NQ, q = x - s * NQ, ax = q >= Q0, k = ax ? q - Q0 : q;
    real t = real(0);
    if (s <= (ax ? m.N1 : m.N0))
      t = F32 ? real((ax ? m.tab1f : m.tab0f)[k * MAXN + s]) : real((ax ? m.tab1 : m.tab0)[k * MAXN + s]);
    tab[x] = t;
  }
  real p0[R], p1[R], rw[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int v = lane + 32 * r, i = v / Q1, j = v - i * Q1;
    p0[r] = F32 ? real(m.p0f[i]) : real(m.p0[i]);
    p1[r] = F32 ? real(m.p1f[j]) : real(m.p1[j]);
    rw[r] = F32 ? real(m.w0f[i]) * real(m.w1f[j]) : real(m.w0[i] * m.w1[j]);
  }
  __syncthreads();
  grid_dependency_wait();
  for (long long c = (long long)blockIdx.x * 4 + w; c < cells; c += (long long)gridDim.x * 4) {
    P f[R];
#pragma unroll
    for (int r = 0; r < R; ++r) f[r] = p_load(Fprev + (c * V + lane + 32 * r) * 2);
    // the instance of the cell (its Kn, tau convention and dt): the last with cell0 <= c
    int ii = 0;
    for (int b0 = 0; b0 < n_inst; b0 += 32) {
      const bool in = b0 + lane < n_inst && inst[b0 + lane].cell0 <= c;
      const unsigned bal = __ballot_sync(0xffffffffu, in);
      if (bal) ii = b0 + 31 - __clz(bal);
      if (bal != 0xffffffffu) break;
    }
    real a = real(0), b = real(0), g = real(0);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      f[r] = p_add(f[r], p_set(rw[r]));  // F = D + R
      a += f[r].x;
      b += p0[r] * f[r].x;
      g += p1[r] * f[r].x;
    }
    const real n = group_sum<32>(a), in_ = rcp_rn(n), u0 = group_sum<32>(b) * in_, u1 = group_sum<32>(g) * in_;
    // 3 n T = sum (xi0^2 + xi1^2) f' + f'',  q = sum [(xi0^2 + xi1^2) f' + f''] xi / 2
    a = b = g = real(0);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const real x0 = p0[r] - u0, x1 = p1[r] - u1;
      const real e = (x0 * x0 + x1 * x1) * f[r].x + f[r].y;
      a += e;
      b += e * x0;
      g += e * x1;
    }
    const real T = group_sum<32>(a) * in_ * (real(1) / real(3)), iT = rcp_rn(T);
    const real hq = real(0.5) * iT * iT, a0 = group_sum<32>(b) * hq, a1 = group_sum<32>(g) * hq;
    const InstDesc& d = inst[ii];
    const real rate = kn_fixed > 0.0 ? n * T * rcp_rn(real(kn_fixed))
                                     : relaxation_rate<real>(d.tau_mode, rcp_rn(real(d.kn)), n, T);
    const real coef = real(cc * d.dt * omp) * rate;
    if (lane < 4) {  // (axis, side): side 0 the positive semi-axis (or the whole line), side 1 the negative
      const int kind = lane & 2 ? m.kind1 : m.kind0;
      const real u = lane & 2 ? u1 : u0;
      const real v = (kind == 1 && (lane & 1)) ? -u : u;
      real M[MAXN];
      eq_moments_fast<real>(kind, nmax, v, T, M);
      const real half = kind == 1 ? real(1) : real(0);
      // boundary terms T (-v)^{k-1} N(0; v, T), from M_1 = v M_0 + T N(0)
      const real bt = half * (M[1] - v * M[0]);
      const real sg = (kind == 1 && (lane & 1)) ? real(-1) : real(1);  // (p - u)^k on the negative semi-axis
      real l1 = real(0), l2 = real(0), l0 = real(0);  // entries s - 1 of k = 1, 2, 0
#pragma unroll
      for (int s = 0; s < MAXN; ++s) {
        if (s > nmax) break;
        const real fs = kind == 1 ? real(s) : (s > 0 ? real(1) : real(0));
        const real z = s == 0 ? bt : real(0);
        const real k1 = T * fs * l0 + z;
        const real k2 = T * (fs * l1 + M[s]) - v * z;
        const real k3 = T * (fs * l2 + real(2) * k1) + v * v * z;
        OV[w][lane][0][s] = M[s];
        OV[w][lane][1][s] = sg * k1;
        OV[w][lane][2][s] = k2;
        OV[w][lane][3][s] = sg * k3;
        l0 = M[s], l1 = k1, l2 = k2;
      }
    }
    __syncwarp();
    for (int x = lane; x < 4 * NQ; x += 32) {
      const int k = x / NQ, q = x - k * NQ, ax = q >= Q0, node = ax ? q - Q0 : q, nq = ax ? Q1 : Q0;
      const int side = ((ax ? m.kind1 : m.kind0) == 1 && node >= nq / 2) ? 1 : 0;
      const real* o = OV[w][ax * 2 + side][k];
      real z = real(0);
      for (int s = 0; s <= nmax; ++s) z += tab[s * NQ + q] * o[s];
      if (ax) PB[w][node][k == 0 ? 0 : k == 1 ? 2 : k == 2 ? 1 : 3] = z;
      else PA[w][node][k == 0 ? 3 : k == 1 ? 1 : k == 2 ? 2 : 0] = z * (k & 1 ? a0 : a1);
    }
    __syncwarp();
    const real c1 = coef * real(0.2) * iT, c2 = coef * real(-0.8), c3 = coef * real(0.2), c4 = coef * real(-0.4) * T;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int v = lane + 32 * r, i = v / Q1, j = v - i * Q1;
      const real* x = PA[w][i];
      const real* y = PB[w][j];
      const real t = x[0] * y[0] + x[1] * y[1] + x[2] * y[2] + x[3] * y[3];
      const real l = x[1] * y[0] + x[3] * y[2];
      real* o = Fout + (c * V + v) * 2;
      const P h = p_load(o);
      p_store(o, p_make(h.x + (c1 * t + c2 * l), h.y + (c3 * t + c4 * l)));
    }
    __syncwarp();  // OV, PA, PB of this warp are rewritten for its next cell
  }
}

// Launched as dependent on the stage, as the next stage is on it.  In double precision only where its CTAs
// come to an eighth of the SMs at most: the device places a dependent grid's CTAs while the other's still
// hold some SMs, and those that are free take more than their share, which a kernel of 1/64-rate
// operations does not make up for (a step replayed from a graph, 8 x 8 velocities: 1600 cells 718 us
// dependent, 471 not; 8 x 8, 2560 cells 784 and 603; 16 x 20, 608 cells 436 and 342; 8 x 4, 8 cells 98 and
// 104).  From six CTAs a SM it evens out, and the correction is dependent again.
template <typename real>
cudaError_t launch_shakhov(real* Fout, const real* Fprev, long long cells, int Vp, const ModelArgs& m,
                           const InstDesc* inst, int n_inst, double cc, double one_minus_pr, double kn_fixed, int sms,
                           cudaStream_t s) {
  long long blocks = (cells + 3) / 4;
  if (blocks > 152 * 16) blocks = 152 * 16;
  const bool early = sizeof(real) == 4 || blocks <= sms / 8, dependent = early || blocks > 6ll * sms;
  const dim3 g(static_cast<unsigned>(blocks > 0 ? blocks : 1));
#define VLB_SHAKHOV(q0, q1)                                                                                          \
  if (m.nq0 == q0 && m.nq1 == q1)                                                                                    \
    return launch_ordered(dependent, shakhov_fixed_kernel<real, q0, q1>, g, 128, 0, s, Fout, Fprev, cells, m, inst, \
                          n_inst, cc, one_minus_pr, kn_fixed, early);
  VLB_SHAKHOV(16, 20) VLB_SHAKHOV(16, 12) VLB_SHAKHOV(8, 4)
#undef VLB_SHAKHOV
  return launch_ordered(dependent, shakhov_kernel<real>, g, 128, 0, s, Fout, Fprev, cells, Vp, m, inst, n_inst, cc,
                        one_minus_pr, kn_fixed, early);
}

// ---------------------------------------------------------------- caller layout <-> device layout
// Caller rows hold f' then f'' (V values each); device rows hold the deviation
// from R as interleaved (f', f'') pairs of Vp velocities.  Bound by HBM (one read and one
// write of the distribution): one warp per cell row, each lane holding NV neighbouring
// velocities of every chunk of 32 NV, so that a chunk is two contiguous accesses of the
// caller's row (f', f'') and one of the device row, and the rest state of the lane's
// velocities stays in registers over all rows of the warp.  A row is read whole before any of
// it is written, so src and dst may be the same buffer when V == Vp and the map is the identity.
//
// F -/+ R is rounded once.  In single precision R (53 bits) is a sum of three floats, and the sum with F
// stays on the FP32 pipe, where one in double cost three operations of the 1/64-rate FP64 pipe per
// value: its bounds from directed sums of the low parts round to the same value nearly always, and the
// others (near rest, where F and R nearly cancel, or next to a tie) are gathered exactly.  (A pair of
// floats alone would lose the last five bits of R, near rest a quarter of a unit in the deviation's last
// place.)  In double precision R = w_i w_j is not rounded before the sum.  2048 x 512 x 192 channel
// (1.6 GB), both directions together: 5.5 ms with the sum in double, 1.15 ms so (6.4 GB moved: 0.82 of
// the measured copy bandwidth; 1.28 ms at rest).
template <typename real>
struct RestValue;  // of one velocity, with the sign of the sum
template <>
struct RestValue<float> {
  float hi, mid, lo;
  __device__ __forceinline__ void set(double w0, double w1) {
    const double R = w0 * w1;
    hi = float(R);
    mid = float(R - double(hi));
    lo = float(R - double(hi) - double(mid));
  }
};
template <>
struct RestValue<double> {
  double w0, w1;
  __device__ __forceinline__ void set(double a, double b) { w0 = a, w1 = b; }
};
// x + R where both bounds round to the same value; else out is set
__device__ __forceinline__ float add_rest(float x, RestValue<float> r, bool& out) {
  float s, e;
  two_sum(x, r.hi, s, e);
  const float d = __fadd_rn(s, __fadd_rd(__fadd_rd(e, r.mid), r.lo));
  const float u = __fadd_rn(s, __fadd_ru(__fadd_ru(e, r.mid), r.lo));
  out = out || !(d == u);
  return d;
}
__device__ __forceinline__ double add_rest(double x, RestValue<double> r, bool&) { return fma(r.w0, r.w1, x); }
// a + b rounded to odd: of the two neighbours of an inexact sum the one with the last bit set, so that a
// further rounding to fewer bits sees which side of a tie the sum lies on
__device__ __forceinline__ float add_odd(float a, float b) {
  const float d = __fadd_rd(a, b), u = __fadd_ru(a, b);
  return __float_as_uint(d) & 1u ? d : u;
}
__device__ __forceinline__ float add_rest_exact(float x, RestValue<float> r) {
  float s, e, v, f, t, q;
  two_sum(x, r.hi, s, e);
  two_sum(e, r.mid, v, f);
  two_sum(s, v, t, q);
  const float z = __fadd_rn(t, add_odd(q, add_odd(f, r.lo)));
  return fabsf(s) <= 3.402823466e38f ? z : s;  // Inf and NaN stay what the plain sum gives
}
__device__ __forceinline__ double add_rest_exact(double x, RestValue<double> r) { return fma(r.w0, r.w1, x); }

template <typename real, int NV, int CH>
__global__ void __launch_bounds__(256) deviation_kernel(const real* src, real* dst, long long cells, int Vp,
                                                        const __grid_constant__ ModelArgs m, int to_dev, CellMap map) {
  using P = pair_t<real>;
  // (the weights by way of shared memory: an index per lane into the parameters is serialised; then R,
  // whose parts take FP64-pipe operations, once per CTA)
  __shared__ double sw[2][MAXQ];
  __shared__ RestValue<real> sr[32 * CH * NV];
  if (threadIdx.x < 2 * MAXQ) sw[threadIdx.x / MAXQ][threadIdx.x % MAXQ] = (threadIdx.x < MAXQ ? m.w0 : m.w1)[threadIdx.x % MAXQ];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int V = m.nq0 * m.nq1;
  for (int v = threadIdx.x; v < 32 * CH * NV; v += blockDim.x) {
    const int i = v < V ? v / m.nq1 : 0, j = v < V ? v - i * m.nq1 : 0;
    sr[v].set(to_dev ? -sw[0][i] : sw[0][i], sw[1][j]);
  }
  __syncthreads();
  RestValue<real> R[CH][NV];
#pragma unroll
  for (int k = 0; k < CH; ++k)
#pragma unroll
    for (int q = 0; q < NV; ++q) R[k][q] = sr[(32 * k + lane) * NV + q];
  const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long c = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); c < cells; c += nw) {
    const long long cc = caller_cell(map, c);  // device cell c is the caller's cell cc
    const real* a = src + (to_dev ? cc * 2 * V : c * 2 * Vp);
    real* o = dst + (to_dev ? c * 2 * Vp : cc * 2 * V);
    P x[CH][NV];
#pragma unroll
    for (int k = 0; k < CH; ++k) {
      const int v = (32 * k + lane) * NV;
#pragma unroll
      for (int q = 0; q < NV; ++q) x[k][q] = p_set(real(0));
      if (v < V) {
        if (to_dev) {
          if constexpr (NV == 2) {
            const P f1 = p_load(a + v), f2 = p_load(a + V + v);
            x[k][0] = p_make(f1.x, f2.x), x[k][1] = p_make(f1.y, f2.y);
          } else {
            x[k][0] = p_make(a[v], a[V + v]);
          }
        } else {
          if constexpr (NV == 2) {
            const float4 y = *reinterpret_cast<const float4*>(a + 2 * v);
            x[k][0] = p_make(y.x, y.y), x[k][1] = p_make(y.z, y.w);
          } else {
            x[k][0] = p_load(a + 2 * v);
          }
        }
      }
    }
#pragma unroll
    for (int k = 0; k < CH; ++k) {
      if (32 * k * NV >= V) break;
      P y[NV];
      bool out = false;
#pragma unroll
      for (int q = 0; q < NV; ++q)
        y[q] = p_make(add_rest(x[k][q].x, R[k][q], out), add_rest(x[k][q].y, R[k][q], out));
      if (__any_sync(0xffffffffu, out)) {
#pragma unroll
        for (int q = 0; q < NV; ++q)
          y[q] = p_make(add_rest_exact(x[k][q].x, R[k][q]), add_rest_exact(x[k][q].y, R[k][q]));
      }
#pragma unroll
      for (int q = 0; q < NV; ++q)
        if ((32 * k + lane) * NV < V) x[k][q] = y[q];  // (the padding velocities stay zero)
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < CH; ++k) {
      const int v = (32 * k + lane) * NV;
      if (to_dev) {
        if (v < Vp) {  // the padding velocities are zero
          if constexpr (NV == 2)
            *reinterpret_cast<float4*>(o + 2 * v) = make_float4(x[k][0].x, x[k][0].y, x[k][1].x, x[k][1].y);
          else p_store(o + 2 * v, x[k][0]);
        }
      } else if (v < V) {
        if constexpr (NV == 2) {
          p_store(o + v, p_make(x[k][0].x, x[k][1].x));
          p_store(o + V + v, p_make(x[k][0].y, x[k][1].y));
        } else {
          o[v] = x[k][0].x, o[V + v] = x[k][0].y;
        }
      }
    }
    __syncwarp();
  }
}

template <typename real, int NV>
static cudaError_t go_deviation(const real* src, real* dst, long long cells, int Vp, const ModelArgs& m, int to_dev,
                                cudaStream_t s, CellMap map) {
  // eight warps a CTA, up to eight CTAs an SM, a row's loads in flight in each warp
  long long blocks = (cells + 7) / 8;
  if (blocks > 152 * 8) blocks = 152 * 8;
  const int g = int(blocks > 0 ? blocks : 1), chunks = (Vp + 32 * NV - 1) / (32 * NV);
  if (chunks <= 4) deviation_kernel<real, NV, 4><<<g, 256, 0, s>>>(src, dst, cells, Vp, m, to_dev, map);
  else if (chunks <= 8) deviation_kernel<real, NV, 8><<<g, 256, 0, s>>>(src, dst, cells, Vp, m, to_dev, map);
  else if (chunks <= 16) deviation_kernel<real, NV, 16><<<g, 256, 0, s>>>(src, dst, cells, Vp, m, to_dev, map);
  else if constexpr (NV == 1) deviation_kernel<real, 1, 32><<<g, 256, 0, s>>>(src, dst, cells, Vp, m, to_dev, map);
  else return cudaErrorInvalidValue;  // MAXQ^2 velocities are 16 chunks of 64
  return cudaGetLastError();
}

template <typename real>
cudaError_t launch_deviation(const real* src, real* dst, long long cells, int Vp, const ModelArgs& m,
                             int to_deviation, cudaStream_t s, CellMap map) {
  // two velocities a lane (8- and 16-byte accesses) where the caller's rows and buffer allow it
  if constexpr (sizeof(real) == 4) {
    const void* caller = to_deviation ? static_cast<const void*>(src) : static_cast<const void*>(dst);
    if (m.nq0 * m.nq1 == Vp && reinterpret_cast<uintptr_t>(caller) % 8 == 0)
      return go_deviation<real, 2>(src, dst, cells, Vp, m, to_deviation, s, map);
  }
  return go_deviation<real, 1>(src, dst, cells, Vp, m, to_deviation, s, map);
}

// ---------------------------------------------------------------- moments (FP64), one warp per cell
template <typename real>
__global__ void moments_kernel(const real* F, long long cells, int Vp, const __grid_constant__ ModelArgs m,
                               double* out, CellMap map) {
  const int lane = threadIdx.x & 31;
  const long long warp0 = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  const int nq1 = m.nq1, V = m.nq0 * m.nq1;
  for (long long c = warp0; c < cells; c += nwarps) {
    const real* f = F + c * 2 * Vp;
    double sn = 0, s0 = 0, s1 = 0;
    for (int v = lane; v < V; v += 32) {
      const int i = v / nq1, j = v - i * nq1;
      const double f1 = double(f[2 * v]) + m.w0[i] * m.w1[j];  // F = D + R
      sn += f1;
      s0 += m.p0[i] * f1;
      s1 += m.p1[j] * f1;
    }
    sn = warp_sum<real>(sn);
    s0 = warp_sum<real>(s0);
    s1 = warp_sum<real>(s1);
    const double n = sn, u0 = s0 / n, u1 = s1 / n;
    double t00 = 0, t01 = 0, t11 = 0, tr2 = 0, q0 = 0, q1 = 0;
    for (int v = lane; v < V; v += 32) {
      const int i = v / nq1, j = v - i * nq1;
      const double r = m.w0[i] * m.w1[j];
      const double f1 = double(f[2 * v]) + r, f2 = double(f[2 * v + 1]) + r;
      const double x0 = m.p0[i] - u0, x1 = m.p1[j] - u1;
      t00 += x0 * x0 * f1;
      t01 += x0 * x1 * f1;
      t11 += x1 * x1 * f1;
      tr2 += f2;
      const double e = 0.5 * (x0 * x0 + x1 * x1) * f1 + 0.5 * f2;
      q0 += e * x0;
      q1 += e * x1;
    }
    t00 = warp_sum<real>(t00);
    t01 = warp_sum<real>(t01);
    t11 = warp_sum<real>(t11);
    tr2 = warp_sum<real>(tr2);
    q0 = warp_sum<real>(q0);
    q1 = warp_sum<real>(q1);
    if (lane == 0) {
      double* o = out + caller_cell(map, c) * 9;  // in the caller's cell order
      o[0] = n;
      o[1] = u0;
      o[2] = u1;
      o[3] = (t00 + t11 + tr2) / (3.0 * n);
      o[4] = t00;
      o[5] = t01;
      o[6] = t11;
      o[7] = q0;
      o[8] = q1;
    }
  }
}

template <typename real>
cudaError_t launch_moments(const real* F, long long cells, int Vp, const ModelArgs& m, double* out, cudaStream_t s,
                           CellMap map) {
  long long blocks = (cells * 32 + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  if (blocks < 1) blocks = 1;
  moments_kernel<real><<<int(blocks), 256, 0, s>>>(F, cells, Vp, m, out, map);
  return cudaGetLastError();
}

template int stage_variants<VLB_REAL>(int, int, StageVariant*);
template size_t stage_smem_bytes<VLB_REAL>(StageVariant, int);
template bool stage_split_tables<VLB_REAL>(int, int);
template cudaError_t launch_stage<VLB_REAL>(StageVariant, const StageArgs<VLB_REAL>&, const ModelArgs&,
                                            const KArgs<VLB_REAL>&, int, cudaStream_t, bool);
template cudaError_t launch_init_equilibrium<VLB_REAL>(VLB_REAL*, long long, int, const ModelArgs&, double, double,
                                                       double, double, cudaStream_t);
template cudaError_t channel_kernels<VLB_REAL>(int, int, int, bool, ChanKernel*, int*);
template cudaError_t launch_channel<VLB_REAL>(const ChanArgs<VLB_REAL>&, const void*, int, int, int, int, int,
                                              cudaStream_t, bool);
template bool channel_force_pairs<VLB_REAL>(int, int, const AxisTables*, std::vector<unsigned char>*);
template bool channel_tables<VLB_REAL>(int, int, const ModelArgs&, double, std::vector<unsigned char>*);
template cudaError_t launch_seed<VLB_REAL>(VLB_REAL*, long long, int, const ModelArgs&, const double*,
                                           const double*, const double*, const double*, const double*, cudaStream_t,
                                           CellMap);
template cudaError_t stage_config<VLB_REAL>(StageVariant, const ModelArgs&, int, int*, int*, bool);
template cudaError_t launch_deviation<VLB_REAL>(const VLB_REAL*, VLB_REAL*, long long, int, const ModelArgs&, int,
                                                cudaStream_t, CellMap);
template cudaError_t launch_moments<VLB_REAL>(const VLB_REAL*, long long, int, const ModelArgs&, double*,
                                              cudaStream_t, CellMap);
template cudaError_t launch_shakhov<VLB_REAL>(VLB_REAL*, const VLB_REAL*, long long, int, const ModelArgs&,
                                              const InstDesc*, int, double, double, double, int, cudaStream_t);

}  // namespace vlb
