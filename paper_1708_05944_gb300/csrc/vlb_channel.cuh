// One TVD-RK3 stage of the gradually expanding channel in the vielbein frame
// (Sec. VII.A-C, Eq. canalie_boltz), as a marching kernel: each CTA owns a
// strip of TP = 4 adjacent xi-columns and walks up a segment of lambda rows
// (wall-normal).  A thread owns one velocity on all four columns (on one, see ChanSmem).  Step s of the march
//
//   - reconstructs the five xi interfaces of row s in one walk along the strip (the row and its
//     halo come from a shared-memory ring that bulk copies fill) and the lambda interface of
//     every column from the column's window of differences, kept in registers, so that each
//     lambda interface is reconstructed once and each xi interface once per strip;
//   - combines advection, force, BGK relaxation and the RK3 weights of row s and stores it
//     straight to global memory;
//   - prepares the rows ahead, by warp role: the momentum-space force of row s + 1, the moments
//     and truncated equilibria of row s + 3, the inflow factors of row s + 2 and the reservoir
//     ghost cells of row s + 1.
//
// One CTA barrier a step; two CTAs a SM overlap each other's barriers and serial parts (single
// precision).  What bounds it: latency, with 12 warps a SM at 168 registers each; then the FP32
// pipe (half busy: about 290 of its cycles per warp and cell-velocity row, of which the ten
// reconstructions of a row of four columns take 160).  Why four columns a thread: the strip's xi
// walk and the windows cost 34 packed operations an interface where five cells loaded afresh cost
// 44 (windows of two columns or of raw rows in shared memory, twice the warps or half the
// registers, measured 13.0 - 14.1 ms a step where this took 9.85); why unrolled: the same loop rolled
// halves the reconstructions in flight (14.5).  A barrier at the step's end keeps the warps on
// the same instructions; waiting later, at the next combine, lost more to instruction fetches
// (12.5).  2048 x 512 x 192, single precision, a step of three stages: 20.3 ms for one thread per
// (column, velocity) with 1024 threads of 64 registers, 9.9 ms now (1.30 TB/s algorithmic a
// stage); double precision, 256 x 64: 10.9 and 6.7 ms; Cartesian split, 512 x 256: 2.39 and 1.19.
//
// Boundaries: the centreline mirror (Sec. VII.C.3) at the bottom of the march, the diffuse wall
// (Sec. VII.C.4) at its top with n_w per column from the zero-mass-flux balance, and the
// inlet/outlet reservoirs as halo cells of the first and last strip.
//
// Distribution buffers hold the deviation D = F - R from the rest state
// (ModelArgs), with (f', f'') interleaved per velocity: a cell row is
// 2 Q0 Q1 reals, element (i, j, d) at 2 (i Q1 + j) + d.
#pragma once
#include "vlb_device.cuh"

namespace vlb {

// Per-cell geometry of the channel (Sec. VII.A): V^lambda = a p^lambda and V^xi = b p^xi - c p^lambda
// at the interfaces, 1/d chi^xi_p and the discrete connection coefficients.  The interface factors
// of lambda carry 1/d lambda_s, and what multiplies a pair is stored twice (the operand of a
// packed operation).
template <typename T>
struct ChanCell {
  T ap[2], nam[2], idx[2];  // a / d lambda at s+1/2, -a / d lambda at s-1/2, 1 / d chi_p
  T bm, cm, bp, cp;         // b, c at p-1/2, p+1/2
  T glxl, glxx;             // Gamma_{l x l}, Gamma_{l x x}
};
static_assert(sizeof(ChanCell<float>) == 48 && sizeof(ChanCell<double>) == 96, "bulk-copied geometry rows");

template <int Q0, int Q1>
struct ChanShape {
  static constexpr int V = Q0 * Q1;
  static constexpr int ROW = 2 * V;        // reals per cell row
  static constexpr int NW = V / 32;        // warps: one thread per velocity
  static constexpr int TP = 4;             // columns per strip
  // per-cell equilibrium record, in pairs: n g0_i twice, g1_j twice, (1, T), -1/tau twice, (u^xi, 0)
  static constexpr int EQW = 2 * (Q0 + Q1 + 3);
  static_assert(V % 32 == 0 && Q0 % 2 == 0 && Q1 % 2 == 0, "velocity set shape of the channel kernel");
  static_assert(Q0 % 8 == 0 && Q0 + Q1 <= 32, "eight lanes per cell, four equilibrium factors each");
};

// Model tables of a channel context, in device memory, copied into each CTA's shared memory.
// gw0/gw1 are the factors of f_eq(1, 0, T0), the wall and reservoir equilibrium at rest (they
// change with T0); sc0 sc1 is the power-of-two scale of the WENO walk (WenoWin) per velocity.
template <typename real, int Q0, int Q1>
struct alignas(16) ChanTables {
  real p0[Q0], p1[Q1], w0[Q0], w1[Q1], sc0[Q0], sc1[Q1], isc0[Q0], isc1[Q1];
  real tab[MAXN * (Q0 + Q1)];  // equilibrium tables of both axes, [s][k] (zero beyond an axis' order)
  real gw0[Q0], gw1[Q1];
  double wall_den;  // sum over p^lambda < 0 of gw0 p^lambda times sum of gw1: incoming flux of f_eq(1, 0, T0)
  double ref_flux_pos;  // sum over p^lambda > 0 of p^lambda R (ModelArgs)
  // sums of R (ModelArgs: n, rho u0, rho u1, energy) as (hi, lo) in the bulk type (lo = 0 in
  // double), and the sum of the products w0_i w1_j of the bulk-type weights, the part of the mass
  // that the stage's f_eq - R subtracts
  real ref_hi[4], ref_lo[4], ref_sum[2];
  int nmax, kind1, pad[2];  // the larger expansion order; axis 1 half range
};

// Host-side description of a channel context: grid size, Kn, time step, reservoirs,
// and the flow-rate ends (flow = 1: the parabolic profiles of Q0 replace the reservoirs).
struct ChanDesc {
  int nl, nx;
  double kn, dt, n_in, n_out, T0;
  float knf, dtf, n_inf, n_outf, T0f;
  int flow;
  double q0;
};

template <typename real>
struct ChanArgs {
  const real* Fprev;  // distribution L acts on
  const real* Fl;     // F_l of the step (read when ca != 0)
  real* Fout;
  const void* tables;  // ChanTables of the context's shape
  const ChanCell<real>* geo;
  double* nw;  // per column
  unsigned* err;
  int nl, nx;
  int seglen;  // rows per lambda segment (the last one may be shorter, >= 3 rows)
  int nseg;
  // Fout = F_prev + ca (F_l - F_prev) + ccdt L[F_prev] (see StageArgs), each twice; ca = 0: no F_l
  pair_t<real> ca, ccdt;
  real ikn, n_in, n_out, T0;  // 1/Kn, reservoir densities, wall and reservoir temperature
  unsigned long long max_polls;
  // flow-rate ends (Sec. VII.C.1-2), when flow != 0: per end e and row s,
  // qflow[(2 e) nl + s] = Q_s (the inflow equilibrium's u^xi) and
  // qflow[(2 e + 1) nl + s] = (1 + phi) Q_s (the particle flux through the end interface)
  const real* qflow;
  int flow;
};

// Shared-memory carve-up of a CTA, identical on host and device.  The ring holds
// rows s .. s+4 of the strip, each with its xi-halo (TP + 6 cells): row s for the xi
// reconstruction and the combine, s+1 for the force, s+2 and s+3 for the lambda windows and the
// moments, s+4 in flight (issued when step s begins, after the barrier that ends the use of row s-1).  Cells are padded so that the force tasks of neighbouring cells fall on consecutive
// banks: cell stride = Q1 pairs modulo 128 bytes.
//
// CG: groups of threads that share the strip's columns; XW: warps beside those that own velocities.  A
// small velocity set (one warp) takes a warp per column and three for the roles of the rows ahead where
// the grid leaves SMs idle: a step then takes the time of its longest part, not of their sum, and double
// precision gets all of an SM's FP64 units.  The xi walk of a single column reconstructs two interfaces,
// five for four columns, so it costs a sixth more arithmetic; the values are the same.
template <typename real, int Q0, int Q1, int CG, int XW>
struct ChanSmem {
  using S = ChanShape<Q0, Q1>;
  using Tab = ChanTables<real, Q0, Q1>;
  static constexpr bool F32 = sizeof(real) == 4;
  static constexpr int TP = S::TP;
  static constexpr int NT = S::V * CG + 32 * XW;
  static constexpr int NRING = 5;
  static constexpr int RC = TP + 6;  // cells of a ring row
  static constexpr int NEQ = 4;      // equilibrium records (rows s .. s+3)
  static constexpr int NRES = 2;     // inflow factors (rows s+1, s+2)
  static constexpr size_t al(size_t x) { return (x + 15) & ~size_t(15); }
  static constexpr size_t rowb = size_t(S::ROW) * sizeof(real);
  static constexpr size_t pad = (size_t(Q1) * 2 * sizeof(real)) % 128;
  static constexpr int CS = int((rowb + pad) / sizeof(real));  // reals from cell to cell, in the ring and in lbl
  static constexpr int XS = 2 * Q1 + 2;                        // reals from row i to row i+1 of a cell in lbx
  static constexpr size_t bar_off = 0;  // one mbarrier per ring slot
  static constexpr size_t tab_off = 64;
  static constexpr size_t ring_off = al(tab_off + sizeof(Tab));
  static constexpr size_t geo_off = ring_off + size_t(NRING) * RC * CS * sizeof(real);
  static constexpr size_t lbl_off = geo_off + size_t(NRING) * TP * sizeof(ChanCell<real>);
  static constexpr size_t lbx_off = lbl_off + size_t(2) * TP * CS * sizeof(real);
  static constexpr size_t eq_off = al(lbx_off + size_t(2) * TP * Q0 * XS * sizeof(real));
  static constexpr size_t res_off = al(eq_off + size_t(NEQ) * TP * S::EQW * sizeof(real));
  static constexpr size_t resn_off = al(res_off + size_t(NRES) * 2 * Q1 * sizeof(real));
  static constexpr size_t mvs_off = al(resn_off + size_t(NRES) * 2 * sizeof(real));
  static constexpr size_t wred_off = al(mvs_off + size_t(TP + 2) * 4 * MAXN * sizeof(real));
  static constexpr size_t nwv_off = al(wred_off + size_t(2) * TP * S::NW * sizeof(real));  // two wall sums
  static constexpr size_t bytes = al(nwv_off + size_t(TP) * sizeof(double));
  static_assert(rowb % 128 == 0 && pad % 16 == 0, "cells are bulk copies");
  static_assert((TP * sizeof(ChanCell<real>)) % 16 == 0, "geometry rows are bulk copies");
  static_assert(ring_off % 16 == 0 && geo_off % 16 == 0 && lbl_off % 16 == 0 && lbx_off % 16 == 0, "alignment");
  static_assert(NRING * sizeof(uint64_t) <= tab_off, "mbarriers fit before the tables");
  static_assert((NEQ & (NEQ - 1)) == 0 && (NRES & (NRES - 1)) == 0, "record slots by mask");
  // CTAs a SM the registers are sized for (228 KB of shared memory, 1 KB of it per CTA; single
  // precision: 168 registers a thread for four columns, 80 for one).  How many the device holds is
  // asked of the driver (channel_kernels).
  static constexpr int fit = int((228 * 1024) / (bytes + 1024));
  static constexpr int regs = CG == 1 ? 168 : 96;
  static constexpr int min_ctas = sizeof(real) == 8 ? 1 : (fit * NT * regs <= 65536 ? fit : 65536 / (NT * regs));
};

// Coefficients of a packed contraction: single precision holds each duplicated into a pair, the
// operand of a packed fma over (f', f''); double precision holds them once.
template <typename real>
struct CoefOf {
  using type = float2;
};
template <>
struct CoefOf<double> {
  using type = double;
};
__device__ __forceinline__ float2 k_mul(float2 k, float2 x) { return p_mul(k, x); }
__device__ __forceinline__ float2 k_fma(float2 k, float2 x, float2 a) { return p_fma(k, x, a); }
__device__ __forceinline__ double2 k_mul(double k, double2 x) { return p_mul(p_set(k), x); }
__device__ __forceinline__ double2 k_fma(double k, double2 x, double2 a) { return p_fma(p_set(k), x, a); }

// Force matrices of the channel.  On each axis K = d/dp and Kt = d/dp (p .) of the projected
// expansions satisfy
//   Kt = K diag(p) + z v^T:
// multiplying the expansion by p raises its degree by one, and its top term is a multiple of the
// polynomial that vanishes on the nodes; on the full range its derivative is projected out
// (z = 0), on the half range the projection of the jump at p = 0 leaves a rank-1 term.  So
//   wa K f + wb Kt f = K ((wa + wb p) f) + wb (v . f) z,
// one contraction in place of two.  K is split by the reflection of its axis (see KArgs): with J
// the permutation p -> -p, K J = -J K, and with e = f + J f, o = f - J f (k over half the nodes)
//   P[i][k] = (K[i][k] + K[i][Jk]) / 2,  M[i][k] = (K[i][k] - K[i][Jk]) / 2,
//   (K f)_i = P e + M o,  (K f)_Ji = M o - P e;  z and v are odd (v_Jk = -v_k).
// The block travels as a kernel parameter: the coefficients are uniform constant-bank operands.
template <typename real, int Q0, int Q1>
struct ChanKP {
  using C = typename CoefOf<real>::type;
  static constexpr int H0 = Q0 / 2, H1 = Q1 / 2;
  C P0[H0 * H0], M0[H0 * H0], p0[H0], v0[H0], z0[H0];
  C P1[H1 * H1], M1[H1 * H1], p1[H1], v1[H1], z1[H1];
};

// wa K f + wb Kt f of one line of 2 H nodes: node k of the first half at F + k sF, its mirror at
// Fm + k sM; results likewise to O, Om.  Everything is in pairs (f', f'').
template <typename real, int H, bool RANK1, typename C>
__device__ __forceinline__ void force_line(const C* __restrict__ Pm, const C* __restrict__ Mm, const C* __restrict__ pk,
                                           const C* __restrict__ vk, const C* __restrict__ zk, const real* F,
                                           const real* Fm, int sF, int sM, real wa, real wb, real* O, real* Om, int sO,
                                           int sOm) {
  using P = pair_t<real>;
  const P WA = p_set(wa), WB = p_set(wb), NWB = p_set(-wb);
  P e[H], o[H], t = p_set(real(0));
#pragma unroll
  for (int k = 0; k < H; ++k) {
    const P f = p_load(F + k * sF), g = p_load(Fm + k * sM);
    // (wa + wb p) f at the node, (wa - wb p) g at its mirror
    const P a = p_mul(k_fma(pk[k], WB, WA), f), b = k_fma(pk[k], NWB, WA);
    e[k] = p_fma(b, g, a);
    o[k] = p_sub(a, p_mul(b, g));
    if constexpr (RANK1) t = k_fma(vk[k], p_sub(f, g), t);
  }
  if constexpr (RANK1) t = p_mul(t, WB);
#pragma unroll
  for (int i = 0; i < H; ++i) {
    P A, B = k_mul(Mm[i * H], o[0]);
    if constexpr (RANK1) A = k_fma(Pm[i * H], e[0], k_mul(zk[i], t));
    else A = k_mul(Pm[i * H], e[0]);
#pragma unroll
    for (int k = 1; k < H; ++k) {
      A = k_fma(Pm[i * H + k], e[k], A);
      B = k_fma(Mm[i * H + k], o[k], B);
    }
    p_store(O + i * sO, p_add(B, A));
    p_store(Om + i * sOm, p_sub(B, A));
  }
}

// Moments (Eq. macro_red), tau = Kn / (n T) (Eq. canalie_tau) and the normalised truncated
// equilibrium (Sec. IV.D, reading 18) of four cells by one warp, eight lanes each: row holds the
// lane's cell's V pairs, mv is 4 MAXN reals of scratch, rec its record.  The mass sum is
// compensated in single precision.  Serial per cell, so it takes the whole warp's latency: four
// cells at once cost what one does.
template <typename real, int Q0, int Q1>
__device__ __forceinline__ void channel_equilibrium(const ChanTables<real, Q0, Q1>& tb, const real* row, real* mv,
                                                    real* rec, real ikn) {
  constexpr bool F32 = sizeof(real) == 4;
  constexpr int RP = Q0 / 8, FP = (Q0 + Q1 + 7) / 8;  // rows i and factors per lane
  const int h = threadIdx.x & 7;
  // sum over the lane's rows i = h + 8 r: the p^xi weights are uniform, p^lambda enters per row
  real sn = 0, sr = 0, sp = 0, se = 0;
#pragma unroll
  for (int r = 0; r < RP; ++r) {
    const real* f = row + 2 * (h + 8 * r) * Q1;
    const real pr = tb.p0[h + 8 * r];
    real n = 0;
#pragma unroll
    for (int j = 0; j < Q1; ++j) {
      const pair_t<real> x = p_load(f + 2 * j);
      const real pj = tb.p1[j], t = pj * x.x;
      n += x.x;
      sp += t;
      se += pj * t + x.y;
    }
    sn += n;
    sr += pr * n;
    se += pr * pr * n;
  }
  sr = group_sum<8>(sr), sp = group_sum<8>(sp), se = group_sum<8>(se);
  real nn, th, tl;  // th + tl: the cell's mass that f_eq - R has to carry
  if constexpr (F32) {
    float e = 0.f, nh, nlo;
    group_sum_comp<8>(sn, e);
    two_sum(sn, tb.ref_hi[0], nh, nlo);
    nn = nh + (nlo + (e + tb.ref_lo[0]));
    two_sum(sn, tb.ref_sum[0], th, tl);
    tl = tl + (e + tb.ref_sum[1]);
  } else {
    nn = group_sum<8>(sn) + tb.ref_hi[0];
    th = nn, tl = 0.0;
  }
  const real inv = rcp_rn(nn);
  const real u0 = (sr + (tb.ref_hi[1] + tb.ref_lo[1])) * inv, u1 = (sp + (tb.ref_hi[2] + tb.ref_lo[2])) * inv;
  const real T = ((se + (tb.ref_hi[3] + tb.ref_lo[3])) * inv - (u0 * u0 + u1 * u1)) * (real(1) / real(3));
  if (h < 4) {  // moment vectors [axis][side]; axis 0 is half range
    const real u = (h & 2 ? u1 : u0) * (h & 1 ? real(-1) : real(1));
    eq_moments_fast<real>(h & 2 ? tb.kind1 : 1, tb.nmax, u, T, mv + h * MAXN);
  }
  __syncwarp();
  real g[FP], a0 = real(0), a1 = real(0);
  const real* m[FP];
#pragma unroll
  for (int q = 0; q < FP; ++q) {
    const int k = h + 8 * q;  // axis 0 for q < RP
    g[q] = real(0);
    m[q] = mv + (q < RP ? (k >= Q0 / 2 ? 1 : 0) : 2 + (tb.kind1 == 1 && k - Q0 >= Q1 / 2 ? 1 : 0)) * MAXN;
  }
#pragma unroll 1
  for (int s = 0; s <= tb.nmax; ++s)
#pragma unroll
    for (int q = 0; q < FP; ++q)
      if (h + 8 * q < Q0 + Q1) g[q] += tb.tab[s * (Q0 + Q1) + h + 8 * q] * m[q][s];
#pragma unroll
  for (int q = 0; q < FP; ++q) {
    if (q < RP) g[q] *= nn, a0 += g[q];
    else a1 += g[q];
  }
  a0 = group_sum<8>(a0), a1 = group_sum<8>(a1);
  // g0 <- g0 target / (sum g0 sum g1); single precision: g0 (1 - delta), the target in float-float
  real scale;
  if constexpr (F32) {
    const float Ah = a0 * a1, Al = fmaf(a0, a1, -Ah);
    scale = (__fsub_rn(Ah, th) + (Al - tl)) * rcp_rn(Ah);
  } else {
    scale = th / (a0 * a1);
  }
#pragma unroll
  for (int q = 0; q < FP; ++q) {
    real val = g[q];
    if (q < RP) {
      if constexpr (F32) val = fmaf(-val, scale, val);
      else val *= scale;
    }
    if (h + 8 * q < Q0 + Q1) p_store(rec + 2 * (h + 8 * q), p_make(val, val));
  }
  if (h == 0) {
    const real nit = -(nn * T * ikn);
    p_store(rec + 2 * (Q0 + Q1), p_make(real(1), T));
    p_store(rec + 2 * (Q0 + Q1) + 2, p_make(nit, nit));
    p_store(rec + 2 * (Q0 + Q1) + 4, p_make(u1, real(0)));
  }
  __syncwarp();
}

// ------------------------------------------------------------------ the stage kernel
// Device cell (s, p) of the channel is s * n_xi + p (xi fastest).
//
// HX: axis 1 is half range (its mirror node is k + Q1/2 and its Kt has the rank-1 term).
//
// CLB runs the Cartesian-split formulation (Sec. VII.G, Eq. canalie_coord_beq_cons) on the
// same march: momenta (p^x, p^y) on the model's axes, no force term, fluxes of F = D + R, and
// the geometry record read as V^lambda = am p^x - glxl p^y at s - 1/2 and ap p^x - glxx p^y at
// s + 1/2 (a = 1 / (1 + phi), glxl / glxx = a lambda phi' at the interfaces), V^xi = b p^y
// (c = 0).  The lambda upwind side and the wall's incoming half-plane (Eq. canalie_coord_nw)
// then depend on the column and the interface: the lambda window holds the six cells around an
// interface and the walk's terms are formed per interface from the five of the upwind side.
template <typename real, int Q0, int Q1, int CG, int XW, bool CLB, bool HX>
__global__ void __launch_bounds__(ChanSmem<real, Q0, Q1, CG, XW>::NT, ChanSmem<real, Q0, Q1, CG, XW>::min_ctas)
    channel_stage_kernel(const __grid_constant__ ChanArgs<real> a, const __grid_constant__ ChanKP<real, Q0, Q1> kp) {
  using S = ChanShape<Q0, Q1>;
  using L = ChanSmem<real, Q0, Q1, CG, XW>;
  using Tab = ChanTables<real, Q0, Q1>;
  using P = pair_t<real>;
  constexpr int V = S::V, ROW = S::ROW, EQW = S::EQW, TP = S::TP, NW = S::NW, CPT = TP / CG;
  constexpr int NRING = L::NRING, RC = L::RC, CS = L::CS, XS = L::XS;
  extern __shared__ __align__(128) unsigned char smem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool col = XW == 0 || tid < V * CG;  // owns a velocity of CPT columns, from c0
  const int v = !col ? lane : CG == 1 ? tid : tid % V;
  const int c0 = CG == 1 || !col ? 0 : tid / V * CPT;
  const int i = v / Q1, j = v - i * Q1;

  const int nl = a.nl, nx = a.nx;
  const int nstrips = nx / TP;
  const int strip = blockIdx.x % nstrips, seg = blockIdx.x / nstrips;
  const int p0 = strip * TP;
  const int sA = seg * a.seglen, sB = min(sA + a.seglen, nl);
  const bool inlet = p0 == 0, outlet = p0 + TP == nx;
  const bool need_fl = a.ca.x != real(0);
  const int rlast = min(sB + 2, nl - 1);  // last row a segment reads
  const int pa = max(p0 - 3, 0), pb = min(p0 + TP + 3, nx);  // xi cells of a ring row in memory

  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + L::bar_off);  // [NRING]: the row of the slot has landed
  const Tab& tb = *reinterpret_cast<const Tab*>(smem + L::tab_off);
  real* ring = reinterpret_cast<real*>(smem + L::ring_off);                      // [NRING][RC][CS]
  ChanCell<real>* gring = reinterpret_cast<ChanCell<real>*>(smem + L::geo_off);  // [NRING][TP]
  real* lbl = reinterpret_cast<real*>(smem + L::lbl_off);                        // [2][TP][CS]: lambda force
  real* lbx = reinterpret_cast<real*>(smem + L::lbx_off);                        // [2][TP][Q0][XS]: xi force
  real* eqr = reinterpret_cast<real*>(smem + L::eq_off);                         // [NEQ][TP][EQW]
  real* resr = reinterpret_cast<real*>(smem + L::res_off);                       // [NRES][2][Q1]
  real* resn = reinterpret_cast<real*>(smem + L::resn_off);                      // [NRES][2] inflow densities
  real* mvs = reinterpret_cast<real*>(smem + L::mvs_off);                        // [TP+2][4][MAXN]
  real* wred = reinterpret_cast<real*>(smem + L::wred_off);                      // [2][TP][NW]
  double* nwv = reinterpret_cast<double*>(smem + L::nwv_off);                    // [TP]

  auto dcell = [&](int s, int p) -> size_t { return size_t(s) * nx + p; };
  auto slot = [&](int r) -> int { return (r - sA) % NRING; };
  // cell cc in [-3, TP + 3) of ring slot k
  auto cell = [&](int k, int cc) -> real* { return ring + (k * RC + cc + 3) * CS; };
  int issued = -1;  // warp 0: the last row whose copies it has started
  // row r with its halo (one bulk copy per cell: cells are padded) and its geometry, by warp 0
  auto row_issue = [&](int r) {
    const int k = slot(r), n = pb - pa;
    issued = r;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (lane == 0) mbar_expect_tx(bar + k, unsigned(n * L::rowb + TP * sizeof(ChanCell<real>)));
    __syncwarp();
    if (lane < n) bulk_g2s(cell(k, pa - p0 + lane), a.Fprev + dcell(r, pa + lane) * ROW, unsigned(L::rowb), bar + k);
    if (lane == n) bulk_g2s(gring + k * TP, a.geo + dcell(r, p0), unsigned(TP * sizeof(ChanCell<real>)), bar + k);
  };
  auto row_wait = [&](int r) -> bool { return mbar_wait(bar + slot(r), unsigned((r - sA) / NRING) & 1u, a.max_polls); };

  // ---- prologue: tables and rows sA .. sA+3 (the tables are no kernel's output; the rows and
  // everything below are read and written once the launch before this one is complete)
  grid_launch_dependents();
  if (tid == 0) {
    for (int k = 0; k < NRING; ++k) mbar_init(bar + k, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  {
    const uint4* src = reinterpret_cast<const uint4*>(a.tables);
    uint4* dst = reinterpret_cast<uint4*>(smem + L::tab_off);
    for (int x = tid; x < int(sizeof(Tab) / 16); x += L::NT) dst[x] = src[x];
  }
  __syncthreads();
  grid_dependency_wait();
  if (warp == 0)
    for (int r = sA; r <= min(sA + 3, rlast); ++r) row_issue(r);

  // per-thread constants; the walks' values are scaled by sc, their results by isc
  const real isc = tb.isc0[i] * tb.isc1[j];
  const P SC = p_set(tb.sc0[i] * tb.sc1[j]);
  const real pl = tb.p0[i], px = tb.p1[j];
  const real plI = pl * isc, pxI = px * isc;
  const P PLI = p_set(plI);
  const real Rij = tb.w0[i] * tb.w1[j];
  const P NR = p_set(-Rij);
  const bool lpos = pl >= real(0);
  const int off = lpos ? 0 : 1;  // the lambda window of step s is centred on row s + off
  const real T0 = a.T0;
  WenoSide<real> wl;
  wl.set(CLB || lpos);  // (the Cartesian split's windows are in upwind order)

  bool good = true;  // every wait of this thread so far ended in time
  // a wait ran out: let the copies in flight land (bounded), then leave together
  auto give_up = [&]() {
    if (tid == 0) {
      atomicOr(a.err, ERR_TIMEOUT);
      for (int r = max(sA, issued - NRING + 1); r <= issued; ++r) row_wait(r);
    }
    __syncthreads();
  };
  for (int r = sA; r <= min(sA + 3, rlast); ++r) good = row_wait(r) && good;
  if (!__syncthreads_and(good)) {
    give_up();
    return;
  }

  // ---- the roles of the rows ahead, by warp: with six warps, 0 and 1 contract along lambda, 2 and 3
  // along xi, 4 takes the equilibria, 5 the inflow factors; with extra warps they share the same;
  // else the one warp takes all in turn.
  constexpr bool SPLIT = NW >= 6;
  static_assert(CG == 1 || XW == 3, "column groups come with extra warps");
  static_assert(XW == 0 || XW == 3, "extra warps: lambda, xi, equilibria and inflow");
  constexpr int CW = NW * CG;  // column warps
  constexpr int WL = SPLIT ? 0 : XW ? CW : 0, WX = SPLIT ? 2 : XW ? CW + 1 : 0, WE = SPLIT ? 4 : XW ? CW + 2 : 0,
                WR = SPLIT ? 5 : WE, FW = SPLIT ? 2 : 1;  // their first warps; warps of a contraction
  auto force_row = [&](int r) {
    if constexpr (!CLB) {
      const int k = slot(r);
      real* ol = lbl + (r & 1) * TP * CS;
      real* ox = lbx + (r & 1) * TP * Q0 * XS;
      // Eq. (canalie_boltz): G_lxx (p^xi)^2 K0 f + G_lxl p^xi Kt0 f along lambda,
      // -G_lxl (p^lambda)^2 K1 f - G_lxx p^lambda Kt1 f along xi
      if (warp >= WL && warp < WL + FW)
        for (int t = tid - 32 * WL; t < TP * Q1; t += 32 * FW) {
          const int cc = t / Q1, jj = t - cc * Q1;
          const ChanCell<real>& g = gring[k * TP + cc];
          const real pj = tb.p1[jj];
          const real* F = cell(k, cc) + 2 * jj;
          real* O = ol + cc * CS + 2 * jj;
          force_line<real, Q0 / 2, true>(kp.P0, kp.M0, kp.p0, kp.v0, kp.z0, F, F + Q0 * Q1, 2 * Q1, 2 * Q1,
                                         g.glxx * pj * pj, g.glxl * pj, O, O + Q0 * Q1, 2 * Q1, 2 * Q1);
        }
      if (warp >= WX && warp < WX + FW)
        for (int t = tid - 32 * WX; t < TP * Q0; t += 32 * FW) {
          const int cc = t / Q0, ii = t - cc * Q0;
          const ChanCell<real>& g = gring[k * TP + cc];
          const real pi = tb.p0[ii];
          const real* F = cell(k, cc) + 2 * ii * Q1;
          real* O = ox + (cc * Q0 + ii) * XS;
          constexpr int M = HX ? Q1 : 2 * (Q1 - 1), sM = HX ? 2 : -2;  // mirror of node 0, step
          force_line<real, Q1 / 2, HX>(kp.P1, kp.M1, kp.p1, kp.v1, kp.z1, F, F + M, 2, sM, -g.glxl * pi * pi,
                                       -g.glxx * pi, O, O + M, 2, sM);
        }
    }
  };
  auto eq_row = [&](int r) {
    if (warp != WE) return;
    const int cc = lane >> 3;
    channel_equilibrium<real, Q0, Q1>(tb, cell(slot(r), cc), mvs + cc * 4 * MAXN,
                                      eqr + ((r & (L::NEQ - 1)) * TP + cc) * EQW, a.ikn);
  };
  // inflow factors g_xi(u^xi, T0) of row r at one end: reservoirs, u^xi of the adjacent
  // cell; flow-rate ends, u^xi = Q_s and the density n_s of Eq. (canalie_inlet_s)
  auto res_job = [&](int r, int end) {
    const int cc = end == 0 ? 0 : TP - 1, rs = r & (L::NRES - 1);
    const real ures = a.flow ? a.qflow[(2 * end) * nl + r] : eqr[((r & (L::NEQ - 1)) * TP + cc) * EQW + 2 * (Q0 + Q1) + 4];
    real* mv = mvs + (TP + end) * 4 * MAXN;
    if (lane < 2) eq_moments_fast<real>(tb.kind1, tb.nmax, lane ? -ures : ures, T0, mv + lane * MAXN);
    __syncwarp();
    if (lane < Q1) {
      const real* m = mv + ((tb.kind1 == 1 && lane >= Q1 / 2) ? 1 : 0) * MAXN;
      real g = real(0);
      for (int s = 0; s <= tb.nmax; ++s) g += tb.tab[s * (Q0 + Q1) + Q0 + lane] * m[s];
      resr[(rs * 2 + end) * Q1 + lane] = g;
    }
    __syncwarp();
    if (a.flow) {
      // n_s sum_{entering} V f'_eq(1, (0, Q_s), T0) + sum_{leaving} V f'_adjacent = (1 + phi) Q_s,
      // V = b p^xi - c p^lambda of the end interface (the decision of fill_ghosts); FP64 sums as for n_w
      const int k = slot(r);
      const ChanCell<real>& gk = gring[k * TP + cc];
      const real bb = end == 0 ? gk.bm : gk.bp, cq = end == 0 ? gk.cm : gk.cp;
      const real* Fa = cell(k, cc);
      const real* gr = resr + (rs * 2 + end) * Q1;
      double lv = 0.0, en = 0.0;
      for (int vv = lane; vv < V; vv += 32) {
        const int ii = vv / Q1, jj = vv - ii * Q1;
        const real Vx = bb * tb.p1[jj] - cq * tb.p0[ii];
        const bool into = end == 0 ? (Vx > real(0)) : (Vx < real(0));
        if (into) en += double(Vx) * double(tb.gw0[ii] * gr[jj]);
        else lv += double(Vx) * (double(Fa[2 * vv]) + double(tb.w0[ii]) * double(tb.w1[jj]));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        lv += __shfl_xor_sync(0xffffffffu, lv, o);
        en += __shfl_xor_sync(0xffffffffu, en, o);
      }
      if (lane == 0) resn[rs * 2 + end] = real((double(a.qflow[(2 * end + 1) * nl + r]) - lv) / en);
      __syncwarp();
    }
  };
  auto res_row = [&](int r) {
    if (!(inlet || outlet) || warp != WR) return;
#pragma unroll 1
    for (int end = 0; end < 2; ++end)
      if (end == 0 ? inlet : outlet) res_job(r, end);
  };
  // reservoir halo cells of row r past an end strip (the bulk copy leaves them out): populations
  // entering the domain see f_eq(n_res, (0, u^xi), T0) - R, the others the adjacent cell (zeroth order)
  auto fill_ghosts = [&](int r) {
    const int k = slot(r), rs = r & (L::NRES - 1);
#pragma unroll
    for (int end = 0; end < 2; ++end) {
      if (!(end == 0 ? inlet : outlet) || (CG > 1 && c0 != (end == 0 ? 0 : TP - CPT))) continue;
      const int ce = end == 0 ? 0 : TP - 1;
      const ChanCell<real>& g = gring[k * TP + ce];
      const real Vx = end == 0 ? g.bm * px - g.cm * pl : g.bp * px - g.cp * pl;
      P q;
      if (end == 0 ? (Vx > real(0)) : (Vx < real(0))) {
        const real nres = a.flow ? resn[rs * 2 + end] : (end == 0 ? a.n_in : a.n_out);
        const real e = nres * tb.gw0[i] * resr[(rs * 2 + end) * Q1 + j];
        q = p_make(e - Rij, e * T0 - Rij);
      } else {
        q = p_load(cell(k, ce) + 2 * v);
      }
      for (int d = 1; d <= 3; ++d) p_store(cell(k, end == 0 ? -d : TP - 1 + d) + 2 * v, q);
    }
  };

  // ---- lambda windows.  Value of row r of column c at or below row sA + 2: the ring, global
  // memory below the segment, the centreline mirror below row 0 (ghost 1-k of cell k,
  // p^lambda -> -p^lambda, Sec. VII.C.3)
  auto low_row = [&](int r, int c) -> P {
    if (r >= sA) return p_load(cell(slot(r), c) + 2 * v);
    if (r >= 0) return p_load(a.Fprev + dcell(r, p0 + c) * ROW + 2 * v);
    return p_load(cell(slot(-1 - r), c) + 2 * (refl(1, Q0, i) * Q1 + j));
  };
  // vielbein: the window centred on row s + off; Cartesian split: F(s-2 .. s+3) of step s (scaled).
  // Before the march's pass sA - 1, which brings in one row more and reconstructs interface sA - 1/2.
  WenoWin<real, !L::F32> win[CLB ? 1 : CPT];
  P raw[CLB ? CPT : 1][6];
  P flo[CPT];  // lambda interface s - 1/2 (scaled)
  if (col)
#pragma unroll
  for (int c = 0; c < CPT; ++c) {
    const int cc = c0 + c;
    if constexpr (CLB) {
#pragma unroll
      for (int q = 1; q < 6; ++q) raw[c][q] = p_mul(low_row(sA - 4 + q, cc), SC);
    } else {
      const int b = sA - 3 + off;
      const P x = p_mul(low_row(b, cc), SC);  // (its lower neighbour's terms leave the window at once)
      win[c].start(x, x, p_mul(low_row(b + 1, cc), SC), p_mul(low_row(b + 2, cc), SC), p_mul(low_row(b + 3, cc), SC));
    }
    flo[c] = p_set(real(0));
  }
  // Cartesian split: the window of the interface between w[2] and w[3] in upwind order
  auto clb_win = [](const P* w, bool up) -> WenoWin<real, false> {
    WenoWin<real, false> t;
    t.start(p_sel(up, w[0], w[5]), p_sel(up, w[1], w[4]), p_sel(up, w[2], w[3]), p_sel(up, w[3], w[2]),
            p_sel(up, w[4], w[1]));
    return t;
  };
  // ---- the wall (Sec. VII.C.4), when the march first needs row nl: n_w per column from the
  // zero-mass-flux balance; rows nl-3 .. nl-1 stay in the ring from there on
  auto wall_out = [&](int c) -> bool {  // this velocity leaves through the wall
    if constexpr (CLB) {
      const ChanCell<real>& gw = gring[slot(nl - 1) * TP + c];
      return gw.ap[0] * pl - gw.glxx * px > real(0);
    } else {
      return pl > real(0);
    }
  };
  // any row of the lambda stencils, once wall_density has run where it lies beyond the wall
  auto any_row = [&](int r, int c) -> P {
    if (r >= nl) return p_load(cell(slot(min(r, nl + 1)), c) + 2 * v);
    const int vv = r < 0 ? refl(1, Q0, i) * Q1 + j : v;
    return p_load(a.Fprev + dcell(r < 0 ? -1 - r : r, p0 + c) * ROW + 2 * vv);
  };
  // ghosts of rows nl (G1) and nl+1, nl+2 (G2) of the populations leaving column c: quadratic
  // extrapolation (Eq. extrapol)
  auto extrapolate = [&](int c, P& G1, P& G2) {
    const P F3 = p_load(cell(slot(nl - 3), c) + 2 * v), F2 = p_load(cell(slot(nl - 2), c) + 2 * v),
            F1 = p_load(cell(slot(nl - 1), c) + 2 * v);
    G1 = p_add(p_sub(p_mul(p_set(real(3)), F1), p_mul(p_set(real(3)), F2)), F3);
    G2 = p_add(p_sub(p_mul(p_set(real(6)), F1), p_mul(p_set(real(8)), F2)), p_mul(p_set(real(3)), F3));
  };
  // The wall's n_w, and its ghost rows into the ring slots of rows nl and nl + 1 (rows nl-5 and
  // nl-4 have left them; row nl + 2 reads as nl + 1): each thread its own velocity
  auto wall_density = [&]() {
    if (col)
#pragma unroll 1
    for (int c = c0; c < c0 + CPT; ++c) {
      real fl = real(0), fd = real(0);
      const bool out = wall_out(c);
      real Vw = pl;
      if constexpr (CLB) {
        // V^lambda at the wall interface (row nl-1's upper face); the outgoing flux is of F = D + R,
        // the incoming one of f_eq(1, 0, T0), both over this column's half-planes (Eq. canalie_coord_nw)
        const ChanCell<real>& gw = gring[slot(nl - 1) * TP + c];
        Vw = gw.ap[0] * pl - gw.glxx * px;
        if (!out) fd = tb.gw0[i] * tb.gw1[j] * Vw;
      }
      if (out) {
        WenoWin<real, false> t;
        P G1, G2;
        extrapolate(c, G1, G2);
        t.start(p_mul(p_load(cell(slot(nl - 3), c) + 2 * v), SC), p_mul(p_load(cell(slot(nl - 2), c) + 2 * v), SC),
                p_mul(p_load(cell(slot(nl - 1), c) + 2 * v), SC), p_mul(G1, SC), p_mul(G2, SC));
        fl = (t.face_any(true).x * isc + (CLB ? Rij : real(0))) * Vw;
      }
      __syncwarp();
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        fl += __shfl_xor_sync(0xffffffffu, fl, o);
        if constexpr (CLB) fd += __shfl_xor_sync(0xffffffffu, fd, o);
      }
      if (lane == 0) wred[c * NW + (v >> 5)] = fl, wred[(TP + c) * NW + (v >> 5)] = fd;
    }
    __syncthreads();
    if (tid < TP) {
      double num = CLB ? 0.0 : tb.ref_flux_pos;  // vielbein: the outgoing flux of R, then of D
      double den = CLB ? 0.0 : tb.wall_den;
      for (int w = 0; w < NW; ++w) {
        num += double(wred[v * NW + w]);
        if (CLB) den += double(wred[(TP + v) * NW + w]);
      }
      const double nwc = -num / den;  // Eq. (nw) / (canalie_coord_nw)
      nwv[v] = nwc;
      a.nw[p0 + v] = nwc;
      if (!isfinite(nwc)) atomicOr(a.err, ERR_NONFINITE);
    }
    __syncthreads();
    if (col)
#pragma unroll 1
    for (int c = c0; c < c0 + CPT; ++c) {
      P G1, G2;
      if (wall_out(c)) {
        extrapolate(c, G1, G2);
      } else {  // f_eq(n_w, 0, T0) - R (Eq. weno_populate)
        const real e = real(nwv[c]) * tb.gw0[i] * tb.gw1[j];
        G1 = G2 = p_make(e - Rij, e * T0 - Rij);
      }
      p_store(cell(slot(nl), c) + 2 * v, G1);
      p_store(cell(slot(nl + 1), c) + 2 * v, G2);
    }
  };

  // this thread's F_l and F_out of the strip's first cell in row s; F_l is loaded one step ahead
  const real* Fl = a.Fl + dcell(sA, p0 + c0) * ROW + 2 * v;
  real* Fo = a.Fout + dcell(sA, p0 + c0) * ROW + 2 * v;
  const size_t rstep = size_t(nx) * ROW;
  P flr[CPT];
#pragma unroll
  for (int c = 0; c < CPT; ++c) {
    flr[c] = p_set(real(0));
    if (need_fl && col) flr[c] = p_load(Fl + c * ROW);
  }
  __syncthreads();

  // ---- the march.  Its first three passes only run the roles of the first rows; the third also
  // reconstructs the lambda interfaces sA - 1/2.
#pragma unroll 1
  for (int s = sA - 3; s < sB; ++s) {
    if (s >= sA - 1) {
    const bool full = s >= sA;
    if (full && warp == 0 && s + 4 <= rlast) row_issue(s + 4);
    if (s > sA && s + 3 <= rlast) good = row_wait(s + 3) && good;
    if (s == nl - 3) wall_density();
    if (col) {
    const int k0 = full ? slot(s) : 0;
    const int k3 = slot(min(s + 2 + (CLB ? 1 : off), nl + 1));  // the row that joins the lambda windows
    const ChanCell<real>* geo = gring + k0 * TP + c0;
    const P R2 = p_set(CLB ? Rij * SC.x : real(0));

    // ---- xi: V F (CLB: of F = D + R) at the five interfaces of the strip in one walk.  V^xi = b p^xi
    // - c p^lambda (Eq. canalie_V), times isc; an interface's upwind cell follows the last one's,
    // unless V^xi changes its sign between the two.
    P dphi[CPT];
    if (full) {
      auto xi_load = [&](int cc) -> P { return p_mul(p_load(cell(k0, c0 + cc) + 2 * v), SC); };
      auto xi_vel = [&](int c) -> real {
        const P bc = p_load(c < CPT ? &geo[c].bm : &geo[CPT - 1].bp);
        return bc.x * pxI - bc.y * plI;
      };
      auto flux = [&](real V, P f) -> P { return p_mul(p_set(V), CLB ? p_add(f, R2) : f); };
      WenoWin<real, true> wx;
      WenoSide<real> sx;
      WenoRange<real> range;
      real V = xi_vel(0);
      bool up = V >= real(0);
      sx.set(up);
      const real* q = cell(k0, c0 + (up ? -3 : -2)) + 2 * v;
      wx.start(p_mul(p_load(q), SC), p_mul(p_load(q + CS), SC), p_mul(p_load(q + 2 * CS), SC),
               p_mul(p_load(q + 3 * CS), SC), p_mul(p_load(q + 4 * CS), SC));
      P phi[CPT + 1];
      phi[0] = flux(V, wx.face(sx, range));
#pragma unroll
      for (int c = 1; c <= CPT; ++c) {
        V = xi_vel(c);
        if ((V >= real(0)) == up) {
          wx.push(p_mul(p_load(q + (4 + c) * CS), SC));
        } else {
          up = !up;
          sx.set(up);
          q += up ? -CS : CS;
          wx.start(p_mul(p_load(q + c * CS), SC), p_mul(p_load(q + (1 + c) * CS), SC), p_mul(p_load(q + (2 + c) * CS), SC),
                   p_mul(p_load(q + (3 + c) * CS), SC), p_mul(p_load(q + (4 + c) * CS), SC));
        }
        phi[c] = flux(V, wx.face(sx, range));
      }
      if (__any_sync(0xffffffffu, !range.ok())) {  // a face does not hold (see weno_holds)
#pragma unroll 1
        for (int c = 0; c <= CPT; ++c) {
          V = xi_vel(c);
          up = V >= real(0);
          const int n = up ? c - 1 : c;
          wx.start(xi_load(n - 2), xi_load(n - 1), xi_load(n), xi_load(n + 1), xi_load(n + 2));
          const P x = flux(V, wx.face_any(up));
          const int to = wx.in_range(up) ? -1 : c;
#pragma unroll
          for (int k = 0; k <= CPT; ++k) phi[k] = p_sel(k == to, x, phi[k]);
        }
      }
#pragma unroll
      for (int c = 0; c < CPT; ++c) dphi[c] = p_mul(p_load(geo[c].idx), p_sub(phi[c + 1], phi[c]));
    }

    // ---- lambda interface s + 1/2 of every column
    P fhi[CPT];
    WenoRange<real> range;
    auto lam_up = [&](int c) -> bool {  // upwind side of interface s + 1/2, Cartesian split
      const ChanCell<real>& g = geo[c];
      return (full ? g.ap[0] * pl - g.glxx * px : -(g.nam[0] * pl + g.glxl * px)) >= real(0);
    };
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
      const P fnew = p_mul(p_load(cell(k3, c0 + c) + 2 * v), SC);
      if constexpr (CLB) {
#pragma unroll
        for (int q = 0; q < 5; ++q) raw[c][q] = raw[c][q + 1];
        raw[c][5] = fnew;
        fhi[c] = clb_win(raw[c], lam_up(c)).face(wl, range);
      } else {
        win[c].push(fnew);
        fhi[c] = win[c].face(wl, range);
      }
    }
    if (__any_sync(0xffffffffu, !range.ok())) {
#pragma unroll 1
      for (int c = 0; c < CPT; ++c) {
        // from memory: the windows' older terms are not kept
        const bool up = CLB ? lam_up(c) : lpos;
        const int b = s + (up ? 0 : 1) - 2, cc = c0 + c;
        WenoWin<real, false> w;
        w.start(p_mul(any_row(b, cc), SC), p_mul(any_row(b + 1, cc), SC), p_mul(any_row(b + 2, cc), SC),
                p_mul(any_row(b + 3, cc), SC), p_mul(any_row(b + 4, cc), SC));
        const P x = w.face_any(up);
        const int to = w.in_range(up) ? -1 : c;
#pragma unroll
        for (int k = 0; k < CPT; ++k) fhi[k] = p_sel(k == to, x, fhi[k]);
      }
    }

    // ---- the combine of row s
    if (full) {
      const real* rec = eqr + ((s & (L::NEQ - 1)) * TP + c0) * EQW;
      const real* fb = lbl + ((s & 1) * TP + c0) * CS + 2 * v;
      const real* xb = lbx + (((s & 1) * TP + c0) * Q0 + i) * XS + 2 * j;
#pragma unroll
      for (int c = 0; c < CPT; ++c) {
        const ChanCell<real>& g = geo[c];
        P adv;
        if constexpr (CLB) {
          // Eq. (canalie_coord_beq_cons): fluxes of F = D + R, V^lambda per interface (no force term
          // balances the rest state's advection here)
          const real Vlm = g.nam[0] * plI + g.glxl * pxI, Vlp = g.ap[0] * plI - g.glxx * pxI;
          adv = p_add(p_fma(p_set(Vlp), p_add(fhi[c], R2), p_mul(p_set(Vlm), p_add(flo[c], R2))), dphi[c]);
        } else {
          // chi flux differences (Sec. VII.B)
          adv = p_fma(PLI, p_fma(p_load(g.ap), fhi[c], p_mul(p_load(g.nam), flo[c])), dphi[c]);
        }
        // L = -advection + force - (F - f_eq) / tau
        const real* rc = rec + c * EQW;
        const P deq = p_fma(p_mul(p_load(rc + 2 * i), p_load(rc + 2 * (Q0 + j))), p_load(rc + 2 * (Q0 + Q1)), NR);
        const P F = p_load(cell(k0, c0 + c) + 2 * v);
        P Lv = p_sub(p_mul(p_sub(F, deq), p_load(rc + 2 * (Q0 + Q1) + 2)), adv);
        if constexpr (!CLB) Lv = p_add(Lv, p_add(p_load(fb + c * CS), p_load(xb + c * Q0 * XS)));
        P o = p_fma(a.ccdt, Lv, F);
        if (need_fl) o = p_fma(a.ca, p_sub(flr[c], F), o);
        p_store(Fo + c * ROW, o);
      }
      Fl += rstep;
      Fo += rstep;
      if (need_fl && s + 1 < sB)
#pragma unroll
        for (int c = 0; c < CPT; ++c) flr[c] = p_load(Fl + c * ROW);
    }
#pragma unroll
    for (int c = 0; c < CPT; ++c) flo[c] = fhi[c];
    }
    }
    // ---- the rows ahead
    if (s + 3 < sB) eq_row(s + 3);
    if (s + 2 >= sA && s + 2 < sB) res_row(s + 2);
    if (s + 1 >= sA && s + 1 < sB) {
      force_row(s + 1);
      if (col && (inlet || outlet)) fill_ghosts(s + 1);
    }
    if (!__syncthreads_and(good)) {
      give_up();
      return;
    }
  }
}

}  // namespace vlb
