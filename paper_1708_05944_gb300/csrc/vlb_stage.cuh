// One TVD-RK3 stage of the chi-formulation circular Couette update, fused into
// one kernel per tile of up to TC cells of one instance (all momenta of those cells):
//
//   bulk-copy the tile, its three-cell halo and its cells' geometry to shared memory
//   -> moments per cell (Eq. macro_red), truncated equilibrium and tau; meanwhile,
//      on the warps without a cell, the inertial force
//      (1/R)[(p^phi)^2 K^R f - p^R K~^phi f] (Eq. boltz_couette_kom)
//   -> walls: extrapolated outgoing ghosts (Eq. extrapol), wall flux, n_w
//      (Eq. nw), incoming ghosts f_eq(n_w, u_w, T_w) (Eq. weno_populate)
//   -> WENO-5 fluxes along the cells, chi flux difference, BGK, RK3 combine
//      (Eqs. weno5_flux, flux_kom_R / flux_kom_eta, BGK, rk3) -> global.
//
// Every distribution buffer holds the deviation D = F - R from the rest state
// (ModelArgs): the operator is linear in R's part, which it leaves unchanged.
// A cell row holds Vp velocity pairs (f', f'') interleaved (see pair_t).
//
// What bounds it: latency (36 - 42 % of the issue slots, 35 % of the FP32 pipe, 20 warps a SM).  The
// walk of phase D takes WENO-5 on shared differences (WenoWin), phase A sums a row of nodes per
// lane: 285 -> 204 instructions per warp and cell-velocity row.  Single precision, 16 x 20
// velocities, a step: 256 instances of 64 .. 1024 cells 1.90 -> 1.51 ms, 5 x 1024 cells 90 -> 72 us;
// double precision 5 x 1024 cells 2.62 -> 1.84 ms.
#pragma once
#include <type_traits>

#include "vlb_device.cuh"

namespace vlb {

template <typename real>
struct StageArgs {
  const real* Fprev;  // distribution L acts on
  const real* Fl;     // F_l of the step (read when ca != 0)
  real* Fout;
  // Fout = ca F_l + (1 - ca) F_prev + cc dt L[F_prev], evaluated as
  // F_prev + ca (F_l - F_prev) + cc dt L so that the weights on F sum to exactly
  // one in any precision (float(1/3) + float(2/3) = 1 + 3e-8 would add that much
  // mass every step).
  double ca, cc;
  float caf, ccf;  // single-precision copies
  const InstDesc* inst;
  const TileDesc* tiles;
  int n_tiles;
  const GeoCell* geo;    // per global cell
  const GeoCellF* geof;  // single-precision copy
  double* nw;          // 2 per instance: inner, outer wall density
  const WallEq* wall;  // 2 per instance: inner, outer wall equilibrium
  const real* halo;    // 2 x 3 rows per instance: ghost cells of slab halo ends (InstDesc::halo)
  // the f~ formulation (the FT kernels): sqrt(g) per global cell and the inertial term of R per
  // velocity; geo / geof then hold e_{s+-1/2} / (d eta sqrt(g)) as cp / cm and 1 / R_s as inv_rbar
  const real* sqrtg;
  const real* forceR;
  unsigned* err;
  int Vp;              // velocities per cell row, padded (>= nq0 nq1, multiple of 4); a row holds 2 Vp reals
  int nbuf;            // tile buffers: 1, or 2 when a persistent CTA stages its next tile during this one
  unsigned long long max_polls;
};

// Shared-memory carve-up, identical on host and device: two mbarriers, nbuf tile
// buffers (the TC + 6 rows of a tile with its halo, then the geometry of its TC
// cells), the force buffer (TC rows), then doubles and reals.
template <typename real, int TC, int NT>
struct StageSmem {
  static constexpr int NW = NT / 32;
  using Geo = typename std::conditional<sizeof(real) == 4, GeoCellF, GeoCell>::type;
  __host__ __device__ static size_t tile_off() { return 16; }
  __host__ __device__ static size_t geo_off(int Vp) { return size_t(TC + 6) * 2 * Vp * sizeof(real); }
  __host__ __device__ static size_t buf_bytes(int Vp) { return geo_off(Vp) + size_t(TC) * sizeof(Geo); }
  __host__ __device__ static size_t lbuf_off(int Vp, int nbuf) { return tile_off() + size_t(nbuf) * buf_bytes(Vp); }
  __host__ __device__ static size_t dbl_off(int Vp, int nbuf) {
    size_t o = lbuf_off(Vp, nbuf) + size_t(TC) * 2 * Vp * sizeof(real);
    return (o + 15) & ~size_t(15);
  }
  // doubles: p0, p1 (MAXQ each), reduction (NW*4), wall equilibrium factors (2*MAXQ), scalars (16)
  static constexpr size_t n_dbl = 2 * MAXQ + NW * 4 + 2 * MAXQ + 16;
  __host__ __device__ static size_t real_off(int Vp, int nbuf) { return dbl_off(Vp, nbuf) + n_dbl * sizeof(double); }
  // reals: p0, p1, the two WENO scales (MAXQ each), tab0, tab1 (MAXQ*MAXN each), then pairs: n g_R and g_phi
  // (TC*MAXQ each), six pairs of per-cell values (TC); then moment vectors (TC*4*MAXN),
  // w0, w1 (MAXQ each)
  static constexpr size_t n_real = 4 * MAXQ + 2 * MAXQ * MAXN + 4 * TC * MAXQ + 12 * TC + TC * 4 * MAXN + 2 * MAXQ;
  __host__ __device__ static size_t bytes(int Vp, int nbuf) { return real_off(Vp, nbuf) + n_real * sizeof(real); }
};

// CTAs per SM the register allocation is sized for, where shared memory would
// allow them but the compiler, left alone, takes too many registers a thread.  A
// single-precision CTA of 256 to 384 threads needs at most about 64 KB of shared
// memory for tiles up to 8 cells (three fit on an SM) and about 100 KB for 16
// (two fit) with the model shapes that have fixed node counts.  In double precision the sets of
// up to 64 velocities run on CTAs of 64 threads, whose latency only other CTAs hide: left alone the
// compiler takes 172 to 184 registers, four CTAs a SM where shared memory holds five to seven
// (64 instances of 80 cells, 8 x 8 velocities, a step: 904 us, and 836 with five).
constexpr int stage_min_ctas(int real_bytes, int tc, int nt) {
  return real_bytes == 8 ? (nt == 64 ? 6 : 1) : nt >= 256 && nt <= 384 ? (tc <= 8 ? 3 : 2) : 1;
}

// FT: the f~ formulation (Sec. VI.B, Eqs. boltz_couette_cons / boltz_couette_str_cons).  The
// stencils act on F~ = sqrt(g) (D + R), held during phase D as F~ - R so that the walls' ghost
// rows (stored the same way) need no sqrt(g); the walls extrapolate F~; the flux difference
// takes e / (d eta sqrt(g)) and the force 1 / R_s, with the rest state's own advection and
// inertial term added (F~ is not a deviation).  The moments, equilibrium and BGK act on D.
template <typename real, int TC, int Q0MAX, int Q1MAX, int NT, bool EXACT, bool FT = false>
__global__ void __launch_bounds__(NT, stage_min_ctas(int(sizeof(real)), TC, NT))
    couette_stage_kernel(const __grid_constant__ StageArgs<real> a, const __grid_constant__ ModelArgs m,
                         const __grid_constant__ KArgs<real> kk) {
  using L = StageSmem<real, TC, NT>;
  constexpr int NW = L::NW;
  constexpr int VPC = (Q0MAX * Q1MAX + 3) / 4 * 4;
  extern __shared__ __align__(128) unsigned char smem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // exact instantiations fix node counts and strides at compile time; the generic one reads them
  const int nq0 = EXACT ? Q0MAX : m.nq0;
  const int nq1 = EXACT ? Q1MAX : m.nq1;
  const int V = nq0 * nq1;
  const int Vp = EXACT ? VPC : a.Vp;
  const int row = 2 * Vp;

  const int nbuf = a.nbuf;
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem);  // one mbarrier per tile buffer
  real* tile0 = reinterpret_cast<real*>(smem + L::tile_off());
  const size_t bstride = L::buf_bytes(Vp) / sizeof(real);  // reals per tile buffer
  real* lbuf = reinterpret_cast<real*>(smem + L::lbuf_off(Vp, nbuf));
  double* p0d = reinterpret_cast<double*>(smem + L::dbl_off(Vp, nbuf));
  double* p1d = p0d + MAXQ;
  double* red = p1d + MAXQ;
  double* gw0 = red + NW * 4;  // wall equilibrium factors
  double* gw1 = gw0 + MAXQ;
  double* mw = gw1 + MAXQ;     // [0] incoming equilibrium flux, [1] n_w
  real* p0r = reinterpret_cast<real*>(smem + L::real_off(Vp, nbuf));
  real* p1r = p0r + MAXQ;
  real* iw0 = p1r + MAXQ;  // powers of two next to 1 / w_i and 1 / w_j: the scale of the WENO walk
  real* iw1 = iw0 + MAXQ;
  real* tabr0 = iw1 + MAXQ;  // equilibrium tables in the bulk type, [s][k]
  real* tabr1 = tabr0 + MAXQ * MAXN;
  // per-cell values of phase D as ready pairs (both lanes of a packed operand)
  using P2 = pair_t<real>;
  P2* gRn = reinterpret_cast<P2*>(tabr1 + MAXQ * MAXN);  // [t][i] n_t g_{R,i} twice
  P2* gP = gRn + TC * MAXQ;                              // [t][j] g_{phi,j} twice
  // per cell: cp twice, -cm twice, 1/Rbar twice, -1/tau twice, (1, T), pad (16-byte loads)
  enum { C_CP = 0, C_NCM, C_IR, C_NTAU, C_1T, C_N = 6 };
  P2* crec = gP + TC * MAXQ;
  real* mv = reinterpret_cast<real*>(crec + C_N * TC);   // [t][axis*2 + side][s]
  real* w0r = mv + TC * 4 * MAXN;  // weights: R_ij = w0_i w1_j in the bulk type
  real* w1r = w0r + MAXQ;

  grid_launch_dependents();
  if (tid == 0) {
    mbar_init(bar, 1);
    mbar_init(bar + 1, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  constexpr bool F32 = sizeof(real) == 4;
  for (int x = tid; x < MAXQ; x += NT) {
    p0d[x] = m.p0[x];
    p1d[x] = m.p1[x];
    if constexpr (F32) {
      p0r[x] = m.p0f[x];
      p1r[x] = m.p1f[x];
      iw0[x] = x < nq0 ? weno_pow2_dev(m.iw0f[x]) : 1.0f;
      iw1[x] = x < nq1 ? weno_pow2_dev(m.iw1f[x]) : 1.0f;
      w0r[x] = m.w0f[x];
      w1r[x] = m.w1f[x];
    } else {
      p0r[x] = m.p0[x];
      p1r[x] = m.p1[x];
      iw0[x] = x < nq0 ? weno_pow2_dev(m.iw0[x]) : 1.0;
      iw1[x] = x < nq1 ? weno_pow2_dev(m.iw1[x]) : 1.0;
      w0r[x] = m.w0[x];
      w1r[x] = m.w1[x];
    }
  }
  for (int x = tid; x < MAXQ * MAXN; x += NT) {
    const int y = (x % MAXN) * MAXQ + x / MAXN;
    tabr0[y] = sizeof(real) == 4 ? real(m.tab0f[x]) : real(m.tab0[x]);
    tabr1[y] = sizeof(real) == 4 ? real(m.tab1f[x]) : real(m.tab1[x]);
  }
  // the next tile's descriptor is read during the current tile (its load latency hidden); it and the
  // instances are no kernel's output
  TileDesc td_next = blockIdx.x < a.n_tiles ? a.tiles[blockIdx.x] : TileDesc{0, 0, 0};
  asm volatile("prefetch.global.L1 [%0];" ::"l"(a.inst + td_next.inst));
  __syncthreads();
  // what the launch before this one wrote is read and what it read is written from here on
  // (dependent launches, see launch_dependent)
  grid_dependency_wait();
  const bool need_fl = a.caf != 0.0f;
  using Geo = typename L::Geo;
  const Geo* geo_src =
      reinterpret_cast<const Geo*>(F32 ? static_cast<const void*>(a.geof) : static_cast<const void*>(a.geo));
  // warp 0 stages tile tx (cells lo..hi-1 at slots lo-c0+3 ..., then its cells' geometry) into
  // buffer b with bulk copies that complete on the buffer's mbarrier
  auto stage_tile = [&](const TileDesc& t, int b) {
    const InstDesc i = a.inst[t.inst];
    const int lo = max(t.c0 - 3, 0), hi = min(t.c0 + t.nc + 3, i.n_cells);
    real* dst = tile0 + b * bstride;
    const unsigned rbytes = unsigned(row * sizeof(real)), gbytes = unsigned(t.nc * sizeof(Geo));
    if (lane == 0) mbar_expect_tx(bar + b, rbytes * unsigned(hi - lo) + gbytes);
    __syncwarp();
    for (int c = lo + lane; c < hi; c += 32)
      bulk_g2s(dst + (c - t.c0 + 3) * row, a.Fprev + size_t(i.cell0 + c) * row, rbytes, bar + b);
    if (lane == 0) bulk_g2s(dst + L::geo_off(Vp) / sizeof(real), geo_src + i.cell0 + t.c0, gbytes, bar + b);
  };
  unsigned phase = 0;  // bit b: parity of buffer b's next completion
  if (nbuf == 2 && warp == 0 && blockIdx.x < a.n_tiles) stage_tile(td_next, 0);
  // one tile per iteration: a launch with one CTA per tile runs the body once, a persistent
  // launch (grid sized by occupancy) walks the tile list, with two buffers staging the next
  // tile while this one is computed
  for (int tix = blockIdx.x, it = 0; tix < a.n_tiles; tix += gridDim.x, ++it) {
  const int b = nbuf == 2 ? (it & 1) : 0;
  real* tile = tile0 + b * bstride;
  const TileDesc td = td_next;
  const InstDesc in = a.inst[td.inst];
  const int n = in.n_cells, c0 = td.c0;
  const int TCe = td.nc;  // the host sizes tiles (1 <= nc <= TC) to fill the launch in whole rounds
  if (nbuf == 1 && warp == 0) stage_tile(td, 0);
  bool ok = mbar_wait(bar + b, (phase >> b) & 1u, a.max_polls);
  ok = __syncthreads_and(ok);
  if (!ok) {
    if (tid == 0) atomicOr(a.err, ERR_TIMEOUT);
    mbar_wait(bar + b, (phase >> b) & 1u, a.max_polls);  // let the copies land before the CTA exits
    if (tid == 0) bulk_wait_all();                        // and the stores read their source
    return;
  }
  phase ^= 1u << b;
  {  // the cells' geometry as pairs for phase D
    const Geo* g = reinterpret_cast<const Geo*>(tile + L::geo_off(Vp) / sizeof(real));
    for (int t = tid; t < TCe; t += NT) {
      crec[C_N * t + C_CP] = p_set(real(g[t].cp));
      crec[C_N * t + C_NCM] = p_set(real(-g[t].cm));
      crec[C_N * t + C_IR] = p_set(real(g[t].inv_rbar));
    }
  }

  // ==== phase A: per cell, LPC lanes of a warp with no CTA barrier: moments (Eq. macro_red), tau,
  // the equilibrium moment vectors and factors (Sec. IV.D) and their mass normalisation.  Each
  // shuffle level and each per-cell scalar step serves all the warp's cells (eight lanes and four
  // cells where the node counts are fixed, else a half-warp and two); warps without a cell go on
  // to the force contractions below.
  // (single-precision tiles of four cells and less keep two cells a warp: with one warp for all
  // four, the f~ stage's critical path grew by 3 %)
  constexpr bool BYROW = EXACT && 16 % Q0MAX == 0 && Q0MAX >= 8 && Q1MAX % 2 == 0;
  constexpr int LPC = BYROW && !(F32 && TC < 8) ? 8 : 16, CPW = 32 / LPC;
  constexpr int NF0 = (Q0MAX + LPC - 1) / LPC, NF1 = (Q1MAX + LPC - 1) / LPC;  // factors per lane and axis
  const int NA = (TCe + CPW - 1) / CPW;  // warps with cells
  for (int wa = warp; wa < NA; wa += NW) {
    const int hl = lane & (LPC - 1);
    const int tc = CPW * wa + lane / LPC;
    const bool has = tc < TCe;         // the last warp's groups beyond the tile have no cell: they
    const int t = has ? tc : TCe - 1;  // repeat the last one's and write nothing
    const real* F = tile + (t + 3) * row;
    real sn = 0, sr = 0, sp = 0, se = 0;  // the lane's partial sums
    if constexpr (BYROW) {
      // lane hl sums nodes j of its rows i (all of them, or its share where a row has several lanes):
      // the p^phi weights are uniform operands and p^R enters once per row (a third of the
      // instructions of the general form); row by row, for the rounding of short sums
      constexpr int PARTS = LPC / Q0MAX > 0 ? LPC / Q0MAX : 1, JN = Q1MAX / PARTS, RP = Q0MAX * PARTS / LPC;
#pragma unroll
      for (int r = 0; r < RP; ++r) {
        const int i = hl % Q0MAX + LPC * r, jb = (hl / Q0MAX) * JN;
        const real* f = F + 2 * (i * Q1MAX + jb);
        const real pr = p0r[i];
        real n = 0, q = 0, e = 0;
#pragma unroll
        for (int j = 0; j < JN; ++j) {
          const pair_t<real> x = p_load(f + 2 * j);
          const real pj = PARTS > 1 ? p1r[jb + j] : F32 ? real(m.p1f[j]) : real(m.p1[j]), u = pj * x.x;
          n += x.x;
          q += u;
          e += pj * u + x.y;
        }
        const real u = pr * n;
        sn += n;
        sr += u;
        sp += q;
        se += pr * u + e;
      }
    } else {
#pragma unroll 4
      for (int v = hl; v < V; v += LPC) {
        const int i = v / nq1, j = v - i * nq1;
        const pair_t<real> f = p_load(F + 2 * v);
        const real f1 = f.x, f2 = f.y, pr = p0r[i], pp = p1r[j];
        sn += f1;
        sr += pr * f1;
        sp += pp * f1;
        se += (pr * pr + pp * pp) * f1 + f2;
      }
    }
    // sums over the cell's lanes; then the sums of D plus those of R and the derived fields
    real nn, u0, u1, T;
    double dn = 0.0;  // FP64 path: sum of D (n - sum R)
    float en = 0.f;   // FP32 path: rounding error of the mass sum sn (float-float sn + en)
    if constexpr (F32) {
      // compensated FP32 butterflies leave the same sums on every lane of the cell; n in
      // float-float, the other fields in FP32 through one reciprocal: no FP64 and no
      // broadcast on the dependency chain
      float er = 0.f, ep = 0.f, ee = 0.f;
      group_sum_comp<LPC>(sn, en);
      group_sum_comp<LPC>(sr, er);
      group_sum_comp<LPC>(sp, ep);
      group_sum_comp<LPC>(se, ee);
      float nh, nl;
      two_sum(sn, m.ref_nf[0], nh, nl);
      nn = nh + (nl + (en + m.ref_nf[1]));
      const float inv = rcp_rn(nn);
      u0 = (sr + (er + m.ref_rf)) * inv;
      u1 = (sp + (ep + m.ref_pf)) * inv;
      T = ((se + (ee + m.ref_ef)) * inv - (u0 * u0 + u1 * u1)) * (1.0f / 3.0f);
    } else {
      dn = group_sum<LPC>(double(sn));
      const double dr = group_sum<LPC>(double(sr)), dpp = group_sum<LPC>(double(sp)), de = group_sum<LPC>(double(se));
      nn = real(dn + m.ref_n);
      const real inv = rcp_rn(nn);
      u0 = real(dr + m.ref_r) * inv, u1 = real(dpp + m.ref_p) * inv;
      T = (real(de + m.ref_e) * inv - (u0 * u0 + u1 * u1)) * (real(1) / real(3));
    }
    if (hl == 0 && has) {
      crec[C_N * t + C_1T] = p_make(real(1), T);
      crec[C_N * t + C_NTAU] = p_set(-relaxation_rate<real>(in.tau_mode, rcp_rn(F32 ? real(in.kn_f) : real(in.kn)), nn, T));
    }
    real* mt = mv + t * 4 * MAXN;  // moment vectors [axis * 2 + side][s]
    if (hl < 4 && has) {
      const int ax = hl >> 1, side = hl & 1;
      const real u = (ax ? u1 : u0) * (side ? real(-1) : real(1));
      eq_moments_fast<real>(ax ? m.kind1 : m.kind0, ax ? m.N1 : m.N0, u, T, mt + hl * MAXN);
    }
    __syncwarp();
    // equilibrium factors: lane hl takes g_R[k] and g_phi[k] for k = hl, hl + LPC, ...
    real gr[NF0], gp[NF1], sgr = real(0), sgp = real(0);
#pragma unroll
    for (int q = 0; q < NF0; ++q) {
      const int k = hl + LPC * q;
      gr[q] = real(0);
      if (k < nq0) {
        const real* mm = mt + ((m.kind0 == 1 && p0r[k] < real(0)) ? 1 : 0) * MAXN;
        for (int s2 = 0; s2 <= m.N0; ++s2) gr[q] += tabr0[s2 * MAXQ + k] * mm[s2];
        gr[q] *= nn;
      }
    }
#pragma unroll
    for (int q = 0; q < NF1; ++q) {
      const int k = hl + LPC * q;
      gp[q] = real(0);
      if (k < nq1) {
        const real* mm = mt + (2 + ((m.kind1 == 1 && p1r[k] < real(0)) ? 1 : 0)) * MAXN;
        for (int s2 = 0; s2 <= m.N1; ++s2) gp[q] += tabr1[s2 * MAXQ + k] * mm[s2];
      }
    }
    // rescale g_R so that sum_i g_R sum_j g_phi is exactly the target sum D + sum R (f_eq - R
    // of phase D then carries the cell's mass).  In exact arithmetic the truncated equilibrium has this
    // sum (Sec. IV.D); in single precision the table contraction misses it by some 1e-7, and the BGK
    // term would turn that into a mass source of (dt / tau) 1e-7 n every step.  g_R <- g_R (1 - delta)
    real scale0;  // FP64 path: the factor of g_R
    float delta = 0.f;
    if constexpr (F32) {
      // A = sum g_R sum g_phi and the target sum D + sum R, both in float-float;
      // delta = (A - target) / A, where A_hi - target_hi is exact (the two are close)
      float a0 = gr[0], a0e = 0.f, a1 = gp[0], a1e = 0.f, t1, er;
#pragma unroll
      for (int q = 1; q < NF0; ++q) two_sum(a0, gr[q], t1, er), a0 = t1, a0e += er;
#pragma unroll
      for (int q = 1; q < NF1; ++q) two_sum(a1, gp[q], t1, er), a1 = t1, a1e += er;
      group_sum_comp<LPC>(a0, a0e);
      group_sum_comp<LPC>(a1, a1e);
      const float Ah = a0 * a1;
      const float Al = fmaf(a0, a1e, fmaf(a0e, a1, fmaf(a0, a1, -Ah)));
      float th, tl;
      two_sum(sn, m.ref_sumf[0], th, tl);
      tl = tl + (en + m.ref_sumf[1]);
      delta = (__fsub_rn(Ah, th) + (Al - tl)) * rcp_rn(Ah);
      scale0 = real(0);
    } else {
#pragma unroll
      for (int q = 0; q < NF0; ++q) sgr += gr[q];
#pragma unroll
      for (int q = 0; q < NF1; ++q) sgp += gp[q];
      scale0 = real((dn + m.ref_n) / (group_sum<LPC>(double(sgr)) * group_sum<LPC>(double(sgp))));
    }
    if (has) {
#pragma unroll
      for (int q = 0; q < NF0; ++q) {
        const int k = hl + LPC * q;
        if (k < nq0) gRn[t * MAXQ + k] = p_set(F32 ? real(fmaf(-float(gr[q]), delta, float(gr[q]))) : gr[q] * scale0);
      }
#pragma unroll
      for (int q = 0; q < NF1; ++q) {
        const int k = hl + LPC * q;
        if (k < nq1) gP[t * MAXQ + k] = p_set(gp[q]);
      }
    }
  }
  // Single-precision fixed-shape kernels contract both fields of a velocity in one task
  // (packed FP32x2 against duplicated coefficients); the others one field per task.
  constexpr bool PAIRED = F32 && EXACT;
  constexpr int TPF = PAIRED ? 1 : 2;  // tasks per (cell, column) and per (cell, row)
  constexpr int HQ = KArgs<real>::HQ;
  // lbuf = -(p^phi)^2 K^R f (one task per (cell, [field,] j): a column of nq0 values)
  auto force_R = [&](int x) {
    if constexpr (PAIRED) {  // even and odd parts under the reflection of axis 0 (KArgs)
      constexpr int H = Q0MAX / 2;
      const int j = x % Q1MAX, t = x / Q1MAX;
      const real* F = tile + (t + 3) * row;
      real* Lr = lbuf + t * row;
      // node k of the first half and its mirror refl(k) = k + H (half range) or Q - 1 - k
      // (full range): the mirror's pair sits at r0 + k rs
      const int rs = m.kind0 == 1 ? 2 * Q1MAX : -2 * Q1MAX;
      const int r0 = 2 * refl(m.kind0, Q0MAX, 0) * Q1MAX + 2 * j;
      pair_t<real> e[H], o[H];
#pragma unroll
      for (int k = 0; k < H; ++k) {
        const pair_t<real> fk = p_load(F + 2 * j + 2 * k * Q1MAX), fr = p_load(F + r0 + k * rs);
        e[k] = p_add(fk, fr);
        o[k] = p_sub(fk, fr);
      }
      const pair_t<real> w = p_set(-p1r[j] * p1r[j]);
#pragma unroll
      for (int i = 0; i < H; ++i) {
        pair_t<real> pe = p_set(real(0)), mo = p_set(real(0));
#pragma unroll
        for (int k = 0; k < H; ++k) {
          pe = p_fma(kk.pairs.P0[i * HQ + k], e[k], pe);
          mo = p_fma(kk.pairs.M0[i * HQ + k], o[k], mo);
        }
        p_store(Lr + 2 * j + 2 * i * Q1MAX, p_mul(w, p_add(mo, pe)));
        p_store(Lr + r0 + i * rs, p_mul(w, p_sub(mo, pe)));
      }
    } else {
      const int j = x % nq1, td2 = x / nq1, d = td2 & 1, t = td2 >> 1;
      const real* F = tile + (t + 3) * row + d;
      real* Lr = lbuf + t * row + d;
      const real w = -p1r[j] * p1r[j];
      if constexpr (EXACT) {  // as above, one field
        constexpr int H = Q0MAX / 2;
        const int rs = m.kind0 == 1 ? 2 * Q1MAX : -2 * Q1MAX;
        const int r0 = 2 * refl(m.kind0, Q0MAX, 0) * Q1MAX + 2 * j;
        real e[H], o[H];
#pragma unroll
        for (int k = 0; k < H; ++k) {
          const real fk = F[2 * j + 2 * k * Q1MAX], fr = F[r0 + k * rs];
          e[k] = fk + fr;
          o[k] = fk - fr;
        }
#pragma unroll
        for (int i = 0; i < H; ++i) {
          real pe = 0, mo = 0;
#pragma unroll
          for (int k = 0; k < H; ++k) {
            pe += kk.split.P0[i * HQ + k] * e[k];
            mo += kk.split.M0[i * HQ + k] * o[k];
          }
          Lr[2 * j + 2 * i * Q1MAX] = w * (mo + pe);
          Lr[r0 + i * rs] = w * (mo - pe);
        }
      } else {
        real col[Q0MAX];
#pragma unroll
        for (int ip = 0; ip < Q0MAX; ++ip) col[ip] = ip < nq0 ? F[2 * (ip * nq1 + j)] : real(0);
#pragma unroll
        for (int i = 0; i < Q0MAX; ++i) {
          if (i < nq0) {
            real acc = 0;
#pragma unroll
            for (int ip = 0; ip < Q0MAX; ++ip)
              if (ip < nq0) acc += kk.full.K0[i * MAXQ + ip] * col[ip];
            Lr[2 * (i * nq1 + j)] = w * acc;
          }
        }
      }
    }
  };
  // lbuf += p^R K~^phi f (one task per (cell, [field,] i): a row of nq1 values)
  auto force_phi = [&](int x) {
    if constexpr (PAIRED) {  // even and odd parts under the reflection of axis 1 (KArgs)
      constexpr int H = Q1MAX / 2;
      const int i = x % Q0MAX, t = x / Q0MAX;
      const real* F = tile + (t + 3) * row + 2 * i * Q1MAX;
      real* Lr = lbuf + t * row + 2 * i * Q1MAX;
      const int rs = m.kind1 == 1 ? 2 : -2;  // the mirror of node k sits at r0 + k rs
      const int r0 = 2 * refl(m.kind1, Q1MAX, 0);
      pair_t<real> e[H], o[H];
#pragma unroll
      for (int k = 0; k < H; ++k) {
        const pair_t<real> fk = p_load(F + 2 * k), fr = p_load(F + r0 + k * rs);
        e[k] = p_add(fk, fr);
        o[k] = p_sub(fk, fr);
      }
      const pair_t<real> pr = p_set(p0r[i]);
#pragma unroll
      for (int j = 0; j < H; ++j) {
        pair_t<real> pe = p_set(real(0)), mo = p_set(real(0));
#pragma unroll
        for (int k = 0; k < H; ++k) {
          pe = p_fma(kk.pairs.P1[j * HQ + k], e[k], pe);
          mo = p_fma(kk.pairs.M1[j * HQ + k], o[k], mo);
        }
        p_store(Lr + 2 * j, p_fma(pr, p_add(pe, mo), p_load(Lr + 2 * j)));
        p_store(Lr + r0 + j * rs, p_fma(pr, p_sub(pe, mo), p_load(Lr + r0 + j * rs)));
      }
    } else {
      const int i = x % nq0, td2 = x / nq0, d = td2 & 1, t = td2 >> 1;
      const real* F = tile + (t + 3) * row + d + 2 * i * nq1;
      real* Lr = lbuf + t * row + d + 2 * i * nq1;
      const real pr = p0r[i];
      if constexpr (EXACT) {  // as above, one field
        constexpr int H = Q1MAX / 2;
        const int rs = m.kind1 == 1 ? 2 : -2;
        const int r0 = 2 * refl(m.kind1, Q1MAX, 0);
        real e[H], o[H];
#pragma unroll
        for (int k = 0; k < H; ++k) {
          const real fk = F[2 * k], fr = F[r0 + k * rs];
          e[k] = fk + fr;
          o[k] = fk - fr;
        }
#pragma unroll
        for (int j = 0; j < H; ++j) {
          real pe = 0, mo = 0;
#pragma unroll
          for (int k = 0; k < H; ++k) {
            pe += kk.split.P1[j * HQ + k] * e[k];
            mo += kk.split.M1[j * HQ + k] * o[k];
          }
          Lr[2 * j] += pr * (pe + mo);
          Lr[r0 + j * rs] += pr * (pe - mo);
        }
      } else {
        real rw[Q1MAX];
#pragma unroll
        for (int jp = 0; jp < Q1MAX; ++jp) rw[jp] = jp < nq1 ? F[2 * jp] : real(0);
#pragma unroll
        for (int j = 0; j < Q1MAX; ++j) {
          if (j < nq1) {
            real acc = 0;
#pragma unroll
            for (int jp = 0; jp < Q1MAX; ++jp)
              if (jp < nq1) acc += kk.full.Kt1[j * MAXQ + jp] * rw[jp];
            Lr[2 * j] += pr * acc;
          }
        }
      }
    }
  };
  // Both contractions read only the owned cells, which phase A does not change.  When
  // some warps have no cell and the tasks come to at most six per idle thread, those
  // warps run all of them during phase A (the K~^phi tasks after a barrier among those
  // warps only); otherwise every thread takes K^R tasks after phase A and K~^phi tasks
  // after a CTA barrier.
  const int nR = TCe * TPF * nq1, nP = TCe * TPF * nq0;
  const int nfree = NA < NW ? NT - 32 * NA : 0;
  const bool early = nR + nP <= 6 * nfree;  // uniform across the CTA
  const bool runs = !early || warp >= NA;
  const int f0 = early ? tid - 32 * NA : tid, fs = early ? nfree : NT;
  if (runs)
    for (int x = f0; x < nR; x += fs) force_R(x);
  if (!early) __syncthreads();
  else if (runs) asm volatile("bar.sync 1, %0;" ::"r"(nfree) : "memory");
  if (runs)
    for (int x = f0; x < nP; x += fs) force_phi(x);
  __syncthreads();

  if (tix + int(gridDim.x) < a.n_tiles) td_next = a.tiles[tix + gridDim.x];

  // stage the next tile into the other buffer, the source of the previous tile's store
  if (nbuf == 2 && warp == 0 && tix + int(gridDim.x) < a.n_tiles) {
    if (lane == 0) bulk_wait_read_all();
    __syncwarp();
    stage_tile(td_next, b ^ 1);
  }

  // ==== phase B: the walls
  for (int wall = 0; wall < 2; ++wall) {
    // every tile whose stencils reach a ghost cell fills the ghosts itself
    const bool active = wall == 0 ? (c0 < 3) : (c0 + TCe + 3 > n);
    if (!active) continue;  // uniform across the CTA
    if (in.halo & (1 << wall)) {
      // a slab end: the three ghost cells are the neighbouring slab's, in increasing
      // radius (below the slab at the inner end, above it at the outer end)
      const real* hb = a.halo + (size_t(td.inst) * 2 + wall) * 3 * row;
      const int sA = wall == 0 ? 3 - c0 : (n - 1 - c0 + 3);  // slot of the edge cell
      for (int x = tid; x < 3 * V; x += NT) {
        const int q = x / V, v = x - q * V;  // ghost q (increasing radius), velocity v
        const int slot = wall == 0 ? sA - 3 + q : sA + 1 + q;
        if (slot >= 0 && slot < TC + 6) p_store(tile + slot * row + 2 * v, p_load(hb + q * row + 2 * v));
      }
      continue;
    }
    const double Tw = wall == 0 ? in.T_in : in.T_out;
    const double sgn = wall == 0 ? 1.0 : -1.0;  // incoming half: p^R > 0 at the inner wall
    __syncthreads();
    {  // the wall's equilibrium factors and incoming flux, computed by the host
      const WallEq& we = a.wall[td.inst * 2 + wall];
      for (int k = tid; k < nq0 + nq1; k += NT) {
        if (k < nq0) gw0[k] = we.g0[k];
        else gw1[k - nq0] = we.g1[k - nq0];
      }
      if (tid == 0) mw[0] = we.in_flux;
    }
    __syncthreads();
    // outgoing wall flux of f' (field 0) and the incoming equilibrium flux, FP64 sums
    const int sA = wall == 0 ? 3 - c0 : (n - 1 - c0 + 3);  // slot of the wall-adjacent cell
    const int dir = wall == 0 ? 1 : -1;                // towards the interior
    double num = 0;
    for (int v = tid; v < V; v += NT) {
      const int i = v / nq1, j = v - i * nq1;
      if (!(sgn * p0d[i] < 0.0)) continue;
      // the same pair reconstruction as phase D (field 0 enters n_w)
      pair_t<real> F0 = p_load(tile + sA * row + 2 * v);
      pair_t<real> F1 = p_load(tile + (sA + dir) * row + 2 * v);
      pair_t<real> F2 = p_load(tile + (sA + 2 * dir) * row + 2 * v);
      if constexpr (FT) {  // F~ of the three wall-adjacent cells
        const long long e0 = in.cell0 + (wall == 0 ? 0 : n - 1);
        const pair_t<real> R2 = p_set(w0r[i] * w1r[j]);
        F0 = p_mul(p_add(F0, R2), p_set(a.sqrtg[e0]));
        F1 = p_mul(p_add(F1, R2), p_set(a.sqrtg[e0 + dir]));
        F2 = p_mul(p_add(F2, R2), p_set(a.sqrtg[e0 + 2 * dir]));
      }
      const pair_t<real> G0 = p_fma(F1, p_set(real(-3)), p_fma(F0, p_set(real(3)), F2));
      const pair_t<real> G1 = p_fma(F1, p_set(real(-8)), p_fma(F0, p_set(real(6)), p_mul(F2, p_set(real(3)))));
      // chi: bit for bit phase D's value (the same cell, side and order).  f~: phase D walks F~ - R, formed
      // by one fma, which agrees with this F~ to rounding; differences of F~ itself are kept here, since
      // where sqrt(g) is far from one F~ - R is larger than F~ and n_w would carry its rounding
      const real sc = iw0[i] * iw1[j];
      const pair_t<real> SC = p_set(sc);
      WenoWin<real, false> w;
      WenoSide<real> ws;
      ws.set(wall != 0);
      w.start(p_mul(wall ? F2 : G1, SC), p_mul(wall ? F1 : G0, SC), p_mul(F0, SC), p_mul(wall ? G0 : F1, SC),
              p_mul(wall ? G1 : F2, SC));
      num += double(w.face_checked(ws).x * rcp_rn(sc)) * p0d[i];
    }
    num = warp_sum<real>(num);
    if (lane == 0) red[warp] = num;
    __syncthreads();
    if (tid == 0) {
      double sacc = FT ? 0.0 : (wall == 0 ? m.ref_flux_neg : m.ref_flux_pos);  // chi: the outgoing flux of R
      for (int w = 0; w < NW; ++w) sacc += red[w];
      const double nwv = -sacc / mw[0];
      mw[1] = nwv;
      a.nw[td.inst * 2 + wall] = nwv;
      if (!isfinite(nwv)) atomicOr(a.err, ERR_NONFINITE);
    }
    __syncthreads();
    const double nwd = mw[1];
    for (int v = tid; v < V; v += NT) {
      const int i = v / nq1, j = v - i * nq1;
      pair_t<real> g1, g2, g3;  // ghosts at distance 1, 2, 3 from the wall
      if (sgn * p0d[i] < 0.0) {
        pair_t<real> F0 = p_load(tile + sA * row + 2 * v);
        pair_t<real> F1 = p_load(tile + (sA + dir) * row + 2 * v);
        pair_t<real> F2 = p_load(tile + (sA + 2 * dir) * row + 2 * v);
        if constexpr (FT) {
          const long long e0 = in.cell0 + (wall == 0 ? 0 : n - 1);
          const pair_t<real> R2 = p_set(w0r[i] * w1r[j]);
          F0 = p_mul(p_add(F0, R2), p_set(a.sqrtg[e0]));
          F1 = p_mul(p_add(F1, R2), p_set(a.sqrtg[e0 + dir]));
          F2 = p_mul(p_add(F2, R2), p_set(a.sqrtg[e0 + 2 * dir]));
        }
        g1 = p_fma(F1, p_set(real(-3)), p_fma(F0, p_set(real(3)), F2));
        g2 = p_fma(F1, p_set(real(-8)), p_fma(F0, p_set(real(6)), p_mul(F2, p_set(real(3)))));
        if constexpr (FT) {  // stored as F~ - R
          const pair_t<real> nR = p_set(-(w0r[i] * w1r[j]));
          g1 = p_add(g1, nR);
          g2 = p_add(g2, nR);
        }
        g3 = g2;  // never read by an outgoing stencil
      } else {  // f_eq(n_w, u_w, T_w) - R
        const double e = nwd * gw0[i] * gw1[j], r = m.w0[i] * m.w1[j];
        g1 = g2 = g3 = p_make(real(e - r), real(e * Tw - r));
      }
      const int s1 = sA - dir, s2 = sA - 2 * dir, s3 = sA - 3 * dir;
      if (s1 >= 0 && s1 < TC + 6) p_store(tile + s1 * row + 2 * v, g1);
      if (s2 >= 0 && s2 < TC + 6) p_store(tile + s2 * row + 2 * v, g2);
      if (s3 >= 0 && s3 < TC + 6) p_store(tile + s3 * row + 2 * v, g3);
    }
  }
  // phase D reads the ghost rows the walls wrote; an interior tile wrote nothing since the
  // barrier after phase A (warp 0's staging goes to the other buffer)
  if (c0 < 3 || c0 + TCe + 3 > n) __syncthreads();  // uniform across the CTA
  real* sgs = nullptr;  // f~: sqrt(g) of the tile's slots, 1 past the walls (ghost rows hold F~ - R)
  if constexpr (FT) {
    __shared__ real sgs_[TC + 6];
    sgs = sgs_;
    for (int q = tid; q < TC + 6; q += NT) {
      const int cell = c0 - 3 + q;
      sgs_[q] = (cell >= 0 && cell < n) ? a.sqrtg[in.cell0 + cell] : real(1);
    }
    __syncthreads();
  }

  // ==== phase D: WENO-5 fluxes along the cells, flux difference, BGK, RK3 combine (in place)
  const real dtr = F32 ? real(in.dt_f) : real(in.dt);
  const real ca = F32 ? real(a.caf) : real(a.ca);
  const real cc = (F32 ? real(a.ccf) : real(a.cc)) * dtr;
  using P = pair_t<real>;
  for (int v = tid; v < V; v += NT) {  // one velocity, both fields, walking the tile's cells
    const int i = v / nq1, j = v - i * nq1;
    const real pr = p0r[i];
    const bool up = pr >= real(0);
    const real sc = iw0[i] * iw1[j];
    const P nrij = p_set(-(w0r[i] * w1r[j]));
    const P SC = p_set(sc);
    const P npr = p_set(-pr * rcp_rn(sc));  // interface values carry the scale sc (a power of two)
    WenoSide<real> side;
    side.set(up);
    real* S = tile + 2 * v;
    const real* Fl = a.Fl + size_t(in.cell0 + c0) * row + 2 * v;  // F_l of the owned cells, read once
    // the advected value of slot q, scaled: D (chi), F~ - R = (D + R) sqrt(g) - R (f~)
    const real Rr = w0r[i] * w1r[j];
    auto adv_val = [&](int q) -> P {
      const P x = p_load(S + q * row);
      if constexpr (FT) return p_mul(p_fma(x, p_set(sgs[q]), p_set(Rr * (sgs[q] - real(1)))), SC);
      else return p_mul(x, SC);
    };
    P FRv = p_set(real(0));  // f~: the inertial term of R for this velocity
    if constexpr (FT) FRv = p_set(a.forceR[v]);
    // the upwind cell of interface s + 1/2 is s for p^R >= 0, s + 1 otherwise: the walk runs one cell ahead
    const int o = up ? 0 : 1;
    WenoWin<real, true> win;
    win.start(adv_val(o), adv_val(o + 1), adv_val(o + 2), adv_val(o + 3), adv_val(o + 4));
    P fm = win.face_checked(side);
    // F_l of the next cell is loaded one cell ahead (a global load, the only one of the walk)
    P fl_next = need_fl ? p_load(Fl) : p_set(real(0));
// (all cells in one body, left by a break at the last: two cells a pass under a guard issue 56e6 ALU
// and 177e6 instructions a launch at a batch of 128 instances, this 34e6 and 145e6 -- the walk's state
// changes its names, not its registers; 4.96 ms a call at a batch of 256, 4.82 ms so)
#pragma unroll
    for (int t = 0; t < TC; ++t) {
      if (t >= TCe) break;
      const P fl = fl_next;
      if (need_fl && t + 1 < TCe) fl_next = p_load(Fl + (t + 1) * row);
      win.push(adv_val(t + 5 + o));
      const P fp = win.face_checked(side);
      // -adv = -p^R (cp F_{s+1/2} - cm F_{s-1/2}); per-cell factors: shared-memory broadcasts
      P cp, ncm, ir, ntau;
      const P2* cr = crec + C_N * t;
      if constexpr (F32) {
        const float4 x = *reinterpret_cast<const float4*>(cr + C_CP), y = *reinterpret_cast<const float4*>(cr + C_IR);
        cp = p_make(x.x, x.y), ncm = p_make(x.z, x.w), ir = p_make(y.x, y.y), ntau = p_make(y.z, y.w);
      } else {
        cp = cr[C_CP], ncm = cr[C_NCM], ir = cr[C_IR], ntau = cr[C_NTAU];
      }
      P nadv = p_mul(p_fma(fp, cp, p_mul(fm, ncm)), npr);
      const P Dc = p_load(S + (t + 3) * row);  // the cell's D
      if constexpr (FT) nadv = p_fma(p_set(-pr * Rr), p_add(cp, ncm), nadv);  // the advection of R
      // f_eq - R for both fields: (g, T g) - R
      const P deq = p_fma(p_mul(gRn[t * MAXQ + i], gP[t * MAXQ + j]), cr[C_1T], nrij);
      P force = p_load(lbuf + t * row + 2 * v);
      if constexpr (FT) force = p_sub(force, FRv);
      // L = -adv + force / Rbar - (D - D_eq) / tau
      const P Lv = p_fma(p_sub(Dc, deq), ntau, p_fma(force, ir, nadv));
      P o = p_fma(Lv, p_set(cc), Dc);
      if (need_fl) o = p_fma(p_sub(fl, Dc), p_set(ca), o);
      p_store(S + (t + 3) * row, o);  // in place: this column's slot t+3 is not read again
      fm = fp;
    }
  }
  // ---- bulk store of the owned cells (generic-proxy writes made visible to the async proxy first)
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  if (tid == 0) {
    bulk_s2g(a.Fout + size_t(in.cell0 + c0) * row, tile + 3 * row, unsigned(TCe * row * sizeof(real)));
    bulk_commit();
    if (nbuf == 1) bulk_wait_read_all();
  }
  if (nbuf == 1) __syncthreads();  // the next tile is staged into this buffer
  }
  if (tid == 0) bulk_wait_all();  // the stores have read their source before the CTA exits
}

}  // namespace vlb
