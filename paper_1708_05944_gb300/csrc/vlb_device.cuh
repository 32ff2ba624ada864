// Device-side building blocks shared by the libvlb kernels: descriptors,
// WENO-5 interface values, equilibrium moment vectors, bounded mbarrier waits.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace vlb {

constexpr int MAXQ = 32;  // nodes per momentum axis
constexpr int MAXN = 8;   // equilibrium expansion order + 1

// Error bits set by kernels in a device word the host reads back.
enum : unsigned { ERR_TIMEOUT = 1u, ERR_NONFINITE = 2u };

struct InstDesc {
  long long cell0;  // first global cell of the instance
  int n_cells;
  int tau_mode;     // vlb_tau_mode
  double kn, dt;
  double u_in, T_in, u_out, T_out;  // walls: tangential speed, temperature
  float kn_f, dt_f;                 // single-precision copies
  int halo;                         // bit e set: end e (0 inner, 1 outer) is a slab halo, not a wall
  int pad;
};

// Diffuse-wall equilibrium f_eq(1, (0, u_w), T_w) of one wall (Eq. weno_populate):
// its factors per axis and its incoming particle flux, sum over the incoming
// half of g0_i p_i times sum_j g1_j.  They depend on the wall only, so the host
// computes them when the walls are set.
struct WallEq {
  double g0[MAXQ], g1[MAXQ];
  double in_flux;
  double pad;
};

struct TileDesc {
  int inst;
  int c0;  // first cell (within the instance) owned by the tile
  int nc;  // cells owned (1 .. the kernel's TC)
};

// (f', f'') pair of one velocity in the bulk type (see the pair operations below).
template <typename real>
struct PairOf;
template <>
struct PairOf<float> {
  using type = float2;
};
template <>
struct PairOf<double> {
  using type = double2;
};
template <typename real>
using pair_t = typename PairOf<real>::type;

// Per-cell chi-formulation factors (Eqs. flux_kom_R, flux_kom_eta):
//   advection = p^R (cp * Flux_{s+1/2} - cm * Flux_{s-1/2}),
//   cp = 2 R_{s+1/2} / (R_{s+1/2}^2 - R_{s-1/2}^2), cm = 2 R_{s-1/2} / (...),
//   inv_rbar = 2 / (R_{s+1/2} + R_{s-1/2}) multiplies the inertial force.
struct GeoCell {
  double cp, cm, inv_rbar, wres;
};

// Single-precision copy of the advection and force factors (cp, cm, inv_rbar, unused).
struct GeoCellF {
  float cp, cm, inv_rbar, pad;
};

// Momentum-space tables of the model (copied into shared memory by each CTA).
struct ModelArgs {
  int nq0, nq1, N0, N1, kind0, kind1;
  double p0[MAXQ], p1[MAXQ];
  double w0[MAXQ], w1[MAXQ];  // quadrature weights
  double tab0[MAXQ * MAXN], tab1[MAXQ * MAXN];  // [k][s] with stride MAXN
  float tab0f[MAXQ * MAXN], tab1f[MAXQ * MAXN];  // single-precision copies for the FP32-bulk path
  float p0f[MAXQ], p1f[MAXQ], iw0f[MAXQ], iw1f[MAXQ];  // nodes and inverse weights, single precision
  double iw0[MAXQ], iw1[MAXQ];                         // inverse weights, double precision
  float w0f[MAXQ], w1f[MAXQ];                          // weights, single precision
  // Device distributions hold the deviation D = F - R from the rest state
  // R_ij = w0_i w1_j (f_eq(1, 0, 1), the same for f' and f'').  R is a steady
  // state of the discrete equations (advection and force cancel on it, BGK
  // vanishes) and WENO-5 is unchanged by adding a constant, so the stage
  // operator applied to D is the operator applied to F; storing D keeps the
  // rounding of each update relative to |F - R| instead of |F|.  Sums of R:
  double ref_n, ref_r, ref_p, ref_e;  // sum R, sum p0 R, sum p1 R, sum (p0^2 + p1^2) R + sum R
  double ref_sum_f;                   // sum of the single-precision products float(w0_i) float(w1_j)
  double ref_flux_pos, ref_flux_neg;  // sum over p0 > 0 (p0 < 0) of p0 R
  // single-precision copies: ref_n and ref_sum_f as (hi, lo) float pairs, the others rounded
  float ref_nf[2], ref_sumf[2];
  float ref_rf, ref_pf, ref_ef;
};

// Momentum-space kernels of the inertial force (Eq. boltz_couette_kom): K0 =
// d/dp^0 on axis 0 and Kt1 = d/dp^1 (p^1 .) on axis 1.  The generic kernels read
// the full matrices; the fixed-shape kernels read the split blocks below (as
// duplicated pairs in single precision).  The split uses that each commutes with the
// reflection of its axis, up to sign: with J the node permutation p_k -> -p_k
// (see refl), K0 J = -J K0 and Kt1 J = J Kt1.  Each then splits into two
// half-size blocks acting on the even and odd parts e_k = f_k + f_Jk,
// o_k = f_k - f_Jk (k over the first half of the nodes):
//   P[i][k] = (K[i][k] + K[i][Jk]) / 2,   M[i][k] = (K[i][k] - K[i][Jk]) / 2,
//   axis 0: (K0 f)_i = P e + M o,  (K0 f)_Ji = M o - P e;
//   axis 1: (Kt1 f)_j = P e + M o, (Kt1 f)_Jj = P e - M o.
template <typename real>
struct KArgs {
  static constexpr int HQ = MAXQ / 2;
  struct Full {
    real K0[MAXQ * MAXQ];   // [i][i'] stride MAXQ
    real Kt1[MAXQ * MAXQ];  // [j][j'] stride MAXQ
  };
  struct Split {
    real P0[HQ * HQ], M0[HQ * HQ];  // [i][k] stride HQ
    real P1[HQ * HQ], M1[HQ * HQ];  // [j][k] stride HQ
  };
  struct SplitPairs {  // the same blocks with every coefficient duplicated, for packed
    pair_t<real> P0[HQ * HQ], M0[HQ * HQ];  // contraction of both fields of a velocity
    pair_t<real> P1[HQ * HQ], M1[HQ * HQ];
  };
  union {
    Full full;
    Split split;
    SplitPairs pairs;
  };
};

// Index of the node at -p_k on an axis of nq nodes: half-range axes list the
// positive nodes first and their mirror images after them (kind 1); full-range
// axes are symmetric about their middle (kind 0).
__host__ __device__ __forceinline__ int refl(int kind, int nq, int k) {
  return kind == 1 ? (k < nq / 2 ? k + nq / 2 : k - nq / 2) : nq - 1 - k;
}

// Type-exact helpers: float arguments must not be promoted to double (the
// FP64 pipe of GB300 runs at a small fraction of the FP32 rate).
__device__ __forceinline__ float vmax(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double vmax(double a, double b) { return fmax(a, b); }
__device__ __forceinline__ float vmin(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ double vmin(double a, double b) { return fmin(a, b); }
// 1 / x correctly rounded (single precision: the reciprocal intrinsic, cheaper than a division).
__device__ __forceinline__ float rcp_rn(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double rcp_rn(double x) { return 1.0 / x; }
// x / y; single precision uses the fast divide (2 ulp), valid for |y| < 2^126.
__device__ __forceinline__ float vdiv(float x, float y) { return __fdividef(x, y); }
__device__ __forceinline__ double vdiv(double x, double y) { return x / y; }

// ---------------------------------------------------------------- WENO-5
// Interface value from the upwind-ordered stencil (a, b, c, d, e) =
// (F_{s-2}, F_{s-1}, F_s, F_{s+1}, F_{s+2}) (Eqs. weno5_flux, weno5_omega,
// weno_sigma) with the epsilon-free weights delta_q / sigma_q^2.
//
// The normalised weights do not change when the stencil is multiplied by a
// constant, so the indicators are computed on the stencil times sc (callers
// pass 1 / (w_i w_j), which brings the weighted populations of every velocity
// to order one and keeps sigma_q inside the single-precision range).  The
// weights are evaluated as delta_q prod_{r != q} sigma_r^2 over their sum,
// with the indicators scaled by their maximum; this form is exact for one
// vanishing indicator (Table IV: that stencil gets weight one).  When the
// products all vanish or are not finite -- two or three zero indicators
// (Table IV), or products below the single-precision range -- a slow path
// uses Table IV for exact zeros and delta_q (sigma_min / sigma_q)^2 otherwise.
template <typename real>
__device__ __noinline__ void weno5_weights_slow(real s1, real s2, real s3, real* w) {
  const real d1 = real(0.1), d2 = real(0.6), d3 = real(0.3);
  if (s1 == real(0) || s2 == real(0) || s3 == real(0)) {
    w[0] = s1 == real(0) ? d1 : real(0);
    w[1] = s2 == real(0) ? d2 : real(0);
    w[2] = s3 == real(0) ? d3 : real(0);
  } else {  // IEEE division: the indicators here may be subnormal or beyond 2^126
    const real mn = vmin(s1, vmin(s2, s3));
    const real r1 = mn / s1, r2 = mn / s2, r3 = mn / s3;
    w[0] = d1 * r1 * r1;
    w[1] = d2 * r2 * r2;
    w[2] = d3 * r3 * r3;
  }
}

// ---------------------------------------------------------------- pairs (f', f'') of one velocity
// Device rows interleave the two reduced distributions of Sec. II: element
// (field d, velocity v) of a cell row sits at 2 v + d, so one 8- or 16-byte
// access moves both fields of a velocity.  The WENO-5 reconstruction, the
// BGK relaxation and the RK3 combine treat f' and f'' alike, and run on the
// pair: single precision through the packed FP32x2 add / multiply / fma of
// sm_100 and later (each lane rounds as the scalar instruction does), double
// precision as two scalar operations.  p_add and p_mul are never contracted
// into an fma (the packed intrinsics round per lane like __fadd_rn and
// __fmul_rn), so an expression of them rounds the same wherever it is inlined.

__device__ __forceinline__ float2 p_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 p_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 p_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 p_set(float s) { return make_float2(s, s); }
__device__ __forceinline__ float2 p_make(float x, float y) { return make_float2(x, y); }
__device__ __forceinline__ double2 p_add(double2 a, double2 b) {
  return make_double2(__dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y));
}
__device__ __forceinline__ double2 p_mul(double2 a, double2 b) {
  return make_double2(__dmul_rn(a.x, b.x), __dmul_rn(a.y, b.y));
}
__device__ __forceinline__ double2 p_fma(double2 a, double2 b, double2 c) {
  return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
__device__ __forceinline__ double2 p_set(double s) { return make_double2(s, s); }
__device__ __forceinline__ double2 p_make(double x, double y) { return make_double2(x, y); }

// a - b on the pair (packed FP32x2 subtract; rounded, never contracted)
__device__ __forceinline__ float2 p_sub(float2 a, float2 b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;"
      : "=l"(r)
      : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)));
  return *reinterpret_cast<float2*>(&r);
}
__device__ __forceinline__ double2 p_sub(double2 a, double2 b) {
  return make_double2(__dsub_rn(a.x, b.x), __dsub_rn(a.y, b.y));
}

template <typename real>
__device__ __forceinline__ pair_t<real> p_load(const real* p) {
  return *reinterpret_cast<const pair_t<real>*>(p);
}
template <typename real>
__device__ __forceinline__ void p_store(real* p, pair_t<real> v) {
  *reinterpret_cast<pair_t<real>*>(p) = v;
}
template <typename P>
__device__ __forceinline__ P p_sel(bool c, P a, P b) {
  return c ? a : b;
}

// Rounded multiply and add that the compiler may not fuse: the weights below are
// inlined at every cell position of an unrolled loop, and a cell must get the
// same bits whichever position (tile shape) it falls at.
__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double radd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double rfma(double a, double b, double c) { return __fma_rn(a, b, c); }

// The reconstruction on a pair of fields: the candidates, the indicators
// (times 4, which the normalisation removes) and the weights run on the pair;
// only the maxima, the reciprocals and the test for the slow path are per
// field.  The weighted sum is normalised once at the end.  The weights are
// products and sums of p_mul / p_add, so a cell gets the same bits at every
// position of an unrolled walk and the result does not depend on the tile shape.
//
// The reconstruction of both fields from their indicators and candidates, as the
// fast path of weno5p computes it, with the Table IV weights of weno5_weights_slow
// for each field whose fast-path denominator den is out of range (fast holds the
// fast-path result, kept for the other field).
template <typename real>
__device__ __noinline__ pair_t<real> weno5p_slow(pair_t<real> s1, pair_t<real> s2, pair_t<real> s3, pair_t<real> F1,
                                                 pair_t<real> F2, pair_t<real> F3, pair_t<real> den,
                                                 pair_t<real> fast) {
  real r[2] = {fast.x, fast.y};
  const real S1[2] = {s1.x, s1.y}, S2[2] = {s2.x, s2.y}, S3[2] = {s3.x, s3.y};
  const real G1[2] = {F1.x, F1.y}, G2[2] = {F2.x, F2.y}, G3[2] = {F3.x, F3.y}, Dn[2] = {den.x, den.y};
  for (int c = 0; c < 2; ++c) {
    if (Dn[c] > real(1e-30) && Dn[c] < real(1e30)) continue;
    real w[3];
    weno5_weights_slow<real>(S1[c], S2[c], S3[c], w);
    const real iden = vdiv(real(1), radd(radd(w[0], w[1]), w[2]));
    r[c] = rmul(rfma(w[0], G1[c], rfma(w[1], G2[c], rmul(w[2], G3[c]))), iden);
  }
  return p_make(r[0], r[1]);
}

template <typename real>
__device__ __forceinline__ pair_t<real> weno5p(pair_t<real> a, pair_t<real> b, pair_t<real> c, pair_t<real> d,
                                               pair_t<real> e, real sc) {
  using P = pair_t<real>;
  const P F1 = p_fma(a, p_set(real(1) / real(3)), p_fma(b, p_set(real(-7) / real(6)), p_mul(c, p_set(real(11) / real(6)))));
  const P F2 = p_fma(b, p_set(real(-1) / real(6)), p_fma(c, p_set(real(5) / real(6)), p_mul(d, p_set(real(1) / real(3)))));
  const P F3 = p_fma(c, p_set(real(1) / real(3)), p_fma(d, p_set(real(5) / real(6)), p_mul(e, p_set(real(-1) / real(6)))));
  const P S = p_set(sc);
  const P A = p_mul(a, S), B = p_mul(b, S), C = p_mul(c, S), D = p_mul(d, S), E = p_mul(e, S);
  const P k = p_set(real(13) / real(3));  // 4 * 13/12: sigma_q times 4
  const P t1 = p_fma(B, p_set(real(-2)), p_add(A, C));
  const P u1 = p_fma(B, p_set(real(-4)), p_fma(C, p_set(real(3)), A));
  const P t2 = p_fma(C, p_set(real(-2)), p_add(B, D));
  const P u2 = p_fma(D, p_set(real(-1)), B);
  const P t3 = p_fma(D, p_set(real(-2)), p_add(C, E));
  const P u3 = p_fma(D, p_set(real(-4)), p_fma(C, p_set(real(3)), E));
  const P s1 = p_fma(p_mul(t1, k), t1, p_mul(u1, u1));
  const P s2 = p_fma(p_mul(t2, k), t2, p_mul(u2, u2));
  const P s3 = p_fma(p_mul(t3, k), t3, p_mul(u3, u3));
  // delta_q prod_{r != q} x_r^2 with x = sigma / max sigma (exact for one vanishing indicator)
  const P r = p_make(vdiv(real(1), vmax(s1.x, vmax(s2.x, s3.x))), vdiv(real(1), vmax(s1.y, vmax(s2.y, s3.y))));
  const P x1 = p_mul(s1, r), x2 = p_mul(s2, r), x3 = p_mul(s3, r);
  const P q1 = p_mul(x1, x1), q2 = p_mul(x2, x2), q3 = p_mul(x3, x3);
  P w1 = p_mul(p_set(real(0.1)), p_mul(q2, q3));
  P w2 = p_mul(p_set(real(0.6)), p_mul(q1, q3));
  P w3 = p_mul(p_set(real(0.3)), p_mul(q1, q2));
  const P den = p_add(p_add(w1, w2), w3);
  const P iden = p_make(vdiv(real(1), den.x), vdiv(real(1), den.y));
  const P res = p_mul(p_fma(w1, F1, p_fma(w2, F2, p_mul(w3, F3))), iden);
  // the fast path needs a normal-range denominator (the reciprocals are
  // single-precision fast divides); anything else -- vanishing or non-finite
  // products, indicators out of range -- takes the slow path of Table IV for
  // that field: one test for both fields and one rarely taken branch
  const bool ok = (den.x > real(1e-30)) & (den.x < real(1e30)) & (den.y > real(1e-30)) & (den.y < real(1e30));
  if (__builtin_expect(!ok, 0)) return weno5p_slow<real>(s1, s2, s3, F1, F2, F3, den, res);
  return res;
}

// ---------------------------------------------------------------- WENO-5 on shared differences
// The same reconstruction for kernels that walk along a line of cells, in the form whose terms
// neighbouring interfaces share.  With G a cell value times an exact power of two close to
// 1 / (w_i w_j), D = G_{k+1} - G_k, S_k = D_{k+1/2} - D_{k-1/2} and the three stencils of the
// upwind cell c centred on c - 1, c, c + 1:
//   u_- = 2 D_{c-1/2} + S_{c-1},  u_0 = D_{c-1/2} + D_{c+1/2},  u_+ = 2 D_{c+1/2} - S_{c+1},
//   sigma_q = 13/3 S_q^2 + u_q^2   (Eq. weno_sigma, times 4, which the weights do not see),
//   candidate_q = G_c + (3 side u_q + S_q) / 12,
// side = +1 for the value at c + 1/2 (velocity >= 0, ideal weights 1/10, 6/10, 3/10 on -, 0, +)
// and -1 for the value at c - 1/2 (velocity < 0, the mirrored weights).  So one cell-centred
// formula serves both upwind sides with three constants per velocity (the ideal weights relative
// to the middle one), a new cell of the walk adds one difference, one S and one 13/3 S^2, and the
// value is the cell's own plus a correction.
// (A constant far below any non-zero indicator stands for an exact zero in 13/3 S^2, so that a
// uniform stretch, all three indicators zero, takes the ideal weights and the value of its cells
// on the fast path, and one or two zeros get all the weight.)
// Power-of-two scaling keeps the scaled values exact; a face value is scaled back by its inverse.
// 34 packed operations per interface against 52 of weno5p, whose bound (the FP32 pipe, 128 fma
// per clock and SM, packed or not) it shares.
template <typename real>
struct WenoSide {  // per velocity: 3 side and the ideal weights of the - and + stencils over the middle one's
  pair_t<real> h3, dm, dp;
  __device__ __forceinline__ void set(bool up) {
    h3 = p_set(up ? real(3) : real(-3));
    dm = p_set(up ? real(1) / real(6) : real(0.5));
    dp = p_set(up ? real(0.5) : real(1) / real(6));
  }
};

// A power of two next to 1 / w.
inline double weno_pow2(double inv_w) {
  int e = 0;
  frexp(inv_w, &e);
  return ldexp(1.0, e);
}

// The same from 1 / w on the device, at most 2^62 (a product of two axes' stays in single precision)
__device__ __forceinline__ float weno_pow2_dev(float inv_w) {
  return fminf(__int_as_float(__float_as_int(inv_w) & 0x7f800000), 4.6116860e18f);
}
__device__ __forceinline__ double weno_pow2_dev(double inv_w) {
  return __hiloint2double(__double2hiint(inv_w) & 0x7ff00000, 0);
}

// A power of two close to 1 / sqrt(s1 s2), s1 and s2 the two largest of three positive numbers: half
// the sum of their bit patterns is the bit pattern of about sqrt(s1 s2).  With it the largest product of
// two scaled numbers lies in [1/4, 9/8], however far apart the three are, and the weights never leave
// the range: over a resting field, where two of three indicators vanish at many faces, scaling by the
// largest one sent whole warps to weno_corr_slow (2048 x 512 x 192 channel from rest, a step: 19.2 ms
// with that, 10.1 so).  (Double precision: the high words; the comparison instructions of the FP64
// pipe run at its 1/64 rate.)  Inf, NaN and two numbers in the top binade give a sum of weights of 0,
// Inf or NaN, and so a face of NaN (0 * Inf).
__device__ __forceinline__ unsigned inv_sqrt_bits(unsigned a, unsigned b, unsigned c, unsigned twice_inv, unsigned exponent) {
  return ((twice_inv - (a + b + c) + min(a, min(b, c))) >> 1) & exponent;
}
__device__ __forceinline__ float inv_pow2_top(float a, float b, float c) {
  return __uint_as_float(inv_sqrt_bits(__float_as_uint(a), __float_as_uint(b), __float_as_uint(c), 0xfe000000u, 0x7f800000u));
}
__device__ __forceinline__ double inv_pow2_top(double a, double b, double c) {
  return __hiloint2double(int(inv_sqrt_bits(__double2hiint(a), __double2hiint(b), __double2hiint(c), 0xffc00000u, 0x7ff00000u)), 0);
}
__device__ __forceinline__ float2 p_rcp(float2 x) {  // 1 / x of normal numbers, about 1 ulp
  float2 r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(x.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(x.y));
  return r;
}
// One reciprocal for both, x.x x.y a normal number: the hardware's approximation (20 bits) and two
// steps of Newton's iteration, r <- r + r (1 - x r).  The product, the last step and the last multiply
// round once each: about 2 ulp.  Seven operations of the FP64 pipe in place of two divisions.
__device__ __forceinline__ double2 p_rcp(double2 x) {
  const double y = __dmul_rn(x.x, x.y);
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(y));
  r = fma(r, fma(-y, r, 1.0), r);
  r = fma(r, fma(-y, r, 1.0), r);
  return make_double2(__dmul_rn(r, x.y), __dmul_rn(r, x.x));
}
// Whether the fast weights gave both values of a face (see inv_pow2_top).  (Double precision: the
// fields share a reciprocal, p_rcp, so that one tells for both; its high word, for the reason above.)
__device__ __forceinline__ bool weno_holds(float2 f) {
  unsigned nan;
  asm("{\n .reg .pred p;\n setp.nan.f32 p, %1, %2;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(nan) : "f"(f.x), "f"(f.y));
  return nan == 0;
}
__device__ __forceinline__ bool weno_holds(double2 f) {
  return (unsigned(__double2hiint(f.x)) & 0x7fffffffu) < 0x7ff80000u;
}

// 13/3 S^2, an exact zero raised to a constant that no other indicator comes near
template <typename real>
__device__ __forceinline__ pair_t<real> weno_sq(pair_t<real> s) {
  return p_fma(p_mul(s, p_set(real(13) / real(3))), s, p_set(sizeof(real) == 4 ? real(1e-40) : real(1e-280)));
}

// The five terms of a face (see above): S on the three stencils and the cell's two differences.
template <typename real>
struct WenoTerms {
  pair_t<real> sm, s0, sp, dm, dc;
};

// num / s for 0 <= num <= s, s > 0 of any size (single precision: the reciprocal instruction wants a
// normal operand; both are scaled by the same power of two)
__device__ __forceinline__ float ratio_to(float num, float s) {
  const float f = s < 1e-20f ? 1.8446744e19f : (s > 1e20f ? 5.4210109e-20f : 1.0f);  // 2^64, 2^-64
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(s * f));
  return (num * f) * r;
}
__device__ __forceinline__ double ratio_to(double num, double s) { return num / s; }

// sum_q w_q (candidate_q - G_c) / sum_q w_q, the correction of the cell value, where the fast weights do not
// hold: Table IV for vanishing indicators, delta_q (sigma_min / sigma_q)^2 otherwise.
template <typename real>
__device__ __forceinline__ real weno_corr_slow1(real sm, real s0, real sp, real dm, real dc, bool up) {
  const real k = real(13) / real(3);
  const real um = radd(radd(dm, dm), sm), u0 = radd(dm, dc), uc = radd(radd(dc, dc), -sp);
  const real bm = rfma(um, um, rmul(rmul(sm, k), sm)), b0 = rfma(u0, u0, rmul(rmul(s0, k), s0)),
             bp = rfma(uc, uc, rmul(rmul(sp, k), sp));
  const real h3 = up ? real(3) : real(-3), lm = up ? real(0.1) : real(0.3), lp = up ? real(0.3) : real(0.1);
  const real qm = rfma(um, h3, sm), q0 = rfma(u0, h3, s0), qp = rfma(uc, h3, sp);
  const real mn = vmin(bm, vmin(b0, bp));
  real wm, w0, wp;
  if (mn == real(0)) {
    wm = bm == real(0) ? lm : real(0);
    w0 = b0 == real(0) ? real(0.6) : real(0);
    wp = bp == real(0) ? lp : real(0);
  } else {
    const real rm = ratio_to(mn, bm), r0 = ratio_to(mn, b0), rp = ratio_to(mn, bp);
    wm = lm * rm * rm, w0 = real(0.6) * r0 * r0, wp = lp * rp * rp;
  }
  return vdiv(rfma(wm, qm, rfma(w0, q0, rmul(wp, qp))), radd(radd(wm, w0), wp)) * (real(1) / real(12));
}
template <typename real>
__device__ __forceinline__ pair_t<real> weno_corr_slow(const WenoTerms<real>& t, bool up) {
  return p_make(weno_corr_slow1<real>(t.sm.x, t.s0.x, t.sp.x, t.dm.x, t.dc.x, up),
                weno_corr_slow1<real>(t.sm.y, t.s0.y, t.sp.y, t.dm.y, t.dc.y, up));
}

// Whether the fast weights hold for several faces.  (A test and a rarely taken branch at every face
// cost registers, code and issue slots.)
template <typename real>
struct WenoRange {
  bool good = true;
  __device__ __forceinline__ void add(pair_t<real> f) { good = good && weno_holds(f); }
  __device__ __forceinline__ bool ok() const { return good; }
};
// The value of a face from the cell's and its terms by the fast weights, NaN where they do not hold;
// K = false: k* are not read, 13/3 S^2 is formed here.
template <typename real, bool K>
__device__ __forceinline__ pair_t<real> weno_face(pair_t<real> g0, const WenoTerms<real>& t, pair_t<real> km,
                                                  pair_t<real> k0, pair_t<real> kp, const WenoSide<real>& w) {
  using P = pair_t<real>;
  const P um = p_add(p_add(t.dm, t.dm), t.sm), u0 = p_add(t.dm, t.dc), up = p_sub(p_add(t.dc, t.dc), t.sp);
  auto sq = [](P s) { return weno_sq<real>(s); };
  const P bm = p_fma(um, um, K ? km : sq(t.sm)), b0 = p_fma(u0, u0, K ? k0 : sq(t.s0)),
          bp = p_fma(up, up, K ? kp : sq(t.sp));
  const P r = p_make(inv_pow2_top(bm.x, b0.x, bp.x), inv_pow2_top(bm.y, b0.y, bp.y));
  const P xm = p_mul(bm, r), x0 = p_mul(b0, r), xp = p_mul(bp, r);
  const P A = p_mul(x0, xp), B = p_mul(xm, xp), C = p_mul(xm, x0);
  const P wm = p_mul(p_mul(A, A), w.dm), w0 = p_mul(B, B), wp = p_mul(p_mul(C, C), w.dp);
  const P den = p_add(p_add(wm, w0), wp);
  const P qm = p_fma(um, w.h3, t.sm), q0 = p_fma(u0, w.h3, t.s0), qp = p_fma(up, w.h3, t.sp);
  const P num = p_fma(wm, qm, p_fma(w0, q0, p_mul(wp, qp)));
  const P i = p_rcp(den);
  return p_fma(num, p_make(i.x * (real(1) / real(12)), i.y * (real(1) / real(12))), g0);
}

// The walk's state around the upwind cell: cell values g0 (the cell), g1, g2 (the next two), the
// differences dm (c - 1/2), dc (c + 1/2), dn (c + 3/2), S on c - 1, c, c + 1, and with K also 13/3 S^2
// there (six registers more, four operations less).
template <typename real, bool K>
struct WenoWin {
  using P = pair_t<real>;
  P g0, g1, g2, dm, dc, dn, sm, s0, sp, km, k0, kp;
  // five neighbouring cells in walk order, centred on c
  __device__ __forceinline__ void start(P a, P b, P c, P d, P e) {
    const P d0 = p_sub(b, a);
    g0 = c, g1 = d, g2 = e;
    dm = p_sub(c, b), dc = p_sub(d, c), dn = p_sub(e, d);
    sm = p_sub(dm, d0), s0 = p_sub(dc, dm), sp = p_sub(dn, dc);
    if constexpr (K) km = weno_sq<real>(sm), k0 = weno_sq<real>(s0), kp = weno_sq<real>(sp);
  }
  __device__ __forceinline__ void push(P f) {  // one cell on
    g0 = g1, g1 = g2;
    dm = dc, dc = dn, dn = p_sub(f, g2);
    g2 = f;
    sm = s0, s0 = sp, sp = p_sub(dn, dc);
    if constexpr (K) km = k0, k0 = kp, kp = weno_sq<real>(sp);
  }
  __device__ __forceinline__ WenoTerms<real> terms() const { return WenoTerms<real>{sm, s0, sp, dm, dc}; }
  __device__ __forceinline__ P fast(const WenoSide<real>& w) const {
    if constexpr (K) return weno_face<real, true>(g0, terms(), km, k0, kp, w);
    else return weno_face<real, false>(g0, terms(), sm, sm, sm, w);
  }
  // the interface value on the cell's side w (times the scale of G), where the range stays ok
  __device__ __forceinline__ P face(const WenoSide<real>& w, WenoRange<real>& range) const {
    const P f = fast(w);
    range.add(f);
    return f;
  }
  __device__ __forceinline__ bool in_range(bool up) const {  // whether face() holds for this face
    WenoSide<real> w;
    w.set(up);
    return weno_holds(fast(w));
  }
  // the value, checked at once
  __device__ __forceinline__ P face_checked(const WenoSide<real>& w) const {
    P f = fast(w);
    if (__builtin_expect(!weno_holds(f), 0)) f = face_any(w.h3.x > real(0));
    return f;
  }
  // the value in any case
  __device__ __forceinline__ P face_any(bool up) const { return p_add(g0, weno_corr_slow<real>(terms(), up)); }
};

// ---------------------------------------------------------------- equilibrium
// Moment vector m_s of the truncated equilibrium factor g_{a,k} = sum_s tab[k][s] m_s
// (Sec. IV.D).  Full range (Eq. eq_gak_H): m_l = E[He_l(X)] / l!, X ~ N(u, T),
// from l m_l = u m_{l-1} + (T - 1) m_{l-2} (generating function
// exp(t u + t^2 (T - 1) / 2)).  Half range (Eq. eq_gak_hh): m_s are the
// half-line moments int_0^inf x^s N(x; u, T) dx, from
// M_0 = (1 + erf(u / sqrt(2T))) / 2, M_1 = u M_0 + T N(0; u, T),
// M_s = u M_{s-1} + (s - 1) T M_{s-2} (integration by parts); the negative
// semi-axis uses u -> -u.
template <typename T_>
__device__ __forceinline__ T_ erf_t(T_ x);
template <>
__device__ __forceinline__ float erf_t<float>(float x) { return erff(x); }
template <>
__device__ __forceinline__ double erf_t<double>(double x) { return erf(x); }
__device__ __forceinline__ float exp_t(float x) { return expf(x); }
__device__ __forceinline__ double exp_t(double x) { return exp(x); }
__device__ __forceinline__ float rsqrt_t(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsqrt_t(double x) { return rsqrt(x); }

template <typename R>
__device__ __forceinline__ void eq_moment_vector(int kind, int N, R u, R T, R* m) {
  if (kind == 0) {
    m[0] = R(1);
    if (N >= 1) m[1] = u;
    for (int l = 2; l <= N; ++l) m[l] = (u * m[l - 1] + (T - R(1)) * m[l - 2]) * (R(1) / R(l));
  } else {
    const R g0 = exp_t(-u * u / (R(2) * T)) * rsqrt_t(R(2) * R(3.14159265358979323846) * T);
    m[0] = R(0.5) * (R(1) + erf_t<R>(u * rsqrt_t(R(2) * T)));
    if (N >= 1) m[1] = u * m[0] + T * g0;
    for (int s = 2; s <= N; ++s) m[s] = u * m[s - 1] + R(s - 1) * T * m[s - 2];
  }
}

// 1 / sqrt(2 pi T), the peak of the unit Gaussian of variance T.  Every half-range equilibrium factor
// carries it, so a rounding that is the same in all cells would not average out: in single
// precision 2 pi T is held as a pair (the constant alone rounds by 2.8e-8; 1 / sqrt(pi) by
// 5.2e-8) and one step of Newton's iteration takes the rest of it and the instruction's error out.
__device__ __forceinline__ float gauss_peak(float T) {
  const float hi = 6.2831854820251464844f, lo = -1.7484555e-7f;  // 2 pi = hi + lo
  const float y = __fmul_rn(hi, T), yl = __fmaf_rn(lo, T, __fmaf_rn(hi, T, -y));
  const float r = rsqrtf(y), yr = __fmul_rn(y, r);
  const float e = __fmaf_rn(-yr, r, 1.0f) - __fmaf_rn(__fmaf_rn(y, r, -yr), r, yl * (r * r));
  return __fmaf_rn(0.5f * r, e, r);
}
__device__ __forceinline__ double gauss_peak(double T) { return rsqrt(6.28318530717958647692 * T); }

// Moment vector of the truncated equilibrium on one axis (the recurrences of eq_moment_vector),
// every entry up to order nmax, with the 1/l factors as constants.
template <typename R>
__device__ __forceinline__ void eq_moments_fast(int kind, int nmax, R u, R T, R* m) {
  R a, b, c;  // m_l = (u m_{l-1} + h c m_{l-2}) f: h = 1, f = 1 / l (full range) or h = l - 1, f = 1
  if (kind == 0) {
    a = R(1), b = u, c = T - R(1);
  } else {
    const R x = u * rsqrt_t(R(2) * T);
    const R g0 = exp_t(-x * x) * gauss_peak(T);  // N(0; u, T)
    a = R(0.5) * (R(1) + erf_t<R>(x));
    b = u * a + T * g0, c = T;
  }
  m[0] = a;
  m[1] = b;
#pragma unroll
  for (int l = 2; l < MAXN; ++l) {
    if (l > nmax) break;
    const R x = (u * b + (kind == 0 ? R(1) : R(l - 1)) * c * a) * (kind == 0 ? R(1.0 / l) : R(1));
    m[l] = x;
    a = b;
    b = x;
  }
}

// 1 / tau of the conventions of relaxation_time, ikn = 1 / Kn
template <typename R>
__device__ __forceinline__ R relaxation_rate(int mode, R ikn, R n, R T) {
  const R r = n * ikn;
  return mode == 0 ? r * T : mode == 1 ? r * R(1.5957691216057307117) : r;  // sqrt(8 / pi)
}

template <typename R>
__device__ __forceinline__ R relaxation_time(int mode, R kn, R n, R T) {
  if (mode == 0) return kn / (n * T);
  if (mode == 1) return R(0.62665706865775012560) * kn / n;  // sqrt(pi / 8)
  return kn / n;
}

// ---------------------------------------------------------------- bulk copy + mbarrier
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

// One-dimensional bulk copy global -> shared completing on the mbarrier (16-byte
// aligned addresses, size a multiple of 16).
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// One-dimensional bulk copy shared -> global (bulk-group completion).
__device__ __forceinline__ void bulk_s2g(void* dst, const void* src, unsigned bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)),
               "r"(bytes)
               : "memory");
}

// Commit the issued bulk stores as a group; wait until every
// committed group of this thread has read its shared-memory source; wait until
// every committed group has completed.
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Programmatic dependent launch (launch_dependent in vlb_launch.h): a grid launched as dependent starts
// once every CTA of the grid before it has called grid_launch_dependents (or ended), and its
// grid_dependency_wait returns when that grid has completed and its writes are visible; before it
// only the launch's own parameters and tables that no kernel writes are read.  Without such a
// launch both do nothing.
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Bounded wait for the phase with the given parity; false on timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity, unsigned long long max_polls) {
  uint32_t done = 0;
  for (unsigned long long it = 0; it < max_polls; ++it) {
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// Knuth's TwoSum: s = fl(a + b) and the exact rounding error err = a + b - s.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& err) {
  s = __fadd_rn(a, b);
  const float bp = __fsub_rn(s, a);
  err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
}

// Compensated butterfly sum over each group of W neighbouring lanes in single precision.  Each step
// adds the partner's value with TwoSum, and the errors accumulate in e.  On return every lane of a
// group holds the same (s, e), whose sum s + e carries about twice the float precision, so a
// reduction that would otherwise need the 1/64-rate FP64 pipe stays on FP32.
template <int W>
__device__ __forceinline__ void group_sum_comp(float& s, float& e) {
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) {
    const float s2 = __shfl_xor_sync(0xffffffffu, s, o), e2 = __shfl_xor_sync(0xffffffffu, e, o);
    float t, err;
    two_sum(s, s2, t, err);
    s = t;
    e = __fadd_rn(__fadd_rn(e, e2), err);
  }
}

// Plain sum over each group of W neighbouring lanes.
template <int W, typename T>
__device__ __forceinline__ T group_sum(T v) {
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <typename real>
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

}  // namespace vlb
