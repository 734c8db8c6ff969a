// Device-side building blocks of the adaptive D2Q21 LBM step (sm_103a).
//
// The lattice, the 8-moment numerical equilibrium and its FP64 Newton solve,
// the shift criterion and Grad's reconstruction, written for one node per
// thread. Loops over velocities are fully unrolled with compile-time velocity
// components, so every multiplication by a zero component disappears and the
// sums below touch only the velocities that contribute.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "alb_cvt.cuh"

namespace alb {

constexpr int Q = 21;   // D2Q21
constexpr int NM = 8;   // 8-moment constraint set (Eq. 8moments)
constexpr int NPLANES = 2 * Q;  // f and g planes

// D2Q21 velocity set (Fig. 1 / Tab. 3 reading): rest, axis 1, diagonal 1,
// axis 2, diagonal 2, axis 3. The index order is part of the C ABI
// (alb_velocities, alb_equilibrium).
__host__ __device__ __forceinline__ constexpr int XI_X(int i) {
  return i == 1 ? 1 : i == 3 ? -1 : i == 5 ? 1 : i == 6 ? -1 : i == 7 ? -1 : i == 8 ? 1
       : i == 9 ? 2 : i == 11 ? -2 : i == 13 ? 2 : i == 14 ? -2 : i == 15 ? -2 : i == 16 ? 2
       : i == 17 ? 3 : i == 19 ? -3 : 0;
}
__host__ __device__ __forceinline__ constexpr int XI_Y(int i) {
  return i == 2 ? 1 : i == 4 ? -1 : i == 5 ? 1 : i == 6 ? 1 : i == 7 ? -1 : i == 8 ? -1
       : i == 10 ? 2 : i == 12 ? -2 : i == 13 ? 2 : i == 14 ? 2 : i == 15 ? -2 : i == 16 ? -2
       : i == 18 ? 3 : i == 20 ? -3 : 0;
}
// Monomial k of the 8-moment set at velocity i: 1, x, y, x^2, xy, y^2, x|xi|^2, y|xi|^2.
__host__ __device__ __forceinline__ constexpr int PM(int k, int i) {
  return k == 0 ? 1 : k == 1 ? XI_X(i) : k == 2 ? XI_Y(i) : k == 3 ? XI_X(i) * XI_X(i)
       : k == 4 ? XI_X(i) * XI_Y(i) : k == 5 ? XI_Y(i) * XI_Y(i)
       : k == 6 ? XI_X(i) * (XI_X(i) * XI_X(i) + XI_Y(i) * XI_Y(i))
       : XI_Y(i) * (XI_X(i) * XI_X(i) + XI_Y(i) * XI_Y(i));
}

// Lattice code of a shift U in [-3, 3]^2: one byte per node.
__host__ __device__ __forceinline__ int lat_code(int ux, int uy) { return (ux + 3) + 7 * (uy + 3); }
__host__ __device__ __forceinline__ int lat_ux(int c) { return c % 7 - 3; }
__host__ __device__ __forceinline__ int lat_uy(int c) { return c / 7 - 3; }

// A double in the population precision P: FP32 rounded on the integer pipe
// (cvt_f32_rn, the hardware rounding for every value of FP32's normal range),
// FP64 unchanged.
template <typename P>
__device__ __forceinline__ P to_p(double v);
template <>
__device__ __forceinline__ float to_p<float>(double v) { return cvt_f32_rn(v); }
template <>
__device__ __forceinline__ double to_p<double>(double v) { return v; }

// Smallest cap on the iterations (Params::maxit) under which a solve may take its
// early steps in FP32: from one start such a solve takes at most 30 FP32 steps and
// 7 residuals in 64 bits (it may try two starts, as the FP64 iteration does, whose
// cap is per start too). What does not converge under a smaller cap has to fail.
constexpr int MIXED_MAXIT = 37;

// Physical and numerical parameters of one flow, passed by value.
struct Params {
  int nx, ny;
  int umax;
  int bcx, bcy;      // 0 periodic, 1 zero-gradient
  int sensor;
  int maxit;
  int warm;          // 1: solves start from the previous step's multipliers
  int rule;          // where ranges overlap: 0 history, 1 neighbourhood
  int moments;       // constraint set: 8, or 4 (reduced model)
  int mixed64;       // FP64 plain: 1, the early Newton steps run in FP32
  int shakhov;       // 1: Pr != 1, heat-flux term of App. E in the collision
  double nu, gamma, n0, tol;
  double prandtl;    // Pr: tau_Pr = 1/2 + (nu/Pr)/T, kappa = rho Cp nu / Pr
  double overlap;    // widening of the current shift's range (0: Eq. criterion)
  double cv, cp;     // Cv = 1/(gamma-1), Cp = gamma Cv
  double half_gm1;   // (gamma - 1) / 2 = 1 / (2 Cv)
  double icp, kappa_nu;  // 1 / Cp, nu / Pr (heat conduction: kappa = rho Cp nu / Pr)
  double seps[3], salpha[3];
  double skx[4], sky[4];  // sensor knots: log10(eps) and alpha (host-computed)
  double thr[6];          // criterion thresholds (t + 1) - n0, t = -umax .. umax - 1
  double wlo[7], whi[7];  // widened range of shift n = j - 3: ((n - n0) - w, ((n + 1) - n0) + w]
};

// Comparisons of the criterion on the integer pipe: an FP64 compare takes a slot
// of the FP64 pipe, which bounds FP64 plain. order_key maps a double's
// bits to a signed integer in IEEE order (negative values have their
// magnitude bits flipped). Integer order then equals IEEE order for all
// non-NaN values except +0 against -0, which cannot meet here: the host's
// thresholds are differences of distinct values, never -0, and a velocity
// ubar + U with an integer U is never -0. A NaN u compares false both ways,
// as in IEEE.
__device__ __forceinline__ long long order_key(double v) {
  const long long b = __double_as_longlong(v);
  return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ bool not_nan(double v) {
  return (__double_as_longlong(v) & 0x7fffffffffffffffLL) <= 0x7ff0000000000000LL;
}
__device__ __forceinline__ bool gt_order(double u, double v) {  // u > v
  return not_nan(u) && order_key(u) > order_key(v);
}
__device__ __forceinline__ bool le_order(double u, double v) {  // u <= v
  return not_nan(u) && order_key(u) <= order_key(v);
}

// Eq. criterion with the host-computed thresholds of Params (the same IEEE
// values as select_shift computes).
__device__ __forceinline__ int select_shift_thr(double u, const Params& pr) {
  int n = -pr.umax;
#pragma unroll
  for (int t = 0; t < 6; ++t)
    if (t < 2 * pr.umax && gt_order(u, pr.thr[t])) ++n;
  return n;
}

// Overlapping ranges chosen by history (Sec. III.A.2): keep the current shift
// while current - n0 - w < u <= current + 1 - n0 + w, else Eq. criterion.
// The widened bounds come from the host (same IEEE operations as the oracle).
__device__ __forceinline__ int select_shift_kept(double u, int current, const Params& pr) {
  if (order_key(pr.overlap) > 0 && gt_order(u, pr.wlo[current + 3]) &&
      le_order(u, pr.whi[current + 3]))
    return current;
  return select_shift_thr(u, pr);
}

// Overlapping ranges chosen by the neighbourhood (Sec. III.A.2): among the
// shifts whose widened range holds u, the one most of the eight surrounding
// nodes use (component `axis` of their lattice codes nb[0..7]); the
// criterion's shift unless another candidate is used by strictly more.
__device__ __forceinline__ int select_shift_neighbours(double u, int axis, const uint8_t nb[8],
                                                       const Params& pr) {
  const int c = select_shift_thr(u, pr);
  int cnt[7] = {0, 0, 0, 0, 0, 0, 0};  // neighbours per shift n = j - 3
#pragma unroll
  for (int j = 0; j < 8; ++j) cnt[(axis ? lat_uy(nb[j]) : lat_ux(nb[j])) + 3] += 1;
  int best = c, best_count = cnt[c + 3];
  // with w <= 1 only the criterion's neighbours c - 1 and c + 1 can also hold u
#pragma unroll
  for (int d = -1; d <= 1; d += 2) {
    const int n = c + d;
    if (n < -pr.umax || n > pr.umax) continue;
    if (!(gt_order(u, pr.wlo[n + 3]) && le_order(u, pr.whi[n + 3]))) continue;
    if (cnt[n + 3] > best_count) {
      best = n;
      best_count = cnt[n + 3];
    }
  }
  return best;
}

// Product rounded by itself. The compiler may fuse a product and a sum into one
// FMA or not, depending on the code around them; in the code that several
// kernels share (single-flow and batched variants) every FMA is therefore
// written out and every other product is one of these, so that a node's update
// gives the same bits in all of them.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// s + c * v with c a compile-time integer after unrolling: the zero and unit
// cases fold away, keeping IEEE semantics for the rest.
template <typename R>
__device__ __forceinline__ R madd(R s, R v, int c) {
  if (c == 0) return s;
  if (c == 1) return s + v;
  if (c == -1) return s - v;
  return fma(v, (R)c, s);
}

// Eq. criterion with offset n0: U = n iff n - n0 < u <= n + 1 - n0, clamped.
__device__ __forceinline__ int select_shift(double u, double n0, int umax) {
  int n = -umax;
  // count the thresholds n + 1 - n0 (n = -umax .. umax-1) that u lies above
  for (int t = -umax; t < umax; ++t) {
    const double hi = (double)(t + 1) - n0;
    if (u > hi) n = t + 1;
  }
  return n;
}

// alpha(eps_Kn) of the kinetic sensor (Sec. IV.A.2): 1 up to seps[0], then
// continuous and piecewise linear in log10(eps) through (seps[1], salpha[0]),
// (seps[2], salpha[1]), (10 seps[2], salpha[2]), constant beyond. Evaluated
// in the population precision P.
template <typename P>
__device__ __forceinline__ P sensor_alpha(const Params& pr, P eps) {
  if (!(eps > to_p<P>(pr.seps[0]))) return (P)1;
  const P l = log10(eps);
#pragma unroll
  for (int k = 0; k < 3; ++k)
    if (l <= (P)pr.skx[k + 1])
      return (P)pr.sky[k] + mul_rn((P)pr.sky[k + 1] - (P)pr.sky[k], l - (P)pr.skx[k]) /
                                ((P)pr.skx[k + 1] - (P)pr.skx[k]);
  return (P)pr.sky[3];
}

// Targets of Eqs. G0_8mom..G3yaa_8mom per unit density, lattice frame.
__device__ __forceinline__ void targets(double ubx, double uby, double T, double m[NM]) {
  const double u2 = fma(ubx, ubx, mul_rn(uby, uby)), q = fma(4.0, T, u2);
  m[0] = 1.0;
  m[1] = ubx;
  m[2] = uby;
  m[3] = fma(ubx, ubx, T);
  m[4] = mul_rn(ubx, uby);
  m[5] = fma(uby, uby, T);
  m[6] = mul_rn(ubx, q);
  m[7] = mul_rn(uby, q);
}

// p_i = exp(-(1 + lambda . P(xi_i))) for all 21 velocities (Eq. exponential / rho).
__device__ __forceinline__ void exp_family(const double lam[NM], double p[Q]) {
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    double s = 1.0 + lam[0];
#pragma unroll
    for (int k = 1; k < NM; ++k) s = madd(s, lam[k], PM(k, i));
    p[i] = exp(-s);
  }
}

enum { NEWTON_OK = 0, NEWTON_MAXIT = 1, NEWTON_SINGULAR = 2, NEWTON_UNREALIZABLE = 3 };

// Maxwellian starting multipliers, lambda_0 from the normalisation sum p = 1.
__device__ __forceinline__ void maxwellian_guess(double ubx, double uby, double T, double lam[NM]) {
  const double iT = 1.0 / T;
#pragma unroll
  for (int k = 0; k < NM; ++k) lam[k] = 0.0;
  lam[1] = -ubx * iT;
  lam[2] = -uby * iT;
  lam[3] = 0.5 * iT;
  lam[5] = 0.5 * iT;
  double p[Q];
  exp_family(lam, p);
  double Z = 0.0;
#pragma unroll
  for (int i = 0; i < Q; ++i) Z += p[i];
  lam[0] = log(Z);
}

// exp(-(1 + lambda . P(xi_i))) for one velocity given at run time.
__device__ __forceinline__ double exp_family_one(const double lam[NM], int cx, int cy) {
  const double x = cx, y = cy, r2 = cx * cx + cy * cy;
  double s = 1.0 + lam[0];
  s = fma(lam[1], x, s);
  s = fma(lam[2], y, s);
  s = fma(lam[3], x * x, s);
  s = fma(lam[4], x * y, s);
  s = fma(lam[5], y * y, s);
  s = fma(lam[6], x * r2, s);
  s = fma(lam[7], y * r2, s);
  return exp(-s);
}

// Grad's factors (Eqs. GradGeneral_f, GradGeneral_g) for cbar = c_i - u:
// phi_f = phi_s + phi_q with phi_s the traceless viscous stress part (mu =
// rho nu) and phi_q the Fourier heat-flux part (kappa = rho Cp nu / Pr), and
// phi_g. phi_q has the shape of the heat-flux term of App. E.
__device__ __forceinline__ void grad_phi(const Params& pr, double rho, double T, double cbx,
                                         double cby, const double du[2][2], const double dT[2],
                                         double* phi_f, double* phi_g, double* phi_q) {
  // two reciprocals serve all quotients (an FP64 division is some nine
  // operations of the FP64 pipe)
  const double iT = 1.0 / T, irho = 1.0 / rho;
  const double mu = mul_rn(rho, pr.nu);
  const double kappa = mul_rn(mul_rn(rho, pr.cp), pr.kappa_nu);
  const double div = du[0][0] + du[1][1];
  const double sxx = mul_rn(-mu, fma(2.0, du[0][0], -div));
  const double syy = mul_rn(-mu, fma(2.0, du[1][1], -div));
  const double sxy = mul_rn(-mu, du[0][1] + du[1][0]);
  const double qx = mul_rn(-kappa, dT[0]);
  const double qy = mul_rn(-kappa, dT[1]);
  const double cxx = mul_rn(cbx, cbx), cyy = mul_rn(cby, cby);
  const double c2 = cxx + cyy;
  const double qc = fma(qx, cbx, mul_rn(qy, cby));
  const double irc = mul_rn(irho, pr.icp);
  const double iT2 = mul_rn(iT, iT);
  const double ps = mul_rn(fma(sxx, cxx, fma(mul_rn(2.0, sxy), mul_rn(cbx, cby), mul_rn(syy, cyy))),
                           mul_rn(mul_rn(0.5, iT2), irho));
  const double pq = mul_rn(mul_rn(qc, mul_rn(iT2, irc)), fma(mul_rn(0.5, c2), iT, -pr.cp));
  *phi_f = ps + pq;
  *phi_q = pq;
  *phi_g = mul_rn(mul_rn(2.0, qc), irc);
}

// Grad's factors as polynomials of the lattice velocity xi = c_i - U: with cbar = xi
// - ubar, phi_f has the eight monomials P_k (a), phi_g is linear (g). All 21
// factors then take some 100 operations instead of 30 each.
__device__ __forceinline__ void grad_poly(const Params& pr, double rho, double T, double ubx,
                                          double uby, const double du[2][2], const double dT[2],
                                          double a[NM], double g[3]) {
  const double iT = 1.0 / T, irho = 1.0 / rho;
  const double mu = rho * pr.nu, kappa = rho * pr.cp * pr.kappa_nu;
  const double div = du[0][0] + du[1][1];
  const double irc = irho * pr.icp, iT2 = iT * iT;
  const double s0 = 0.5 * iT2 * irho;
  // stress: A cx^2 + B cx cy + C cy^2
  const double A = -s0 * mu * (2.0 * du[0][0] - div), C = -s0 * mu * (2.0 * du[1][1] - div);
  const double Bq = -2.0 * s0 * mu * (du[0][1] + du[1][0]);
  // heat flux: (Qx cx + Qy cy) (h |cbar|^2 - cp), with cbar expanded as
  // (Qx x + Qy y - L0) (h r^2 - n1 x - n2 y + n0)
  const double k1 = -iT2 * irc * kappa, h = 0.5 * iT;
  const double Qx = k1 * dT[0], Qy = k1 * dT[1];
  const double L0 = Qx * ubx + Qy * uby;
  const double n1 = 2.0 * h * ubx, n2 = 2.0 * h * uby;
  const double n0 = h * (ubx * ubx + uby * uby) - pr.cp;
  a[0] = A * ubx * ubx + Bq * ubx * uby + C * uby * uby - L0 * n0;
  a[1] = -2.0 * A * ubx - Bq * uby + Qx * n0 + L0 * n1;
  a[2] = -2.0 * C * uby - Bq * ubx + Qy * n0 + L0 * n2;
  a[3] = A - Qx * n1 - L0 * h;
  a[4] = Bq - Qx * n2 - Qy * n1;
  a[5] = C - Qy * n2 - L0 * h;
  a[6] = Qx * h;
  a[7] = Qy * h;
  const double k2 = -2.0 * irc * kappa;
  g[1] = k2 * dT[0];
  g[2] = k2 * dT[1];
  g[0] = -(g[1] * ubx + g[2] * uby);
}

// Resolve a coordinate along one axis: periodic wrap or zero-gradient clamp.
__device__ __forceinline__ int resolve(int x, int n, int bc, bool* ghost) {
  if (bc == 0) {
    if ((unsigned)x < (unsigned)n) return x;  // inside: no remainder needed
    int r = x % n;
    if (r < 0) r += n;
    return r;
  }
  if (x < 0) { *ghost = true; return 0; }
  if (x >= n) { *ghost = true; return n - 1; }
  return x;
}

// Warp-aggregated counter increment (all lanes of the warp must call it).
__device__ __forceinline__ void warp_count(unsigned long long* ctr, unsigned v) {
  const unsigned s = __reduce_add_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0 && s) atomicAdd(ctr, (unsigned long long)s);
}

}  // namespace alb
