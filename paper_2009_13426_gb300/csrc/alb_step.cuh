// Per-node update of the adaptive D2Q21 LBM step (Sec. IV.A.3), shared by the
// single-flow and the batched kernels.
//
// One thread updates one node. Its pulled populations (42, precision P) and
// the 21 equilibrium values per unit density of its latest equilibrium solve
// (64 bits each: FP64, or Q63 fixed point from the FP32 form's solver) sit in
// two columns of the block's dynamic shared memory, with the block size as
// stride.
#pragma once

#include <type_traits>

#include "alb_internal.h"
#include "alb_mixed.cuh"

namespace alb {

constexpr int BLOCK = 128;

// Dynamic shared memory of a block: the tables of the exponentials (FP64, and
// fixed-point in the FP32 form), then the two columns of every thread.
template <typename P>
constexpr size_t table_bytes() {
  return EXPT_N * sizeof(double) +
         (std::is_same<P, float>::value ? FIXT_N * sizeof(uint64_t) : 0);
}
template <typename P, int B = BLOCK>
constexpr size_t smem_bytes() {
  return table_bytes<P>() + (size_t)NPLANES * B * sizeof(P) + (size_t)Q * B * sizeof(double);
}

// Shared columns of this thread: populations (P) and equilibrium (double),
// both with stride B (the block size); the tables of the solves.
template <typename P, int B>
struct Columns {
  P* pop;
  double* eq;
  const uint64_t* fixtab;
  const double* exptab;
  // All threads of the block construct it (it includes a barrier).
  __device__ __forceinline__ explicit Columns(unsigned char* smem) {
    fixtab = reinterpret_cast<const uint64_t*>(smem + EXPT_N * sizeof(double));
    exptab = reinterpret_cast<const double*>(smem);
    if constexpr (std::is_same<P, float>::value) load_fixtab(const_cast<uint64_t*>(fixtab));
    load_exptab(const_cast<double*>(exptab));
    pop = reinterpret_cast<P*>(smem + table_bytes<P>()) + threadIdx.x;
    eq = reinterpret_cast<double*>(smem + table_bytes<P>() + (size_t)NPLANES * B * sizeof(P)) +
         threadIdx.x;
  }
};

// A node: density, velocity in the lattice frame, temperature, next lattice.
struct NodeState {
  double rho, ubx, uby, T;
  int code2;
};

// A solve as handed to the function that is not inlined. What the caller keeps
// across that call is kept small: values live across a call are spilled around it
// on every path, also where the call is not taken.
struct SolveIO {
  double ubx, uby, T;
  float lam[NM];
  bool warm, fixed;
};

// Counts of a solve, added to the flow's counters by the lanes that made one. Which
// lanes of the warp run this together does not matter: each of them goes on to the
// sum with the mask that names them, and every lane's count is in one such sum.
__device__ __forceinline__ void lanes_count(unsigned long long* ctr, unsigned v) {
  const unsigned m = __activemask();
  const unsigned sum = __reduce_add_sync(m, v);
  if ((int)(threadIdx.x & 31) == __ffs(m) - 1 && sum) atomicAdd(ctr, (unsigned long long)sum);
}

// Solves of the FP32 form outside its inlined path: the reduced model, and the
// states the fixed-point refinement does not take.
template <int B>
static __device__ __noinline__ int solve_other(const Params& pr, const double* exptab,
                                               const uint64_t* fixtab, double* eq, SolveIO* io,
                                               unsigned long long* ctr) {
  const double ubx = io->ubx, uby = io->uby, T = io->T;
  const bool warm = io->warm;
  float lam[NM];
  SolveCount cnt;
  int st;
#pragma unroll
  for (int k = 0; k < NM; ++k) lam[k] = io->lam[k];
  io->fixed = false;
  if (pr.moments == 4) {
    // (under a small cap on the iterations, the FP64 Newton alone)
    int it32 = 0, ev = 0, up = 0;
    st = NEWTON_MAXIT;
    if (pr.maxit >= MIXED_MAXIT)
      st = solve4_fix(ubx, uby, T, (float)pr.tol, warm, fixtab, reinterpret_cast<uint64_t*>(eq), B,
                      lam, &it32, &ev, &up);
    cnt.fp32_iters = it32;
    cnt.fp64_evals = ev;
    cnt.fp64_updates = up;
    io->fixed = st == NEWTON_OK;
    if (st != NEWTON_OK) {
      double w8[NM], l8[NM];
      int it = 0;
#pragma unroll
      for (int k = 0; k < NM; ++k) w8[k] = warm ? (double)io->lam[k] : 0.0;
      st = newton4_fp64g(ubx, uby, T, pr.tol, pr.maxit, exptab, eq, B, l8, &it, &ev,
                         warm ? w8 : nullptr);
      cnt.fp64_iters += it;
      cnt.fp64_evals += ev;
      if (warm && st != NEWTON_OK && st != NEWTON_UNREALIZABLE) {
        st = newton4_fp64g(ubx, uby, T, pr.tol, pr.maxit, exptab, eq, B, l8, &it, &ev, nullptr);
        cnt.fp64_iters += it;
        cnt.fp64_evals += ev;
      }
#pragma unroll
      for (int k = 0; k < NM; ++k) lam[k] = (float)l8[k];
    }
  } else {
    st = equilibrium_mixed(ubx, uby, T, pr.tol, pr.maxit, exptab, warm ? io->lam : nullptr, eq, B,
                           lam, nullptr, &cnt);
  }
  if (ctr) {
    lanes_count(ctr + CTR_FP32_ITERS, cnt.fp32_iters);
    lanes_count(ctr + CTR_NEWTON_ITERS, cnt.fp64_iters);
    lanes_count(ctr + CTR_FP64_EVALS, cnt.fp64_evals);
    lanes_count(ctr + CTR_FP64_UPDATES, cnt.fp64_updates);
  }
  if (st == NEWTON_OK)
#pragma unroll
    for (int k = 0; k < NM; ++k) io->lam[k] = lam[k];
  return st;
}

// Counts of one node update, added to the flow's counters warp by warp.
template <typename P>
struct NodeCount {
  unsigned n = 0;    // rebuilt pulls (10 bits), those that fell back (10), solves (11), failed (1)
  unsigned fix = 0;  // FP32 form: counts of solve_fix
  SolveCount solve;  // FP64 plain
};
constexpr unsigned N_REC = 1u, N_REC_FAIL = 1u << 10, N_CALLS = 1u << 20, N_FAIL = 1u << 31;

// Equilibrium of one node in the storage precision P: FP32 Newton steps and FP64
// residuals for the FP64 plain path (or all FP64 steps: Params::mixed64), FP32
// Newton with the fixed-point refinement for the FP32 form (solve_other where
// that does not reach). If `warm` is set, both start from the multipliers that
// load(lam) gives. The equilibrium per unit density lands in the thread's column
// (Q63 instead of FP64 where *fixed is set), the multipliers (in the precision P
// the warm start keeps them in) in lam; after a failure lam is the warm start
// again. ctr (or null) counts the solves of solve_other.
template <typename P, int B, typename Load>
__device__ __forceinline__ int node_equilibrium(const Params& pr, const Columns<P, B>& cl,
                                                const NodeState& s, bool warm, Load load, P lam[NM],
                                                NodeCount<P>* nc, unsigned long long* ctr,
                                                bool* fixed) {
  *fixed = false;
  const double ubx = s.ubx, uby = s.uby, T = s.T;
  if (warm) load(lam);
  if (!(s.rho > 0.0) || !(T > 0.0) || !isfinite(T) || !isfinite(ubx) || !isfinite(uby))
    return NEWTON_UNREALIZABLE;
  if constexpr (std::is_same<P, float>::value) {
    int st = NEWTON_SINGULAR;
    if (pr.moments == 8)
      st = solve_fix(ubx, uby, T, (float)pr.tol, warm, cl.fixtab,
                     reinterpret_cast<uint64_t*>(cl.eq), B, lam, &nc->fix);
    *fixed = st == NEWTON_OK;
    if (st != NEWTON_OK) {
      // A refinement that did not take the state leaves multipliers that the FP32
      // phase has converged: the other solve starts there (states near the edge
      // of what the lattice carries take up to 30 FP32 steps, and have the
      // exponents the fixed-point range ends at).
      SolveIO io;
      io.ubx = ubx;
      io.uby = uby;
      io.T = T;
      const bool converged = st == NEWTON_MAXIT;
      io.warm = warm || converged;
      if (converged)
#pragma unroll
        for (int k = 0; k < NM; ++k) io.lam[k] = lam[k];
      else if (warm)
        load(io.lam);
      st = solve_other<B>(pr, cl.exptab, cl.fixtab, cl.eq, &io, ctr);
      *fixed = io.fixed;
      if (st == NEWTON_OK || !warm)
#pragma unroll
        for (int k = 0; k < NM; ++k) lam[k] = io.lam[k];
      else
        load(lam);
    }
    return st;
  } else {
    int it = 0, ev = 0, st = NEWTON_SINGULAR;
    double w[NM];
#pragma unroll
    for (int k = 0; k < NM; ++k) w[k] = lam[k];
    if (pr.moments == 4) {
      st = newton4_fp64g(ubx, uby, T, pr.tol, pr.maxit, cl.exptab, cl.eq, B, lam, &it, &ev,
                         warm ? w : nullptr);
      nc->solve.fp64_iters += it;
      nc->solve.fp64_evals += ev;
      if (warm && st != NEWTON_OK && st != NEWTON_UNREALIZABLE) {
        st = newton4_fp64g(ubx, uby, T, pr.tol, pr.maxit, cl.exptab, cl.eq, B, lam, &it, &ev,
                           nullptr);
        nc->solve.fp64_iters += it;
        nc->solve.fp64_evals += ev;
      }
    } else {
      if (pr.mixed64) {
        int it32 = 0;
        st = solve_mixed64(ubx, uby, T, pr.tol, warm, cl.exptab, cl.eq, B, lam, &it32, &it, &ev);
        nc->solve.fp32_iters += it32;
        nc->solve.fp64_iters += it32 + it;
        nc->solve.fp64_evals += ev;
      }
      if (st != NEWTON_OK) {
        st = newton_fp64g(ubx, uby, T, pr.tol, pr.maxit, cl.exptab, cl.eq, B, lam, &it, &ev,
                          warm ? w : nullptr);
        nc->solve.fp64_iters += it;
        nc->solve.fp64_evals += ev;
      }
      if (warm && st != NEWTON_OK && st != NEWTON_UNREALIZABLE) {
        // the previous multipliers led nowhere: start again from the Maxwellian
        st = newton_fp64g(ubx, uby, T, pr.tol, pr.maxit, cl.exptab, cl.eq, B, lam, &it, &ev,
                          nullptr);
        nc->solve.fp64_iters += it;
        nc->solve.fp64_evals += ev;
      }
    }
    if (st != NEWTON_OK) {
#pragma unroll
      for (int k = 0; k < NM; ++k) lam[k] = w[k];
    }
    return st;
  }
}

// Moment accumulation: plain in FP64; Neumaier-compensated in FP32.
template <typename P>
struct Acc {
  double s = 0.0;
  __device__ __forceinline__ void add(double v) { s += v; }
  __device__ __forceinline__ void add_times(double v, int w) { s = fma(v, (double)w, s); }
  __device__ __forceinline__ double val() const { return s; }
};
template <>
struct Acc<float> {
  float s = 0.0f, c = 0.0f;
  __device__ __forceinline__ void add(float v) {
    const float t = s + v;
    if (fabsf(s) >= fabsf(v))
      c += (s - t) + v;
    else
      c += (v - t) + s;
    s = t;
  }
  // Products by 3 and 9 round once, by themselves. The sums decide a node's next
  // lattice: with another rounding a velocity beside a threshold falls on the
  // other side, which changes that node's result by far more than FP32's
  // rounding. (Sums that keep the products' errors too change the last bit of 15 %
  // of the primitives in a step.)
  __device__ __forceinline__ void add_times(float v, int w) { add(mul_rn(v, (float)w)); }
  __device__ __forceinline__ double val() const { return cvt_f64(s + c); }
};

// Multipliers stored for node k (8 planes of L), moved into the frame of
// lattice (Ux, Uy) from the lattice code they were computed in.
template <typename L>
__device__ __forceinline__ void load_warm(const L* lam, size_t ps, size_t k, int code_from,
                                          int Ux, int Uy, L w[NM]) {
  L l[NM];
#pragma unroll
  for (int j = 0; j < NM; ++j) l[j] = lam[j * ps + k];
  const int dx = lat_ux(code_from) - Ux, dy = lat_uy(code_from) - Uy;
  if (dx == 0 && dy == 0) {
#pragma unroll
    for (int j = 0; j < NM; ++j) w[j] = l[j];
  } else {
    shift_multipliers<L>(l, (L)dx, (L)dy, w);
  }
}

// One value of an equilibrium column in FP64.
template <typename P>
__device__ __forceinline__ double eq_f64(double v, bool fixed) {
  if constexpr (std::is_same<P, float>::value) {
    if (fixed) return fix_to_f64((uint64_t)__double_as_longlong(v));
  }
  return v;
}

// Grad rebuild of a missing pull (Sec. III.B.2, IV.A.3): the post-collision
// population of velocity i = (cx, cy) in the receiver's lattice (Upx, Upy),
// built from the sender's moments at (sx, sy) (possibly a ghost), their
// central differences and the sender's relaxation time:
// h* = h^eq (1 + (1 - 1/tau) phi_h), plus (1/tau - 1/tau_Pr) h^eq phi_h,q for
// Pr != 1 (the collision of App. E applied to the Grad population). `eq` is the
// equilibrium per unit density of velocity i from the solve of this sender in
// this lattice; ok is false if that solve failed: then the value of the
// Maxwellian guess is taken.
template <typename P>
__device__ __forceinline__ void rebuild_value(const Params& pr, const P* __restrict__ mom,
                                              size_t ps, int cx, int cy, int Upx, int Upy, int sx,
                                              int sy, double eq, bool ok, double* fi, double* gi) {
  bool gh = false;
  const int rx = resolve(sx, pr.nx, pr.bcx, &gh);
  const int ry = resolve(sy, pr.ny, pr.bcy, &gh);
  const int xp = resolve(sx + 1, pr.nx, pr.bcx, &gh);
  const int xm = resolve(sx - 1, pr.nx, pr.bcx, &gh);
  const int yp = resolve(sy + 1, pr.ny, pr.bcy, &gh);
  const int ym = resolve(sy - 1, pr.ny, pr.bcy, &gh);
  const size_t nx = (size_t)pr.nx;
  const size_t ks = ry * nx + rx;
  const size_t kxp = ry * nx + xp, kxm = ry * nx + xm, kyp = yp * nx + rx, kym = ym * nx + rx;
  const P* mux = mom + ps;
  const P* muy = mom + 2 * ps;
  const P* mT = mom + 3 * ps;
  const double rho = (double)mom[ks], ux = (double)mux[ks], uy = (double)muy[ks],
               T = (double)mT[ks];
  const double gfac = mul_rn(fma(2.0, pr.cv, -2.0), T);
  if (!ok) {
    if (T > 0.0) {
      double lam[NM];
      maxwellian_guess(ux - Upx, uy - Upy, T, lam);
      *fi = mul_rn(rho, exp_family_one(lam, cx, cy));
    } else {
      *fi = 0.0;
    }
    *gi = mul_rn(gfac, *fi);
    return;
  }
  double du[2][2], dT[2];
  du[0][0] = mul_rn(0.5, (double)mux[kxp] - (double)mux[kxm]);
  du[1][0] = mul_rn(0.5, (double)mux[kyp] - (double)mux[kym]);
  du[0][1] = mul_rn(0.5, (double)muy[kxp] - (double)muy[kxm]);
  du[1][1] = mul_rn(0.5, (double)muy[kyp] - (double)muy[kym]);
  dT[0] = mul_rn(0.5, (double)mT[kxp] - (double)mT[kxm]);
  dT[1] = mul_rn(0.5, (double)mT[kyp] - (double)mT[kym]);
  const double tau = 0.5 + pr.nu / T;
  const double omega = 1.0 - 1.0 / tau;
  const double feq = mul_rn(rho, eq);
  const double cbx = (double)(cx + Upx) - ux;
  const double cby = (double)(cy + Upy) - uy;
  double phf, phg, phq;
  grad_phi(pr, rho, T, cbx, cby, du, dT, &phf, &phg, &phq);
  double ff = fma(omega, phf, 1.0), fg = fma(omega, phg, 1.0);
  if (pr.shakhov) {
    const double w = 1.0 / tau - 1.0 / (0.5 + pr.kappa_nu / T);
    ff = fma(w, phq, ff);
    fg = fma(w, phg, fg);
  }
  *fi = mul_rn(feq, ff);
  *gi = mul_rn(mul_rn(gfac, feq), fg);
}

// The equilibrium column (values per unit density at stride B) in the
// population precision. In the FP32 form every value is rounded to FP32 once,
// in place, into the first word of its slot (the 64-bit value is not read
// again), so that the sensor, the BGK update and the App. E term read the
// same float; the rounding runs on the integer pipe (fix_to_f32, or cvt_f32_rn
// of a column in FP64), not the FP64 pipe. Element i is then at
// [i * eq_stride<P, B>()].
template <typename P, int B>
__device__ __forceinline__ const P* eq_in_precision(double* eq, bool fixed) {
  if constexpr (std::is_same<P, float>::value) {
    float* v = reinterpret_cast<float*>(eq);
    if (fixed) {
#pragma unroll
      for (int i = 0; i < Q; ++i)
        v[2 * i * B] = fix_to_f32((uint64_t)__double_as_longlong(eq[i * B]));
    } else {
#pragma unroll 1
      for (int i = 0; i < Q; ++i) v[2 * i * B] = cvt_f32_rn(eq[i * B]);
    }
    return v;
  } else {
    return eq;
  }
}
template <typename P, int B>
__host__ __device__ constexpr int eq_stride() {
  return std::is_same<P, float>::value ? 2 * B : B;
}

// |f - fe| / fe of the kinetic sensor (Eq. DeltaAvg): a fast division in
// FP32 (its relative error, about 1e-7, is that of the FP32 populations
// themselves, and alpha is continuous in eps), IEEE division in FP64.
__device__ __forceinline__ float rel_dev(float f, float fe) {
  return __fdividef(fabsf(f - fe), fe);
}
__device__ __forceinline__ double rel_dev(double f, double fe) { return fabs(f - fe) / fe; }

// What the collision needs of a node's moments, in the population precision: the
// velocity (bx, by) in the lattice frame is that of the rounded absolute one.
template <typename P>
struct NodeFields {
  P rho, T, bx, by;
};

// Store of a collided node for Pr != 1: BGK plus the heat-flux term of App. E
// (Eqs. Shakhov, prandtlPoly),
//   f* += (1/tau - 1/tau_Pr) q.cbar / (rho Cp T^2) (|cbar|^2 / (2T) - Cp) f^eq,
//   g* += (1/tau - 1/tau_Pr) 2 q.cbar / (rho Cp) g^eq,
// with q_a = 1/2 sum_i cbar_ia (|cbar_i|^2 f_i + g_i) of the pre-collision
// populations st, cbar_i = xi_i - (u - U) (lattice frame, U of lattice
// `code`), tau_Pr = 1/2 + (nu/Pr)/T, both relaxation times scaled by the
// sensor factor tau / (1/2 + nu/T).
template <typename P, int B>
__device__ __forceinline__ void store_shakhov(const Params& pr, const P* st, const P* eqv,
                                              const NodeFields<P>& nf, P tau, size_t k,
                                              size_t ps, P* __restrict__ pop_out) {
  const P Tp = nf.T, rp = nf.rho, bx = nf.bx, by = nf.by;
  const P cp = (P)pr.cp;
  const P gp = mul_rn(fma((P)2, (P)pr.cv, (P)-2), Tp);
  const P tau_pr = mul_rn((P)0.5 + (P)pr.kappa_nu / Tp, tau / ((P)0.5 + (P)pr.nu / Tp));
  const P om = (P)1 / tau;
  const P w = om - (P)1 / tau_pr;
  P qx = 0, qy = 0;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const P cx = (P)XI_X(i) - bx, cy = (P)XI_Y(i) - by;
    const P e = fma(fma(cx, cx, mul_rn(cy, cy)), st[i * B], st[(Q + i) * B]);
    qx = fma(cx, e, qx);
    qy = fma(cy, e, qy);
  }
  qx = mul_rn(qx, (P)0.5);
  qy = mul_rn(qy, (P)0.5);
  const P rc = mul_rn(rp, cp);
  const P af = w / mul_rn(mul_rn(rc, Tp), Tp);
  const P ag = mul_rn(w, (P)2) / rc;
  const P h = (P)0.5 / Tp;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const P fe = mul_rn(eqv[i * eq_stride<P, B>()], rp);
    const P ge = mul_rn(gp, fe);
    const P f = st[i * B];
    const P g = st[(Q + i) * B];
    const P cx = (P)XI_X(i) - bx, cy = (P)XI_Y(i) - by;
    const P c2 = fma(cx, cx, mul_rn(cy, cy));
    const P qc = fma(qx, cx, mul_rn(qy, cy));
    __stcs(&pop_out[i * ps + k],
           fma(mul_rn(mul_rn(af, qc), fma(c2, h, -cp)), fe, fma(om, fe - f, f)));
    __stcs(&pop_out[(Q + i) * ps + k], fma(mul_rn(ag, qc), ge, fma(om, ge - g, g)));
  }
}

// Moments of one node whose 42 pre-collision populations sit in its shared
// column, and the lattice of its next pull.
template <typename P, int B>
__device__ __forceinline__ NodeState node_moments(const Params& pr, const Columns<P, B>& cl,
                                                  int code, const uint8_t* nb) {
  const P* st = cl.pop;
  const int Ux = lat_ux(code), Uy = lat_uy(code);
  Acc<P> ar, ajx, ajy, ae;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const P f = st[i * B];
    const P g = st[(Q + i) * B];
    ar.add(f);
    if (XI_X(i) != 0) ajx.add_times(XI_X(i) > 0 ? f : -f, abs(XI_X(i)));
    if (XI_Y(i) != 0) ajy.add_times(XI_Y(i) > 0 ? f : -f, abs(XI_Y(i)));
    const int c2 = XI_X(i) * XI_X(i) + XI_Y(i) * XI_Y(i);
    if (c2 != 0) ae.add_times(f, c2);
    ae.add(g);
  }
  // Moments (Eq. polyTemp). The velocity and temperature that define the
  // equilibrium's targets are formed in FP64 from the (FP32 or FP64) sums, so
  // that the collision conserves the sums to their own precision; the next
  // lattice (Eq. criterion) is chosen from u = (rho u) / rho in FP64.
  const double rho = ar.val();
  double ubx, uby, T;
  if constexpr (std::is_same<P, float>::value) {
    // FP32 sums: one FP64 reciprocal serves the three quotients (their last
    // FP64 bit lies far below the sums' own precision); 1/(2 Cv) = (gamma-1)/2
    const double ir = 1.0 / rho;
    ubx = mul_rn(ajx.val(), ir);
    uby = mul_rn(ajy.val(), ir);
    T = mul_rn(mul_rn(fma(-rho, fma(ubx, ubx, mul_rn(uby, uby)), ae.val()), ir), pr.half_gm1);
  } else {
    ubx = ajx.val() / rho;
    uby = ajy.val() / rho;
    T = fma(-rho, fma(ubx, ubx, mul_rn(uby, uby)), ae.val()) / mul_rn(2.0 * rho, pr.cv);
  }
  const double ux = ubx + cvt_f64(Ux), uy = uby + cvt_f64(Uy);
  // next lattice: Eq. criterion, or overlapping ranges chosen by history or
  // by the neighbours' current lattices nb[0..7]
  const bool by_nb = order_key(pr.overlap) > 0 && pr.rule == 1 && nb;
  const int code2 = by_nb ? lat_code(select_shift_neighbours(ux, 0, nb, pr),
                                     select_shift_neighbours(uy, 1, nb, pr))
                          : lat_code(select_shift_kept(ux, Ux, pr), select_shift_kept(uy, Uy, pr));
  return NodeState{rho, ubx, uby, T, code2};
}

// Stores a node's moments and lattices; done before the solve, so that little
// of the node is live across it.
template <typename P>
__device__ __forceinline__ NodeFields<P> node_publish(int code, const NodeState& s, size_t k,
                                                      size_t ps, P* __restrict__ mom_out,
                                                      uint8_t* lat_out, uint8_t* nxt_out) {
  const double Ux = cvt_f64(lat_ux(code)), Uy = cvt_f64(lat_uy(code));
  const double ux = s.ubx + Ux, uy = s.uby + Uy;
  const NodeFields<P> f{to_p<P>(s.rho), to_p<P>(s.T), to_p<P>(ux - Ux), to_p<P>(uy - Uy)};
  mom_out[k] = f.rho;
  mom_out[ps + k] = to_p<P>(ux);
  mom_out[2 * ps + k] = to_p<P>(uy);
  mom_out[3 * ps + k] = f.T;
  lat_out[k] = (uint8_t)code;
  nxt_out[k] = (uint8_t)s.code2;
  return f;
}

// Collision of a node (BGK, or App. E for Pr != 1) with the equilibrium in its
// column (solve status ns, multipliers lam: the warm start's after a failure),
// then the store of its populations and multipliers. Returns false if the solve
// failed: the node is then left uncollided.
template <typename P, int B>
__device__ __forceinline__ bool node_store(const Params& pr, const Columns<P, B>& cl,
                                           const NodeFields<P>& nf, int ns, bool fixed, bool warm,
                                           const P lam[NM], size_t k, size_t ps,
                                           P* __restrict__ pop_out, P* lam_out) {
  const P* st = cl.pop;
  // multipliers for the next step's warm start, if stored
  if (lam_out) {
#pragma unroll
    for (int j = 0; j < NM; ++j)
      lam_out[j * ps + k] =
          ns == NEWTON_OK || warm ? lam[j] : (j == 3 || j == 5 ? (P)0.5 : (P)0);
  }
  if (ns == NEWTON_OK) {
    // f^eq = rho p, g^eq = (2 Cv - D) T f^eq and tau = 1/2 + nu/T in the
    // population precision (in the FP32 form from the FP64 equilibrium)
    const P Tp = nf.T, rp = nf.rho;
    const P gp = mul_rn(fma((P)2, to_p<P>(pr.cv), (P)-2), Tp);
    P tau = (P)0.5 + to_p<P>(pr.nu) / Tp;
    const P* eqv = eq_in_precision<P, B>(cl.eq, fixed);
    constexpr int es = eq_stride<P, B>();
    if (pr.sensor) {
      P eps = 0;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const P fe = mul_rn(eqv[i * es], rp);
        eps += rel_dev(st[i * B], fe);
      }
      eps /= (P)Q;
      tau = mul_rn(tau, sensor_alpha<P>(pr, eps));
    }
    if (pr.shakhov) {
      store_shakhov<P, B>(pr, st, eqv, nf, tau, k, ps, pop_out);
    } else {
      const P om = (P)1 / tau;
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        // (g^eq - g rounds once)
        const P fe = mul_rn(eqv[i * es], rp);
        const P f = st[i * B];
        const P g = st[(Q + i) * B];
        __stcs(&pop_out[i * ps + k], fma(om, fe - f, f));
        __stcs(&pop_out[(Q + i) * ps + k], fma(om, fma(gp, fe, -g), g));
      }
    }
    return true;
  }
#pragma unroll
  for (int i = 0; i < NPLANES; ++i) pop_out[i * ps + k] = st[i * B];
  return false;
}

// Current lattices of the eight nodes around (x, y) (boundary rule for
// positions outside the grid), in a fixed order.
__device__ __forceinline__ void neighbour_codes(const Params& pr, const uint8_t* cur, int x, int y,
                                                uint8_t nb[8]) {
  int m = 0;
#pragma unroll
  for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
    for (int dx = -1; dx <= 1; ++dx) {
      if (dx == 0 && dy == 0) continue;
      bool gh = false;
      const int rx = resolve(x + dx, pr.nx, pr.bcx, &gh);
      const int ry = resolve(y + dy, pr.ny, pr.bcy, &gh);
      nb[m++] = cur[(size_t)ry * pr.nx + rx];
    }
}

template <typename P>
__device__ __forceinline__ void flush_counts(unsigned long long* ctr, const NodeCount<P>& c) {
  if constexpr (std::is_same<P, float>::value) {
    warp_count(ctr + CTR_FP32_ITERS, c.fix & ((1u << WORK_EVALS) - 1u));
    warp_count(ctr + CTR_FP64_EVALS, (c.fix >> WORK_EVALS) & 1023u);
    warp_count(ctr + CTR_FP64_UPDATES, c.fix >> WORK_UPDATES);
  } else {
    warp_count(ctr + CTR_NEWTON_ITERS, c.solve.fp64_iters);
    warp_count(ctr + CTR_FP64_EVALS, c.solve.fp64_evals);
    warp_count(ctr + CTR_FP32_ITERS, c.solve.fp32_iters);
    warp_count(ctr + CTR_FP64_UPDATES, c.solve.fp64_updates);
  }
  warp_count(ctr + CTR_NEWTON_CALLS, (c.n >> 20) & 2047u);
  warp_count(ctr + CTR_NEWTON_FAIL, c.n >> 31);
  warp_count(ctr + CTR_REC, c.n & 1023u);
  warp_count(ctr + CTR_REC_FAIL, (c.n >> 10) & 1023u);
}

// Shared state of a block's rebuilds. The missing pulls are numbered in (thread,
// velocity) order by a prefix sum of the threads' counts and handled in chunks of
// CHUNK; an entry is found again from its number (the thread by bisection, the
// velocity from the thread's mask). Within a chunk, every distinct (sender,
// receiver lattice) is entered once into a hash table and solved once. The table
// keeps key and solve in one word: with these sizes two blocks of the FP32 form
// leave 60 KB of an SM to L1, where their stack lives (28 KB with a list of the
// entries and separate arrays).
template <typename P, int B>
struct RebuildQueue {
  static constexpr bool LARGE = std::is_same<P, float>::value && B > 128;
  static constexpr int PER = LARGE ? 2 : 3;        // entries per thread and chunk
  static constexpr int CHUNK = PER * B;
  static constexpr int HASH = (LARGE ? 3 : 4) * B; // positions: at most 3/4 used
  static constexpr int KEY_BITS = 20;
  static_assert(CHUNK < 1 << (32 - KEY_BITS), "solve numbers");
  unsigned hash[HASH];          // key (20 bits) and solve (12 bits) of a position, or EMPTY
  unsigned short spos[CHUNK];   // position of each solve
  unsigned miss[B];             // velocities missing at each thread's node
  unsigned short start[B];      // number of the thread's first entry
  unsigned char state[B];       // of the solves of a round: 1 failed, 2 column in Q63
  int wsum[B / 32];             // missing pulls per warp
  int count, nsolve;

  // Thread (upper bits) and velocity (5 bits) of entry e.
  __device__ __forceinline__ unsigned entry(int e) const {
    int o = 0;
#pragma unroll
    for (int d = B > 256 ? 256 : B > 128 ? 128 : 64; d > 0; d >>= 1)
      if (o + d < B && start[o + d] <= e) o += d;
    unsigned m = miss[o];
    for (int j = e - start[o]; j > 0; --j) m &= m - 1;
    return (unsigned)o << 5 | (unsigned)(__ffs(m) - 1);
  }
};
constexpr unsigned RB_EMPTY = 0xffffffffu, RB_KEY = (1u << 20) - 1u;

// Key of a rebuild solve: receiver lattice (below 49) and sender position in the
// frame of a tile of 2^lg by B >> lg nodes. The sender lies within 6 nodes of the
// tile (|xi| <= 3, |U| <= 3); 49 (2^lg + 16) ((B >> lg) + 16) stays below 2^18.
__device__ __forceinline__ unsigned rebuild_key(int code, int sx, int sy, int lg) {
  return (unsigned)code + 49u * (unsigned)(sx + 8 + (sy + 8) * ((1 << lg) + 16));
}

// Asynchronous copy of one population from global into shared memory, evicted
// first from L2 (populations are read once and written once per step; L2 is
// kept for the lattice codes and the threads' stack).
template <typename P>
__device__ __forceinline__ void copy_async(P* dst, const P* src, unsigned long long policy) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global.L2::cache_hint [%0], [%1], %2, %3;" ::"r"(d), "l"(src),
               "n"(sizeof(P)), "l"(policy)
               : "memory");
}
__device__ __forceinline__ void async_copies_wait() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

static __constant__ signed char c_xi[Q][2] = {
    {0, 0},  {1, 0},   {0, 1},   {-1, 0}, {0, -1}, {1, 1},  {-1, 1}, {-1, -1}, {1, -1}, {2, 0}, {0, 2},
    {-2, 0}, {0, -2},  {2, 2},   {-2, 2}, {-2, -2}, {2, -2}, {3, 0},  {0, 3},   {-3, 0}, {0, -3}};

// Starts the pulls of node (x, y) in its lattice (Upx, Upy): the 42 populations
// of its senders are copied into its shared-memory column by asynchronous
// copies (all in flight together, without the 42 registers that loads would
// hold), whether or not a sender turns out to live in this lattice. Returns the
// mask of those that do; the others' entries are overwritten by their rebuilds.
// Inside the grid the addresses are a common base plus one uniform offset per
// velocity; at the grid's edges a rolled loop resolves each coordinate (an
// index is inside the grid even for a ghost: resolve clamps it).
template <typename P, int B>
__device__ __forceinline__ unsigned pull_node(const StepArgs<P>& a, const Columns<P, B>& cl, int x,
                                              int y, int code, int Upx, int Upy, bool inside) {
  const Params& pr = a.prm;
  const size_t ps = a.ps;
  unsigned long long policy;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  unsigned own = 0;
  if (inside) {
    const size_t ks = (size_t)(y - Upy) * pr.nx + (x - Upx);
    const P* src = a.pop_in + ks;
    const uint8_t* lat = a.lat_in + ks;
    int sc[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const ptrdiff_t off = -((ptrdiff_t)XI_Y(i) * pr.nx + XI_X(i));
      sc[i] = lat[off];
      copy_async(cl.pop + i * B, src + (off + (ptrdiff_t)(i * ps)), policy);
      copy_async(cl.pop + (Q + i) * B, src + (off + (ptrdiff_t)((Q + i) * ps)), policy);
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) own |= (sc[i] == code ? 1u : 0u) << i;
  } else {
#pragma unroll 1
    for (int i = 0; i < Q; ++i) {
      bool gh = false;
      const int rx = resolve(x - c_xi[i][0] - Upx, pr.nx, pr.bcx, &gh);
      const int ry = resolve(y - c_xi[i][1] - Upy, pr.ny, pr.bcy, &gh);
      const size_t ks = (size_t)ry * pr.nx + rx;
      copy_async(cl.pop + i * B, a.pop_in + (i * ps + ks), policy);
      copy_async(cl.pop + (Q + i) * B, a.pop_in + ((Q + i) * ps + ks), policy);
      // a ghost sender is always rebuilt
      if (!gh && a.lat_in[ks] == code) own |= 1u << i;
    }
  }
  return own;
}

// One time step of the nodes of a tile (Sec. IV.A.3), one node per thread:
// thread t updates node (x0 + (t & (2^lg - 1)), y0 + (t >> lg)) if it lies in
// the grid. Phase 1 pulls every population whose sender lives in the node's
// new lattice and queues the missing ones; phase 2 rebuilds the queued pulls
// with all threads of the block (each distinct sender is a full equilibrium
// solve, so spreading them keeps the warps of interface nodes from waiting on
// a few lanes); phase 3 collides and stores. A rebuilt value depends only on
// its inputs, not on the thread that computes it. All threads of the block
// must call this (it holds barriers).
template <typename P, int B>
__device__ __forceinline__ void tile_step(const StepArgs<P>& a, int x0, int y0, int lg,
                                          const Columns<P, B>& cl, RebuildQueue<P, B>& rq,
                                          NodeCount<P>& nc) {
  const Params& pr = a.prm;
  const size_t ps = a.ps;
  const int t = threadIdx.x;
  const int mask = (1 << lg) - 1;
  const int x = x0 + (t & mask), y = y0 + (t >> lg);
  const bool active = x < pr.nx && y < pr.ny;
  size_t k = 0;
  int code = 0;
  unsigned own = 0;  // bit i: the sender of velocity i lives in lattice `code`
  // all senders of the tile lie in the grid (|xi| <= 3 and |U| <= 3)
  const bool inside = x0 >= 6 && x0 + mask + 6 < pr.nx && y0 >= 6 && y0 + (B >> lg) + 5 < pr.ny;
  if (active) {
    k = (size_t)y * pr.nx + x;
    code = a.nxt_in[k];
    const int Upx = lat_ux(code), Upy = lat_uy(code);
    own = pull_node<P, B>(a, cl, x, y, code, Upx, Upy, inside);
  }
  async_copies_wait();
  // Number the missing pulls: a block-wide prefix sum of the threads' counts, so
  // that their order does not depend on scheduling. A tile without missing pulls
  // passes one barrier and skips the rest.
  int nq = 0;
  {
    const unsigned miss = active ? (~own & ((1u << Q) - 1u)) : 0u;
    const int nmiss = __popc(miss), lane = t & 31, warp = t >> 5;
    int incl = nmiss;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += u;
    }
    if (lane == 31) rq.wsum[warp] = incl;
    if (__syncthreads_or(nmiss)) {
      int end = incl;
      for (int w = 0; w < warp; ++w) end += rq.wsum[w];
      rq.miss[t] = miss;
      rq.start[t] = (unsigned short)(end - nmiss);
      if (t == B - 1) rq.count = end;
      __syncthreads();
      nq = rq.count;
    }
  }
  // Rebuild rounds, then the round of the node itself: the equilibrium solve is
  // one inlined piece of code that both share. The distinct solves of a chunk
  // run B at a time in the columns of threads 0, 1, ...; every entry then takes
  // its value from the column of its solve (which entry comes first into the
  // table, and which thread solves it, changes no value).
  static_assert(B % 32 == 0 && B <= 512, "whole warps; 14 bits for an entry");
  using RQ = RebuildQueue<P, B>;
  P* const pop0 = cl.pop - t;  // column 0 of the block
  int base = 0, round = 0, nsolve = 0;  // chunk, its solves done, its solves
  unsigned ent[RQ::PER];                // this thread's entries: hash position << 16 | entry
#pragma unroll 1
  for (;;) {
    const bool rebuild = base < nq;
    if (rebuild && round == 0) {
      for (int j = t; j < RQ::HASH; j += B) rq.hash[j] = RB_EMPTY;
      if (t == 0) rq.nsolve = 0;
      __syncthreads();
#pragma unroll
      for (int j = 0; j < RQ::PER; ++j) {
        const int e = base + j * B + t;
        ent[j] = 0;
        if (e >= nq) continue;
        const unsigned en = rq.entry(e);
        const int owner = en >> 5, i = en & 31;
        const int ox = owner & mask, oy = owner >> lg;
        const int oc = a.nxt_in[(size_t)(y0 + oy) * pr.nx + (x0 + ox)];
        const unsigned key =
            rebuild_key(oc, ox - c_xi[i][0] - lat_ux(oc), oy - c_xi[i][1] - lat_uy(oc), lg);
        // Knuth's multiplicative hash, scaled to the positions
        unsigned h = __umulhi(key * 2654435761u, (unsigned)RQ::HASH);
        for (;; h = h + 1 < RQ::HASH ? h + 1 : 0) {
          const unsigned old = atomicCAS(&rq.hash[h], RB_EMPTY, key);
          if (old == RB_EMPTY) {
            const unsigned slot = (unsigned)atomicAdd(&rq.nsolve, 1);
            rq.spos[slot] = (unsigned short)h;
            rq.hash[h] = key | slot << RQ::KEY_BITS;
            break;
          }
          if ((old & RB_KEY) == key) break;
        }
        ent[j] = h << 16 | en;
      }
      __syncthreads();
      nsolve = rq.nsolve;
    }
    // what to solve: the round's (sender, lattice) pairs, or the node; wk and wc
    // are the node whose multipliers start the solve and the solve's lattice
    NodeState s;
    NodeFields<P> nf;
    P lam[NM];
    unsigned wk = (unsigned)k;
    int wc = code;
    bool solve = !rebuild && active;
    if (rebuild) {
      if (round + t < nsolve) {
        const unsigned key = rq.hash[rq.spos[round + t]] & RB_KEY;
        const int at = (int)(key / 49u), w = (1 << lg) + 16;
        wc = (int)(key % 49u);
        bool gh = false;
        const int rx = resolve(x0 + at % w - 8, pr.nx, pr.bcx, &gh);
        const int ry = resolve(y0 + at / w - 8, pr.ny, pr.bcy, &gh);
        wk = (unsigned)ry * (unsigned)pr.nx + (unsigned)rx;
        s.rho = (double)a.mom_in[wk];
        s.ubx = (double)a.mom_in[ps + wk] - lat_ux(wc);
        s.uby = (double)a.mom_in[2 * ps + wk] - lat_uy(wc);
        s.T = (double)a.mom_in[3 * ps + wk];
        solve = true;
      }
    } else if (active) {
      uint8_t nb[8];
      const bool by_nb = order_key(pr.overlap) > 0 && pr.rule == 1;
      if (by_nb) neighbour_codes(pr, a.nxt_in, x, y, nb);
      s = node_moments<P, B>(pr, cl, code, by_nb ? nb : nullptr);
      nf = node_publish<P>(code, s, k, ps, a.mom_out, a.lat_out, a.nxt_out);
    }
    int st = NEWTON_UNREALIZABLE;
    bool fixed = false;
    if (solve) {
      nc.n += N_CALLS;
      st = node_equilibrium<P, B>(
          pr, cl, s, pr.warm,
          [&](P* l) { load_warm<P>(a.lam_in, ps, wk, a.lat_in[wk], lat_ux(wc), lat_uy(wc), l); },
          lam, &nc, a.ctr, &fixed);
    }
    if (!rebuild) {
      if (active && !node_store<P, B>(pr, cl, nf, st, fixed, pr.warm, lam, k, ps, a.pop_out,
                                      a.lam_out))
        nc.n |= N_FAIL;
      break;
    }
    rq.state[t] = (unsigned char)((st == NEWTON_OK ? 0 : 1) | (fixed ? 2 : 0));
    __syncthreads();
#pragma unroll 1
    for (int j = 0; j < RQ::PER; ++j) {
      if (base + j * B + t >= nq) break;
      const unsigned en = j == 0 ? ent[0] : j == 1 ? ent[1] : ent[RQ::PER - 1];
      const int j0 = (int)(rq.hash[en >> 16] >> RQ::KEY_BITS) - round;
      if (j0 < 0 || j0 >= B) continue;  // solved in another round
      const int owner = (en >> 5) & 511, i = en & 31;
      const int ox = x0 + (owner & mask), oy = y0 + (owner >> lg);
      const int oc = a.nxt_in[(size_t)oy * pr.nx + ox];
      const int Upx = lat_ux(oc), Upy = lat_uy(oc);
      const int cx = c_xi[i][0], cy = c_xi[i][1];
      const int state = rq.state[j0];
      const bool ok = !(state & 1);
      const double eq = ok ? eq_f64<P>(cl.eq[i * B - t + j0], state & 2) : 0.0;
      double fd, gd;
      rebuild_value<P>(pr, a.mom_in, ps, cx, cy, Upx, Upy, ox - cx - Upx, oy - cy - Upy, eq, ok,
                       &fd, &gd);
      nc.n += ok ? N_REC : N_REC + N_REC_FAIL;
      pop0[i * B + owner] = (P)fd;
      pop0[(Q + i) * B + owner] = (P)gd;
    }
    // the next round reuses the columns, the next chunk the table; after the
    // last one the rebuilt pulls are in place before the collisions
    __syncthreads();
    round += B;
    if (round >= nsolve) {
      round = 0;
      base += RQ::CHUNK;
    }
  }
}

}  // namespace alb
