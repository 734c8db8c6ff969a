// Solvers of the numerical equilibrium: FP32 Newton phase, residuals in fixed
// point (solve_fix, FP32 form) or FP64 (solve_mixed64, FP64 plain; refine_fp64,
// the FP32 form's states outside the fixed-point range), FP64 Newton throughout
// (newton_fp64g), and the reduced model.
//
// The multipliers of Eq. feqNum_8Mom solve G(lambda) = 0 (Eqs. G0_8mom..
// G3yaa_8mom). On GB300 the FP64 pipe runs at 1/62 of the FP32 rate, so the
// Newton iterations run in FP32 (exponentials, exact Jacobian, Cholesky
// factor), and 64 bits are used only where the accuracy of the result comes
// from: the residual. The refinement evaluates the 21 exponentials and the 8
// constraint residuals in 64-bit integers (alb_fix.cuh) or FP64 and corrects
// lambda with the FP32 Cholesky factor (iterative refinement of the Newton
// step) until max_k |G_k| / rho <= tol, the same criterion as the full FP64
// Newton. If the FP32 phase or the refinement fails, the full FP64 Newton takes
// over.
//
// The FP64 exponential is table-driven (Tang, ACM TOMS 15(2), 1989):
// exp(-s) = 2^(n/256) exp(r), n = round(-256 s / ln 2), |r| <= ln2/512, with
// 2^(j/256) from a 256-entry table and exp(r) by its degree-4 Taylor
// polynomial (constants in exp_table.h, generated by gen_exp_table.py).
//
// Every pass over the velocities streams through the symmetric groups of the
// D2Q21 set (the rest velocity, the axis pairs +-a, the diagonal quadruples):
// a group's exponents are built from shared even and odd parts, exponentiated
// and folded into the sums at once, so no per-velocity array stays live. The
// FP64 constraint sums use the butterfly of each group (sums and differences
// formed once for all moments).
#pragma once

#include <type_traits>

#include "alb_device.cuh"
#include "alb_fix.cuh"
#include "exp_table.h"

namespace alb {

// Calls v.rest(s_0), v.pair<a, axis, i+, i->(s_+, s_-) and
// v.quad<a, i++, i-+, i--, i+->(...) with the exponents
// s_i = base + lambda . P(xi_i) of every group (index order of XI_X / XI_Y);
// base is 1 for the exponents of Eq. exponential, 0 for the change of the
// exponents under a step of the multipliers.
template <typename R, typename V>
__device__ __forceinline__ void visit_groups(const R l[NM], V& v, R base = (R)1) {
  const R c = base + l[0];
  v.rest(c);
  {  // axis, |xi| = 1
    const R ex = c + l[3], ox = l[1] + l[6];
    v.template pair<1, 0, 1, 3>(ex + ox, ex - ox);
    const R ey = c + l[5], oy = l[2] + l[7];
    v.template pair<1, 1, 2, 4>(ey + oy, ey - oy);
  }
  {  // axis, |xi| = 2
    const R ex = fma((R)4, l[3], c), ox = fma((R)8, l[6], (R)2 * l[1]);
    v.template pair<2, 0, 9, 11>(ex + ox, ex - ox);
    const R ey = fma((R)4, l[5], c), oy = fma((R)8, l[7], (R)2 * l[2]);
    v.template pair<2, 1, 10, 12>(ey + oy, ey - oy);
  }
  {  // axis, |xi| = 3
    const R ex = fma((R)9, l[3], c), ox = fma((R)27, l[6], (R)3 * l[1]);
    v.template pair<3, 0, 17, 19>(ex + ox, ex - ox);
    const R ey = fma((R)9, l[5], c), oy = fma((R)27, l[7], (R)3 * l[2]);
    v.template pair<3, 1, 18, 20>(ey + oy, ey - oy);
  }
  const R l35 = l[3] + l[5];
  {  // diagonal (+-1, +-1): s = E + sx sy Z + sx X + sy Y
    const R E = c + l35;
    const R X = fma((R)2, l[6], l[1]), Y = fma((R)2, l[7], l[2]);
    const R Ep = E + l[4], Em = E - l[4];
    const R XpY = X + Y, XmY = X - Y;
    v.template quad<1, 5, 6, 7, 8>(Ep + XpY, Em - XmY, Ep - XpY, Em + XmY);
  }
  {  // diagonal (+-2, +-2)
    const R E = fma((R)4, l35, c);
    const R X = fma((R)16, l[6], (R)2 * l[1]), Y = fma((R)16, l[7], (R)2 * l[2]);
    const R Z = (R)4 * l[4];
    const R Ep = E + Z, Em = E - Z;
    const R XpY = X + Y, XmY = X - Y;
    v.template quad<2, 13, 14, 15, 16>(Ep + XpY, Em - XmY, Ep - XpY, Em + XmY);
  }
}

// The same groups as a loop over the speed a = 1, 2, 3 (pairs of the x and y
// axis, and the diagonal quadruple for a < 3), for the passes of the FP32 form:
// v.pair_x(g, k, s_+, s_-), v.pair_y(...) and v.quad(g, k, s_++, s_-+, s_--, s_+-)
// with g = a - 1 and k the powers of a. The loop is kept rolled: the FP32 form's
// node update is one long straight run of code per node, and instruction fetch
// takes issue slots from it (23 % of the stalls at 2048^2 with the groups
// unrolled).
template <typename R>
struct Pow {
  R a, a2, a3;
};
template <typename R, typename V>
__device__ __forceinline__ void visit_speeds(const R l[NM], V& v, R base) {
  const R c = base + l[0];
  v.rest(c);
  const R l35 = l[3] + l[5];
#pragma unroll 1
  for (int g = 0; g < 3; ++g) {
    Pow<R> k;
    k.a = (R)(g + 1);
    k.a2 = mul_rn(k.a, k.a);
    k.a3 = mul_rn(k.a2, k.a);
    {
      const R ex = fma(k.a2, l[3], c), ox = fma(k.a3, l[6], mul_rn(k.a, l[1]));
      v.pair_x(g, k, ex + ox, ex - ox);
      const R ey = fma(k.a2, l[5], c), oy = fma(k.a3, l[7], mul_rn(k.a, l[2]));
      v.pair_y(g, k, ey + oy, ey - oy);
    }
    if (g < 2) {
      const R E = fma(k.a2, l35, c);
      const R t3 = k.a3 + k.a3;
      const R X = fma(t3, l[6], mul_rn(k.a, l[1])), Y = fma(t3, l[7], mul_rn(k.a, l[2]));
      const R Z = mul_rn(k.a2, l[4]);
      const R Ep = E + Z, Em = E - Z;
      const R XpY = X + Y, XmY = X - Y;
      v.quad(g, k, Ep + XpY, Em - XmY, Ep - XpY, Em + XmY);
    }
  }
}
// Index of a group's first point: pairs x: PX + 8 g (and + 2), pairs y: PY + 8 g
// (and + 2), quadruples: PQ + 8 g .. + 3.
constexpr int PX = 1, PY = 2, PQ = 5;
static_assert(XI_X(PX + 16) == 3 && XI_X(PX + 18) == -3 && XI_Y(PY + 8) == 2 &&
                  XI_Y(PY + 10) == -2 && XI_X(PQ + 9) == -2 && XI_Y(PQ + 11) == -2,
              "index pattern of the velocity groups");

// 2^(j/N), j = 0..N-1 (N = EXPT_N); kernels copy it to shared memory (lanes
// index it freely). In global memory: consecutive threads copy consecutive
// entries, which constant memory would serve one by one.
static __device__ const double g_exptab[EXPT_N] = {ALB_EXPT_TABLE_VALUES};

// Copy the table into a block's shared array of EXPT_N doubles (all threads;
// includes a barrier).
__device__ __forceinline__ void load_exptab(double* s_tab) {
  for (int j = threadIdx.x; j < EXPT_N; j += blockDim.x) s_tab[j] = g_exptab[j];
  __syncthreads();
}

// 2^63 2^(-j/512): the fixed-point exponential's table (alb_fix.cuh), in global
// memory (consecutive threads copy consecutive entries).
static __device__ const uint64_t g_fixtab[FIXT_N] = {ALB_FIXT_TABLE_VALUES};

// Copy it into a block's shared array of FIXT_N entries (all threads; no barrier).
__device__ __forceinline__ void load_fixtab(uint64_t* s_fix) {
  for (int j = threadIdx.x; j < FIXT_N; j += blockDim.x) s_fix[j] = g_fixtab[j];
}

// q 2^(n/N) from the table, 0 below 2^-1022 (no subnormal results) and +inf from
// 2^1024 on; q need not be finite there. Integer operations and one product.
__device__ __forceinline__ double exp_scaled(double q, int n, const double* tab) {
  const int e = n >> EXPT_BITS;
  const int ec = e < -1100 ? -1100 : (e > 1100 ? 1100 : e);  // keeps the shift defined
  const long long bits = __double_as_longlong(tab[n & (EXPT_N - 1)]) + ((long long)ec << 52);
  const double v = q * __longlong_as_double(bits);
  return e < -1022 ? 0.0 : (e > 1023 ? __longlong_as_double(0x7ff0000000000000LL) : v);
}

// Table-driven FP64 exp(-s) (Tang's method with an N = 256 table): n nearest
// to -s N / ln2, r = -s - n ln2/N in two parts, exp(r) by its degree-4 Taylor
// polynomial, times 2^(n/N) = 2^(n >> 8) tab[n & 255].
// n comes from an FP32 copy of s: within |s| <= 745 (past which the result is 0
// or +inf anyway) FP32 holds s N / ln2 to 0.031, so n is the nearest integer or
// its neighbour near a tie, |r| <= 0.531 ln2/256, and the polynomial's remainder
// stays below 5.2e-17. The copy, n and its way back run on the integer pipe: 7 FP64
// operations (9 with the index rounded in FP64). Past |s| of 5.8e6 the
// float-to-int rounding saturates and the limits hold; a NaN gives n = 0 and
// passes through the polynomial.
__device__ __forceinline__ double exp_neg(double s, const double* tab) {
  const int n = __float2int_rn(mul_rn(-cvt_f32_rn(s), (float)EXPT_INV_L));
  const double nd = cvt_f64(n);
  double r = fma(nd, -EXPT_L_HI, -s);
  r = fma(nd, -EXPT_L_LO, r);
  double q = fma(r, EXPT_C4, EXPT_C3);
  q = fma(q, r, EXPT_C2);
  q = fma(q, r, 1.0);
  q = fma(q, r, 1.0);
  return exp_scaled(q, n, tab);
}

// exp(-s) for the FP32 form's refinement: the same table, the reduction in
// one step with ln2/N rounded, and the degree-2 Taylor polynomial. Its
// accuracy does not enter the convergence test: each residual is summed
// exactly (in FP64) over the column of values this function fills, so
// max|G|/rho <= 1e-12 holds for the populations returned. It only sets how
// closely those populations follow the exponential family of the returned
// multipliers: to 5e-10 relative here, next to the ~1e-10 the multiplicative
// updates leave, both far below the FP32 storage of the populations.
// The table index n nearest to -s N / ln2 comes from s32, an FP32 value of
// the same exponent: within |s| <= 745 (past which the result is 0 or +inf
// anyway) FP32 holds s N / ln2 to 0.031, so n is the nearest integer or its
// neighbour near a tie and |r| stays below 0.531 ln2/N (truncation r^3/3! below
// 5e-10). 4 FP64 operations: the reduction, the
// polynomial and the scaling (n reaches FP64 exactly on the integer pipe).
// For |s32 N / ln2| >= 2^31 the float-to-int rounding saturates and e takes
// the limits; a NaN gives n = 0 and passes through the polynomial.
__device__ __forceinline__ double exp_neg_refine(double s, float s32, const double* tab) {
  const int n = __float2int_rn(-s32 * (float)EXPT_INV_L);
  const double r = fma(cvt_f64(n), -EXPT_L, -s);
  double q = fma(r, EXPT_C2, 1.0);
  q = fma(q, r, 1.0);
  return exp_scaled(q, n, tab);
}

// An exponent held twice: in FP64 and in FP32 (the FP32 copy picks the
// table index of exp_neg_refine). visit_groups runs on it unchanged; its
// operators live in a namespace of their own, found by argument-dependent
// lookup, so that they hide no FP64 fma.
namespace dual {
struct Exp2 {
  double d;
  float f;
  Exp2() = default;
  __device__ __forceinline__ Exp2(double d_, float f_) : d(d_), f(f_) {}
  __device__ __forceinline__ explicit Exp2(double c) : d(c), f((float)c) {}
};
__device__ __forceinline__ Exp2 operator+(Exp2 a, Exp2 b) { return Exp2(a.d + b.d, a.f + b.f); }
__device__ __forceinline__ Exp2 operator-(Exp2 a, Exp2 b) { return Exp2(a.d - b.d, a.f - b.f); }
__device__ __forceinline__ Exp2 operator*(Exp2 a, Exp2 b) { return Exp2(a.d * b.d, a.f * b.f); }
__device__ __forceinline__ Exp2 fma(Exp2 a, Exp2 b, Exp2 c) {
  return Exp2(::fma(a.d, b.d, c.d), fmaf(a.f, b.f, c.f));
}
}  // namespace dual
using dual::Exp2;

// Maximum that is NaN if either argument is (fmaxf drops a NaN, so that residuals
// that are all NaN would have the maximum 0 and pass for converged).
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// Packed lower triangle of the 8x8 Jacobian: entry (a, b), b <= a.
__host__ __device__ constexpr int tri(int a, int b) { return a * (a + 1) / 2 + b; }

// exp(v) for the FP32 Newton's passes: two instructions, relative error about
// |v| 2^-24 + 2^-22, of the size that the FP32 rounding of the exponent itself
// leaves; results below FP32's normal range are zero.
__device__ __forceinline__ float exp_fast(float v) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(mul_rn(v, 1.44269504f)));
  return r;
}

// G = sum p P and H = sum p P P^T (packed lower triangle) from the sums over the
// speeds (see PassGH32).
template <typename R>
__device__ __forceinline__ void assemble_moments(R p0, const R X[7], const R Y[7], const R E[7],
                                                 const R O[7], const R Py[7], R G[NM], R H[36]) {
  const R x3 = X[3] + O[3], y3 = Y[3] + Py[3];  // x^3, y^3
  G[0] = p0 + X[0] + Y[0] + E[0];
  G[1] = X[1] + O[1];
  G[2] = Y[1] + Py[1];
  G[3] = X[2] + E[2];
  G[4] = O[2];
  G[5] = Y[2] + E[2];
  G[6] = x3 + O[3];  // x^3 + x y^2
  G[7] = y3 + Py[3];
#pragma unroll
  for (int k = 0; k < NM; ++k) H[tri(k, 0)] = G[k];
  H[tri(1, 1)] = G[3];
  H[tri(2, 1)] = G[4];
  H[tri(2, 2)] = G[5];
  H[tri(3, 1)] = x3;
  H[tri(3, 2)] = Py[3];
  H[tri(3, 3)] = X[4] + E[4];
  H[tri(4, 1)] = Py[3];
  H[tri(4, 2)] = O[3];
  H[tri(4, 3)] = O[4];
  H[tri(4, 4)] = E[4];
  H[tri(5, 1)] = O[3];
  H[tri(5, 2)] = y3;
  H[tri(5, 3)] = E[4];
  H[tri(5, 4)] = O[4];
  H[tri(5, 5)] = Y[4] + E[4];
  H[tri(6, 1)] = fma((R)2, E[4], X[4]);
  H[tri(6, 2)] = (R)2 * O[4];
  H[tri(6, 3)] = fma((R)2, O[5], X[5]);
  H[tri(6, 4)] = (R)2 * Py[5];
  H[tri(6, 5)] = (R)2 * O[5];
  H[tri(6, 6)] = fma((R)4, E[6], X[6]);
  H[tri(7, 1)] = (R)2 * O[4];
  H[tri(7, 2)] = fma((R)2, E[4], Y[4]);
  H[tri(7, 3)] = (R)2 * Py[5];
  H[tri(7, 4)] = (R)2 * O[5];
  H[tri(7, 5)] = fma((R)2, Py[5], Y[5]);
  H[tri(7, 6)] = (R)4 * O[6];
  H[tri(7, 7)] = fma((R)4, E[6], Y[6]);
}

// FP32 pass: F = sum p, G = sum p P and H = sum p P P^T at the visited
// multipliers. Every entry is a moment sum p x^m y^n with m + n <= 6. On this
// velocity set it comes from 27 sums over the speeds a: of a symmetric pair's
// sum (even powers of a) and difference (odd powers), and of a diagonal
// quadruple's four parity combinations (even or odd in x and in y). They take
// half the operations of accumulating G and H entry by entry, and half the
// registers (36 + 9 accumulators spilled at 128 registers a thread).
struct PassGH32 {
  float p0;
  float X[7], Y[7];      // pairs: sum a^n (p+ + p-) for even n, (p+ - p-) for odd n
  float E[7], O[7];      // quadruples: even/even (n even); x odd (n odd), x and y odd (n even)
  float Py[7];           // quadruples: y odd (n odd)
  __device__ __forceinline__ PassGH32() {
    p0 = 0.0f;
#pragma unroll
    for (int n = 0; n < 7; ++n) X[n] = Y[n] = E[n] = O[n] = Py[n] = 0.0f;
  }
  __device__ __forceinline__ void rest(float s) { p0 = exp_fast(-s); }
  static __device__ __forceinline__ void add_pair(float M[7], const Pow<float>& k, float pp,
                                                  float pm) {
    const float S = pp + pm, D = mul_rn(k.a, pp - pm);
    const float S2 = mul_rn(k.a2, S), D3 = mul_rn(k.a2, D);
    M[0] += S;
    M[1] += D;
    M[2] += S2;
    M[3] += D3;
    M[4] = fmaf(k.a2, S2, M[4]);
    M[5] = fmaf(k.a2, D3, M[5]);
    M[6] = fmaf(mul_rn(k.a2, k.a2), S2, M[6]);
  }
  __device__ __forceinline__ void pair_x(int, const Pow<float>& k, float sp, float sm) {
    add_pair(X, k, exp_fast(-sp), exp_fast(-sm));
  }
  __device__ __forceinline__ void pair_y(int, const Pow<float>& k, float sp, float sm) {
    add_pair(Y, k, exp_fast(-sp), exp_fast(-sm));
  }
  __device__ __forceinline__ void quad(int, const Pow<float>& k, float spp, float smp, float smm,
                                       float spm) {
    const float ppp = exp_fast(-spp), pmp = exp_fast(-smp), pmm = exp_fast(-smm), ppm = exp_fast(-spm);
    const float Ap = ppp + ppm, Bm = pmp + pmm, Cp = ppp - ppm, Dm = pmp - pmm;
    const float a4 = mul_rn(k.a2, k.a2);
    const float ee = Ap + Bm, oe = mul_rn(k.a, Ap - Bm), eo = mul_rn(k.a, Cp + Dm);
    const float oo = mul_rn(k.a2, Cp - Dm), e2 = mul_rn(k.a2, ee);
    E[0] += ee;
    E[2] += e2;
    E[4] = fmaf(k.a2, e2, E[4]);
    E[6] = fmaf(a4, e2, E[6]);
    O[1] += oe;
    O[3] = fmaf(k.a2, oe, O[3]);
    O[5] = fmaf(a4, oe, O[5]);
    Py[1] += eo;
    Py[3] = fmaf(k.a2, eo, Py[3]);
    Py[5] = fmaf(a4, eo, Py[5]);
    O[2] += oo;
    O[4] = fmaf(k.a2, oo, O[4]);
    O[6] = fmaf(a4, oo, O[6]);
  }
  __device__ __forceinline__ float F() const { return p0 + X[0] + Y[0] + E[0]; }
  __device__ __forceinline__ void scale(float z) {
    p0 = mul_rn(p0, z);
#pragma unroll
    for (int n = 0; n < 7; ++n) {
      X[n] = mul_rn(X[n], z);
      Y[n] = mul_rn(Y[n], z);
      E[n] = mul_rn(E[n], z);
      O[n] = mul_rn(O[n], z);
      Py[n] = mul_rn(Py[n], z);
    }
  }
  __device__ __forceinline__ void assemble(float G[NM], float H[36]) const {
    assemble_moments(p0, X, Y, E, O, Py, G, H);
  }
};

// FP64 constraint sums M = sum p P over the groups of the velocity set, the
// grouping of PassG64: a symmetric pair enters through its sum and
// difference, a diagonal quadruple through its four parity combinations.
struct SumsG64 {
  double M[NM];
  // The sums start at -m (the targets), so that they end as the residual
  // G = sum p P - m without a separate subtraction.
  __device__ __forceinline__ explicit SumsG64(const double m[NM]) {
#pragma unroll
    for (int k = 0; k < NM; ++k) M[k] = -m[k];
  }
  __device__ __forceinline__ void add_rest(double p) { M[0] += p; }
  template <int A, int AX>
  __device__ __forceinline__ void add_pair(double pp, double pm) {
    const double S = pp + pm, D = pp - pm;
    M[0] += S;
    if (AX == 0) {
      M[1] = madd(M[1], D, A);
      M[3] = madd(M[3], S, A * A);
      M[6] = madd(M[6], D, A * A * A);
    } else {
      M[2] = madd(M[2], D, A);
      M[5] = madd(M[5], S, A * A);
      M[7] = madd(M[7], D, A * A * A);
    }
  }
  template <int A>
  __device__ __forceinline__ void add_quad(double ppp, double pmp, double pmm, double ppm) {
    const double Ap = ppp + ppm, Bm = pmp + pmm;  // sx = +1, sx = -1
    const double Cp = ppp - ppm, Dm = pmp - pmm;
    const double sum = Ap + Bm, xs = Ap - Bm, ys = Cp + Dm, xys = Cp - Dm;
    M[0] += sum;
    M[1] = madd(M[1], xs, A);
    M[2] = madd(M[2], ys, A);
    M[3] = madd(M[3], sum, A * A);
    M[4] = madd(M[4], xys, A * A);
    M[5] = madd(M[5], sum, A * A);
    M[6] = madd(M[6], xs, 2 * A * A * A);
    M[7] = madd(M[7], ys, 2 * A * A * A);
  }
};

// FP64 pass: the constraint sums M = sum p P with p = exp(-s) in FP64, each p
// also written to the caller's shared column (p_i at col[i * stride]);
// REFINE selects the cheaper exponential of the FP32 form's refinement.
template <bool REFINE>
struct PassG64 {
  double M[NM];
  const double* tab;
  double* col;
  int stride;
  __device__ __forceinline__ PassG64(const double* t, double* c, int s) : tab(t), col(c), stride(s) {
#pragma unroll
    for (int k = 0; k < NM; ++k) M[k] = 0.0;
  }
  // sums started at -m: they end as the residual G = sum p P - m
  __device__ __forceinline__ PassG64(const double* t, double* c, int s, const double m[NM])
      : tab(t), col(c), stride(s) {
#pragma unroll
    for (int k = 0; k < NM; ++k) M[k] = -m[k];
  }
  // exponents: double, or Exp2 (FP64 with an FP32 copy) in the refinement
  using S = typename std::conditional<REFINE, Exp2, double>::type;
  __device__ __forceinline__ double ex(double s) const { return exp_neg(s, tab); }
  __device__ __forceinline__ double ex(Exp2 s) const { return exp_neg_refine(s.d, s.f, tab); }
  __device__ __forceinline__ void rest(S s) {
    const double p = ex(s);
    col[0] = p;
    M[0] += p;
  }
  template <int A, int AX, int IP, int IM>
  __device__ __forceinline__ void pair(S sp, S sm) {
    const double pp = ex(sp), pm = ex(sm);
    col[IP * stride] = pp;
    col[IM * stride] = pm;
    const double S = pp + pm, D = pp - pm;
    M[0] += S;
    if (AX == 0) {
      M[1] = madd(M[1], D, A);
      M[3] = madd(M[3], S, A * A);
      M[6] = madd(M[6], D, A * A * A);
    } else {
      M[2] = madd(M[2], D, A);
      M[5] = madd(M[5], S, A * A);
      M[7] = madd(M[7], D, A * A * A);
    }
  }
  template <int A, int IPP, int IMP, int IMM, int IPM>
  __device__ __forceinline__ void quad(S spp, S smp, S smm, S spm) {
    const double ppp = ex(spp), pmp = ex(smp);
    const double pmm = ex(smm), ppm = ex(spm);
    col[IPP * stride] = ppp;
    col[IMP * stride] = pmp;
    col[IMM * stride] = pmm;
    col[IPM * stride] = ppm;
    const double Ap = ppp + ppm, Bm = pmp + pmm;  // sx = +1, sx = -1
    const double Cp = ppp - ppm, Dm = pmp - pmm;
    const double sum = Ap + Bm, xs = Ap - Bm, ys = Cp + Dm, xys = Cp - Dm;
    M[0] += sum;
    M[1] = madd(M[1], xs, A);
    M[2] = madd(M[2], ys, A);
    M[3] = madd(M[3], sum, A * A);
    M[4] = madd(M[4], xys, A * A);
    M[5] = madd(M[5], sum, A * A);
    M[6] = madd(M[6], xs, 2 * A * A * A);
    M[7] = madd(M[7], ys, 2 * A * A * A);
  }
};

// Multiplicative pass of the FP32 form's refinement: after a step dl of the
// multipliers, p_i(lambda + dl) = p_i(lambda) exp(-d_i) with d_i = dl . P(xi_i)
// (Eq. exponential), so the populations in the column are updated in place,
// p_i <- p_i + p_i (exp(-d_i) - 1), and the FP64 sums taken again. d_i and
// exp(-d_i) - 1 = -d (1 - d/2 + d^2/6) are formed in FP32 (the step is an FP32
// vector); for |d_i| <= 1e-3 (checked by the caller) the update's factor has
// a relative error of about 1e-10, so the column stays an exponential-family
// member to that level, while the sums that decide convergence are exact FP64
// sums of the column. One FP64 operation per velocity (the factor reaches
// FP64 exactly on the integer pipe) instead of an exponent and an
// exponential.
struct PassMul64 : SumsG64 {
  double* col;
  int stride;
  __device__ __forceinline__ PassMul64(double* c, int s, const double m[NM])
      : SumsG64(m), col(c), stride(s) {}
  __device__ __forceinline__ double upd(int i, float d) const {
    const float e = d * fmaf(d, fmaf(d, -1.0f / 6.0f, 0.5f), -1.0f);
    double* q = col + (size_t)i * stride;
    const double p = fma(*q, cvt_f64(e), *q);
    *q = p;
    return p;
  }
  __device__ __forceinline__ void rest(float d) { add_rest(upd(0, d)); }
  template <int A, int AX, int IP, int IM>
  __device__ __forceinline__ void pair(float dp, float dm) {
    add_pair<A, AX>(upd(IP, dp), upd(IM, dm));
  }
  template <int A, int IPP, int IMP, int IMM, int IPM>
  __device__ __forceinline__ void quad(float dpp, float dmp, float dmm, float dpm) {
    add_quad<A>(upd(IPP, dpp), upd(IMP, dmp), upd(IMM, dmm), upd(IPM, dpm));
  }
};

// Exponents in Q25 octaves (alb_fix.cuh); visit_speeds runs on them unchanged.
// Arithmetic modulo 2^32; the operators live in a namespace of their own, found
// by argument-dependent lookup.
namespace fixe {
struct Oct {
  uint32_t v;
  Oct() = default;
  __device__ __forceinline__ explicit Oct(int c) : v((uint32_t)c) {}
};
__device__ __forceinline__ Oct oct(uint32_t v) {
  Oct o;
  o.v = v;
  return o;
}
__device__ __forceinline__ Oct operator+(Oct a, Oct b) { return oct(a.v + b.v); }
__device__ __forceinline__ Oct operator-(Oct a, Oct b) { return oct(a.v - b.v); }
__device__ __forceinline__ Oct mul_rn(Oct a, Oct b) { return oct(a.v * b.v); }
__device__ __forceinline__ Oct fma(Oct a, Oct b, Oct c) { return oct(a.v * b.v + c.v); }
}  // namespace fixe
using fixe::Oct;

// Q63 constraint sums over the groups of the velocity set, started at -m
// (modulo 2^64), so that they end as the residual G = sum p P - m: the grouping
// of SumsG64. A weighted term is one 32 x 32 + 64 multiply-add and one 32-bit one.
struct SumsFix {
  uint64_t M[NM];
  __device__ __forceinline__ explicit SumsFix(const uint64_t mneg[NM]) {
#pragma unroll
    for (int k = 0; k < NM; ++k) M[k] = mneg[k];
  }
  __device__ __forceinline__ void add_rest(uint64_t p) { M[0] += p; }
  template <int AX>
  __device__ __forceinline__ void add_pair(int g, uint64_t pp, uint64_t pm) {
    const uint32_t a = g + 1;
    const uint64_t S = pp + pm, D = pp - pm;
    M[0] += S;
    M[AX == 0 ? 1 : 2] += a * D;
    M[AX == 0 ? 3 : 5] += (a * a) * S;
    M[AX == 0 ? 6 : 7] += (a * a * a) * D;
  }
  __device__ __forceinline__ void add_quad(int g, uint64_t ppp, uint64_t pmp, uint64_t pmm,
                                           uint64_t ppm) {
    const uint32_t a = g + 1;
    const uint64_t Ap = ppp + ppm, Bm = pmp + pmm;  // sx = +1, sx = -1
    const uint64_t Cp = ppp - ppm, Dm = pmp - pmm;
    const uint64_t sum = Ap + Bm, xs = Ap - Bm, ys = Cp + Dm, xys = Cp - Dm;
    M[0] += sum;
    M[1] += a * xs;
    M[2] += a * ys;
    M[3] += (a * a) * sum;
    M[4] += (a * a) * xys;
    M[5] += (a * a) * sum;
    M[6] += (2 * a * a * a) * xs;
    M[7] += (2 * a * a * a) * ys;
  }
};

// Evaluation: Q63 populations of the exponents into the column, their sums, and
// the largest exponent (as an unsigned number, so that one below zero shows
// too).
struct PassFix : SumsFix {
  const uint64_t* tab;
  uint64_t* col;
  int stride;
  uint32_t ymax;
  __device__ __forceinline__ PassFix(const uint64_t* t, uint64_t* c, int s, const uint64_t mneg[NM])
      : SumsFix(mneg), tab(t), col(c), stride(s), ymax(0) {}
  __device__ __forceinline__ uint64_t ex(int i, Oct y) {
    ymax = ymax > y.v ? ymax : y.v;
    const uint64_t p = fix_exp(y.v, tab);
    col[(size_t)i * stride] = p;
    return p;
  }
  __device__ __forceinline__ void rest(Oct y) { add_rest(ex(0, y)); }
  __device__ __forceinline__ void pair_x(int g, const Pow<Oct>&, Oct p, Oct m) {
    add_pair<0>(g, ex(PX + 8 * g, p), ex(PX + 2 + 8 * g, m));
  }
  __device__ __forceinline__ void pair_y(int g, const Pow<Oct>&, Oct p, Oct m) {
    add_pair<1>(g, ex(PY + 8 * g, p), ex(PY + 2 + 8 * g, m));
  }
  __device__ __forceinline__ void quad(int g, const Pow<Oct>&, Oct pp, Oct mp, Oct mm, Oct pm) {
    add_quad(g, ex(PQ + 8 * g, pp), ex(PQ + 1 + 8 * g, mp), ex(PQ + 2 + 8 * g, mm),
             ex(PQ + 3 + 8 * g, pm));
  }
};

// Multiplicative pass after a small step dl of the multipliers, in place in the
// column: p_i <- p_i exp(-d_i), d_i = dl . P(xi_i) in FP32, and the sums again
// (the fixed-point form of PassMul64).
struct PassMulFix : SumsFix {
  uint64_t* col;
  int stride;
  FixStep fs;
  __device__ __forceinline__ PassMulFix(uint64_t* c, int s, const uint64_t mneg[NM], float bound)
      : SumsFix(mneg), col(c), stride(s), fs(fix_step(bound)) {}
  __device__ __forceinline__ uint64_t upd(int i, float d) const {
    uint64_t* q = col + (size_t)i * stride;
    const uint64_t p = fix_scale(*q, d, fs);
    *q = p;
    return p;
  }
  __device__ __forceinline__ void rest(float d) { add_rest(upd(0, d)); }
  __device__ __forceinline__ void pair_x(int g, const Pow<float>&, float p, float m) {
    add_pair<0>(g, upd(PX + 8 * g, p), upd(PX + 2 + 8 * g, m));
  }
  __device__ __forceinline__ void pair_y(int g, const Pow<float>&, float p, float m) {
    add_pair<1>(g, upd(PY + 8 * g, p), upd(PY + 2 + 8 * g, m));
  }
  __device__ __forceinline__ void quad(int g, const Pow<float>&, float pp, float mp, float mm, float pm) {
    add_quad(g, upd(PQ + 8 * g, pp), upd(PQ + 1 + 8 * g, mp), upd(PQ + 2 + 8 * g, mm),
             upd(PQ + 3 + 8 * g, pm));
  }
};

// Cholesky factor of the Jacobian, FP32: the packed lower triangle L with the
// reciprocals of its diagonal entries in the diagonal slots, so that the
// solves multiply. No diagonal (Jacobi) scaling: the backward error of the
// Cholesky factorisation does not depend on it, and on the 4096^2 layer the
// unscaled factor gave the same iteration counts (and 1 % more MLUPS).
struct Fact32 {
  float L[36];
};

// Approximate reciprocal square root without the handling of subnormal inputs.
__device__ __forceinline__ float rsqrt_fast(float v) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}

__device__ __forceinline__ bool factor32(const float H[36], Fact32& fc) {
  bool ok = true;
#pragma unroll
  for (int j = 0; j < NM; ++j) {
    float dj = H[tri(j, j)];
#pragma unroll
    for (int k = 0; k < j; ++k) dj = fmaf(-fc.L[tri(j, k)], fc.L[tri(j, k)], dj);
    ok = ok && (dj > 0.0f);
    const float il = rsqrt_fast(fmaxf(dj, 1e-30f));
    fc.L[tri(j, j)] = il;
#pragma unroll
    for (int i = j + 1; i < NM; ++i) {
      float s = H[tri(i, j)];
#pragma unroll
      for (int k = 0; k < j; ++k) s = fmaf(-fc.L[tri(i, k)], fc.L[tri(j, k)], s);
      fc.L[tri(i, j)] = mul_rn(s, il);
    }
  }
  return ok;
}

// delta = H^-1 g with the factor (forward and backward substitution).
__device__ __forceinline__ void solve32(const Fact32& fc, const float g[NM], float dl[NM]) {
  float y[NM];
#pragma unroll
  for (int i = 0; i < NM; ++i) {
    float s = g[i];
#pragma unroll
    for (int k = 0; k < i; ++k) s = fmaf(-fc.L[tri(i, k)], y[k], s);
    y[i] = mul_rn(s, fc.L[tri(i, i)]);
  }
#pragma unroll
  for (int i = NM - 1; i >= 0; --i) {
    float s = y[i];
#pragma unroll
    for (int k = i + 1; k < NM; ++k) s = fmaf(-fc.L[tri(k, i)], y[k], s);
    y[i] = mul_rn(s, fc.L[tri(i, i)]);
  }
#pragma unroll
  for (int i = 0; i < NM; ++i) dl[i] = y[i];
}

// Multipliers in the frame of another lattice: lam'.P(u) = lam.P(u - d) for
// every velocity u, where d = U - U' (a velocity xi relative to lattice U is
// xi - d relative to U'). Exact for the exponential; it serves as the starting
// point of the Newton iteration after a change of lattice.
template <typename R>
__device__ __forceinline__ void shift_multipliers(const R l[NM], R dx, R dy, R o[NM]) {
  // (dx, dy and their products are small integers, exact)
  const R xx = mul_rn(dx, dx), xy = mul_rn(dx, dy), yy = mul_rn(dy, dy), d2 = xx + yy;
  const R x3 = fma((R)2, xx, d2), y3 = fma((R)2, yy, d2);
  R t = fma(-l[1], dx, l[0]);
  t = fma(-l[2], dy, t);
  t = fma(l[3], xx, t);
  t = fma(l[4], xy, t);
  t = fma(l[5], yy, t);
  t = fma(-l[6], mul_rn(dx, d2), t);
  o[0] = fma(-l[7], mul_rn(dy, d2), t);
  t = fma(mul_rn((R)-2, l[3]), dx, l[1]);
  t = fma(-l[4], dy, t);
  t = fma(l[6], x3, t);
  o[1] = fma(mul_rn((R)2, l[7]), xy, t);
  t = fma(-l[4], dx, l[2]);
  t = fma(mul_rn((R)-2, l[5]), dy, t);
  t = fma(mul_rn((R)2, l[6]), xy, t);
  o[2] = fma(l[7], y3, t);
  o[3] = fma(-l[7], dy, fma(mul_rn((R)-3, l[6]), dx, l[3]));
  o[4] = fma(mul_rn((R)-2, l[7]), dx, fma(mul_rn((R)-2, l[6]), dy, l[4]));
  o[5] = fma(mul_rn((R)-3, l[7]), dy, fma(-l[6], dx, l[5]));
  o[6] = l[6];
  o[7] = l[7];
}

// FP32 phase: damped Newton from lam (warm start) or, if warm is false, from
// the Maxwellian; on success fc holds the factor of the Jacobian at the
// returned multipliers or one near step before them. Returns NEWTON_OK or
// NEWTON_SINGULAR (non-finite values or a non-positive pivot).
//
// Written as one loop with a single evaluation pass and a single
// factorisation, so that the pass exists once in the code: each turn evaluates
// the point lam and then acts on it according to why it was evaluated (a
// start, a line-search trial, the point a failed line search returns to).
//
// Inlined into each solver (once), so that the factor stays in registers
// between this phase and the refinement. What is live across a pass is kept
// small for the same reason: the last step's direction and length but not its
// start, and the three inputs instead of the eight targets. *gres is the
// residual maximum (FP32) at the last evaluated point, *stale says that the
// factor is of the point before the returned one.
//
// FACTOR = false is the prelude of the FP64 plain path: it stops, without a
// factor, at the first point from which the predicted decrease of the dual lies
// below FP32's resolution (residuals around 1e-3) or whose residual is at most
// 1e-4. That point is one that the Newton iteration itself passes, to FP32's
// rounding, with two or three steps still to go. One FP32 step more would be
// 20 % faster, but its rounding then shows in the last step: the tube parted
// from the oracle by 1.1e-10 in 1000 steps where it stays below 1e-11 so.
//
// FRESH = true evaluates and factorises once more after the last step, so that
// the factor is of the returned point: for the refinement in FP64, whose residuals
// cost the most (2.4 a solve instead of 3.8 on random states; 200,000 solves of
// alb_equilibrium 291 instead of 366 us).
template <bool FACTOR, bool FRESH = false>
__device__ __forceinline__ int newton_fp32(float ubx, float uby, float T, int maxit, bool warm,
                                           float lam[NM], Fact32& fc, int* iters, float* gres,
                                           bool* stale) {
  enum { START_WARM, START_MAXWELL, TRIAL, RETURNED, FULL_STEP };
  *iters = 0;
  *stale = false;
  // Maxwellian multipliers with lambda_0 = 0 (fixed from the normalisation
  // once evaluated)
  auto maxwell = [&]() {
    const float iT = 1.0f / T;
#pragma unroll
    for (int k = 0; k < NM; ++k) lam[k] = 0.0f;
    lam[1] = mul_rn(-ubx, iT);
    lam[2] = mul_rn(-uby, iT);
    lam[3] = mul_rn(0.5f, iT);
    lam[5] = lam[3];
  };
  int mode = START_WARM;
  if (!warm) {
    maxwell();
    mode = START_MAXWELL;
  }
  float dl[NM];
  float Fd = 0.0f, gd = 0.0f, t = 1.0f;
  int it = 0, ls = 0;
#pragma unroll 1
  for (;;) {
    PassGH32 pc;
    visit_speeds<float>(lam, pc, 1.0f);
    float F = pc.F();
    if (mode == START_WARM) {
      if (!(isfinite(F) && F > 0.0f)) {
        maxwell();
        mode = START_MAXWELL;
        continue;
      }
    } else if (mode == START_MAXWELL) {
      // the pass at lambda_0 = 0 gives Z = F; all its sums scale by 1/Z
      const float iz = 1.0f / F;
      lam[0] = logf(F);
      pc.scale(iz);
      F = pc.F();
    }
    // targets, formed again in every turn (the empty statement keeps the
    // compiler from carrying them across the pass)
    float ux = ubx, uy = uby, Tt = T;
    asm volatile("" : "+f"(ux), "+f"(uy), "+f"(Tt));
    float m[NM];
    {
      const float u2 = fmaf(ux, ux, mul_rn(uy, uy)), q = fmaf(4.0f, Tt, u2);
      m[0] = 1.0f; m[1] = ux; m[2] = uy;
      m[3] = fmaf(ux, ux, Tt); m[4] = mul_rn(ux, uy); m[5] = fmaf(uy, uy, Tt);
      m[6] = mul_rn(ux, q); m[7] = mul_rn(uy, q);
    }
#pragma unroll
    for (int k = 0; k < NM; ++k) F = fmaf(lam[k], m[k], F);  // the dual
    if (mode == TRIAL) {
      if (!(isfinite(F) && F <= fmaf(4e-7f, fabsf(Fd), fmaf(mul_rn(-1e-4f, t), gd, Fd)))) {
        // halve the step; with no acceptable one, back to its start for the
        // factor there
        const bool back = ++ls >= 12;
        const float dt = back ? t : mul_rn(0.5f, t);
#pragma unroll
        for (int k = 0; k < NM; ++k) lam[k] = fmaf(-dt, dl[k], lam[k]);
        t -= dt;
        if (back) mode = RETURNED;
        continue;
      }
      ++it;
    }
    // accepted point: the Newton step there
    Fd = F;
    float G[NM], H[36];
    pc.assemble(G, H);
    float gmax = 0.0f;
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      G[k] -= m[k];
      gmax = max_nan(gmax, fabsf(G[k]));
    }
    *gres = gmax;
    if (!FACTOR && gmax <= 1e-4f) break;
    if (!isfinite(gmax) || !factor32(H, fc)) return NEWTON_SINGULAR;
    // FP32 exit at 1e-6, five times the FP32 residual's own noise (about
    // 2e-7): below that the FP32 steps only chase rounding, and the
    // refinement contracts by about 1e-4 per residual from either level
    if (mode == RETURNED || (FRESH && mode == FULL_STEP) || gmax <= 1e-6f || it >= maxit) break;
    solve32(fc, G, dl);
    gd = 0.0f;
#pragma unroll
    for (int k = 0; k < NM; ++k) gd = fmaf(G[k], dl[k], gd);
    const bool near = gd <= mul_rn(2e-6f, fmaxf(1.0f, fabsf(Fd)));
    if (!(gd > 0.0f) || (!FACTOR && near)) break;
#pragma unroll
    for (int k = 0; k < NM; ++k) lam[k] += dl[k];
    if (near) {
      // The predicted decrease gd/2 of the dual lies below its FP32 resolution:
      // a line search would only compare rounding noise. This close to the root
      // the full Newton step is safe; take it and leave the rest to the
      // refinement, with the factor of the point before it: the exponents moved
      // by some 1e-3, so it still contracts by about that per residual, at
      // 0.6 more residuals a solve than with a fresh factor but without the
      // pass and the factorisation that one takes.
      // (FRESH takes them: the refinement in FP64 is the dearer part there.)
      ++it;
      if (FRESH) {
        mode = FULL_STEP;
        continue;
      }
      *stale = true;
      break;
    }
    mode = TRIAL;
    t = 1.0f;
    ls = 0;
  }
  *iters = it;
  return NEWTON_OK;
}

// max_i |P_k(xi_i)| over the velocity set (compile time).
__host__ __device__ constexpr int pm_max(int k) {
  int m = 0;
  for (int i = 0; i < Q; ++i) m = PM(k, i) > m ? PM(k, i) : (-PM(k, i) > m ? -PM(k, i) : m);
  return m;
}

// Largest |dl . P(xi_i)| over the velocities is at most this bound (FP32);
// the weights are max_i |P_k(xi_i)|, checked at compile time.
static_assert(pm_max(0) == 1 && pm_max(1) == 3 && pm_max(2) == 3 && pm_max(3) == 9 &&
                  pm_max(4) == 4 && pm_max(5) == 9 && pm_max(6) == 27 && pm_max(7) == 27,
              "monomial bounds of the D2Q21 set");
__device__ __forceinline__ float step_exponent_bound(const float dl[NM]) {
  float b = fmaf(3.0f, fabsf(dl[1]) + fabsf(dl[2]), fabsf(dl[0]));
  b = fmaf(4.0f, fabsf(dl[4]), b);
  b = fmaf(9.0f, fabsf(dl[3]) + fabsf(dl[5]), b);
  return fmaf(27.0f, fabsf(dl[6]) + fabsf(dl[7]), b);
}

// FP64 refinement: lambda <- lambda + H32^-1 G64(lambda) until max|G|/rho <= tol.
// The first residual evaluates the 21 exponentials in FP64; after a step whose
// exponent changes are all below 1e-3 in magnitude, the next one updates the
// column multiplicatively instead (PassMul64), else it evaluates them again.
// On NEWTON_OK the FP64 equilibrium per unit density at the returned lambda
// is in col[i * stride] (a shared-memory column of the calling thread).
// The residual is formed in FP64 and its maximum taken on its FP32 copy (the
// one the correction is solved with; FP32 resolves 1e-12 to 6e-8 of itself).
// The corrections are summed in FP32 for lam_out32 (lam32 plus every step:
// the multipliers the warm start stores in FP32) and join the FP64
// multipliers only before a full evaluation and, if lam_out64 is given, at
// the end. *evals counts the full evaluations, *updates the multiplicative
// ones.
static __device__ __noinline__ int refine_fp64(double ubx, double uby, double T, double tol,
                                               int maxr, const float lam32[NM], const Fact32& fc,
                                               const double* tab, double* col, int stride,
                                               float lam_out32[NM], double* lam_out64,
                                               int* evals, int* updates) {
  double m[NM];
  targets(ubx, uby, T, m);
  double lam[NM];  // FP64 multipliers of the last full evaluation
  float acc[NM];   // corrections since then
#pragma unroll
  for (int k = 0; k < NM; ++k) {
    lam[k] = cvt_f64(lam32[k]);
    acc[k] = 0.0f;
    lam_out32[k] = lam32[k];
  }
  const float tolf = (float)tol;
  *evals = 0;
  *updates = 0;
  float dl[NM];
  bool small_step = false;
  for (int r = 0;; ++r) {
    double G[NM];  // residual sum p P - m
    if (small_step) {
      PassMul64 pu(col, stride, m);
      visit_groups<float>(dl, pu, 0.0f);
      ++*updates;
#pragma unroll
      for (int k = 0; k < NM; ++k) G[k] = pu.M[k];
    } else {
      if (r > 0) {
#pragma unroll
        for (int k = 0; k < NM; ++k) {
          lam[k] += cvt_f64(acc[k]);
          acc[k] = 0.0f;
        }
      }
      PassG64<true> ps(tab, col, stride, m);
      Exp2 l2[NM];
#pragma unroll
      for (int k = 0; k < NM; ++k) l2[k] = Exp2(lam[k], lam_out32[k]);
      visit_groups<Exp2>(l2, ps, Exp2(1.0));
      ++*evals;
#pragma unroll
      for (int k = 0; k < NM; ++k) G[k] = ps.M[k];
    }
    float gmax = 0.0f;
    bool finite = true;
    float g32[NM];
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      g32[k] = cvt_f32_rn(G[k]);
      finite = finite && isfinite(g32[k]);
      gmax = fmaxf(gmax, fabsf(g32[k]));
    }
    if (!finite) return NEWTON_SINGULAR;
    if (gmax <= tolf) {
      if (lam_out64)
#pragma unroll
        for (int k = 0; k < NM; ++k) lam_out64[k] = lam[k] + (double)acc[k];
      return NEWTON_OK;
    }
    if (r >= maxr) return NEWTON_MAXIT;
    solve32(fc, g32, dl);
    small_step = step_exponent_bound(dl) <= 1e-3f;
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      acc[k] += dl[k];
      lam_out32[k] += dl[k];
    }
  }
}

// Work counts of one equilibrium solve.
struct SolveCount {
  unsigned fp32_iters = 0, fp64_evals = 0, fp64_iters = 0, fp64_updates = 0;
  __device__ __forceinline__ void add(const SolveCount& o) {
    fp32_iters += o.fp32_iters;
    fp64_evals += o.fp64_evals;
    fp64_iters += o.fp64_iters;
    fp64_updates += o.fp64_updates;
  }
};

// Jacobian H = sum_i p_i P(xi_i) P(xi_i)^T (packed lower triangle) from the
// populations per unit density in col[i * stride], group by group: a
// symmetric pair contributes its sum or difference, a diagonal quadruple one
// of its four parity combinations, with the compile-time value of P_a P_b at
// the group's first point as coefficient.
template <int IP, int IM>
__device__ __forceinline__ void jac_pair(const double* col, int stride, double H[36]) {
  const double pp = col[IP * stride], pm = col[IM * stride];
  const double S = pp + pm, D = pp - pm;
#pragma unroll
  for (int a = 0; a < NM; ++a)
#pragma unroll
    for (int b = 0; b <= a; ++b) {
      const int c = PM(a, IP) * PM(b, IP);
      if (c != 0) H[tri(a, b)] = madd(H[tri(a, b)], PM(a, IM) * PM(b, IM) == c ? S : D, c);
    }
}

template <int IPP, int IMP, int IMM, int IPM>
__device__ __forceinline__ void jac_quad(const double* col, int stride, double H[36]) {
  const double ppp = col[IPP * stride], pmp = col[IMP * stride];
  const double pmm = col[IMM * stride], ppm = col[IPM * stride];
  const double Ap = ppp + ppm, Bm = pmp + pmm, Cp = ppp - ppm, Dm = pmp - pmm;
  const double ee = Ap + Bm, oe = Ap - Bm, eo = Cp + Dm, oo = Cp - Dm;
#pragma unroll
  for (int a = 0; a < NM; ++a)
#pragma unroll
    for (int b = 0; b <= a; ++b) {
      const int c = PM(a, IPP) * PM(b, IPP);
      const bool xodd = PM(a, IMP) * PM(b, IMP) == -c;  // x -> -x flips the sign
      const bool yodd = PM(a, IPM) * PM(b, IPM) == -c;  // y -> -y flips the sign
      if (c != 0)
        H[tri(a, b)] = madd(H[tri(a, b)], xodd ? (yodd ? oo : oe) : (yodd ? eo : ee), c);
    }
}

__device__ __forceinline__ void jacobian_grouped(const double* col, int stride, double H[36]) {
#pragma unroll
  for (int k = 0; k < 36; ++k) H[k] = 0.0;
  H[0] = col[0];  // rest velocity: only P_0 = 1 is non-zero
  jac_pair<1, 3>(col, stride, H);
  jac_pair<2, 4>(col, stride, H);
  jac_pair<9, 11>(col, stride, H);
  jac_pair<10, 12>(col, stride, H);
  jac_pair<17, 19>(col, stride, H);
  jac_pair<18, 20>(col, stride, H);
  jac_quad<5, 6, 7, 8>(col, stride, H);
  jac_quad<13, 14, 15, 16>(col, stride, H);
}

// Evaluation of the exponential family at l: p_i = exp(-(1 + l . P(xi_i)))
// into col, and the moments M_k = sum_i p_i P_k(xi_i) (table-driven FP64
// exponential, grouped exponents and sums).
__device__ __forceinline__ void eval_fp64(const double l[NM], const double* tab, double* col,
                                          int stride, double M[NM]) {
  PassG64<false> pg(tab, col, stride);
  visit_groups<double>(l, pg);
#pragma unroll
  for (int k = 0; k < NM; ++k) M[k] = pg.M[k];
}

// FP64 Newton on the multipliers of the 8-moment equilibrium (Sec. II.C.2,
// App. C): damped by backtracking (Armijo) on the strictly convex dual
// F(lambda) = sum_i p_i + lambda . m, whose gradient is -G/rho and Hessian the
// exact Jacobian sum_i p_i P P^T; stops at max_k |G_k|/rho <= tol. Starts from
// `warm` if given, else (or if warm gives a non-finite dual) from the
// Maxwellian with lambda_0 from the normalisation. The iteration is the
// oracle's; its arithmetic is grouped by the symmetry of the velocity set and
// uses the table-driven exponential. On return col[i * stride] holds the
// equilibrium per unit density at lam; *iters counts Newton steps, *evals
// evaluations of the 21 exponentials.
static __device__ __noinline__ int newton_fp64g(double ubx, double uby, double T, double tol,
                                                int maxit, const double* tab, double* col,
                                                int stride, double lam[NM], int* iters,
                                                int* evals, const double* warm) {
  *iters = 0;
  *evals = 0;
  if (!(T > 0.0) || !isfinite(T) || !isfinite(ubx) || !isfinite(uby)) return NEWTON_UNREALIZABLE;
  double m[NM];
  targets(ubx, uby, T, m);
  double M[NM];
  int ev = 0;
  double F = 0.0;
  if (warm) {
#pragma unroll
    for (int k = 0; k < NM; ++k) lam[k] = warm[k];
    eval_fp64(lam, tab, col, stride, M);
    ev = 1;
    F = M[0];
#pragma unroll
    for (int k = 0; k < NM; ++k) F = fma(lam[k], m[k], F);
  }
  if (!warm || !isfinite(F)) {
    // Maxwellian: lambda_1 = -u/T, lambda_xx = lambda_yy = 1/(2T), lambda_0
    // from sum p = 1 (the exponentials at lambda_0 = 0 divided by their sum)
    const double iT = 1.0 / T;
#pragma unroll
    for (int k = 0; k < NM; ++k) lam[k] = 0.0;
    lam[1] = -ubx * iT;
    lam[2] = -uby * iT;
    lam[3] = 0.5 * iT;
    lam[5] = 0.5 * iT;
    eval_fp64(lam, tab, col, stride, M);
    ev += 1;
    const double Z = M[0];
    lam[0] = log(Z);
    const double iZ = 1.0 / Z;
#pragma unroll
    for (int i = 0; i < Q; ++i) col[i * stride] *= iZ;
#pragma unroll
    for (int k = 0; k < NM; ++k) M[k] *= iZ;
    F = M[0];
#pragma unroll
    for (int k = 0; k < NM; ++k) F = fma(lam[k], m[k], F);
  }
  int it = 0;
  for (;;) {
    double G[NM];
    double gmax = 0.0;
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      G[k] = M[k] - m[k];
      gmax = fmax(gmax, fabs(G[k]));
    }
    if (!isfinite(gmax)) { *iters = it; *evals = ev; return NEWTON_SINGULAR; }
    if (gmax <= tol) { *iters = it; *evals = ev; return NEWTON_OK; }
    if (it >= maxit) { *iters = it; *evals = ev; return NEWTON_MAXIT; }
    // Jacobian, then its Cholesky factor in place (reciprocal pivots kept)
    double H[36], il[NM];
    jacobian_grouped(col, stride, H);
    bool ok = true;
#pragma unroll
    for (int j = 0; j < NM; ++j) {
      double d = H[tri(j, j)];
#pragma unroll
      for (int k = 0; k < j; ++k) d = fma(-H[tri(j, k)], H[tri(j, k)], d);
      ok = ok && (d > 0.0);
      const double l = sqrt(fmax(d, 1e-300));
      il[j] = 1.0 / l;
      H[tri(j, j)] = l;
#pragma unroll
      for (int i = j + 1; i < NM; ++i) {
        double s = H[tri(i, j)];
#pragma unroll
        for (int k = 0; k < j; ++k) s = fma(-H[tri(i, k)], H[tri(j, k)], s);
        H[tri(i, j)] = s * il[j];
      }
    }
    if (!ok) { *iters = it; *evals = ev; return NEWTON_SINGULAR; }
    double d[NM];
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      double s = G[i];
#pragma unroll
      for (int k = 0; k < i; ++k) s = fma(-H[tri(i, k)], d[k], s);
      d[i] = s * il[i];
    }
#pragma unroll
    for (int i = NM - 1; i >= 0; --i) {
      double s = d[i];
#pragma unroll
      for (int k = i + 1; k < NM; ++k) s = fma(-H[tri(k, i)], d[k], s);
      d[i] = s * il[i];
    }
    double gd = 0.0;
#pragma unroll
    for (int k = 0; k < NM; ++k) gd = fma(G[k], d[k], gd);
    // backtracking (Armijo) along lam + t d
    double t = 1.0, Fc = 0.0;
    bool accepted = false;
    double lc[NM];
    for (int ls = 0; ls < 40; ++ls) {
#pragma unroll
      for (int k = 0; k < NM; ++k) lc[k] = fma(t, d[k], lam[k]);
      eval_fp64(lc, tab, col, stride, M);
      ++ev;
      Fc = M[0];
#pragma unroll
      for (int k = 0; k < NM; ++k) Fc = fma(lc[k], m[k], Fc);
      if (isfinite(Fc) && Fc <= F - 1e-4 * t * gd + 1e-15 * fabs(F)) { accepted = true; break; }
      t *= 0.5;
    }
    ++it;
    if (!accepted) {
      eval_fp64(lam, tab, col, stride, M);
      *iters = it;
      *evals = ev + 1;
      return NEWTON_MAXIT;
    }
#pragma unroll
    for (int k = 0; k < NM; ++k) lam[k] = lc[k];
    F = Fc;
  }
}

// FP64 evaluation with the Jacobian: p_i = exp(-(1 + lambda . P(xi_i))) into the
// column and the 27 moment sums of PassGH32, from which both G (less the
// targets) and H follow: 96 operations for the sums, against 68 for the
// constraint sums alone and 150 more for the entries of the Jacobian.
struct PassGH64 {
  double p0, X[7], Y[7], E[7], O[7], Py[7];
  const double* tab;
  double* col;
  int stride;
  __device__ __forceinline__ PassGH64(const double* t, double* c, int s)
      : p0(0.0), tab(t), col(c), stride(s) {
#pragma unroll
    for (int n = 0; n < 7; ++n) X[n] = Y[n] = E[n] = O[n] = Py[n] = 0.0;
  }
  __device__ __forceinline__ double ex(int i, double s) const {
    const double p = exp_neg(s, tab);
    col[i * stride] = p;
    return p;
  }
  __device__ __forceinline__ void rest(double s) { p0 = ex(0, s); }
  template <int A, int AX, int IP, int IM>
  __device__ __forceinline__ void pair(double sp, double sm) {
    const double pp = ex(IP, sp), pm = ex(IM, sm);
    const double S = pp + pm, D = pp - pm;
    double* M = AX == 0 ? X : Y;
    constexpr int A2 = A * A;
    M[0] += S;
    M[1] = madd(M[1], D, A);
    M[2] = madd(M[2], S, A2);
    M[3] = madd(M[3], D, A2 * A);
    M[4] = madd(M[4], S, A2 * A2);
    M[5] = madd(M[5], D, A2 * A2 * A);
    M[6] = madd(M[6], S, A2 * A2 * A2);
  }
  template <int A, int IPP, int IMP, int IMM, int IPM>
  __device__ __forceinline__ void quad(double spp, double smp, double smm, double spm) {
    const double ppp = ex(IPP, spp), pmp = ex(IMP, smp), pmm = ex(IMM, smm), ppm = ex(IPM, spm);
    const double Ap = ppp + ppm, Bm = pmp + pmm, Cp = ppp - ppm, Dm = pmp - pmm;
    const double ee = Ap + Bm, oe = Ap - Bm, eo = Cp + Dm, oo = Cp - Dm;
    constexpr int A2 = A * A;
    E[0] += ee;
    E[2] = madd(E[2], ee, A2);
    E[4] = madd(E[4], ee, A2 * A2);
    E[6] = madd(E[6], ee, A2 * A2 * A2);
    O[1] = madd(O[1], oe, A);
    O[3] = madd(O[3], oe, A2 * A);
    O[5] = madd(O[5], oe, A2 * A2 * A);
    Py[1] = madd(Py[1], eo, A);
    Py[3] = madd(Py[3], eo, A2 * A);
    Py[5] = madd(Py[5], eo, A2 * A2 * A);
    O[2] = madd(O[2], oo, A2);
    O[4] = madd(O[4], oo, A2 * A2);
    O[6] = madd(O[6], oo, A2 * A2 * A2);
  }
  __device__ __forceinline__ void assemble(double G[NM], double H[36]) const {
    assemble_moments(p0, X, Y, E, O, Py, G, H);
  }
};

// Equilibrium of the FP64 plain path: the Newton iteration of newton_fp64g with
// its early steps in FP32. The FP32 phase follows the iteration to a residual of
// about 1e-3; the FP64 steps from there have the residual and the Jacobian in
// FP64, and each step is solved with the FP32 factor and one correction by the
// FP64 Jacobian (1e-10 of the step). The FP32 rounding of the point they start
// from, 1e-7, is squared away by the steps as any other error of it, so that the
// iteration ends where the one in FP64 throughout ends (the same number of steps,
// 5.1 a solve on the 1024^2 layer, and the same error against 64-bit results).
// A step costs 430 operations of the FP64 pipe, which bounds this path, where a
// step of newton_fp64g costs 910: 11.0 -> 4.7 ms a step of the 1024^2 layer,
// 5570 -> 2160 FP64 instructions per node, 80 % of the pipe busy.
// Returns NEWTON_OK with the column and the multipliers (lam: in, the warm
// start if `warm`), or another status: newton_fp64g then solves from the start.
// *steps counts the FP64 steps.
static __device__ __noinline__ int solve_mixed64(double ubx, double uby, double T, double tol,
                                                 bool warm, const double* tab, double* col,
                                                 int stride, double lam[NM], int* it32, int* steps,
                                                 int* evals) {
  float dl[NM];
  Fact32 fc;
  float gres = 0.0f;
  int st;
  *it32 = *steps = *evals = 0;
#pragma unroll
  for (int k = 0; k < NM; ++k) dl[k] = warm ? cvt_f32_rn(lam[k]) : 0.0f;
  for (bool w = warm;; w = false) {
    int it = 0;
    bool stale;
    st = newton_fp32<false>(cvt_f32_rn(ubx), cvt_f32_rn(uby), cvt_f32_rn(T), 30, w, dl, fc, &it,
                            &gres, &stale);
    *it32 += it;
    if (st == NEWTON_OK || !w) break;
  }
  if (st != NEWTON_OK) return st;
  double m[NM];
  targets(ubx, uby, T, m);
#pragma unroll
  for (int k = 0; k < NM; ++k) lam[k] = cvt_f64(dl[k]);
  const float tolf = cvt_f32_rn(tol);
  float last = INFINITY;
#pragma unroll 1
  for (int n = 0;; ++n) {
    PassGH64 pg(tab, col, stride);
    visit_groups<double>(lam, pg);
    *evals += 1;
    double G[NM], H[36];
    pg.assemble(G, H);
    float g32[NM], gmax = 0.0f;
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      G[k] -= m[k];
      g32[k] = cvt_f32_rn(G[k]);
      gmax = max_nan(gmax, fabsf(g32[k]));
    }
    if (gmax <= tolf) return NEWTON_OK;
    // (a NaN residual fails both comparisons)
    if (n >= 6 || !(gmax < last)) return NEWTON_MAXIT;
    last = gmax;
    float h32[36];
#pragma unroll
    for (int k = 0; k < 36; ++k) h32[k] = cvt_f32_rn(H[k]);
    if (!factor32(h32, fc)) return NEWTON_SINGULAR;
    solve32(fc, g32, dl);
    double d[NM];
#pragma unroll
    for (int k = 0; k < NM; ++k) d[k] = cvt_f64(dl[k]);
    float r32[NM];
#pragma unroll
    for (int a = 0; a < NM; ++a) {
      double r = G[a];
#pragma unroll
      for (int b = 0; b < NM; ++b) r = fma(-H[a >= b ? tri(a, b) : tri(b, a)], d[b], r);
      r32[a] = cvt_f32_rn(r);
    }
    solve32(fc, r32, dl);
#pragma unroll
    for (int k = 0; k < NM; ++k) lam[k] += d[k] + cvt_f64(dl[k]);
    *steps += 1;
  }
}

// Reduced model (App. C.2, Eq. feqNum_4Mom): four constraints - mass,
// momentum and the energy trace sum f xi_a xi_a = rho (|ubar|^2 + D T) - and
// the exponential family in (1, xi_x, xi_y, |xi|^2). The multipliers are kept
// in the 8-slot layout of the full set (lambda_xx = lambda_yy = l2, the rest
// 0), so the grouped evaluation, the warm-start planes and the lattice shift
// of the multipliers are shared. The iteration is the oracle's: Maxwellian
// start with lambda_0 from the normalisation (or the warm multipliers),
// Newton on the dual with Armijo backtracking, stop at max|G|/rho <= tol; the
// 4x4 Jacobian takes its entries from the constraint sums of the evaluation
// plus sum p |xi|^4.
__device__ __forceinline__ void expand4(const double l4[4], double l8[NM]) {
  l8[0] = l4[0]; l8[1] = l4[1]; l8[2] = l4[2];
  l8[3] = l4[3]; l8[4] = 0.0; l8[5] = l4[3]; l8[6] = 0.0; l8[7] = 0.0;
}

static __device__ __noinline__ int newton4_fp64g(double ubx, double uby, double T, double tol,
                                                 int maxit, const double* tab, double* col,
                                                 int stride, double lam[NM], int* iters,
                                                 int* evals, const double* warm) {
  *iters = 0;
  *evals = 0;
  if (!(T > 0.0) || !isfinite(T) || !isfinite(ubx) || !isfinite(uby)) return NEWTON_UNREALIZABLE;
  const double m[4] = {1.0, ubx, uby, ubx * ubx + uby * uby + 2.0 * T};
  double l4[4], M[NM];
  int ev = 0;
  double F = 0.0;
  if (warm) {
    l4[0] = warm[0]; l4[1] = warm[1]; l4[2] = warm[2]; l4[3] = warm[3];
    expand4(l4, lam);
    eval_fp64(lam, tab, col, stride, M);
    ev = 1;
    F = M[0];
#pragma unroll
    for (int k = 0; k < 4; ++k) F = fma(l4[k], m[k], F);
  }
  if (!warm || !isfinite(F)) {
    const double iT = 1.0 / T;
    l4[0] = 0.0; l4[1] = -ubx * iT; l4[2] = -uby * iT; l4[3] = 0.5 * iT;
    expand4(l4, lam);
    eval_fp64(lam, tab, col, stride, M);
    ev += 1;
    const double Z = M[0];
    l4[0] = log(Z);
    const double iZ = 1.0 / Z;
#pragma unroll
    for (int i = 0; i < Q; ++i) col[i * stride] *= iZ;
#pragma unroll
    for (int k = 0; k < NM; ++k) M[k] *= iZ;
    F = M[0];
#pragma unroll
    for (int k = 0; k < 4; ++k) F = fma(l4[k], m[k], F);
  }
  int it = 0;
  for (;;) {
    const double G[4] = {M[0] - m[0], M[1] - m[1], M[2] - m[2], (M[3] + M[5]) - m[3]};
    double gmax = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) gmax = fmax(gmax, fabs(G[k]));
    if (!isfinite(gmax)) { expand4(l4, lam); *iters = it; *evals = ev; return NEWTON_SINGULAR; }
    if (gmax <= tol) { expand4(l4, lam); *iters = it; *evals = ev; return NEWTON_OK; }
    if (it >= maxit) { expand4(l4, lam); *iters = it; *evals = ev; return NEWTON_MAXIT; }
    // Jacobian sum p P4 P4^T: all but sum p |xi|^4 are the sums of the last
    // evaluation (P4 = (1, x, y, x^2 + y^2)); |xi|^4 is a^4 on an axis pair and
    // 4 a^4 on a diagonal quadruple of the velocity set
    const double sr4 =
        (col[1 * stride] + col[3 * stride]) + (col[2 * stride] + col[4 * stride]) +
        16.0 * ((col[9 * stride] + col[11 * stride]) + (col[10 * stride] + col[12 * stride])) +
        81.0 * ((col[17 * stride] + col[19 * stride]) + (col[18 * stride] + col[20 * stride])) +
        4.0 * ((col[5 * stride] + col[6 * stride]) + (col[7 * stride] + col[8 * stride])) +
        64.0 * ((col[13 * stride] + col[14 * stride]) + (col[15 * stride] + col[16 * stride]));
    double H[10];
    H[tri(0, 0)] = M[0];
    H[tri(1, 0)] = M[1];
    H[tri(1, 1)] = M[3];
    H[tri(2, 0)] = M[2];
    H[tri(2, 1)] = M[4];
    H[tri(2, 2)] = M[5];
    H[tri(3, 0)] = M[3] + M[5];
    H[tri(3, 1)] = M[6];
    H[tri(3, 2)] = M[7];
    H[tri(3, 3)] = sr4;
    bool ok = true;
    double il[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      double d = H[tri(j, j)];
#pragma unroll
      for (int k = 0; k < j; ++k) d = fma(-H[tri(j, k)], H[tri(j, k)], d);
      ok = ok && (d > 0.0);
      const double l = sqrt(fmax(d, 1e-300));
      il[j] = 1.0 / l;
      H[tri(j, j)] = l;
#pragma unroll
      for (int i = j + 1; i < 4; ++i) {
        double s = H[tri(i, j)];
#pragma unroll
        for (int k = 0; k < j; ++k) s = fma(-H[tri(i, k)], H[tri(j, k)], s);
        H[tri(i, j)] = s * il[j];
      }
    }
    if (!ok) { expand4(l4, lam); *iters = it; *evals = ev; return NEWTON_SINGULAR; }
    double d[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      double s = G[i];
#pragma unroll
      for (int k = 0; k < i; ++k) s = fma(-H[tri(i, k)], d[k], s);
      d[i] = s * il[i];
    }
#pragma unroll
    for (int i = 3; i >= 0; --i) {
      double s = d[i];
#pragma unroll
      for (int k = i + 1; k < 4; ++k) s = fma(-H[tri(k, i)], d[k], s);
      d[i] = s * il[i];
    }
    double gd = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) gd = fma(G[k], d[k], gd);
    double t = 1.0, Fc = 0.0, lc[4];
    bool accepted = false;
    for (int ls = 0; ls < 40; ++ls) {
#pragma unroll
      for (int k = 0; k < 4; ++k) lc[k] = fma(t, d[k], l4[k]);
      expand4(lc, lam);
      eval_fp64(lam, tab, col, stride, M);
      ++ev;
      Fc = M[0];
#pragma unroll
      for (int k = 0; k < 4; ++k) Fc = fma(lc[k], m[k], Fc);
      if (isfinite(Fc) && Fc <= F - 1e-4 * t * gd + 1e-15 * fabs(F)) { accepted = true; break; }
      t *= 0.5;
    }
    ++it;
    if (!accepted) {
      expand4(l4, lam);
      eval_fp64(lam, tab, col, stride, M);
      *iters = it;
      *evals = ev + 1;
      return NEWTON_MAXIT;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) l4[k] = lc[k];
    F = Fc;
  }
}

// The change of the constraint sums under a small step dl of the multipliers, sum
// p_i (exp(-d_i) - 1) P(xi_i), in FP32 (in units of 2^-31): its relative error of
// some 1e-7 lies far below what the step leaves.
struct PassDelta {
  float M[NM];
  const uint64_t* col;
  int stride;
  __device__ __forceinline__ PassDelta(const uint64_t* c, int s) : col(c), stride(s) {
#pragma unroll
    for (int k = 0; k < NM; ++k) M[k] = 0.0f;
  }
  __device__ __forceinline__ float w(int i, float d) const {
    const uint32_t hi = reinterpret_cast<const uint32_t*>(col)[2 * i * stride + 1];
    return mul_rn((float)hi, mul_rn(d, fmaf(d, fmaf(d, -1.0f / 6.0f, 0.5f), -1.0f)));
  }
  __device__ __forceinline__ void rest(float d) { M[0] += w(0, d); }
  template <int AX>
  __device__ __forceinline__ void add_pair(const Pow<float>& k, float p, float m) {
    const float S = p + m, D = p - m;
    M[0] += S;
    M[AX ? 2 : 1] = fmaf(k.a, D, M[AX ? 2 : 1]);
    M[AX ? 5 : 3] = fmaf(k.a2, S, M[AX ? 5 : 3]);
    M[AX ? 7 : 6] = fmaf(k.a3, D, M[AX ? 7 : 6]);
  }
  __device__ __forceinline__ void pair_x(int g, const Pow<float>& k, float dp, float dm) {
    add_pair<0>(k, w(PX + 8 * g, dp), w(PX + 2 + 8 * g, dm));
  }
  __device__ __forceinline__ void pair_y(int g, const Pow<float>& k, float dp, float dm) {
    add_pair<1>(k, w(PY + 8 * g, dp), w(PY + 2 + 8 * g, dm));
  }
  __device__ __forceinline__ void quad(int g, const Pow<float>& k, float dpp, float dmp, float dmm,
                                       float dpm) {
    const float ppp = w(PQ + 8 * g, dpp), pmp = w(PQ + 1 + 8 * g, dmp);
    const float pmm = w(PQ + 2 + 8 * g, dmm), ppm = w(PQ + 3 + 8 * g, dpm);
    const float Ap = ppp + ppm, Bm = pmp + pmm, Cp = ppp - ppm, Dm = pmp - pmm;
    const float sum = Ap + Bm, xs = Ap - Bm, ys = Cp + Dm, xys = Cp - Dm;
    const float t3 = k.a3 + k.a3;
    M[0] += sum;
    M[1] = fmaf(k.a, xs, M[1]);
    M[2] = fmaf(k.a, ys, M[2]);
    M[3] = fmaf(k.a2, sum, M[3]);
    M[4] = fmaf(k.a2, xys, M[4]);
    M[5] = fmaf(k.a2, sum, M[5]);
    M[6] = fmaf(t3, xs, M[6]);
    M[7] = fmaf(t3, ys, M[7]);
  }
};

// Largest exponent |1 + lambda . P(xi_i)| over the velocities is at most this:
// the larger of the axis and the diagonal velocities' bounds.
__device__ __forceinline__ float exponent_bound(const float l[NM]) {
  const float ax = fmaf(9.0f, fabsf(l[3]), fmaf(3.0f, fabsf(l[1]), mul_rn(27.0f, fabsf(l[6]))));
  const float ay = fmaf(9.0f, fabsf(l[5]), fmaf(3.0f, fabsf(l[2]), mul_rn(27.0f, fabsf(l[7]))));
  const float dg = fmaf(4.0f, fabsf(l[3]) + fabsf(l[4]) + fabsf(l[5]),
                        fmaf(2.0f, fabsf(l[1]) + fabsf(l[2]),
                             mul_rn(16.0f, fabsf(l[6]) + fabsf(l[7]))));
  return fabsf(1.0f + l[0]) + max_nan(max_nan(ax, ay), dg);
}

// Refinement of the FP32 form in fixed point: as refine_fp64, lambda <- lambda +
// H32^-1 G(lambda) until max|G|/rho <= tol with G the exact sum of the
// populations in the column, here in Q63 (alb_fix.cuh). Returns NEWTON_OK with
// the Q63 populations in col[i * stride], or another status for the states it
// does not take (an exponent outside the fixed-point range, FP32 residual above
// 1/64: the Q63 residual has to stay below one) and for failures; the caller
// then refines in FP64.
__device__ __forceinline__ int refine_fix(double ubx, double uby, double T, float tolf, int maxr,
                                          float lam[NM], const Fact32& fc, float gres, bool stale,
                                          const uint64_t* tab, uint64_t* col, int stride,
                                          int* evals, int* updates) {
  *evals = 0;
  *updates = 0;
  if (!(gres < 0.015625f)) return NEWTON_MAXIT;
  uint64_t mneg[NM];
  {
    double m[NM];
    targets(ubx, uby, T, m);
    mneg[0] = 1ull << 63;
#pragma unroll
    for (int k = 1; k < NM; ++k) mneg[k] = 0u - fix_of_f64(m[k]);
  }
  float dl[NM];
  float bound = INFINITY;  // of the last step's exponent changes
  for (int r = 0;; ++r) {
    float g32[NM];
    if (bound <= FIX_STEP_MAX) {
      PassMulFix pu(col, stride, mneg, bound);
      visit_speeds<float>(dl, pu, 0.0f);
      ++*updates;
#pragma unroll
      for (int k = 0; k < NM; ++k) g32[k] = fix_residual_f32(pu.M[k]);
    } else {
      if (!(exponent_bound(lam) < FIX_S_MAX)) return NEWTON_MAXIT;
      Oct mu[NM];
      mu[0] = fixe::oct((uint32_t)__float2int_rn(mul_rn(1.0f + lam[0], FIX_SCALE)));
#pragma unroll
      for (int k = 1; k < NM; ++k) mu[k] = fixe::oct((uint32_t)__float2int_rn(mul_rn(lam[k], FIX_SCALE)));
      PassFix ps(tab, col, stride, mneg);
      visit_speeds<Oct>(mu, ps, Oct(0));
      ++*evals;
      if (ps.ymax >= FIX_Y_END) return NEWTON_MAXIT;
#pragma unroll
      for (int k = 0; k < NM; ++k) g32[k] = fix_residual_f32(ps.M[k]);
    }
    float gmax = 0.0f;
#pragma unroll
    for (int k = 0; k < NM; ++k) gmax = fmaxf(gmax, fabsf(g32[k]));
    if (gmax <= tolf) return NEWTON_OK;
    if (r >= maxr) return NEWTON_MAXIT;
    solve32(fc, g32, dl);
    bound = step_exponent_bound(dl);  // (a NaN fails both comparisons)
    if (r == 0 && stale && bound <= FIX_STEP_MAX) {
      // With the factor one step old, this step leaves some 1e-3 of the
      // residual: 1e-10, for a second update. What it leaves is known in FP32
      // from the change of the sums, and a second correction joins the step
      // before the column is updated once (250 operations instead of a pass of
      // some 700).
      PassDelta pd(col, stride);
      visit_speeds<float>(dl, pd, 0.0f);
      float d2[NM];
#pragma unroll
      for (int k = 0; k < NM; ++k) g32[k] = fmaf(pd.M[k], 4.656612873077393e-10f, g32[k]);
      solve32(fc, g32, d2);
#pragma unroll
      for (int k = 0; k < NM; ++k) dl[k] += d2[k];
      bound = step_exponent_bound(dl);
    }
#pragma unroll
    for (int k = 0; k < NM; ++k) lam[k] += dl[k];
  }
}

constexpr int WORK_EVALS = 12, WORK_UPDATES = 22;

// FP32 Newton from the warm start if given, else (or if that fails) from the
// Maxwellian, then the fixed-point refinement: on NEWTON_OK the Q63 column and
// the multipliers in lam. *work collects the counts of a node's solves in one
// register: FP32 steps (at most 62 a solve), evaluations and updates (at most 7)
// in 12, 10 and 10 bits, enough for the 23 solves of a thread and tile.
//
// lam holds the warm start on entry if `warm` is set. Inlined: a call would save
// and restore some sixty registers per thread through local memory, which
// at two blocks of columns per SM leaves L1.
__device__ __forceinline__ int solve_fix(double ubx, double uby, double T, float tolf, bool warm,
                                         const uint64_t* ftab, uint64_t* col, int stride,
                                         float lam[NM], unsigned* work) {
  const float ubx32 = cvt_f32_rn(ubx), uby32 = cvt_f32_rn(uby), T32 = cvt_f32_rn(T);
  Fact32 fc;
  float gres = 0.0f;
  bool stale = false;
  int st, it = 0, ev = 0, up = 0;
  for (bool w = warm;; w = false) {
    int it32 = 0;
    st = newton_fp32<true>(ubx32, uby32, T32, 30, w, lam, fc, &it32, &gres, &stale);
    it += it32;
    if (st == NEWTON_OK || !w) break;
  }
  if (st == NEWTON_OK)
    st = refine_fix(ubx, uby, T, tolf, 6, lam, fc, gres, stale, ftab, col, stride, &ev, &up);
  *work += (unsigned)it + ((unsigned)ev << WORK_EVALS) + ((unsigned)up << WORK_UPDATES);
  return st;
}

// The reduced model (four multipliers: 1, x, y, |xi|^2) in the FP32 form: FP32
// Newton on the 4x4 system and the fixed-point refinement, as solve_fix. The
// multipliers stay in the 8-slot layout (lambda_xx = lambda_yy, the rest 0), so
// the passes are shared; their sums give the four residuals and the Jacobian.
// The FP64 4x4 Newton it replaces here was bound by the FP64 pipe (4.3 FP64
// evaluations a solve): 2.25 -> 0.19 ms a step of the 512^2 shear layer.
struct Fact4 {
  float L[10];
};
__device__ __forceinline__ bool factor4(const float H[10], Fact4& fc) {
  bool ok = true;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float dj = H[tri(j, j)];
#pragma unroll
    for (int k = 0; k < j; ++k) dj = fmaf(-fc.L[tri(j, k)], fc.L[tri(j, k)], dj);
    ok = ok && (dj > 0.0f);
    const float il = rsqrt_fast(fmaxf(dj, 1e-30f));
    fc.L[tri(j, j)] = il;
#pragma unroll
    for (int i = j + 1; i < 4; ++i) {
      float s = H[tri(i, j)];
#pragma unroll
      for (int k = 0; k < j; ++k) s = fmaf(-fc.L[tri(i, k)], fc.L[tri(j, k)], s);
      fc.L[tri(i, j)] = mul_rn(s, il);
    }
  }
  return ok;
}
// The step in the 8-slot layout.
__device__ __forceinline__ void solve4(const Fact4& fc, const float g[4], float dl[NM]) {
  float y[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float s = g[i];
#pragma unroll
    for (int k = 0; k < i; ++k) s = fmaf(-fc.L[tri(i, k)], y[k], s);
    y[i] = mul_rn(s, fc.L[tri(i, i)]);
  }
#pragma unroll
  for (int i = 3; i >= 0; --i) {
    float s = y[i];
#pragma unroll
    for (int k = i + 1; k < 4; ++k) s = fmaf(-fc.L[tri(k, i)], y[k], s);
    y[i] = mul_rn(s, fc.L[tri(i, i)]);
  }
  dl[0] = y[0]; dl[1] = y[1]; dl[2] = y[2]; dl[3] = y[3];
  dl[4] = 0.0f; dl[5] = y[3]; dl[6] = 0.0f; dl[7] = 0.0f;
}

static __device__ __noinline__ int solve4_fix(double ubx, double uby, double T, float tolf,
                                              bool warm, const uint64_t* ftab, uint64_t* col,
                                              int stride, float lam[NM], int* it32, int* evals,
                                              int* updates) {
  *it32 = *evals = *updates = 0;
  const float ux = cvt_f32_rn(ubx), uy = cvt_f32_rn(uby), T32 = cvt_f32_rn(T);
  const float m[4] = {1.0f, ux, uy, fmaf(ux, ux, fmaf(uy, uy, mul_rn(2.0f, T32)))};
  Fact4 fc;
  float dl[NM], l[NM], gres = 0.0f;
  bool done = false;
#pragma unroll 1
  for (bool w = warm; !done; w = false) {
    bool start = true, back = false;  // back: a failed line search returned to its start
    float Fd = 0.0f, gd = 0.0f, t = 1.0f;
    int it = 0, ls = 0;
    const float iT = 1.0f / T32;
#pragma unroll
    for (int k = 0; k < NM; ++k) l[k] = 0.0f;
    l[0] = w ? lam[0] : 0.0f;
    l[1] = w ? lam[1] : mul_rn(-ux, iT);
    l[2] = w ? lam[2] : mul_rn(-uy, iT);
    l[3] = l[5] = w ? lam[3] : mul_rn(0.5f, iT);
    bool bad = false;
#pragma unroll 1
    for (;;) {
      PassGH32 pc;
      visit_speeds<float>(l, pc, 1.0f);
      float F = pc.F();
      if (start && !w) {
        const float iz = 1.0f / F;
        l[0] = logf(F);
        pc.scale(iz);
        F = pc.F();
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) F = fmaf(l[k], m[k], F);
      if (!start && !back) {
        if (!(isfinite(F) && F <= fmaf(4e-7f, fabsf(Fd), fmaf(mul_rn(-1e-4f, t), gd, Fd)))) {
          back = ++ls >= 12;
          const float dt = back ? t : mul_rn(0.5f, t);
#pragma unroll
          for (int k = 0; k < NM; ++k) l[k] = fmaf(-dt, dl[k], l[k]);
          t -= dt;
          continue;
        }
        ++it;
      }
      start = false;
      Fd = F;
      float G8[NM], H8[36];
      pc.assemble(G8, H8);
      const float g[4] = {G8[0] - m[0], G8[1] - m[1], G8[2] - m[2], (G8[3] + G8[5]) - m[3]};
      const float H[10] = {G8[0], G8[1], G8[3], G8[2], G8[4], G8[5], G8[3] + G8[5], G8[6], G8[7],
                           H8[tri(3, 3)] + fmaf(2.0f, H8[tri(5, 3)], H8[tri(5, 5)])};
      gres = fmaxf(fmaxf(fabsf(g[0]), fabsf(g[1])), fmaxf(fabsf(g[2]), fabsf(g[3])));
      if (!isfinite(g[0] + g[1] + g[2] + g[3]) || !factor4(H, fc)) {
        bad = true;
        break;
      }
      if (back || gres <= 1e-6f || it >= 30) break;
      solve4(fc, g, dl);
      gd = fmaf(g[3], dl[3], fmaf(g[2], dl[2], fmaf(g[1], dl[1], mul_rn(g[0], dl[0]))));
      if (!(gd > 0.0f)) break;
#pragma unroll
      for (int k = 0; k < NM; ++k) l[k] += dl[k];
      if (gd <= mul_rn(2e-6f, fmaxf(1.0f, fabsf(Fd)))) {
        ++it;
        break;
      }
      t = 1.0f;
      ls = 0;
    }
    *it32 += it;
    if (!bad) done = true;
    else if (!w) return NEWTON_SINGULAR;
  }
  if (!(gres < 0.015625f)) return NEWTON_MAXIT;
  uint64_t mneg[NM];
#pragma unroll
  for (int k = 0; k < NM; ++k) mneg[k] = 0u;
  mneg[0] = 1ull << 63;
  mneg[1] = 0u - fix_of_f64(ubx);
  mneg[2] = 0u - fix_of_f64(uby);
  mneg[3] = 0u - fix_of_f64(fma(ubx, ubx, fma(uby, uby, mul_rn(2.0, T))));
  float bound = INFINITY;
#pragma unroll 1
  for (int r = 0;; ++r) {
    uint64_t M[4];
    if (bound <= FIX_STEP_MAX) {
      PassMulFix pu(col, stride, mneg, bound);
      visit_speeds<float>(dl, pu, 0.0f);
      ++*updates;
      M[0] = pu.M[0]; M[1] = pu.M[1]; M[2] = pu.M[2]; M[3] = pu.M[3] + pu.M[5];
    } else {
      if (!(exponent_bound(l) < FIX_S_MAX)) return NEWTON_MAXIT;
      Oct mu[NM];
      mu[0] = fixe::oct((uint32_t)__float2int_rn(mul_rn(1.0f + l[0], FIX_SCALE)));
#pragma unroll
      for (int k = 1; k < NM; ++k) mu[k] = fixe::oct((uint32_t)__float2int_rn(mul_rn(l[k], FIX_SCALE)));
      PassFix ps(ftab, col, stride, mneg);
      visit_speeds<Oct>(mu, ps, Oct(0));
      ++*evals;
      if (ps.ymax >= FIX_Y_END) return NEWTON_MAXIT;
      M[0] = ps.M[0]; M[1] = ps.M[1]; M[2] = ps.M[2]; M[3] = ps.M[3] + ps.M[5];
    }
    float g[4], gmax = 0.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      g[k] = fix_residual_f32(M[k]);
      gmax = fmaxf(gmax, fabsf(g[k]));
    }
    if (gmax <= tolf) break;
    if (r >= 6) return NEWTON_MAXIT;
    solve4(fc, g, dl);
    bound = step_exponent_bound(dl);
#pragma unroll
    for (int k = 0; k < NM; ++k) l[k] += dl[k];
  }
#pragma unroll
  for (int k = 0; k < NM; ++k) lam[k] = l[k];
  return NEWTON_OK;
}

// The FP32 phase of the refinement in FP64, with a fresh factor. A function of its
// own: inlined beside the call of the refinement it spills (200,000 solves of
// alb_equilibrium 291 us inlined, 257 us so).
static __device__ __noinline__ int newton_fp32_fresh(float ubx, float uby, float T, bool warm,
                                                     float lam[NM], Fact32& fc, int* iters,
                                                     float* gres) {
  bool stale;
  return newton_fp32<true, true>(ubx, uby, T, 30, warm, lam, fc, iters, gres, &stale);
}

// Equilibrium of the FP32 form by FP32 Newton (from the warm start if given,
// else from the Maxwellian; again from the Maxwellian if the warm start fails),
// FP64 refinement, full FP64 Newton as the last fallback. The FP64 equilibrium
// per unit density lands in col[i * stride]; the multipliers in lam32 (FP32, as
// the warm start keeps them) and, if lam64 is given, in FP64. It serves the
// states solve_fix does not take and the callers that want FP64 multipliers.
static __device__ __noinline__ int equilibrium_mixed(double ubx, double uby, double T, double tol,
                                                     int maxit, const double* tab,
                                                     const float* warm, double* col, int stride,
                                                     float lam32[NM], double* lam64,
                                                     SolveCount* cnt) {
  if (!(T > 0.0) || !isfinite(T) || !isfinite(ubx) || !isfinite(uby)) return NEWTON_UNREALIZABLE;
  float l32[NM];
  Fact32 fc;
  float gres = 0.0f;
  int ev = 0;
  int st = NEWTON_SINGULAR;
  const float ubx32 = cvt_f32_rn(ubx), uby32 = cvt_f32_rn(uby), T32 = cvt_f32_rn(T);
  bool w = warm != nullptr;
  if (w)
#pragma unroll
    for (int k = 0; k < NM; ++k) l32[k] = warm[k];
  for (;;) {
    int it32 = 0;
    st = newton_fp32_fresh(ubx32, uby32, T32, w, l32, fc, &it32, &gres);
    cnt->fp32_iters += it32;
    if (st == NEWTON_OK || !w) break;
    w = false;
  }
  if (st == NEWTON_OK) {
    int up = 0;
    st = refine_fp64(ubx, uby, T, tol, 6, l32, fc, tab, col, stride, lam32, lam64, &ev, &up);
    cnt->fp64_evals += ev;
    cnt->fp64_updates += up;
  }
  if (st != NEWTON_OK) {
    int it = 0;
    double ld[NM];
    st = newton_fp64g(ubx, uby, T, tol, maxit, tab, col, stride, ld, &it, &ev, nullptr);
    cnt->fp64_iters += it;
    cnt->fp64_evals += ev;
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      lam32[k] = (float)ld[k];
      if (lam64) lam64[k] = ld[k];
    }
  }
  return st;
}

}  // namespace alb
