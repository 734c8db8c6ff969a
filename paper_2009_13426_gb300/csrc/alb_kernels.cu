// Kernels of the adaptive D2Q21 LBM step (one node per thread).
//
//  step_kernel   pull (Eq. stream) in the receiver's lattice with Grad rebuild
//                of missing pulls (Eqs. GradGeneral*), moments (Eq. polyTemp),
//                shift for the next pull (Eq. criterion), numerical equilibrium
//                (Eq. feqNum_8Mom), g^eq (Eq. gEq), optional sensor
//                (Eq. DeltaAvg), BGK (Eq. coll), store.
//  init_kernel   Grad-regularised initial populations, then the same collision.
//  export / equilibrium / select kernels for the C ABI.
//
// Layout: structure of arrays. Plane p (f_0..f_20, g_0..g_20) of a buffer is
// a contiguous nx*ny array, x fastest; lattice codes and moments likewise.
// Each thread owns two columns of the block's dynamic shared memory: its 42
// pulled populations (stride BLOCK) and the 21 equilibrium values (64 bits
// each) per unit density of its latest equilibrium solve (stride BLOCK).
#include <type_traits>

#include "alb_step.cuh"
#include "alb_tiles.h"

namespace alb {

// One time step of every node: block (bx, by) updates the tile of 2^lg nodes
// along x by B >> lg rows at (bx << lg, by * (B >> lg)).
template <typename P, int B, int MINB>
__global__ void __launch_bounds__(B, MINB)
    step_kernel(const __grid_constant__ StepArgs<P> a, int lg) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ RebuildQueue<P, B> s_rq;
  const Columns<P, B> cl(smem_raw);  // includes a barrier
  NodeCount<P> nc;
  tile_step<P, B>(a, blockIdx.x << lg, blockIdx.y * (B >> lg), lg, cl, s_rq, nc);
  flush_counts(a.ctr, nc);
}

template <typename P>
struct InitArgs {
  const double *rho, *rhoux, *rhouy, *rhoE;
  P* pop_out;
  P* mom_out;
  uint8_t* lat_out;
  uint8_t* nxt_out;
  P* lam_out;
  size_t ps;
  Params prm;
  unsigned long long* ctr;
};

__device__ __forceinline__ void init_prim(const double* rho, const double* rhoux,
                                          const double* rhouy, const double* rhoE, double cv,
                                          size_t k, double* r, double* ux, double* uy,
                                          double* T) {
  *r = rho[k];
  *ux = rhoux[k] / *r;
  *uy = rhouy[k] / *r;
  *T = (rhoE[k] - 0.5 * (*r) * ((*ux) * (*ux) + (*uy) * (*uy))) / ((*r) * cv);
}

// The same at a neighbour, for the central differences of u and T: one reciprocal
// instead of three divisions (the node's own velocity, which chooses its lattice,
// keeps the divisions).
__device__ __forceinline__ void init_near(const double* rho, const double* rhoux,
                                          const double* rhouy, const double* rhoE, double icv,
                                          size_t k, double* ux, double* uy, double* T) {
  const double ir = 1.0 / rho[k];
  *ux = rhoux[k] * ir;
  *uy = rhouy[k] * ir;
  *T = (rhoE[k] * ir - 0.5 * ((*ux) * (*ux) + (*uy) * (*uy))) * icv;
}

// Visitor that writes the Grad-regularised populations of a node to its column:
// s = 1 + phi_f of every velocity (grad_poly).
template <typename P>
struct GradFill {
  P* pop;
  const double* eq;
  bool fixed;
  double r, gfac, g0, gx, gy;
  __device__ __forceinline__ GradFill(P* p, const double* e, bool fx, double r_, double gf,
                                      const double g[3])
      : pop(p), eq(e), fixed(fx), r(r_), gfac(gf), g0(1.0 + g[0]), gx(g[1]), gy(g[2]) {}
  template <int I>
  __device__ __forceinline__ void put(double s) {
    const double feq = r * eq_f64<P>(eq[I * BLOCK], fixed);
    pop[I * BLOCK] = to_p<P>(feq * s);
    pop[(Q + I) * BLOCK] = to_p<P>(gfac * feq * madd(madd(g0, gx, XI_X(I)), gy, XI_Y(I)));
  }
  __device__ __forceinline__ void rest(double s) { put<0>(s); }
  template <int A, int AX, int IP, int IM>
  __device__ __forceinline__ void pair(double sp, double sm) {
    put<IP>(sp);
    put<IM>(sm);
  }
  template <int A, int IPP, int IMP, int IMM, int IPM>
  __device__ __forceinline__ void quad(double spp, double smp, double smm, double spm) {
    put<IPP>(spp);
    put<IMP>(smp);
    put<IMM>(smm);
    put<IPM>(spm);
  }
};

// Grad-regularised initial condition (Sec. IV.A.1): h = h^eq (1 + phi_h) in the
// lattice chosen from the initial velocity, then the first collision.
template <typename P>
__global__ void __launch_bounds__(BLOCK, (std::is_same<P, float>::value ? 4 : 1))
    init_kernel(const __grid_constant__ InitArgs<P> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Columns<P, BLOCK> cl(smem_raw);
  const Params& pr = a.prm;
  const int x = blockIdx.x * BLOCK + threadIdx.x;
  const int y = blockIdx.y;
  unsigned n_bad = 0, n_fail = 0;
  NodeCount<P> cnt;  // (the initial solves are not step work: only failures are counted)
  if (x < pr.nx) {
    const size_t nx = (size_t)pr.nx;
    const size_t k = (size_t)y * nx + x;
    bool gh = false;
    const int xp = resolve(x + 1, pr.nx, pr.bcx, &gh), xm = resolve(x - 1, pr.nx, pr.bcx, &gh);
    const int yp = resolve(y + 1, pr.ny, pr.bcy, &gh), ym = resolve(y - 1, pr.ny, pr.bcy, &gh);
    double r, ux, uy, T, ux1, uy1, T1, ux2, uy2, T2;
    init_prim(a.rho, a.rhoux, a.rhouy, a.rhoE, pr.cv, k, &r, &ux, &uy, &T);
    double du[2][2], dT[2];
    const double icv = pr.gamma - 1.0;
    init_near(a.rho, a.rhoux, a.rhouy, a.rhoE, icv, y * nx + xp, &ux1, &uy1, &T1);
    init_near(a.rho, a.rhoux, a.rhouy, a.rhoE, icv, y * nx + xm, &ux2, &uy2, &T2);
    du[0][0] = 0.5 * (ux1 - ux2);
    du[0][1] = 0.5 * (uy1 - uy2);
    dT[0] = 0.5 * (T1 - T2);
    init_near(a.rho, a.rhoux, a.rhouy, a.rhoE, icv, yp * nx + x, &ux1, &uy1, &T1);
    init_near(a.rho, a.rhoux, a.rhouy, a.rhoE, icv, ym * nx + x, &ux2, &uy2, &T2);
    du[1][0] = 0.5 * (ux1 - ux2);
    du[1][1] = 0.5 * (uy1 - uy2);
    dT[1] = 0.5 * (T1 - T2);
    const int U0x = select_shift(ux, pr.n0, pr.umax), U0y = select_shift(uy, pr.n0, pr.umax);
    const int code = lat_code(U0x, U0y);
    P lam[NM];
    const bool realizable = (r > 0.0) && (T > 0.0) && isfinite(r) && isfinite(T);
    bool fixed = false;
    const NodeState s0{r, ux - U0x, uy - U0y, T, 0};
    const int ns = realizable
                       ? node_equilibrium<P, BLOCK>(pr, cl, s0, false, [](P*) {}, lam, &cnt, nullptr,
                                                    &fixed)
                       : NEWTON_UNREALIZABLE;
    if (!realizable) n_bad += 1;
    if (ns != NEWTON_OK && realizable) n_fail += 1;
    if (ns == NEWTON_OK) {
      double ca[NM], cg[3];
      grad_poly(pr, r, T, ux - U0x, uy - U0y, du, dT, ca, cg);
      GradFill<P> fill(cl.pop, cl.eq, fixed, r, (2.0 * pr.cv - 2.0) * T, cg);
      visit_groups<double>(ca, fill);
      // the first collision starts from the multipliers just found if the
      // flow starts its solves from previous multipliers
      // with the neighbourhood rule, the neighbours' initial lattices (Eq.
      // criterion on their initial velocities, boundary rule outside the grid)
      uint8_t nb[8];
      if (pr.overlap > 0.0 && pr.rule == 1) {
        int m = 0;
        for (int dy = -1; dy <= 1; ++dy)
          for (int dx = -1; dx <= 1; ++dx) {
            if (dx == 0 && dy == 0) continue;
            bool g2 = false;
            const size_t kk = (size_t)resolve(y + dy, pr.ny, pr.bcy, &g2) * nx +
                              resolve(x + dx, pr.nx, pr.bcx, &g2);
            const double rr = a.rho[kk];
            nb[m++] = (uint8_t)lat_code(select_shift(a.rhoux[kk] / rr, pr.n0, pr.umax),
                                        select_shift(a.rhouy[kk] / rr, pr.n0, pr.umax));
          }
      }
      const NodeState s = node_moments<P, BLOCK>(pr, cl, code, nb);
      const NodeFields<P> nf = node_publish<P>(code, s, k, a.ps, a.mom_out, a.lat_out, a.nxt_out);
      P first[NM];
#pragma unroll
      for (int j = 0; j < NM; ++j) first[j] = lam[j];
      bool fixed2 = false;
      const int n2 = node_equilibrium<P, BLOCK>(
          pr, cl, s, pr.warm,
          [&](P* l) {
#pragma unroll
            for (int j = 0; j < NM; ++j) l[j] = first[j];
          },
          lam, &cnt, nullptr, &fixed2);
      if (!node_store<P, BLOCK>(pr, cl, nf, n2, fixed2, pr.warm, lam, k, a.ps, a.pop_out, a.lam_out))
        n_fail += 1;
    } else {
      for (int i = 0; i < NPLANES; ++i) a.pop_out[i * a.ps + k] = (P)0;
      a.mom_out[k] = (P)r;
      a.mom_out[a.ps + k] = (P)ux;
      a.mom_out[2 * a.ps + k] = (P)uy;
      a.mom_out[3 * a.ps + k] = (P)T;
      a.lat_out[k] = (uint8_t)code;
      a.nxt_out[k] = (uint8_t)code;
      if (a.lam_out)
#pragma unroll
        for (int j = 0; j < NM; ++j) a.lam_out[j * a.ps + k] = j == 3 || j == 5 ? (P)0.5 : (P)0;
    }
  }
  warp_count(a.ctr + CTR_UNREALIZABLE, n_bad);
  warp_count(a.ctr + CTR_NEWTON_FAIL, n_fail);
}

template <typename P>
__global__ void export_moments_kernel(const P* mom, size_t ps, size_t n, double cv, double* rho,
                                      double* rhoux, double* rhouy, double* rhoE) {
  for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n;
       k += (size_t)gridDim.x * blockDim.x) {
    const double r = (double)mom[k], ux = (double)mom[ps + k], uy = (double)mom[2 * ps + k],
                 T = (double)mom[3 * ps + k];
    rho[k] = r;
    rhoux[k] = r * ux;
    rhouy[k] = r * uy;
    rhoE[k] = 0.5 * r * (ux * ux + uy * uy) + r * cv * T;
  }
}

// Planes [p0, p0 + np) of a buffer (population or moment planes, stride ps)
// as FP64 planes of n values each.
template <typename P>
__global__ void export_planes_kernel(const P* src, size_t ps, size_t n, int np, double* dst) {
  const size_t total = (size_t)np * n;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total;
       t += (size_t)gridDim.x * blockDim.x) {
    const size_t p = t / n, k = t - p * n;
    dst[t] = (double)src[p * ps + k];
  }
}

__global__ void export_shifts_kernel(const uint8_t* lat, size_t n, signed char* ux,
                                     signed char* uy) {
  for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n;
       k += (size_t)gridDim.x * blockDim.x) {
    const int c = lat[k];
    ux[k] = (signed char)lat_ux(c);
    uy[k] = (signed char)lat_uy(c);
  }
}

__global__ void __launch_bounds__(BLOCK)
    equilibrium_kernel(const double* rho, const double* ubx, const double* uby, const double* T,
                       int n, double tol, int maxit, int precision, double* feq, double* lambda,
                       int* iters, int* status) {
  __shared__ double s_tab[EXPT_N];
  __shared__ double s_eq[Q * BLOCK];
  load_exptab(s_tab);
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  double* eq = s_eq + threadIdx.x;
  double lam[NM];
  const double r = rho[k];
  SolveCount cnt;
  int st = NEWTON_UNREALIZABLE;
  if (r > 0.0) {
    if (precision == 0) {
      int it = 0, ev = 0;
      st = newton_fp64g(ubx[k], uby[k], T[k], tol, maxit, s_tab, eq, BLOCK, lam, &it, &ev, nullptr);
      cnt.fp64_iters = it;
    } else {
      float l32[NM];  // the FP64 multipliers are asked for here
      st = equilibrium_mixed(ubx[k], uby[k], T[k], tol, maxit, s_tab, nullptr, eq, BLOCK, l32,
                             lam, &cnt);
    }
  }
  for (int i = 0; i < Q; ++i) feq[(size_t)k * Q + i] = st == NEWTON_UNREALIZABLE ? 0.0 : r * eq[i * BLOCK];
  if (lambda)
#pragma unroll
    for (int j = 0; j < NM; ++j) lambda[(size_t)k * NM + j] = lam[j];
  if (iters)
    iters[k] = precision == 0 ? (int)cnt.fp64_iters : (int)(cnt.fp64_evals + cnt.fp64_updates);
  if (status) status[k] = st;
}

template <bool REFINE>
__global__ void exp_neg_kernel(const double* s, int n, double* out) {
  __shared__ double s_tab[EXPT_N];
  load_exptab(s_tab);
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) out[k] = REFINE ? exp_neg_refine(s[k], (float)s[k], s_tab) : exp_neg(s[k], s_tab);
}

__global__ void select_kernel(const double* rho, const double* rhou, int n, double n0, int umax,
                              signed char* out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  out[k] = (signed char)select_shift(rhou[k] / rho[k], n0, umax);
}

// ----------------------------------------------------------------- launchers

static dim3 grid_of(const Params& p) { return dim3((p.nx + BLOCK - 1) / BLOCK, p.ny); }

// Tiles of the step kernel: 2^lg nodes along x, the block's other threads on the
// following rows. 32 nodes (one warp, one 128-byte line) along x rather than a
// whole row: the pulls missing along an interface between two lattices then
// share their senders within a tile, so each is solved fewer times and fewer
// solves follow one another in one block (1021 x 733 shear layer: 0.089 against
// 0.148 rebuild solves per node and 0.81 against 1.35 ms a step for rows of 256;
// 64 wide 0.90 ms; 16 wide 0.80 ms there and 14.37 against 14.41 ms at 4096^2,
// but half a line per row). Narrower or wider where the grid is.
static dim3 step_grid(const Params& p, int block, int* lg) {
  int l = 3;
  while (l < 5 && (1 << l) < p.nx) ++l;
  l = tile_lg(l, block, p.ny);
  *lg = l;
  const int rows = block >> l;
  return dim3((p.nx + (1 << l) - 1) >> l, (p.ny + rows - 1) / rows);
}

// Dynamic shared memory needs an explicit opt-in once static plus dynamic
// shared memory exceed 48 KB; the dynamic size is always declared.
template <typename K>
static cudaError_t allow_smem(K kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

cudaError_t launch_init(FlowDev& f, const double* rho, const double* rhoux, const double* rhouy,
                        const double* rhoE, cudaStream_t s) {
  if (f.q == 49) return launch_init_q49(f, rho, rhoux, rhouy, rhoE, s);
  const int out = f.cur;
  cudaError_t e;
  if (f.precision == 0) {
    InitArgs<double> a{rho, rhoux, rhouy, rhoE, (double*)f.pop[out], (double*)f.mom[out],
                       f.lat[out], f.nxt[out], (double*)f.lam[out], f.ps, f.prm, f.ctr};
    if ((e = allow_smem(init_kernel<double>, smem_bytes<double>())) != cudaSuccess) return e;
    init_kernel<double><<<grid_of(f.prm), BLOCK, smem_bytes<double>(), s>>>(a);
  } else {
    InitArgs<float> a{rho, rhoux, rhouy, rhoE, (float*)f.pop[out], (float*)f.mom[out],
                      f.lat[out], f.nxt[out], (float*)f.lam[out], f.ps, f.prm, f.ctr};
    if ((e = allow_smem(init_kernel<float>, smem_bytes<float>())) != cudaSuccess) return e;
    init_kernel<float><<<grid_of(f.prm), BLOCK, smem_bytes<float>(), s>>>(a);
  }
  return cudaGetLastError();
}

template <typename P, int B, int MINB>
static cudaError_t launch_step_shape(const FlowDev& f, cudaStream_t s) {
  const cudaError_t e = allow_smem(step_kernel<P, B, MINB>, smem_bytes<P, B>());
  if (e != cudaSuccess) return e;
  int lg = 0;
  const dim3 g = step_grid(f.prm, B, &lg);
  step_kernel<P, B, MINB><<<g, B, smem_bytes<P, B>(), s>>>(step_args<P>(f, f.cur), lg);
  return cudaGetLastError();
}

// FP64 plain: blocks of 128 threads, two per SM by shared memory, or up to 512^2
// nodes of 256, where the longer rounds of rebuild solves save more than the
// second block hides (64^2 vortex 0.39 against 0.42 ms, 201^2 Riemann 0.45 / 0.56,
// 512^2 shear 1.44 / 1.46, but 700^2 2.53 / 2.46 and 1400^2 vortex 7.73 / 7.39).
//
// FP32 form, ms a step with 256 threads and 255 registers (one block per SM),
// 384 and 168, and two blocks of 256 and 128, which spill most but keep 16 warps:
//   600^2 shear 0.288 / 0.296 / -        600^2 vortex 0.209 / 0.203 / -
//   800^2 shear 0.441 / 0.423 / -        800^2 Riemann 0.476 / 0.455 / -
//   1030^2 shear 0.674 / 0.643 / 0.613   1030^2 vortex 0.557 / 0.530 / 0.483
//   1400^2 shear 1.08 / 1.01 / 0.93      1400^2 Riemann 1.11 / 1.05 / 1.02
//   2048^2 shear 2.05 / 1.93 / 1.70      2900^2 Riemann 4.15 / 3.96 / 3.75
//   4096^2 shear 7.44 / 7.02 / 6.04
// and below, in an earlier build, 64^2 vortex 0.103 / 0.149 / 0.127, 201^2 Riemann
// 0.105 / 0.121 / 0.131, 512^2 shear 0.260 / 0.277 / 0.283, 700^2 shear 0.376 / 0.368
// / 0.419. Few tiles want the shortest chain through one block, many the most warps.
// Blocks smaller than 256 lose threads for an interface tile's rebuild solves
// (201^2: 0.161 with 128, 0.207 with 64 where 256 took 0.151). Grids of fewer
// than 8 rows do not fill the 32 x 8 tile: 128 threads (2048 x 4 tube 0.048 ms).
constexpr size_t FP64_SMALL = 512 * 512, FP32_SMALL = 512 * 512, FP32_MEDIUM = 1024 * 1024;

cudaError_t launch_step(FlowDev& f, cudaStream_t s) {
  if (f.q == 49) return launch_step_q49(f, s);
  cudaError_t e;
  if (f.precision == 0)
    e = f.n <= FP64_SMALL && f.prm.ny >= 8 ? launch_step_shape<double, 256, 1>(f, s)
                                           : launch_step_shape<double, 128, 1>(f, s);
  else if (f.prm.ny < 8)
    e = launch_step_shape<float, 128, 2>(f, s);
  else if (f.n <= FP32_SMALL)
    e = launch_step_shape<float, 256, 1>(f, s);
  else if (f.n <= FP32_MEDIUM)
    e = launch_step_shape<float, 384, 1>(f, s);
  else
    e = launch_step_shape<float, 256, 2>(f, s);
  if (e == cudaSuccess) f.cur ^= 1;
  return e;
}

cudaError_t launch_export_moments(const FlowDev& f, double* rho, double* rhoux, double* rhouy,
                                  double* rhoE, cudaStream_t s) {
  const int blocks = (int)((f.n + 255) / 256 < 4096 ? (f.n + 255) / 256 : 4096);
  if (f.precision == 0)
    export_moments_kernel<double><<<blocks, 256, 0, s>>>((const double*)f.mom[f.cur], f.ps, f.n,
                                                         f.prm.cv, rho, rhoux, rhouy, rhoE);
  else
    export_moments_kernel<float><<<blocks, 256, 0, s>>>((const float*)f.mom[f.cur], f.ps, f.n,
                                                        f.prm.cv, rho, rhoux, rhouy, rhoE);
  return cudaGetLastError();
}

cudaError_t launch_export_planes(const FlowDev& f, int what, int p0, int np, double* dst,
                                 cudaStream_t s) {
  const int buf = f.cur;
  const void* base = what == 0 ? f.pop[buf] : f.mom[buf];
  const size_t total = (size_t)np * f.n;
  const int blocks = (int)((total + 255) / 256 < 8192 ? (total + 255) / 256 : 8192);
  if (total == 0) return cudaSuccess;
  if (f.precision == 0)
    export_planes_kernel<double><<<blocks, 256, 0, s>>>((const double*)base + p0 * f.ps, f.ps,
                                                        f.n, np, dst);
  else
    export_planes_kernel<float><<<blocks, 256, 0, s>>>((const float*)base + p0 * f.ps, f.ps,
                                                       f.n, np, dst);
  return cudaGetLastError();
}

cudaError_t launch_export_shifts(const FlowDev& f, signed char* ux, signed char* uy,
                                 cudaStream_t s, bool next) {
  const int blocks = (int)((f.n + 255) / 256 < 4096 ? (f.n + 255) / 256 : 4096);
  export_shifts_kernel<<<blocks, 256, 0, s>>>(next ? f.nxt[f.cur] : f.lat[f.cur], f.n, ux, uy);
  return cudaGetLastError();
}

cudaError_t launch_equilibrium(const double* rho, const double* ubx, const double* uby,
                               const double* T, int n, double tol, int maxit, int precision,
                               double* feq, double* lambda, int* iters, int* status,
                               cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  equilibrium_kernel<<<(n + BLOCK - 1) / BLOCK, BLOCK, 0, s>>>(rho, ubx, uby, T, n, tol, maxit,
                                                               precision, feq, lambda, iters,
                                                               status);
  return cudaGetLastError();
}

cudaError_t launch_exp_neg(const double* x, int n, double* out, cudaStream_t s, bool refine) {
  if (n <= 0) return cudaSuccess;
  if (refine)
    exp_neg_kernel<true><<<(n + 255) / 256, 256, 0, s>>>(x, n, out);
  else
    exp_neg_kernel<false><<<(n + 255) / 256, 256, 0, s>>>(x, n, out);
  return cudaGetLastError();
}

cudaError_t launch_select(const double* rho, const double* rhou, int n, double n0, int umax,
                          signed char* out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  select_kernel<<<(n + 255) / 256, 256, 0, s>>>(rho, rhou, n, n0, umax, out);
  return cudaGetLastError();
}

}  // namespace alb
