// Device kernels of the batched Henry-problem solver (sm_103a).
//
// Data layout (per multigrid level k of a batch of B samples, grid nx x ny):
//  * every per-cell array is [B][N] with N = nx ny, sample-major;
//  * inside a sample, cells are stored row by row, and inside each row the
//    cells of colour 0 ((ix + iy) even) come first, then those of colour 1:
//        st(ix, iy) = iy nx + colour (nx / 2) + ix / 2.
//    A red or black Gauss-Seidel half-sweep therefore streams contiguous
//    memory, and the two colours never share a 32-byte sector.
//  * the Jacobian of a level is 6 planes of 2x2 blocks [6][B N]: centre,
//    west, east, south, north, and the inverse of the centre block (so the
//    smoother needs no division); block = {a00, a01, a10, a11}, row = equation
//    (fluid mass, salt), column = unknown (p, c).
//  * states (p, c) and residuals are FP64 double2; the Jacobian, Krylov and
//    multigrid vectors are T (double, or float in the mixed-precision mode).
//
// The discrete equations are the cell-centred finite-volume form of Eqs.
// (e_cont_eq), (e_tran_eq) with Darcy's law (e_Darcy_vel), rho(c) linear
// (e_lin_density), D = phi Dm (e_mol_diff) and the boundary conditions of
// Sec. 2.1 of arXiv 2302.07804; every flux is taken outward from the cell:
//   interior face P|Nb:  rho_f = (rho_P + rho_Nb)/2,
//       q = -(K/mu) ((p_Nb - p_P)/h + sigma rho_f g),  sigma = +1 north, -1 south, 0 east/west
//       F = rho_f q h,  G = F c_up - rho_f phi Dm (c_Nb - c_P),  c_up = c_P if F >= 0 else c_Nb
//   x = 0:  F = -rho0 q_in h,  G = F c_up(c_b = 0) + 2 rho_b phi Dm c_P,  rho_b = (rho_P + rho0)/2
//   x = Lx: q = -(K/mu)(p_b - p_P)/(h/2), p_b = rho1 g (Ly - y_P), rho_b = (rho_P + rho1)/2,
//           F = rho_b q h, c_up = c_P if F >= 0 else 1, G = F c_up - 2 rho_b phi Dm (1 - c_P)
//   R^m = phi (rho - rho_old) h^2/tau + sum F,   R^s = phi (rho c - rho_old c_old) h^2/tau + sum G
// and every residual and Jacobian entry is multiplied by inv_s = 1 / (rho0 h_fine^2 / tau).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

namespace hk {

constexpr int TPB = 256;  // threads per CTA of every cell kernel

struct __align__(32) d4_t { double a00, a01, a10, a11; };
struct __align__(16) f4_t { float a00, a01, a10, a11; };

template <typename T> struct VT;
template <> struct VT<double> { typedef double2 v2; typedef d4_t b4; };
template <> struct VT<float> { typedef float2 v2; typedef f4_t b4; };

template <typename V2, typename T>
__device__ __forceinline__ V2 mk2(T a, T b) { V2 v; v.x = a; v.y = b; return v; }

// Physics constants passed by value.
struct Phys {
  double rho0, rho1, drho, g, Ly, Dm;
  double rho1g;  // rho1 g
};

// Per-sample coefficients: porosity, K / mu, phi * Dm, inflow velocity.
struct Coef {
  double phi, kmu, PD, qin;
};

// Per-sample scalars of BiCGStab.
struct LinScal {
  double rho, alpha, omega, bnorm2;
  double aow;  // alpha / omega
};

// Partial-sum slots of the fine-level reductions: [q][B][nct].
enum { P_RR = 0, P_RN = 1, P_RV = 2, P_TS = 3, P_TT = 4, P_MAX = 5, P_DC = 6, NPART = 7 };

__host__ __device__ __forceinline__ int st_of(int ix, int iy, int nx) {
  return iy * nx + (((ix + iy) & 1) ? (nx >> 1) : 0) + (ix >> 1);
}
// Grid widths and cells per sample are powers of two: indices are split by
// shifts (a 64-bit division is some 70 instructions, a noticeable part of a
// small launch).
__device__ __forceinline__ int lg2(int pow2) { return 31 - __clz(pow2); }
__device__ __forceinline__ int sample_of(int64_t e, int N) { return (int)(e >> lg2(N)); }
__device__ __forceinline__ void xy_of(int st, int nx, int& ix, int& iy) {
  iy = st >> lg2(nx);
  const int r = st - iy * nx, half = nx >> 1;
  const int col = r >= half ? 1 : 0;
  const int j = r - col * half;
  ix = 2 * j + ((col ^ iy) & 1);
}

// Programmatic dependent launch.  The kernels of a solve form one chain; each
// is launched with the programmatic-serialisation attribute, so that its CTAs
// start, split their indices and load what does not come from the kernel
// before while that one drains (measured on GB300 between dependent launches
// of a small kernel: 4.1 -> 1.4 us on a stream, 1.3 -> 0.95 us as graph nodes).
// Rules that keep this safe:
//  * every CTA of every kernel of the chain waits (grid_wait) before it ends,
//    also where its sample has stopped, so a kernel's completion implies its
//    predecessors';
//  * a kernel lets its successor start (grid_start_next) only after its own
//    wait, so when a kernel starts, all kernels but its direct predecessor
//    have completed: what those wrote (operators, right-hand sides, flags) may
//    be read before the wait, what the predecessor writes only after it;
//  * nothing is written before the wait, and pointers to what the
//    predecessor writes carry no __restrict__ (their loads must not become
//    read-only ones that could be moved across the wait).
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_start_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_enter() {
  grid_wait();
  grid_start_next();
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// Deterministic CTA-wide sum; the result is returned to every thread.
__device__ __forceinline__ double block_reduce(double v, double* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    const double u = warp_sum(lane < nw ? sh[lane] : 0.0);
    if (lane == 0) sh[32] = u;
  }
  __syncthreads();
  return sh[32];
}
// The same sum with fewer FP64 instructions: a shared-memory tree (halving
// the active threads each stage) down to one warp, then shuffles.  The FP64
// pipe (2 FMA units per SM on GB300) bounds the Krylov and SpMV kernels, and
// block_reduce's shuffle stage runs its adds in every warp: 5 per warp, 45
// warp instructions per 256-thread CTA, against 12 here.  sh: blockDim.x + 1
// doubles; blockDim.x a power of two >= 64.  Deterministic order.
__device__ __forceinline__ double block_sum_tree(double v, double* sh) {
  const int t = threadIdx.x, n = blockDim.x;
  sh[t] = v;
  __syncthreads();
  for (int s = n >> 1; s >= 32; s >>= 1) {
    if (t < s) sh[t] += sh[t + s];
    __syncthreads();
  }
  if (t < 32) {
    double u = warp_sum(sh[t]);
    if (t == 0) sh[n] = u;
  }
  __syncthreads();
  return sh[n];
}
// Two such sums side by side (CTAs of TPB threads, the same order of additions
// each): the halves of the CTA take one each, so that their dependent
// additions - 8 of 64 cycles - run on different warps.  The first sum is
// returned to thread 0, the second to thread TPB / 2.  sh: 2 TPB doubles.
__device__ __forceinline__ double block_sum_pair(double v1, double v2, double* sh) {
  const int t = threadIdx.x, u = t & (TPB / 2 - 1);
  sh[t] = v1;
  sh[TPB + t] = v2;
  __syncthreads();
  double* q = sh + (t >= TPB / 2 ? TPB : 0);
#pragma unroll
  for (int s = TPB / 2; s >= 32; s >>= 1) {
    if (u < s) q[u] += q[u + s];
    __syncthreads();
  }
  return u < 32 ? warp_sum(q[u]) : 0.0;
}
// CTA-wide max of non-negative doubles without NaNs (+inf allowed) on the
// integer pipes: for such values the IEEE-754 bit patterns order like the
// values, so the max of the 64-bit patterns is the max of the values, with no
// FP64 instruction.
__device__ __forceinline__ double block_max_nonneg(double v, double* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  unsigned long long u = (unsigned long long)__double_as_longlong(v);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long x = __shfl_xor_sync(0xffffffffu, u, o);
    u = x > u ? x : u;
  }
  unsigned long long* su = reinterpret_cast<unsigned long long*>(sh);
  __syncthreads();
  if (lane == 0) su[w] = u;
  __syncthreads();
  if (w == 0) {
    unsigned long long x = lane < nw ? su[lane] : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long y = __shfl_xor_sync(0xffffffffu, x, o);
      x = y > x ? y : x;
    }
    if (lane == 0) su[32] = x;
  }
  __syncthreads();
  return __longlong_as_double((long long)su[32]);
}
// Two sums over a sample's nct partials (slots a and b), computed identically
// by every CTA of the sample: warps 0 and 1 take one each, in a fixed order.
// fin (large grids): the finalised per-sample values instead (one warp per
// sample summed the partials in the same order).
__device__ __forceinline__ void sample_sums(const double* part, const double* fin, int a, int b, int64_t stride, int s,
                                            int nct, double* sh, double& va, double& vb) {
  if (fin) {
    va = fin[(int64_t)s * NPART + a];
    vb = fin[(int64_t)s * NPART + b];
    return;
  }
  const int w = threadIdx.x >> 5;
  if (w < 2) {
    const double* p = part + (w == 0 ? a : b) * stride + (int64_t)s * nct;
    double v = 0.0;
    for (int i = threadIdx.x & 31; i < nct; i += 32) v += p[i];
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) sh[w] = v;
  }
  __syncthreads();
  va = sh[0];
  vb = sh[1];  // the caller's next barrier comes before sh is written again
}
// One warp per sample: fin[s][slot] = sum of the sample's partials of up to
// two slots (slot_b < 0: one), in the order sample_sum uses.
__global__ void k_finalize(int B, int nct, const double* part, int slot_a, int slot_b,
                           double* __restrict__ fin) {
  grid_enter();
  const int s = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (s >= B) return;
  const int64_t stride = (int64_t)B * nct;
  for (int q = 0; q < 2; ++q) {
    const int slot = q == 0 ? slot_a : slot_b;
    if (slot < 0) continue;
    const double* p = part + slot * stride + (int64_t)s * nct;
    double v = 0.0;
    for (int i = lane; i < nct; i += 32) v += p[i];
    v = warp_sum(v);
    if (lane == 0) fin[(int64_t)s * NPART + slot] = v;
  }
}
// Max of a sample's nct non-negative partial maxima, by one warp (lanes
// stride over the partials; a max does not depend on the order), returned
// to every lane.  Wide grids have thousands of partials per sample.
__device__ __forceinline__ double warp_sample_max(const double* p, int nct, int lane) {
  unsigned long long v = 0;  // the bit patterns of non-negative values order like the values
  for (int i = lane; i < nct; i += 32) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(p[i]);
    v = u > v ? u : v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long u = __shfl_xor_sync(0xffffffffu, v, o);
    v = u > v ? u : v;
  }
  return __longlong_as_double((long long)v);
}

// 2x2 block helpers as explicit fused multiply-add chains: two FMAs per row
// (written as r - a x - b y the compiler would issue a MUL, an FMA and an
// ADD, and on GB300 the FP64 pipe is the smoother's bottleneck).
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
template <typename B4, typename T>
__device__ __forceinline__ void bmv_sub(const B4& A, T x0, T x1, T& r0, T& r1) {
  r0 = fma_(-A.a00, x0, fma_(-A.a01, x1, r0));
  r1 = fma_(-A.a10, x0, fma_(-A.a11, x1, r1));
}
template <typename B4, typename T>
__device__ __forceinline__ void bmv_add(const B4& A, T x0, T x1, T& r0, T& r1) {
  r0 = fma_(A.a00, x0, fma_(A.a01, x1, r0));
  r1 = fma_(A.a10, x0, fma_(A.a11, x1, r1));
}
template <typename B4, typename T>
__device__ __forceinline__ void bmv(const B4& A, T x0, T x1, T& y0, T& y1) {
  y0 = fma_(A.a00, x0, A.a01 * x1);
  y1 = fma_(A.a10, x0, A.a11 * x1);
}
// One row of the coarsest grid's explicit inverse times its four unknowns
// (every solver of that grid uses this order).
template <typename T>
__device__ __forceinline__ T coarse_row(const T* m, T v0, T v1, T v2, T v3) {
  return fma_(m[3], v3, fma_(m[2], v2, fma_(m[1], v1, m[0] * v0)));
}
template <typename B4>
__device__ __forceinline__ B4 mkblk(double a00, double a01, double a10, double a11) {
  B4 b;
  b.a00 = a00; b.a01 = a01; b.a10 = a10; b.a11 = a11;
  return b;
}

// Products that the compiler must not contract into multiply-adds, so that the
// assembly's arithmetic is the same at every call site; sign changes and
// comparisons on the integer pipes (an FP64 compare or negation takes the
// FP64 pipe's 64 cycles a warp).
__device__ __forceinline__ double mul_(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double neg_(double a) {
  return __hiloint2double(__double2hiint(a) ^ 0x80000000, __double2loint(a));
}
__device__ __forceinline__ float neg_(float a) { return -a; }
__device__ __forceinline__ bool nonneg(double a) {  // a >= 0 (-0 included)
  const long long u = __double_as_longlong(a);
  return u >= 0 || (u << 1) == 0;
}
__device__ __forceinline__ bool nonneg(float a) { return a >= 0.f; }
// max(|a|, |b|) as a non-negative double; +inf for anything beyond 1e300 or NaN.
__device__ __forceinline__ double abs_max_or_inf(double a, double b) {
  const unsigned long long m = 0x7fffffffffffffffull, lim = 0x7e37e43c8800759cull;  // the bits of 1e300
  const unsigned long long x = (unsigned long long)__double_as_longlong(a) & m;
  const unsigned long long y = (unsigned long long)__double_as_longlong(b) & m;
  const unsigned long long z = x > y ? x : y;
  return __longlong_as_double((long long)(z <= lim ? z : 0x7ff0000000000000ull));
}

// ---------------------------------------------------------------------------
// a4 (and coarse operators by rediscretisation): residual and Jacobian.
//
// A face between a left/lower cell L and a right/upper cell R carries the
// scaled mass and salt fluxes F, G from L to R; L's residuals gain +F, +G and
// R's lose them.  With rho_f = rs / 2 (rs = rho_L + rho_R), K/mu = 2 kh and
// phi Dm = 2 PDh (all scaled by inv_s, the square cells' h in F's favour):
//   F = rs qh,  qh = -kh (p_R - p_L + ghh rs)   (ghh = g h / 2 on a north face, else 0)
//   G = F c_up - rs PDh (c_R - c_L),  c_up = c_L if F >= 0 else c_R  (the tie takes c_L)
//   dF/dp_L = rs kh = -dF/dp_R,  dF/dc_L = dF/dc_R = drho (qh - kh ghh rs),
//   dG/dp = c_up dF/dp,  dG/dc_L = c_up dF/dc + [F if F >= 0] + PD rho_L,
//   dG/dc_R = c_up dF/dc + [F if F < 0] - PD rho_R
// (the diffusive terms because rho_f -+ drho (c_R - c_L) / 2 are rho_L and
// rho_R): 19 operations for a north face, 17 for an east one, derivatives
// included.  The seaside boundary is an east face with twice the cell's
// coefficients (half the distance) to a ghost cell of p_b = rho1 g (Ly - y),
// c = 1; the land side has its prescribed flux (land_side).
//
// What bounds it: the FP64 pipe (a warp instruction takes 17-19 cycles of an
// SM).  Per cell 36 operations of its east and north face, ~4 of re-evaluated
// tile-edge faces, 22 to add four faces, 8 accumulation, ~14 for the inverse
// of the centre block - about 95 instead of 176 before the fluxes were written
// in these terms, with comparisons and sign changes on the integer pipes and
// the scaled coefficients formed once per sample and level.  8192 level-0
// samples, FP64, per call of the event timer: residual and Jacobian 1048 ->
// 639 us, residual alone 468 -> 289 us, coarse operators 68 -> 42 us; the
// solve 440 -> 386 ms; the fused FP32 level-0 solver, 1000 samples, 32.6 ->
// 28.6 ms.
//
// Fluxes and residuals are formed in S (FP64 on the fine grid), derivatives
// and blocks in T; in the mixed mode (T = float) the coarse operators are
// assembled entirely in FP32 (S = T) and the fine Jacobian's derivative terms
// in FP32 from FP64 fluxes.
//
// Scaled coefficients of one sample on one multigrid level of the constant-
// coefficient model (formed by level_coef: k_coefficients for every level, the
// fused solver its own), inv_s included.
struct __align__(64) LevelCoef {
  double kh, kg;    // K / (2 mu), kh g h / 2
  double PD, PDh;   // phi Dm, half of it
  double pv, pvd;   // phi h^2 / tau, that times drho
  double Fl, Flo;   // land side: outward mass flux -rho0 q_in h, and max(Fl, 0)
};
template <typename S>
struct FaceCoef {
  S kh, kg, PD, PDh;
};
template <typename T, typename S, bool JAC = true>
struct FaceData {
  S F, G;              // fluxes L -> R (scaled)
  T dp, dc, dpc;       // dF/dp_L, dF/dc, dG/dp_L
  T gL, gR;            // dG/dc_L, dG/dc_R
};
// Residual-only evaluation (JAC = false): the fluxes alone.
template <typename T, typename S>
struct FaceData<T, S, false> {
  S F, G;
};

// JAC = false: the fluxes only, with exactly the arithmetic of the JAC =
// true form, so both forms give bit-identical residuals.
// DROP: the fallback preconditioner operator - the Jacobian without the
// derivatives of the face densities with respect to c (dF/dc = 0 in both
// rows), an operator whose diagonal blocks stay definite where density
// contrasts over heterogeneous K make point-block Gauss-Seidel diverge.
template <typename T, typename S, bool NORTH, bool DROP, bool JAC = true>
__device__ __forceinline__ void face_eval(S drho, S rho0, S ghh, const FaceCoef<S>& k, S pL, S cL, S pR, S cR,
                                          FaceData<T, S, JAC>& f) {
  const S rhoL = fma_(drho, cL, rho0), rhoR = fma_(drho, cR, rho0);
  const S rs = rhoL + rhoR;
  S u = pR - pL;
  if (NORTH) u = fma_(ghh, rs, u);
  const S qh = mul_(neg_(k.kh), u);
  const S Ff = mul_(rs, qh);
  const bool up = nonneg(Ff);
  const S cup = up ? cL : cR;
  f.F = Ff;
  f.G = fma_(Ff, cup, neg_(mul_(rs, mul_(k.PDh, cR - cL))));
  if constexpr (JAC) {
    const T rsT = (T)rs, cupT = (T)cup, FT = (T)Ff, khT = (T)k.kh, PDT = (T)k.PD, dT = (T)drho;
    // one rounding each; (T)rs - (T)rhoL carries two, one of them of a value twice as
    // large (and saves a conversion: level 0, mixed, 1000 samples 16.93 against 17.01 ms)
    const T rLT = (T)rhoL, rRT = (T)rhoR;
    const T dp = mul_(rsT, khT);
    const T dc = DROP ? (T)0 : mul_(dT, NORTH ? fma_(neg_((T)k.kg), rsT, (T)qh) : (T)qh);
    f.dp = dp;
    f.dc = dc;
    f.dpc = mul_(dp, cupT);
    f.gL = fma_(dc, cupT, (up ? FT : (T)0) + mul_(PDT, rLT));
    f.gR = fma_(dc, cupT, (up ? (T)0 : FT) - mul_(PDT, rRT));
  }
}

// One cell's residual and blocks as its faces are added.
template <typename T, typename S, bool JAC = true>
struct CellSum {
  S Rm, Rs;
  T C[4], Nb[4][4];  // centre block; W, E, S, N blocks
};
// Accumulation terms.
template <typename T, typename S, bool JAC>
__device__ __forceinline__ void cell_begin(S drho, S rho0, S pv, S pvd, S cP, S cO, CellSum<T, S, JAC>& o) {
  const S d = cP - cO;
  o.Rm = mul_(pvd, d);
  o.Rs = mul_(mul_(pv, d), fma_(drho, cP + cO, rho0));
  if constexpr (JAC) {
    o.C[0] = o.C[2] = (T)0;
    o.C[1] = (T)pvd;
    o.C[3] = (T)mul_(pv, fma_((S)2 * drho, cP, rho0));
#pragma unroll
    for (int k = 0; k < 4; ++k) o.Nb[k][0] = o.Nb[k][1] = o.Nb[k][2] = o.Nb[k][3] = (T)0;
  }
}
// The face to neighbour k (0 W, 1 E, 2 S, 3 N); IS_L: the cell is its L.  With
// nb false (the seaside boundary face) no neighbour block.
template <bool IS_L, typename T, typename S, bool JAC>
__device__ __forceinline__ void cell_add(const FaceData<T, S, JAC>& f, int k, CellSum<T, S, JAC>& o, bool nb = true) {
  if (IS_L) {
    o.Rm += f.F;
    o.Rs += f.G;
    if constexpr (JAC) {
      o.C[0] += f.dp;
      o.C[1] += f.dc;
      o.C[2] += f.dpc;
      o.C[3] += f.gL;
      if (nb) {
        o.Nb[k][0] = neg_(f.dp);
        o.Nb[k][1] = f.dc;
        o.Nb[k][2] = neg_(f.dpc);
        o.Nb[k][3] = f.gR;
      }
    }
  } else {
    o.Rm -= f.F;
    o.Rs -= f.G;
    if constexpr (JAC) {
      o.C[0] += f.dp;
      o.C[1] -= f.dc;
      o.C[2] += f.dpc;
      o.C[3] -= f.gR;
      o.Nb[k][0] = neg_(f.dp);
      o.Nb[k][1] = neg_(f.dc);
      o.Nb[k][2] = neg_(f.dpc);
      o.Nb[k][3] = neg_(f.gL);
    }
  }
}
// The land side (ix = 0): prescribed inflow of fresh water, c_b = 0, diffusion
// over half a cell; Fl the outward mass flux, Flo = max(Fl, 0), PD the cell's.
template <typename T, typename S, bool JAC>
__device__ __forceinline__ void land_side(S drho, S rho0, S Fl, S Flo, S PD, S cP, CellSum<T, S, JAC>& o) {
  const S rhoP = fma_(drho, cP, rho0), PDr = mul_(PD, cP);
  o.Rm += Fl;
  o.Rs += fma_(Flo, cP, mul_(rhoP + rho0, PDr));
  if constexpr (JAC) o.C[3] += (T)fma_((S)2 * PD, rhoP, Flo);
}

// A thread's view of its cell's coefficients: the sample's scalars or, with
// FIELDS, cc[st] = (phi, K/mu) of the cell and fc[st] = (K / (2 mu), phi Dm),
// scaled by inv_s, on its east (.x, .y) and north (.z, .w) face (harmonic
// means; zero across the boundary).
template <typename S, bool FIELDS>
struct CellCoefs {
  S pv, pvd, PD, Fl, Flo;
  FaceCoef<S> in;  // of the sample's interior faces (not FIELDS)
  S kc;            // K/mu of the cell, scaled (FIELDS: for the seaside face)

  __device__ __forceinline__ void load(const Phys& ph, const LevelCoef* lc, const Coef* coef, int s, double vt_s,
                                       double inv_s, double h, const double2* cc, int64_t e) {
    if constexpr (FIELDS) {
      const double2 c = cc[e];
      pv = (S)mul_(c.x, vt_s);
      pvd = mul_(pv, (S)ph.drho);
      kc = (S)mul_(c.y, inv_s);
      PD = (S)mul_(mul_(c.x, ph.Dm), inv_s);
      Fl = (S)mul_(mul_(mul_(-ph.rho0, coef[s].qin), inv_s), h);
      Flo = nonneg(Fl) ? Fl : (S)0;
    } else {
      const LevelCoef c = lc[s];
      pv = (S)c.pv;
      pvd = (S)c.pvd;
      PD = (S)c.PD;
      Fl = (S)c.Fl;
      Flo = (S)c.Flo;
      in.kh = (S)c.kh;
      in.kg = (S)c.kg;
      in.PD = (S)c.PD;
      in.PDh = (S)c.PDh;
      kc = in.kh + in.kh;
    }
  }
  // The east or north face of the cell at entry e (its L).
  __device__ __forceinline__ FaceCoef<S> face(bool north, S ghh, const double4_32a* fc, int64_t e) const {
    if constexpr (FIELDS) {
      const double4_32a q = fc[e];
      FaceCoef<S> k;
      k.kh = (S)(north ? q.z : q.x);
      k.PD = (S)(north ? q.w : q.y);
      k.PDh = mul_((S)0.5, k.PD);
      k.kg = mul_(k.kh, ghh);
      return k;
    } else {
      return in;
    }
  }
  // The seaside boundary face: twice the cell's coefficients.
  __device__ __forceinline__ FaceCoef<S> sea() const {
    FaceCoef<S> k;
    k.kh = kc;
    k.kg = (S)0;
    k.PD = PD + PD;
    k.PDh = PD;
    return k;
  }
};
__device__ __forceinline__ double2 sea_ghost(const Phys& ph, double h, int iy) {
  // iy + 1/2 exactly, from the bits of 2^52 + iy (an int conversion takes the FP64 pipe as well)
  const double y = __hiloint2double(0x43300000, iy) - 4503599627370495.5;
  return make_double2(mul_(ph.rho1g, fma(-h, y, ph.Ly)), 1.0);
}

// One cell, all four faces evaluated by its own thread.  `xs`, `xos` point at
// the cell arrays of one sample (storage layout; global or shared memory), cc
// and fc at the sample's (FIELDS), e0 is the sample's first entry (unused
// here: the arrays are sample-relative).
template <typename T, typename S, bool FIELDS = false, bool DROP = false, bool JAC = true>
__device__ __forceinline__ void assemble_cell(const Phys& ph, const CellCoefs<S, FIELDS>& K, int nx, int ny, double h,
                                              const double2* xs, const double2* xos, int st, int ix, int iy,
                                              CellSum<T, S, JAC>& o, const double4_32a* fc = nullptr) {
  const S drho = (S)ph.drho, rho0 = (S)ph.rho0, ghh = (S)(0.5 * ph.g * h);
  const double2 xP = xs[st];
  const S pP = (S)xP.x, cP = (S)xP.y;
  cell_begin<T, S, JAC>(drho, rho0, K.pv, K.pvd, cP, (S)xos[st].y, o);
  FaceData<T, S, JAC> f;
  if (ix > 0) {
    const int w = st_of(ix - 1, iy, nx);
    const double2 xN = xs[w];
    face_eval<T, S, false, DROP, JAC>(drho, rho0, ghh, K.face(false, ghh, fc, w), (S)xN.x, (S)xN.y, pP, cP, f);
    cell_add<false>(f, 0, o);
  }
  {
    const bool sea = ix + 1 == nx;
    const double2 xN = sea ? sea_ghost(ph, h, iy) : xs[st_of(ix + 1, iy, nx)];
    face_eval<T, S, false, DROP, JAC>(drho, rho0, ghh, sea ? K.sea() : K.face(false, ghh, fc, st), pP, cP, (S)xN.x,
                                      (S)xN.y, f);
    cell_add<true>(f, 1, o, !sea);
  }
  if (iy > 0) {
    const int w = st_of(ix, iy - 1, nx);
    const double2 xN = xs[w];
    face_eval<T, S, true, DROP, JAC>(drho, rho0, ghh, K.face(true, ghh, fc, w), (S)xN.x, (S)xN.y, pP, cP, f);
    cell_add<false>(f, 2, o);
  }
  if (iy + 1 < ny) {
    const double2 xN = xs[st_of(ix, iy + 1, nx)];
    face_eval<T, S, true, DROP, JAC>(drho, rho0, ghh, K.face(true, ghh, fc, st), pP, cP, (S)xN.x, (S)xN.y, f);
    cell_add<true>(f, 3, o);
  }
  if (ix == 0) land_side<T, S, JAC>(drho, rho0, K.Fl, K.Flo, K.PD, cP, o);
}

// Store a cell's Jacobian blocks (6 planes with stride `ps`, incl. C^-1).
template <typename T>
__device__ __forceinline__ void store_blocks(typename VT<T>::b4* J, int64_t ps, int64_t i, const T C[4],
                                             const T Nb[4][4]) {
  typedef typename VT<T>::b4 B4;
  J[i] = mkblk<B4>(C[0], C[1], C[2], C[3]);
#pragma unroll
  for (int k = 0; k < 4; ++k) J[(k + 1) * ps + i] = mkblk<B4>(Nb[k][0], Nb[k][1], Nb[k][2], Nb[k][3]);
  const T idet = (T)1 / fma_(C[0], C[3], neg_(mul_(C[1], C[2])));
  const T nd = neg_(idet);
  J[5 * ps + i] = mkblk<B4>(mul_(C[3], idet), mul_(C[1], nd), mul_(C[2], nd), mul_(C[0], idet));
}

// One thread per cell; FINE: CTAs never straddle samples (N % TPB == 0) and
// write the per-CTA max |F| (inf for non-finite) to rmax_part[s][ct].
template <typename T, bool FINE, bool FIELDS = false, bool DROP = false, bool JAC = true>
__global__ void __launch_bounds__(TPB) k_assemble(Phys ph, const Coef* __restrict__ coef,
                                                  const LevelCoef* __restrict__ lc, int B, int nx, int ny,
                                                  double h, double vt_s, double inv_s,
                                                  const double2* x, const double2* xo,
                                                  const int* active, double2* __restrict__ F,
                                                  typename VT<T>::b4* __restrict__ J, int64_t plane,
                                                  double* __restrict__ rmax_part, const double2* __restrict__ cc,
                                                  const double4_32a* __restrict__ fc) {
  typedef typename std::conditional<FINE, double, T>::type S;
  __shared__ double sh[40];
  const int N = nx * ny;
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  const int64_t total = (int64_t)B * N;
  const int s = sample_of(e, N);
  grid_enter();
  if (FINE) {
    if (!active[s]) return;  // uniform over the CTA
  } else {
    if (e >= total || !active[s]) return;
  }
  const int st = (int)(e - (int64_t)s * N);
  int ix, iy;
  xy_of(st, nx, ix, iy);
  const int64_t base = e - st;
  CellCoefs<S, FIELDS> K;
  K.load(ph, lc, coef, s, vt_s, inv_s, h, cc, e);
  CellSum<T, S, JAC> o;
  assemble_cell<T, S, FIELDS, DROP, JAC>(ph, K, nx, ny, h, x + base, xo + base, st, ix, iy, o,
                                         FIELDS ? fc + base : nullptr);
  if (FINE) {
    const double fm = (double)o.Rm, fs = (double)o.Rs;
    if (F) F[e] = make_double2(fm, fs);
    const double bm = block_max_nonneg(abs_max_or_inf(fm, fs), sh);
    if (threadIdx.x == 0) {
      const int nct = N / TPB;
      rmax_part[(int64_t)s * nct + (st / TPB)] = bm;
    }
  }
  if constexpr (JAC) {
    if (J) store_blocks<T>(J, plane, e, o.C, o.Nb);
  }
}

// Tile assembly, the face-once form: every cell evaluates its east and north
// faces into shared memory (phase 1) and then sums its four faces (phase 2);
// a face to a cell of another tile is evaluated again, by the same code.
//
// k_assemble_tile: a CTA holds TPB consecutive cells in storage order, i.e.
// TPB / nx whole rows (nx <= TPB), possibly of several samples.  A cell of the
// tile's first row evaluates the face below it itself.  FINE: N % TPB == 0,
// one sample per CTA.  Shared memory: 2 x TPB faces (28 KB in FP64).
template <typename T, bool FINE, bool FIELDS, bool DROP, bool JAC>
__device__ __forceinline__ void assemble_tile(unsigned blk, const Phys& ph, const Coef* __restrict__ coef,
                                              const LevelCoef* __restrict__ lc, int B, int nx, int ny, double h,
                                              double vt_s, double inv_s, const double2* x, const double2* xo,
                                              const int* active, double2* __restrict__ F,
                                              typename VT<T>::b4* __restrict__ J, int64_t plane,
                                              double* __restrict__ rmax_part, const double2* __restrict__ cc,
                                              const double4_32a* __restrict__ fc) {
  typedef typename std::conditional<FINE, double, T>::type S;
  __shared__ FaceData<T, S, JAC> fE[TPB], fN[TPB];
  __shared__ double sh[40];
  const int N = nx * ny;
  const int64_t e = (int64_t)blk * TPB + threadIdx.x;
  const int64_t total = (int64_t)B * N;
  const int s = sample_of(e, N);
  if (FINE) {
    if (!active[s]) return;  // uniform over the CTA
  }
  const bool on = e < total && active[s];
  const int st = (int)(e - (int64_t)s * N);
  int ix = 0, iy = 0;
  xy_of(st, nx, ix, iy);
  const int64_t base = e - st;
  // tile slot of the cell (ix, row r of the tile); rows hold nx consecutive storage entries
  const int r = threadIdx.x >> lg2(nx);
  const int slot = r * nx + ix;
  const S drho = (S)ph.drho, rho0 = (S)ph.rho0, ghh = (S)(0.5 * ph.g * h);
  CellCoefs<S, FIELDS> K;
  S pP = (S)0, cP = (S)0;
  if (on) {
    K.load(ph, lc, coef, s, vt_s, inv_s, h, cc, e);
    const double2 xP = x[e];
    pP = (S)xP.x;
    cP = (S)xP.y;
    const bool sea = ix + 1 == nx;
    {  // east face (or the seaside boundary), P = L
      const double2 xN = sea ? sea_ghost(ph, h, iy) : x[base + st_of(ix + 1, iy, nx)];
      face_eval<T, S, false, DROP, JAC>(drho, rho0, ghh, sea ? K.sea() : K.face(false, ghh, fc, e), pP, cP, (S)xN.x,
                                        (S)xN.y, fE[slot]);
    }
    if (iy + 1 < ny) {  // north face, P = L
      const double2 xN = x[base + st_of(ix, iy + 1, nx)];
      face_eval<T, S, true, DROP, JAC>(drho, rho0, ghh, K.face(true, ghh, fc, e), pP, cP, (S)xN.x, (S)xN.y, fN[slot]);
    }
  }
  __syncthreads();
  if (!on) return;
  CellSum<T, S, JAC> o;
  cell_begin<T, S, JAC>(drho, rho0, K.pv, K.pvd, cP, (S)xo[e].y, o);
  if (ix > 0) cell_add<false>(fE[slot - 1], 0, o);       // W: P = R
  cell_add<true>(fE[slot], 1, o, ix + 1 < nx);            // E: P = L
  if (iy > 0) {                                           // S: P = R
    if (r > 0) {
      cell_add<false>(fN[slot - nx], 2, o);
    } else {  // the lower cell is in another tile: evaluate the face here
      const int sb = st_of(ix, iy - 1, nx);
      const double2 xN = x[base + sb];
      FaceData<T, S, JAC> f;
      face_eval<T, S, true, DROP, JAC>(drho, rho0, ghh, K.face(true, ghh, fc, base + sb), (S)xN.x, (S)xN.y, pP, cP, f);
      cell_add<false>(f, 2, o);
    }
  }
  if (iy + 1 < ny) cell_add<true>(fN[slot], 3, o);        // N: P = L
  if (ix == 0) land_side<T, S, JAC>(drho, rho0, K.Fl, K.Flo, K.PD, cP, o);
  if (FINE) {
    const double fm = (double)o.Rm, fs = (double)o.Rs;
    if (F) F[e] = make_double2(fm, fs);
    const double bm = block_max_nonneg(abs_max_or_inf(fm, fs), sh);
    if (threadIdx.x == 0) {
      const int nct = N / TPB;
      rmax_part[(int64_t)s * nct + (st / TPB)] = bm;
    }
  }
  if constexpr (JAC) {
    if (J) store_blocks<T>(J, plane, e, o.C, o.Nb);
  }
}

template <typename T, bool FINE, bool FIELDS = false, bool DROP = false, bool JAC = true>
__global__ void __launch_bounds__(TPB) k_assemble_tile(Phys ph, const Coef* __restrict__ coef,
                                                       const LevelCoef* __restrict__ lc, int B, int nx, int ny,
                                                       double h, double vt_s, double inv_s,
                                                       const double2* x, const double2* xo,
                                                       const int* active, double2* __restrict__ F,
                                                       typename VT<T>::b4* __restrict__ J, int64_t plane,
                                                       double* __restrict__ rmax_part,
                                                       const double2* __restrict__ cc,
                                                       const double4_32a* __restrict__ fc) {
  grid_enter();
  assemble_tile<T, FINE, FIELDS, DROP, JAC>(blockIdx.x, ph, coef, lc, B, nx, ny, h, vt_s, inv_s, x, xo, active, F, J,
                                            plane, rmax_part, cc, fc);
}

// The coarse operators of several levels (nx <= TPB) in one launch: a level's
// assembly is one dependent chain of some 95 operations a cell (3 us in FP64
// whatever the grid), and the levels do not depend on one another.
struct AssembleLevels {
  static constexpr int MAX = 12;
  int n;
  unsigned first[MAX + 1];  // first block of each level
  int nx[MAX], ny[MAX];
  double h[MAX], vt_s[MAX];
  const LevelCoef* lc[MAX];
  const double2 *x[MAX], *xo[MAX];
  void* J[MAX];
  int64_t plane[MAX];
  const double2* cc[MAX];
  const double4_32a* fc[MAX];
};
template <typename T, bool FIELDS, bool DROP>
__global__ void __launch_bounds__(TPB) k_assemble_levels(Phys ph, const Coef* __restrict__ coef,
                                                         const __grid_constant__ AssembleLevels A, int B,
                                                         double inv_s, const int* active) {
  grid_enter();
  int l = 0;
  while (l + 1 < A.n && blockIdx.x >= A.first[l + 1]) ++l;
  assemble_tile<T, false, FIELDS, DROP, true>(blockIdx.x - A.first[l], ph, coef, A.lc[l], B, A.nx[l], A.ny[l], A.h[l],
                                              A.vt_s[l], inv_s, A.x[l], A.xo[l], active, nullptr,
                                              (typename VT<T>::b4*)A.J[l], A.plane[l], nullptr, A.cc[l], A.fc[l]);
}

// k_assemble_tile2d: a CTA covers a TILE_W x (TPB / TILE_W) block of cells of
// one sample, mapped by position, not by storage order (nx a multiple of
// TILE_W, ny of TPB / TILE_W).  A cell on the tile's west or south edge
// evaluates that face itself: 2 + 1 / TH + 1 / TILE_W face evaluations per
// cell (TH = TPB / TILE_W rows; 2.5 for 128 x 2, 2.16 for 32 x 8).  The
// per-tile max |F| goes to slot (tile index) of the sample's N / TPB partials.
constexpr int TILE_W_DEFAULT = 128;  // for grids wider than TPB cells
template <typename T, bool FINE, bool FIELDS = false, bool DROP = false, bool JAC = true, int TILE_W = TILE_W_DEFAULT>
__global__ void __launch_bounds__(TPB) k_assemble_tile2d(Phys ph, const Coef* __restrict__ coef,
                                                         const LevelCoef* __restrict__ lc, int B, int nx,
                                                         int ny, double h, double vt_s, double inv_s,
                                                         const double2* x, const double2* xo,
                                                         const int* active, double2* __restrict__ F,
                                                         typename VT<T>::b4* __restrict__ J, int64_t plane,
                                                         double* __restrict__ rmax_part,
                                                         const double2* __restrict__ cc,
                                                         const double4_32a* __restrict__ fc) {
  typedef typename std::conditional<FINE, double, T>::type S;
  constexpr int TH = TPB / TILE_W;
  __shared__ FaceData<T, S, JAC> fE[TPB], fN[TPB];
  __shared__ double sh[40];
  const int N = nx * ny;
  const int tiles = N / TPB;  // per sample
  const int s = blockIdx.x >> lg2(tiles);
  const int tile = (int)(blockIdx.x - (int64_t)s * tiles);
  grid_enter();
  if (s >= B || !active[s]) return;  // uniform over the CTA
  const int tx = threadIdx.x % TILE_W, ty = threadIdx.x / TILE_W;
  const int tpr = nx / TILE_W;  // tiles per row band
  const int ix = (tile & (tpr - 1)) * TILE_W + tx, iy = (tile >> lg2(tpr)) * TH + ty;
  const int64_t base = (int64_t)s * N, e = base + st_of(ix, iy, nx);
  const int slot = threadIdx.x;
  const S drho = (S)ph.drho, rho0 = (S)ph.rho0, ghh = (S)(0.5 * ph.g * h);
  CellCoefs<S, FIELDS> K;
  K.load(ph, lc, coef, s, vt_s, inv_s, h, cc, e);
  const double2 xP = x[e];
  const S pP = (S)xP.x, cP = (S)xP.y;
  const bool sea = ix + 1 == nx;
  {  // east face (or the seaside boundary), P = L
    const double2 xN = sea ? sea_ghost(ph, h, iy) : x[base + st_of(ix + 1, iy, nx)];
    face_eval<T, S, false, DROP, JAC>(drho, rho0, ghh, sea ? K.sea() : K.face(false, ghh, fc, e), pP, cP, (S)xN.x,
                                      (S)xN.y, fE[slot]);
  }
  if (iy + 1 < ny) {  // north face, P = L
    const double2 xN = x[base + st_of(ix, iy + 1, nx)];
    face_eval<T, S, true, DROP, JAC>(drho, rho0, ghh, K.face(true, ghh, fc, e), pP, cP, (S)xN.x, (S)xN.y, fN[slot]);
  }
  __syncthreads();
  CellSum<T, S, JAC> o;
  cell_begin<T, S, JAC>(drho, rho0, K.pv, K.pvd, cP, (S)xo[e].y, o);
  if (ix > 0) {  // W: P = R
    if (tx > 0) {
      cell_add<false>(fE[slot - 1], 0, o);
    } else {
      const int64_t w = base + st_of(ix - 1, iy, nx);
      const double2 xN = x[w];
      FaceData<T, S, JAC> f;
      face_eval<T, S, false, DROP, JAC>(drho, rho0, ghh, K.face(false, ghh, fc, w), (S)xN.x, (S)xN.y, pP, cP, f);
      cell_add<false>(f, 0, o);
    }
  }
  cell_add<true>(fE[slot], 1, o, !sea);  // E: P = L
  if (iy > 0) {                          // S: P = R
    if (ty > 0) {
      cell_add<false>(fN[slot - TILE_W], 2, o);
    } else {
      const int64_t w = base + st_of(ix, iy - 1, nx);
      const double2 xN = x[w];
      FaceData<T, S, JAC> f;
      face_eval<T, S, true, DROP, JAC>(drho, rho0, ghh, K.face(true, ghh, fc, w), (S)xN.x, (S)xN.y, pP, cP, f);
      cell_add<false>(f, 2, o);
    }
  }
  if (iy + 1 < ny) cell_add<true>(fN[slot], 3, o);  // N: P = L
  if (ix == 0) land_side<T, S, JAC>(drho, rho0, K.Fl, K.Flo, K.PD, cP, o);
  if (FINE) {
    const double fm = (double)o.Rm, fs = (double)o.Rs;
    if (F) F[e] = make_double2(fm, fs);
    const double bm = block_max_nonneg(abs_max_or_inf(fm, fs), sh);
    if (threadIdx.x == 0) rmax_part[(int64_t)s * tiles + tile] = bm;
  }
  if constexpr (JAC) {
    if (J) store_blocks<T>(J, plane, e, o.C, o.Nb);
  }
}

// Coarse states: means of the 2x2 children, up to four levels in one launch.
// A CTA takes a tile of TW x TW/2 cells (TW = min(32, nx)) of one sample's
// grid and halves it level by level in shared memory; xc[k] are the sample-
// major arrays of the next levels.
struct RestrictLevels {
  int n;
  double2* xc[4];
};
constexpr int RESTRICT_THREADS = 128;
__global__ void __launch_bounds__(RESTRICT_THREADS) k_restrict_states(int B, int nx, int ny, const double2* xf,
                                                                      const __grid_constant__ RestrictLevels A,
                                                                      const int* active) {
  __shared__ double2 buf[2][RESTRICT_THREADS];
  grid_enter();
  int TW = min(32, nx), TH = TW >> 1;
  const int N = nx * ny, tiles = N / (TW * TH), tpr = nx / TW;
  const int s = blockIdx.x >> lg2(tiles), tile = blockIdx.x - s * tiles;
  if (s >= B || !active[s]) return;
  const int tx = tile & (tpr - 1), ty = tile >> lg2(tpr);
  const double2* x = xf + (int64_t)s * N;
  for (int k = 0; k < A.n; ++k) {
    // the tile's TW/2 x TH/2 coarse cells from its TW x TH cells
    const int cw = TW >> 1, ch = TH >> 1, t = threadIdx.x;
    if (t < cw * ch) {
      const int ly = t >> lg2(cw), lx = t - ly * cw;
      double2 a, b, c, d;
      if (k == 0) {
        const int ix = tx * TW + 2 * lx, iy = ty * TH + 2 * ly;
        a = x[st_of(ix, iy, nx)];
        b = x[st_of(ix + 1, iy, nx)];
        c = x[st_of(ix, iy + 1, nx)];
        d = x[st_of(ix + 1, iy + 1, nx)];
      } else {
        const double2* q = buf[(k + 1) & 1] + 2 * ly * TW + 2 * lx;
        a = q[0];
        b = q[1];
        c = q[TW];
        d = q[TW + 1];
      }
      const double2 m = make_double2(0.25 * (((a.x + b.x) + c.x) + d.x), 0.25 * (((a.y + b.y) + c.y) + d.y));
      buf[k & 1][t] = m;
      const int ncx = nx >> (k + 1);
      A.xc[k][(int64_t)s * (N >> (2 * (k + 1))) + st_of(tx * cw + lx, ty * ch + ly, ncx)] = m;
    }
    __syncthreads();
    TW = cw;
    TH = ch;
  }
}

// a5 (Galerkin option): A_c = R A P with piecewise-constant P, R = P^T.
template <typename T>
__global__ void __launch_bounds__(TPB) k_galerkin(int B, int ncx, int ncy, const typename VT<T>::b4* Jf,
                                                  int64_t plane_f, typename VT<T>::b4* __restrict__ Jc,
                                                  int64_t plane_c, const int* active) {
  typedef typename VT<T>::b4 B4;
  const int Nc = ncx * ncy;
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  grid_enter();
  if (e >= (int64_t)B * Nc) return;
  const int s = sample_of(e, Nc);
  if (!active[s]) return;
  const int stc = (int)(e - (int64_t)s * Nc);
  int IX, IY;
  xy_of(stc, ncx, IX, IY);
  const int nxf = 2 * ncx;
  const int64_t bf = (int64_t)s * Nc * 4;
  const int64_t ia = bf + st_of(2 * IX, 2 * IY, nxf), ib = bf + st_of(2 * IX + 1, 2 * IY, nxf);
  const int64_t ic = bf + st_of(2 * IX, 2 * IY + 1, nxf), id = bf + st_of(2 * IX + 1, 2 * IY + 1, nxf);
  auto ld = [&](int k, int64_t i) { return Jf[k * plane_f + i]; };
  auto add = [](B4& acc, const B4& v) { acc.a00 += v.a00; acc.a01 += v.a01; acc.a10 += v.a10; acc.a11 += v.a11; };
  B4 C = ld(0, ia);
  add(C, ld(0, ib)); add(C, ld(0, ic)); add(C, ld(0, id));
  add(C, ld(2, ia)); add(C, ld(1, ib)); add(C, ld(2, ic)); add(C, ld(1, id));
  add(C, ld(4, ia)); add(C, ld(3, ic)); add(C, ld(4, ib)); add(C, ld(3, id));
  B4 W = ld(1, ia); add(W, ld(1, ic));
  B4 E = ld(2, ib); add(E, ld(2, id));
  B4 S = ld(3, ia); add(S, ld(3, ib));
  B4 Nn = ld(4, ic); add(Nn, ld(4, id));
  Jc[e] = C;
  Jc[plane_c + e] = W;
  Jc[2 * plane_c + e] = E;
  Jc[3 * plane_c + e] = S;
  Jc[4 * plane_c + e] = Nn;
  const double a = C.a00, b = C.a01, c = C.a10, d = C.a11;
  const double idet = 1.0 / (a * d - b * c);
  Jc[5 * plane_c + e] = mkblk<B4>(d * idet, -b * idet, -c * idet, a * idet);
}

// Gauss-Jordan elimination with partial pivoting in FP64 on an n x n matrix,
// one column of [A | I] per lane (c = 0 .. 2n - 1 of a group of W lanes), rows in
// registers: every step is one division and n multiply-adds deep, where one
// thread per matrix runs all 2n columns one after another.  All lanes of the
// warp take part.
template <int N, int W>
__device__ __forceinline__ void gauss_jordan_lanes(double (&M)[N]) {
#pragma unroll
  for (int col = 0; col < N; ++col) {
    double v[N];  // column col
#pragma unroll
    for (int r = 0; r < N; ++r) v[r] = __shfl_sync(0xffffffffu, M[r], col, W);
    int piv = col;
    unsigned long long best = 0;
#pragma unroll
    for (int r = col; r < N; ++r) {  // largest magnitude, the first of equals
      const unsigned long long m = (unsigned long long)__double_as_longlong(v[r]) & 0x7fffffffffffffffull;
      if (r == col || m > best) {
        best = m;
        piv = r;
      }
    }
#pragma unroll
    for (int r = col + 1; r < N; ++r) {
      if (r != piv) continue;
      double t = M[r];
      M[r] = M[col];
      M[col] = t;
      t = v[r];
      v[r] = v[col];
      v[col] = t;
    }
    M[col] *= 1.0 / v[col];
#pragma unroll
    for (int r = 0; r < N; ++r)
      if (r != col) M[r] = fma(neg_(v[r]), M[col], M[r]);
  }
}

// Coarsest grid (2 x 1 cells, 4 unknowns; cells st 0 = (0,0) colour 0, st 1 =
// (1,0) colour 1): explicit inverse by eight lanes.  J: the sample's blocks, ps
// their plane stride; lane c = 4 + j ends with column j of the inverse.
template <typename B4>
__device__ __forceinline__ void coarse_inverse_lanes(const B4* J, int64_t ps, int c, double (&M)[4]) {
  // unknown c = 2 cell + var couples to the equations of cell 0 (rows 0, 1)
  // and cell 1 (rows 2, 3)
  const int cell = (c >> 1) & 1, var = c & 1;
  const B4 up = cell == 0 ? J[0] : J[2 * ps];       // C of cell 0, E of cell 0
  const B4 lo = cell == 0 ? J[ps + 1] : J[1];       // W of cell 1, C of cell 1
  const double a[4] = {(double)(var ? up.a01 : up.a00), (double)(var ? up.a11 : up.a10),
                       (double)(var ? lo.a01 : lo.a00), (double)(var ? lo.a11 : lo.a10)};
#pragma unroll
  for (int r = 0; r < 4; ++r) M[r] = c < 4 ? a[r] : (c - 4 == r ? 1.0 : 0.0);
  gauss_jordan_lanes<4, 8>(M);
}
template <typename T>
__global__ void k_coarse_inverse(int B, const typename VT<T>::b4* J, int64_t plane,
                                 T* __restrict__ Ainv, const int* active) {
  grid_enter();
  const int s = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 3), c = threadIdx.x & 7;
  const bool on = s < B && active[s];
  double M[4];
  coarse_inverse_lanes(J + 2 * (int64_t)(on ? s : 0), plane, c, M);
  if (on && c >= 4)
    for (int i = 0; i < 4; ++i) Ainv[(int64_t)s * 16 + i * 4 + c - 4] = (T)M[i];
}

template <typename T>
__global__ void k_coarse_solve(int B, const T* __restrict__ Ainv, const typename VT<T>::v2* b,
                               typename VT<T>::v2* __restrict__ x, const int* __restrict__ active) {
  typedef typename VT<T>::v2 V2;
  grid_enter();
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= B || !active[s]) return;
  const V2 b0 = b[2 * (int64_t)s], b1 = b[2 * (int64_t)s + 1];
  const T v[4] = {b0.x, b0.y, b1.x, b1.y};
  const T* M = Ainv + (int64_t)s * 16;
  T o[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) o[i] = coarse_row(M + 4 * i, v[0], v[1], v[2], v[3]);
  x[2 * (int64_t)s] = mk2<V2>(o[0], o[1]);
  x[2 * (int64_t)s + 1] = mk2<V2>(o[2], o[3]);
}

// ---- smoother source begin (the measured sweep-traffic record is keyed to the hash of this region)
// a7: one half-sweep of red-black point-block Gauss-Seidel over colour `col`:
//   x_P = C_P^{-1} (b_P - sum_nb A_nb x_nb).
// MODE 0: x = 0 before the sweep (first pre-smoothing sweep: x_P = C_P^{-1} b_P).
// MODE 1: plain sweep.
// MODE 2: first post-smoothing sweep right after the coarse-grid correction:
//         the neighbours' values are read as x_nb + x_c(parent(nb)), which is
//         x += P x_c followed by the sweep (the swept cells' own old values do
//         not enter point Gauss-Seidel, and the other colour is overwritten by
//         the next half-sweep).
// Cell form: J, b, x point at one sample's arrays (plane stride ps), xc at the
// sample's coarse vector; i = storage index of the swept cell (ix, iy).
template <typename T, int MODE>
__device__ __forceinline__ typename VT<T>::v2 sweep_cell(int nx, int ny, int ix, int iy, int i,
                                                         const typename VT<T>::b4* J, int64_t ps,
                                                         const typename VT<T>::v2* b, const typename VT<T>::v2* x,
                                                         const typename VT<T>::v2* xc) {
  typedef typename VT<T>::v2 V2;
  const V2 bb = b[i];
  T r0 = bb.x, r1 = bb.y;
  if (MODE != 0) {
    const int ncx = nx >> 1;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int jx = ix + (k == 0 ? -1 : (k == 1 ? 1 : 0));
      const int jy = iy + (k == 2 ? -1 : (k == 3 ? 1 : 0));
      if (jx < 0 || jx >= nx || jy < 0 || jy >= ny) continue;
      V2 xn = x[st_of(jx, jy, nx)];
      if (MODE == 2) {
        const V2 cc = xc[st_of(jx >> 1, jy >> 1, ncx)];
        xn.x += cc.x;
        xn.y += cc.y;
      }
      bmv_sub(J[(k + 1) * ps + i], xn.x, xn.y, r0, r1);
    }
  }
  T y0, y1;
  bmv(J[5 * ps + i], r0, r1, y0, y1);
  return mk2<V2>(y0, y1);
}

// NT: threads per CTA (any multiple of 32 up to 1024; every thread owns one
// cell).  Every sweep but the first of a level (MODE 0) follows another kernel
// of the cycle, so its blocks and right-hand side are complete when it starts.
// PRE = 1: they are loaded before the wait, which leaves only the neighbours' x
// on the critical path of a small launch but takes 76 registers instead of 32
// in FP64; the rule stands at with_preload (henry_engine.cu).  PRE = 2: the
// blocks alone, where b and the flags come from the kernel before (the black
// sweep after k_bicg_p or k_bicg_s has done the red one).
template <typename T, int MODE, int NT = TPB, int PRE = 0>
__global__ void __launch_bounds__(NT) k_sweep(int B, int nx, int ny, int col, const typename VT<T>::b4* __restrict__ J,
                                               int64_t plane, const typename VT<T>::v2* b,
                                               typename VT<T>::v2* x, const typename VT<T>::v2* xc,
                                               const int* active) {
  typedef typename VT<T>::v2 V2;
  typedef typename VT<T>::b4 B4;
  const int N = nx * ny, halfN = N >> 1, half = nx >> 1;
  const int64_t t = (int64_t)blockIdx.x * NT + threadIdx.x;
  const bool in = t < (int64_t)B * halfN;
  const int s = in ? sample_of(t, halfN) : 0;
  const int u = (int)(t - (int64_t)s * halfN);
  const int iy = u >> lg2(half), j = u - iy * half;
  const int ix = 2 * j + ((col ^ iy) & 1);
  const int64_t base = (int64_t)s * N;
  const int i = iy * nx + col * half + j;
  if constexpr (MODE == 0 || !PRE) {
    grid_enter();
    if (!in || !active[s]) return;
    x[base + i] = sweep_cell<T, MODE>(nx, ny, ix, iy, i, J + base, plane, b + base, x + base,
                                      MODE == 2 ? xc + (int64_t)s * (N >> 2) : nullptr);
  } else {
    bool on = in && (PRE == 2 || active[s]);
    const bool has[4] = {ix > 0, ix + 1 < nx, iy > 0, iy + 1 < ny};
    B4 A[4], Ci;
    V2 bb = mk2<V2>((T)0, (T)0);
    if (on) {
      const B4* Js = J + base + i;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (has[k]) A[k] = Js[(k + 1) * plane];
      Ci = Js[5 * plane];
      if (PRE == 1) bb = b[base + i];
    }
    grid_enter();
    if (PRE == 2) on = on && active[s];
    if (!on) return;
    if (PRE == 2) bb = b[base + i];
    // sweep_cell's arithmetic
    const V2* xs = x + base;
    const V2* xcs = MODE == 2 ? xc + (int64_t)s * (N >> 2) : nullptr;
    const int ncx = nx >> 1;
    V2 xn[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (!has[k]) continue;
      const int jx = ix + (k == 0 ? -1 : (k == 1 ? 1 : 0)), jy = iy + (k == 2 ? -1 : (k == 3 ? 1 : 0));
      xn[k] = xs[st_of(jx, jy, nx)];
      if (MODE == 2) {
        const V2 cc = xcs[st_of(jx >> 1, jy >> 1, ncx)];
        xn[k].x += cc.x;
        xn[k].y += cc.y;
      }
    }
    T r0 = bb.x, r1 = bb.y, y0, y1;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (has[k]) bmv_sub(A[k], xn[k].x, xn[k].y, r0, r1);
    bmv(Ci, r0, r1, y0, y1);
    x[base + i] = mk2<V2>(y0, y1);
  }
}
// ---- smoother source end

// Residual r_P = b_P - (A x)_P of one cell (sample-relative arrays).
template <typename T>
__device__ __forceinline__ void residual_cell(int nx, int ny, int ix, int iy, int i, const typename VT<T>::b4* J,
                                              int64_t ps, const typename VT<T>::v2* b,
                                              const typename VT<T>::v2* x, T& r0, T& r1) {
  typedef typename VT<T>::v2 V2;
  const V2 bb = b[i], xx = x[i];
  r0 = bb.x;
  r1 = bb.y;
  bmv_sub(J[i], xx.x, xx.y, r0, r1);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int jx = ix + (k == 0 ? -1 : (k == 1 ? 1 : 0));
    const int jy = iy + (k == 2 ? -1 : (k == 3 ? 1 : 0));
    if (jx < 0 || jx >= nx || jy < 0 || jy >= ny) continue;
    const V2 xn = x[st_of(jx, jy, nx)];
    bmv_sub(J[(k + 1) * ps + i], xn.x, xn.y, r0, r1);
  }
}

// Residual b - A x restricted by summation over the 2x2 children of coarse
// cell (IX, IY).  After a red-black sweep the black cells' residuals vanish
// (point Gauss-Seidel makes each swept equation hold), so MODE 0 sums the two
// colour-0 children only; MODE 1 (no pre-smoothing, x = 0) restricts b itself.
template <typename T, int MODE>
__device__ __forceinline__ typename VT<T>::v2 restrict_cell(int ncx, int ncy, int IX, int IY,
                                                            const typename VT<T>::b4* J, int64_t ps,
                                                            const typename VT<T>::v2* b,
                                                            const typename VT<T>::v2* x) {
  typedef typename VT<T>::v2 V2;
  const int nx = 2 * ncx, ny = 2 * ncy;
  T s0 = 0, s1 = 0;
  if (MODE == 1) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const V2 bb = b[st_of(2 * IX + (c & 1), 2 * IY + (c >> 1), nx)];
      s0 += bb.x;
      s1 += bb.y;
    }
  } else {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int ix = 2 * IX + c, iy = 2 * IY + c;  // (0,0) and (1,1): colour 0
      T r0, r1;
      residual_cell<T>(nx, ny, ix, iy, st_of(ix, iy, nx), J, ps, b, x, r0, r1);
      s0 += r0;
      s1 += r1;
    }
  }
  return mk2<V2>(s0, s1);
}

// PRE as in k_sweep (the residual form follows a sweep).
template <typename T, int MODE, int NT = TPB, bool PRE = false>  // MODE 0: RED_ONLY, 1: ZERO_X
__global__ void __launch_bounds__(NT) k_residual_restrict(int B, int ncx, int ncy,
                                                           const typename VT<T>::b4* __restrict__ J, int64_t plane,
                                                           const typename VT<T>::v2* b,
                                                           const typename VT<T>::v2* x,
                                                           typename VT<T>::v2* __restrict__ bc,
                                                           const int* active) {
  typedef typename VT<T>::v2 V2;
  typedef typename VT<T>::b4 B4;
  const int Nc = ncx * ncy;
  const int64_t e = (int64_t)blockIdx.x * NT + threadIdx.x;
  const bool in = e < (int64_t)B * Nc;
  const int s = in ? sample_of(e, Nc) : 0;
  const int stc = (int)(e - (int64_t)s * Nc);
  int IX, IY;
  xy_of(stc, ncx, IX, IY);
  const int64_t base = (int64_t)s * Nc * 4;
  if constexpr (MODE == 1 || !PRE) {
    grid_enter();
    if (!in || !active[s]) return;
    bc[e] = restrict_cell<T, MODE>(ncx, ncy, IX, IY, J + base, plane, b + base, x + base);
  } else {
    const bool on = in && active[s];
    const int nx = 2 * ncx, ny = 2 * ncy;
    B4 A[2][5];
    V2 bb[2];
    if (on) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int ix = 2 * IX + c, iy = 2 * IY + c, i = st_of(ix, iy, nx);
        const bool has[4] = {ix > 0, ix + 1 < nx, iy > 0, iy + 1 < ny};
        const B4* Js = J + base + i;
        A[c][0] = Js[0];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (has[k]) A[c][k + 1] = Js[(k + 1) * plane];
        bb[c] = b[base + i];
      }
    }
    grid_enter();
    if (!on) return;
    // restrict_cell's arithmetic
    const V2* xs = x + base;
    T s0 = 0, s1 = 0;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int ix = 2 * IX + c, iy = 2 * IY + c;
      const bool has[4] = {ix > 0, ix + 1 < nx, iy > 0, iy + 1 < ny};
      T r0 = bb[c].x, r1 = bb[c].y;
      const V2 xx = xs[st_of(ix, iy, nx)];
      bmv_sub(A[c][0], xx.x, xx.y, r0, r1);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (!has[k]) continue;
        const V2 xn = xs[st_of(ix + (k == 0 ? -1 : (k == 1 ? 1 : 0)), iy + (k == 2 ? -1 : (k == 3 ? 1 : 0)), nx)];
        bmv_sub(A[c][k + 1], xn.x, xn.y, r0, r1);
      }
      s0 += r0;
      s1 += r1;
    }
    bc[e] = mk2<V2>(s0, s1);
  }
}

// x += P x_c (used only when there is no post-smoothing to fuse it into).
template <typename T, int NT = TPB>
__global__ void __launch_bounds__(NT) k_prolong_add(int B, int nx, int ny, typename VT<T>::v2* x,
                                                    const typename VT<T>::v2* xc,
                                                    const int* active) {
  typedef typename VT<T>::v2 V2;
  const int N = nx * ny;
  const int64_t e = (int64_t)blockIdx.x * NT + threadIdx.x;
  grid_enter();
  if (e >= (int64_t)B * N) return;
  const int s = sample_of(e, N);
  if (!active[s]) return;
  int ix, iy;
  xy_of((int)(e - (int64_t)s * N), nx, ix, iy);
  const V2 c = xc[(int64_t)s * (N >> 2) + st_of(ix >> 1, iy >> 1, nx >> 1)];
  V2 v = x[e];
  v.x += c.x;
  v.y += c.y;
  x[e] = v;
}

template <typename T, int NT = TPB>
__global__ void __launch_bounds__(NT) k_zero(int64_t n, typename VT<T>::v2* __restrict__ x) {
  grid_enter();
  const int64_t e = (int64_t)blockIdx.x * NT + threadIdx.x;
  if (e < n) x[e] = mk2<typename VT<T>::v2>((T)0, (T)0);
}

// ---------------------------------------------------------------------------
// a8: y_P = (A x)_P of one cell (sample-relative arrays).
template <typename T>
__device__ __forceinline__ typename VT<T>::v2 spmv_cell(int nx, int ny, int ix, int iy, int i,
                                                        const typename VT<T>::b4* J, int64_t ps,
                                                        const typename VT<T>::v2* x) {
  typedef typename VT<T>::v2 V2;
  const V2 xx = x[i];
  T r0, r1;
  bmv(J[i], xx.x, xx.y, r0, r1);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int jx = ix + (k == 0 ? -1 : (k == 1 ? 1 : 0));
    const int jy = iy + (k == 2 ? -1 : (k == 3 ? 1 : 0));
    if (jx < 0 || jx >= nx || jy < 0 || jy >= ny) continue;
    const V2 xn = x[st_of(jx, jy, nx)];
    bmv_add(J[(k + 1) * ps + i], xn.x, xn.y, r0, r1);
  }
  return mk2<V2>(r0, r1);
}

// y = A x (fine level, all cells) with per-CTA partial dot products:
//   NDOT 1: <w1, y>;  NDOT 2: <w1, y>, <y, y>.
// b (nullable): x is the result of a V-cycle on this operator for the right-
// hand side b that ended with a black half-sweep.  Point Gauss-Seidel makes
// the swept equations hold, (A x)_P = b_P on every black cell, so those cells
// take b_P and only the red ones form the product: half the operations, and
// 104 instead of 208 bytes a cell.  A warp's cells then have one colour (on 32
// cells wide grids the CTA's eight rows are dealt out by colour).  8192 level-0
// samples, FP64: 145 -> 94 us a call, the solve 384 -> 369 ms (level 2 with
// partners, 33 samples: 192 -> 188; level 3 with partners, mixed, 20 samples:
// 316 -> 314); with the first red half-sweeps in the BiCGStab kernels as well
// 370, 187 and 312 ms.
// PRE as in k_sweep (the kernel follows the sweep that ends a V-cycle).
template <typename T, int NDOT, bool PRE = false>
__global__ void __launch_bounds__(TPB) k_spmv(int B, int nx, int ny, const typename VT<T>::b4* __restrict__ J,
                                              int64_t plane, const typename VT<T>::v2* x,
                                              typename VT<T>::v2* __restrict__ y,
                                              const typename VT<T>::v2* w1, double* __restrict__ part,
                                              int slot1, int slot2, const int* active,
                                              const typename VT<T>::v2* b) {
  typedef typename VT<T>::v2 V2;
  typedef typename VT<T>::b4 B4;
  __shared__ double sh[NDOT == 2 ? 2 * TPB : TPB + 1];
  const int N = nx * ny, nct = N / TPB;
  int lt = threadIdx.x;
  if (b && nx == 32) lt = ((lt & 0x70) << 1) | ((lt >> 7) << 4) | (lt & 15);  // (colour, row, j) -> (row, colour, j)
  const int64_t e = (int64_t)blockIdx.x * TPB + lt;
  const int s = sample_of(e, N);
  const bool on = active[s];  // uniform over the CTA
  const int st = (int)(e - (int64_t)s * N);
  int ix, iy;
  xy_of(st, nx, ix, iy);
  const int64_t base = e - st;
  const bool black = b && (st & (nx - 1)) >= (nx >> 1);
  V2 ww = mk2<V2>((T)0, (T)0), yy;
  if (black) {  // uniform over the warp
    if (on) {
      yy = b[e];
      if (NDOT >= 1 && part) ww = w1[e];
    }
    grid_enter();
    if (!on) return;
  } else if constexpr (PRE) {
    const bool has[4] = {ix > 0, ix + 1 < nx, iy > 0, iy + 1 < ny};
    B4 A[5];
    if (on) {
      A[0] = J[e];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (has[k]) A[k + 1] = J[(k + 1) * plane + e];
      if (NDOT >= 1 && part) ww = w1[e];
    }
    grid_enter();
    if (!on) return;
    // spmv_cell's arithmetic
    const V2* xs = x + base;
    const V2 xx = xs[st];
    T r0, r1;
    bmv(A[0], xx.x, xx.y, r0, r1);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (!has[k]) continue;
      const V2 xn = xs[st_of(ix + (k == 0 ? -1 : (k == 1 ? 1 : 0)), iy + (k == 2 ? -1 : (k == 3 ? 1 : 0)), nx)];
      bmv_add(A[k + 1], xn.x, xn.y, r0, r1);
    }
    yy = mk2<V2>(r0, r1);
  } else {
    grid_enter();
    if (!on) return;
    yy = spmv_cell<T>(nx, ny, ix, iy, st, J + base, plane, x + base);
    if (NDOT >= 1 && part) ww = w1[e];
  }
  y[e] = yy;
  if (NDOT >= 1 && part) {
    // per-cell products in T, widened once for the FP64 CTA reduction
    const double w1y = (double)fma_(ww.x, yy.x, ww.y * yy.y);
    const int64_t pi = (int64_t)s * nct + st / TPB, stride = (int64_t)B * nct;
    if (NDOT == 2) {
      const double d = block_sum_pair(w1y, (double)fma_(yy.x, yy.x, yy.y * yy.y), sh);
      if (threadIdx.x == 0) part[slot1 * stride + pi] = d;
      if (threadIdx.x == TPB / 2) part[slot2 * stride + pi] = d;
    } else {
      const double d = block_sum_tree(w1y, sh);
      if (threadIdx.x == 0) part[slot1 * stride + pi] = d;
    }
  }
}

// ---------------------------------------------------------------------------
// a6: right-preconditioned BiCGStab (Templates book), per sample, on the fine
// level; per-sample scalars live in LinScal, per-CTA partial sums in part.

// r = r_hat = b (= -F), p = v = dx = 0; partials <r_hat, r>, <r, r>.
template <typename T>
__global__ void __launch_bounds__(TPB) k_bicg_init(int B, int N, const double2* F,
                                                   typename VT<T>::v2* __restrict__ r,
                                                   typename VT<T>::v2* __restrict__ rh,
                                                   typename VT<T>::v2* __restrict__ p, typename VT<T>::v2* __restrict__ v,
                                                   typename VT<T>::v2* __restrict__ dx, double* __restrict__ part,
                                                   const int* active) {
  typedef typename VT<T>::v2 V2;
  __shared__ double sh[TPB + 1];
  const int nct = N / TPB;
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  const int s = blockIdx.x / (unsigned)nct;
  grid_enter();
  if (!active[s]) return;
  const double2 f = F[e];
  const V2 rr = mk2<V2>((T)(-f.x), (T)(-f.y));
  const V2 z = mk2<V2>((T)0, (T)0);
  r[e] = rr;
  rh[e] = rr;
  p[e] = z;
  v[e] = z;
  dx[e] = z;
  const double bs = block_sum_tree((double)fma_(rr.x, rr.x, rr.y * rr.y), sh);
  if (threadIdx.x == 0) {
    const int64_t pi = (int64_t)s * nct + (e - (int64_t)s * N) / TPB, stride = (int64_t)B * nct;
    part[P_RR * stride + pi] = bs;
    part[P_RN * stride + pi] = bs;
  }
}

// Start of iteration `it`: rho_it = <r_hat, r>, convergence test on ||r||,
// beta = (rho_it / rho_{it-1}) (alpha / omega), p = r + beta (p - omega v).
// A converged sample's CTA 0 clears lin_active; the last iteration counts
// still-active samples in *n_active and per-sample iterations in iters.
// FIRST: the V-cycle that follows starts with a red half-sweep from zero, x_P =
// C_P^-1 p_P; it is done here (Ci: the fine operator's plane of inverses, ph
// the cycle's vector, nx the grid's width), one launch and one pass over the
// red half of p less.
template <typename T>
__device__ __forceinline__ void first_sweep(const typename VT<T>::b4* Ci, typename VT<T>::v2* x, int nx, int64_t e,
                                            typename VT<T>::v2 b) {
  if (((int)e & (nx - 1)) >= (nx >> 1)) return;  // black
  T y0, y1;
  bmv(Ci[e], b.x, b.y, y0, y1);
  x[e] = mk2<typename VT<T>::v2>(y0, y1);
}
template <typename T, bool FIRST = false>
__global__ void __launch_bounds__(TPB) k_bicg_p(int B, int N, int it, int maxit, double rtol2,
                                                const typename VT<T>::v2* r, typename VT<T>::v2* p,
                                                const typename VT<T>::v2* v, const double* part, LinScal* sc,
                                                int* lin_active, int* __restrict__ iters,
                                                int* __restrict__ status, int* __restrict__ n_active,
                                                unsigned long long* __restrict__ lin_total, const double* fin,
                                                const typename VT<T>::b4* __restrict__ Ci, typename VT<T>::v2* ph,
                                                int nx) {
  typedef typename VT<T>::v2 V2;
  __shared__ double sh[2];
  const int nct = N / TPB;
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  const int s = blockIdx.x / (unsigned)nct;
  grid_enter();
  if (!lin_active[s]) return;
  const int ct = (int)((e - (int64_t)s * N) / TPB);
  const int64_t stride = (int64_t)B * nct;
  double rho, rn2;
  sample_sums(part, fin, P_RR, P_RN, stride, s, nct, sh, rho, rn2);
  // The test and the Krylov scalars once per CTA, by thread 0 (an FP64
  // division is a long FP64-pipe sequence, and every thread would compute
  // the same values); bc = (stop code, beta, omega).
  __shared__ double bc[3];
  if (threadIdx.x == 0) {
    const double bn2 = (it == 0) ? rn2 : sc[s].bnorm2;
    const bool finite = (rn2 <= 1.0e300) && (rho == rho);
    const bool conv = rn2 <= rtol2 * bn2;
    bc[0] = (!finite || conv || it >= maxit) ? (!finite ? -2.0 : (conv ? (double)it : -1.0)) : -3.0;
    if (bc[0] != -3.0) {
      // A sample that reaches maxit keeps its last iterate (inexact Newton
      // step; Newton's own test decides); a non-finite one fails.
      if (ct == 0) {
        lin_active[s] = 0;
        iters[s] = (int)bc[0];
        atomicAdd(lin_total, (unsigned long long)it);
      }
    } else {
      if (ct == 0) {
        atomicAdd(n_active, 1);
        if (it == 0) sc[s].bnorm2 = bn2;
      }
      if (it > 0) {
        const LinScal q = sc[s];
        bc[1] = (rho / q.rho) * q.aow;
        bc[2] = q.omega;
      }
    }
  }
  __syncthreads();
  if (bc[0] != -3.0) return;
  const V2 rr = r[e];
  V2 pn = rr;
  if (it > 0) {
    const V2 pp = p[e], vv = v[e];
    const T bt = (T)bc[1], om = (T)bc[2];
    pn = mk2<V2>(rr.x + bt * (pp.x - om * vv.x), rr.y + bt * (pp.y - om * vv.y));
  }
  p[e] = pn;
  if (FIRST) first_sweep<T>(Ci, ph, nx, e, pn);
}

// alpha = rho / <r_hat, v>; s = r - alpha v.  CTA 0 stores rho and alpha.
// FIRST as in k_bicg_p.
template <typename T, bool FIRST = false>
__global__ void __launch_bounds__(TPB) k_bicg_s(int B, int N, const typename VT<T>::v2* r, const typename VT<T>::v2* v,
                                                typename VT<T>::v2* __restrict__ sv, const double* part,
                                                LinScal* sc, const int* lin_active, const double* fin,
                                                const typename VT<T>::b4* __restrict__ Ci, typename VT<T>::v2* shv,
                                                int nx) {
  typedef typename VT<T>::v2 V2;
  __shared__ double sh[2];
  const int nct = N / TPB;
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  const int s = blockIdx.x / (unsigned)nct;
  grid_enter();
  if (!lin_active[s]) return;
  const int ct = (int)((e - (int64_t)s * N) / TPB);
  const int64_t stride = (int64_t)B * nct;
  double rho, rv;
  sample_sums(part, fin, P_RR, P_RV, stride, s, nct, sh, rho, rv);
  __shared__ double bc;
  if (threadIdx.x == 0) bc = rho / rv;  // once per CTA
  __syncthreads();
  const double alpha = bc;
  if (threadIdx.x == 0 && ct == 0) {
    sc[s].rho = rho;
    sc[s].alpha = alpha;
  }
  const V2 rr = r[e], vv = v[e];
  const T a = (T)alpha;
  const V2 sn = mk2<V2>(rr.x - a * vv.x, rr.y - a * vv.y);
  sv[e] = sn;
  if (FIRST) first_sweep<T>(Ci, shv, nx, e, sn);
}

// omega = <t, s> / <t, t>; dx += alpha p_hat + omega s_hat; r = s - omega t;
// partials <r_hat, r>, <r, r>.  CTA 0 stores omega.
// PRE: everything but t and the matvec's sums is loaded before the wait.
template <typename T, bool PRE = false>
__global__ void __launch_bounds__(TPB) k_bicg_update(int B, int N, typename VT<T>::v2* dx, const typename VT<T>::v2* ph,
                                                     const typename VT<T>::v2* shv, const typename VT<T>::v2* sv,
                                                     const typename VT<T>::v2* t, const typename VT<T>::v2* rh,
                                                     typename VT<T>::v2* __restrict__ r, double* part, LinScal* sc,
                                                     const int* lin_active, const double* fin) {
  typedef typename VT<T>::v2 V2;
  __shared__ double sh[2 * TPB];
  const int nct = N / TPB;
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  const int s = blockIdx.x / (unsigned)nct;
  const bool on = lin_active[s];
  V2 x0, p0, s0, sv0, rh0;
  auto load = [&] {
    x0 = dx[e];
    p0 = ph[e];
    s0 = shv[e];
    sv0 = sv[e];
    rh0 = rh[e];
  };
  if (PRE && on) load();
  grid_enter();
  if (!on) return;
  const int ct = (int)((e - (int64_t)s * N) / TPB);
  const int64_t stride = (int64_t)B * nct;
  double ts, tt;
  sample_sums(part, fin, P_TS, P_TT, stride, s, nct, sh, ts, tt);
  __shared__ double bc;
  if (threadIdx.x == 0) bc = (tt > 0.0) ? ts / tt : 0.0;  // once per CTA
  __syncthreads();
  const double omega = bc;
  const double alpha = sc[s].alpha;
  if (threadIdx.x == 0 && ct == 0) sc[s].omega = omega;
  const T a = (T)alpha, w = (T)omega;
  if (!PRE) load();
  const V2 t0 = t[e];
  dx[e] = mk2<V2>(x0.x + a * p0.x + w * s0.x, x0.y + a * p0.y + w * s0.y);
  const V2 rn = mk2<V2>(sv0.x - w * t0.x, sv0.y - w * t0.y);
  r[e] = rn;
  const double d = block_sum_pair((double)fma_(rh0.x, rn.x, rh0.y * rn.y), (double)fma_(rn.x, rn.x, rn.y * rn.y), sh);
  const int64_t pi = (int64_t)s * nct + ct;
  if (threadIdx.x == 0) part[P_RR * stride + pi] = d;
  if (threadIdx.x == TPB / 2) part[P_RN * stride + pi] = d;
  if (threadIdx.x == TPB - 1 && ct == 0) sc[s].aow = alpha / omega;
}

// Samples whose BiCGStab did not converge (or broke down) in this Newton
// iteration get a second linear solve with the fallback preconditioner.
__global__ void k_mark_retry(int B, const int* newton_active, const int* iters,
                             int* __restrict__ lin_active, int* n_retry) {
  grid_enter();
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= B) return;
  const int r = newton_active[s] && iters[s] < 0;
  lin_active[s] = r;
  if (r) atomicAdd(n_retry, 1);
}

// ---------------------------------------------------------------------------
// a9 / a10: Newton control.

// Per sample, after the fine assembly: converged if max |F| <= atol; a
// non-finite residual fails the sample; counts samples still iterating.
__global__ void k_newton_res_check(int B, int nct, double atol, int maxit, const double* rmax_part,
                                   int* newton_active, int* lin_active, int* newton_it, int* status,
                                   int* n_active, unsigned long long* it_total) {
  grid_enter();
  // one warp per sample
  const int s = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (s >= B) return;
  int act = newton_active[s];
  const double rm = act ? warp_sample_max(rmax_part + (int64_t)s * nct, nct, lane) : 0.0;
  if (lane != 0) return;
  if (act) {
    if (!(rm <= 1.0e300)) {
      status[s] = 3;
      act = 0;
    } else if (rm <= atol) {
      act = 0;
    } else if (newton_it[s] >= maxit) {
      status[s] = status[s] ? status[s] : 1;
      act = 0;
    } else {
      newton_it[s] += 1;
      atomicAdd(n_active, 1);
      atomicAdd(it_total, 1ULL);
    }
  }
  newton_active[s] = act;
  lin_active[s] = act;
}

// Per-CTA maxima of the Newton step: max(|dp| / p_ref, |dc|) (the update
// test) and max |dc| (the step limiter).
template <typename T>
__global__ void __launch_bounds__(TPB) k_newton_step_max(int B, int N, double inv_pref,
                                                         const typename VT<T>::v2* dx,
                                                         double* __restrict__ dmax_part, double* __restrict__ dc_part,
                                                         const int* newton_active) {
  __shared__ double sh[40];
  const int nct = N / TPB;
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  const int s = blockIdx.x / (unsigned)nct;
  grid_enter();
  if (!newton_active[s]) return;
  const auto d = dx[e];
  const double dc = abs_max_or_inf((double)d.y, 0.0);
  const double loc = abs_max_or_inf((double)d.x * inv_pref, dc);
  const double m = block_max_nonneg(loc, sh);
  const double mc = block_max_nonneg(dc, sh);
  if (threadIdx.x == 0) {
    const int64_t i = (int64_t)s * nct + (e - (int64_t)s * N) / TPB;
    dmax_part[i] = m;
    dc_part[i] = mc;
  }
}

// Per sample: theta = min(1, dc_limit / max |dc|) (a step that would change a
// mass fraction by more than dc_limit is shortened; dc_limit <= 0: theta = 1;
// -1 for a sample that does not iterate), and the update test on the full step:
// at most dxtol ends the sample's iteration with this update.  An infinite or
// NaN step has theta = 0 and is still applied, 0 * NaN: the failed sample's
// state and QoIs become NaN.
__global__ void k_newton_theta(int B, int nct, double dc_limit, const double* dc_part, double dxtol,
                               const double* dmax_part, int* newton_active, int* status,
                               double* __restrict__ theta) {
  grid_enter();
  // one warp per sample
  const int s = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (s >= B) return;
  if (!newton_active[s]) {
    if (lane == 0) theta[s] = -1.0;
    return;
  }
  double th = 1.0;
  if (dc_limit > 0.0) {
    const double mc = warp_sample_max(dc_part + (int64_t)s * nct, nct, lane);
    if (mc > dc_limit) th = dc_limit / mc;
  }
  const double dm = warp_sample_max(dmax_part + (int64_t)s * nct, nct, lane);
  if (lane != 0) return;
  theta[s] = th;
  if (!(dm <= 1.0e300)) {
    status[s] = 3;
    newton_active[s] = 0;
  } else if (dm <= dxtol) {
    newton_active[s] = 0;
  }
}

// a9: x += theta dx.
template <typename T>
__global__ void __launch_bounds__(TPB) k_newton_update(int B, int N, double2* x, const typename VT<T>::v2* dx,
                                                       const double* theta) {
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  const int s = blockIdx.x / (unsigned)(N / TPB);
  grid_enter();
  const double th = theta[s];
  if (__double_as_longlong(th) < 0) return;  // the sample does not iterate
  const auto d = dx[e];
  double2 xx = x[e];
  xx.x = fma(th, (double)d.x, xx.x);
  xx.y = fma(th, (double)d.y, xx.y);
  x[e] = xx;
}

// Start of a time step: old state = state; samples that have not failed iterate.
__global__ void __launch_bounds__(TPB) k_step_begin(int64_t n, const double2* x, double2* __restrict__ xo) {
  grid_enter();
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  if (e < n) xo[e] = x[e];
}
// Start of a later time step with a linear-in-time predictor for Newton's
// first iterate: x_old <- x^n, x <- x^n + w (x^n - x^{n-1}) (x^{n-1} is the
// old state of the previous step).  Only the starting point changes; Newton
// still stops on the residual and update tests of the step.
__global__ void __launch_bounds__(TPB) k_step_begin_predict(int64_t n, double w, double2* x, double2* xo) {
  grid_enter();
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  if (e >= n) return;
  const double2 a = x[e], b = xo[e];
  xo[e] = a;
  x[e] = make_double2(fma(w, a.x - b.x, a.x), fma(w, a.y - b.y, a.y));
}
// The quadratic predictor: x^{n+1} ~ x^n + w (2 (x^n - x^{n-1}) - (x^{n-1} -
// x^{n-2})), i.e. 3 x^n - 3 x^{n-1} + x^{n-2} for w = 1 (extrapolation of the
// parabola through the last three states); xoo <- x^{n-1}, xo <- x^n.
__global__ void __launch_bounds__(TPB) k_step_begin_predict2(int64_t n, double w, double2* x, double2* xo,
                                                             double2* xoo) {
  grid_enter();
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  if (e >= n) return;
  const double2 a = x[e], b = xo[e], c = xoo[e];
  xoo[e] = b;
  xo[e] = a;
  const double dx = 2.0 * (a.x - b.x) - (b.x - c.x), dy = 2.0 * (a.y - b.y) - (b.y - c.y);
  x[e] = make_double2(fma(w, dx, a.x), fma(w, dy, a.y));
}
// xoo <- x^{n-1} ahead of a step that still uses the linear predictor, so
// that the next step has three states.
__global__ void __launch_bounds__(TPB) k_copy_d2(int64_t n, const double2* src, double2* __restrict__ dst) {
  grid_enter();
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  if (e < n) dst[e] = src[e];
}
__global__ void k_step_flags(int B, const int* status, int* __restrict__ newton_active,
                             int* __restrict__ newton_it) {
  grid_enter();
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= B) return;
  newton_active[s] = status[s] == 0 ? 1 : 0;
  newton_it[s] = 0;
}

}  // namespace hk
