// Sampling, coefficients, initial state, QoIs, layout conversion and the
// MLMC accumulation kernels (sm_103a).
#pragma once
#include <cooperative_groups.h>

#include "henry_kernels.cuh"

namespace hk {

// ---------------------------------------------------------------------------
// a1: Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): 10 rounds of two
// 32x32->64-bit multiplications whose high halves are XORed with the other
// two counter words and the round key; the key advances by the Weyl
// increments between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
  const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u, W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) {
      k.x += W0;
      k.y += W1;
    }
    const uint32_t hi0 = __umulhi(M0, c.x), lo0 = M0 * c.x;
    const uint32_t hi1 = __umulhi(M1, c.z), lo1 = M1 * c.z;
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
  }
  return c;
}
// Two words -> (2u + 1 - 2^52) 2^-52 with u = (w0 << 20) | (w1 >> 12): an odd
// multiple of 2^-52 in (-1, 1), formed exactly in integers.
__device__ __forceinline__ double words_to_unit(uint32_t w0, uint32_t w1) {
  const int64_t u = ((int64_t)w0 << 20) | (int64_t)(w1 >> 12);
  const int64_t k = 2 * u + 1 - ((int64_t)1 << 52);
  return (double)k * 0x1p-52;
}
__global__ void k_sample_xi(uint64_t seed, int level, uint64_t first, int n, double* __restrict__ xi) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint64_t sidx = first + (uint64_t)i;
  const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
  const uint4 a = philox4x32_10(make_uint4((uint32_t)level, (uint32_t)sidx, (uint32_t)(sidx >> 32), 0u), key);
  const uint4 b = philox4x32_10(make_uint4((uint32_t)level, (uint32_t)sidx, (uint32_t)(sidx >> 32), 1u), key);
  xi[3 * (int64_t)i + 0] = words_to_unit(a.x, a.y);
  xi[3 * (int64_t)i + 1] = words_to_unit(a.z, a.w);
  xi[3 * (int64_t)i + 2] = words_to_unit(b.x, b.y);
}

// a2: phi = phi_mean (1 + phi_amp xi1), K = K_mean exp(logK_amp xi2),
// q_in = qin_mean (1 + qin_amp xi3); stored as (phi, K / mu, phi Dm, q_in).
struct CoefModel {
  double phi_mean, K_mean, qin_mean, phi_amp, logK_amp, qin_amp, mu, Dm;
};
// The assembly's scaled coefficients of each sample on one multigrid level
// (constant-coefficient model): cells of width h, vt_s = h^2 / tau inv_s.
__device__ __forceinline__ LevelCoef level_coef(const Phys& ph, const Coef& c, double h, double vt_s, double inv_s) {
  LevelCoef l;
  l.kh = 0.5 * (c.kmu * inv_s);
  l.kg = l.kh * (0.5 * ph.g * h);
  l.PD = c.PD * inv_s;
  l.PDh = 0.5 * l.PD;
  l.pv = c.phi * vt_s;
  l.pvd = l.pv * ph.drho;
  l.Fl = -ph.rho0 * c.qin * inv_s * h;
  l.Flo = l.Fl >= 0.0 ? l.Fl : 0.0;
  return l;
}
// The multigrid levels whose LevelCoef k_coefficients fills.
struct LevelList {
  static constexpr int MAX = 16;
  int n;
  Phys ph;
  double inv_s, h[MAX], vt_s[MAX];
  LevelCoef* lc[MAX];
};
__global__ void k_coefficients(CoefModel m, int n, const double* __restrict__ xi, Coef* __restrict__ coef,
                               int* __restrict__ status, const __grid_constant__ LevelList L = LevelList{}) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double x1 = xi[3 * (int64_t)i], x2 = xi[3 * (int64_t)i + 1], x3 = xi[3 * (int64_t)i + 2];
  Coef c;
  c.phi = m.phi_mean * (1.0 + m.phi_amp * x1);
  const double K = m.K_mean * exp(m.logK_amp * x2);
  c.kmu = K / m.mu;
  c.PD = c.phi * m.Dm;
  c.qin = m.qin_mean * (1.0 + m.qin_amp * x3);
  coef[i] = c;
  for (int k = 0; k < L.n; ++k) L.lc[k][i] = level_coef(L.ph, c, L.h[k], L.vt_s[k], L.inv_s);
  const bool ok = (c.phi > 0.0) && (c.phi < 1.0) && (K > 0.0) && (K <= 1.0e300) && (c.qin == c.qin) &&
                  (fabs(c.qin) <= 1.0e300);
  status[i] = ok ? 0 : 3;
}

// ---------------------------------------------------------------------------
// Random-field coefficient model (KL expansions of log K and phi, see
// henry_kl.cuh): per sample the inputs are theta_K[terms], theta_phi[terms]
// (iid N(0,1), drawn by the caller) and xi3 (uniform, for q_in).  cc[e] =
// (phi, K / mu) at the cell centre:
//   K = K_mean exp(sigma_K sum_t sqrt(lam_t) theta_K,t psi_t),
//   phi = clip(phi_mean + sigma_phi sum_t sqrt(lam_t) theta_phi,t psi_t, phi_lo, phi_hi),
// psi_t(x, y) = psi_x[ti_t](x) psi_y[tj_t](y) from the 1-D tables of this grid.
struct KLParams {
  int terms, n_in, m;
  double K_mean, sigma_logK, phi_mean, sigma_phi, phi_lo, phi_hi, mu;
};
__global__ void __launch_bounds__(TPB) k_fields_kl(KLParams P, int B, int nx, int ny, const double* __restrict__ inp,
                                                   const int* __restrict__ ti, const int* __restrict__ tj,
                                                   const double* __restrict__ sl, const double* __restrict__ psx,
                                                   const double* __restrict__ psy, double2* __restrict__ cc,
                                                   int* __restrict__ status) {
  const int N = nx * ny;
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  if (e >= (int64_t)B * N) return;
  const int s = (int)(e / N);
  int ix, iy;
  xy_of((int)(e - (int64_t)s * N), nx, ix, iy);
  const double* in = inp + (int64_t)s * P.n_in;
  double gK = 0.0, gp = 0.0;
  for (int t = 0; t < P.terms; ++t) {
    const double mode = psy[(int64_t)tj[t] * ny + iy] * psx[(int64_t)ti[t] * nx + ix];
    gK = fma(sl[t] * in[t], mode, gK);
    gp = fma(sl[t] * in[P.terms + t], mode, gp);
  }
  const double K = P.K_mean * exp(P.sigma_logK * gK);
  const double phi = fmin(fmax(P.phi_mean + P.sigma_phi * gp, P.phi_lo), P.phi_hi);
  cc[e] = make_double2(phi, K / P.mu);
  if (!(K > 0.0 && K <= 1.0e300 && phi == phi)) atomicExch(status + s, 3);
}

// Two-layer porosity of the paper's experiments (Eq. poro_2levels) with the
// Kozeny-Carman permeability (Eq. e_perm_Kozeny_Carman) K = kappa phi^3 /
// (1 - phi^2), kappa fixed by K(E[phi]) = K_mean; the paper's y in [-1, 0]
// is y - Ly here, the layer interface at -0.75 is y = Ly - 0.75.
struct TwoLayerParams {
  int n_in;
  double phi_mean, kappa, mu, Ly, y_if;
};
__global__ void __launch_bounds__(TPB) k_fields_two_layer(TwoLayerParams P, int B, int nx, int ny, double h,
                                                          const double* __restrict__ inp, double2* __restrict__ cc,
                                                          int* __restrict__ status) {
  const int N = nx * ny;
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  if (e >= (int64_t)B * N) return;
  const int s = (int)(e / N);
  int ix, iy;
  xy_of((int)(e - (int64_t)s * N), nx, ix, iy);
  const double* in = inp + (int64_t)s * P.n_in;
  const double xi1 = in[0], xi2 = in[1];
  const double x = (ix + 0.5) * h, yp = (iy + 0.5) * h - P.Ly;  // paper coordinates
  const double pi = 3.14159265358979323846;
  const double c0 = (yp < P.y_if) ? 1.0 + 0.2 * xi1 : 1.0 - 0.2 * xi1;
  const double phi = P.phi_mean * (1.0 + 0.15 * (xi2 * cos(pi * x / 2.0) + xi2 * sin(2.0 * pi * yp) + xi1 * cos(2.0 * pi * x))) * c0;
  const double K = P.kappa * phi * phi * phi / (1.0 - phi * phi);
  cc[e] = make_double2(phi, K / P.mu);
  if (!(phi > 0.0 && phi < 1.0 && K > 0.0 && K <= 1.0e300)) atomicExch(status + s, 3);
}

// Coarse multigrid cells: mean of the children's (phi, K / mu).
__global__ void __launch_bounds__(TPB) k_restrict_cc(int B, int ncx, int ncy, const double2* __restrict__ ccf,
                                                     double2* __restrict__ ccc) {
  const int Nc = ncx * ncy;
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  if (e >= (int64_t)B * Nc) return;
  const int s = (int)(e / Nc);
  int IX, IY;
  xy_of((int)(e - (int64_t)s * Nc), ncx, IX, IY);
  const int nxf = 2 * ncx;
  const int64_t bf = (int64_t)s * Nc * 4;
  const double2 a = ccf[bf + st_of(2 * IX, 2 * IY, nxf)], b = ccf[bf + st_of(2 * IX + 1, 2 * IY, nxf)];
  const double2 c = ccf[bf + st_of(2 * IX, 2 * IY + 1, nxf)], d = ccf[bf + st_of(2 * IX + 1, 2 * IY + 1, nxf)];
  ccc[e] = make_double2(0.25 * (((a.x + b.x) + c.x) + d.x), 0.25 * (((a.y + b.y) + c.y) + d.y));
}

// Face coefficients: harmonic means 2 a b / (a + b) of K / mu (halved) and of
// phi Dm, scaled by inv_s, on the east (.x, .y) and north (.z, .w) face of
// every cell, 0 on the boundary.
__global__ void __launch_bounds__(TPB) k_face_coefs(int B, int nx, int ny, double Dm, double inv_s,
                                                    const double2* __restrict__ cc,
                                                    double4_32a* __restrict__ fc) {
  const int N = nx * ny;
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  if (e >= (int64_t)B * N) return;
  const int s = (int)(e / N);
  const int st = (int)(e - (int64_t)s * N);
  int ix, iy;
  xy_of(st, nx, ix, iy);
  const double2* c = cc + (int64_t)s * N;
  const double2 P = c[st];
  double4_32a f;
  f.x = f.y = f.z = f.w = 0.0;
  auto harm = [](double a, double b) { return 2.0 * a * b / (a + b); };
  if (ix + 1 < nx) {
    const double2 E = c[st_of(ix + 1, iy, nx)];
    f.x = 0.5 * harm(P.y, E.y) * inv_s;
    f.y = harm(P.x * Dm, E.x * Dm) * inv_s;
  }
  if (iy + 1 < ny) {
    const double2 Nn = c[st_of(ix, iy + 1, nx)];
    f.z = 0.5 * harm(P.y, Nn.y) * inv_s;
    f.w = harm(P.x * Dm, Nn.x * Dm) * inv_s;
  }
  fc[e] = f;
}

// a2 for the field models: q_in from its uniform input (index iq).
__global__ void k_coefficients_qin(int n, int n_in, int iq, double qin_mean, double qin_amp,
                                   const double* __restrict__ inp, Coef* __restrict__ coef, int* __restrict__ status) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  Coef c;
  c.phi = 0.0;
  c.kmu = 0.0;
  c.PD = 0.0;
  c.qin = qin_mean * (1.0 + qin_amp * inp[(int64_t)i * n_in + iq]);
  coef[i] = c;
  status[i] = (c.qin == c.qin && fabs(c.qin) <= 1.0e300) ? 0 : 3;
}

// a3: c = 0 and fresh-water hydrostatic pressure rho0 g (Ly - y).
__global__ void __launch_bounds__(TPB) k_init_state(int B, int nx, int ny, double h, double rho0g, double Ly,
                                                    double2* __restrict__ x) {
  const int N = nx * ny;
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  if (e >= (int64_t)B * N) return;
  const int st = (int)(e % N);
  const int iy = st / nx;
  x[e] = make_double2(rho0g * (Ly - (iy + 0.5) * h), 0.0);
}

// a11: QoIs, one CTA per sample, qoi[s][nq]: salt mass sum phi rho c h^2 and c at
// (1.5, 0.25) = mean of the cells (ix0, iy0), (ix0+1, iy0), (ix0, iy0+1),
// (ix0+1, iy0+1) with ix0 = 1.5 / h - 1, iy0 = 0.25 / h - 1.
// With per-cell coefficients (cc != NULL) the porosity weights each cell.
// QS >= 1 (the paper's QoIs, Sec. 2.2 and 4) adds [2] the freshwater integral
// Q_FW of Eq. (integral_fw), the area of the cells with c <= 0.012178, and
// [3..14] c at the 12 points of Eq. (12points) (paper y in [-1, 0], here y +
// Ly) by bilinear interpolation of the four surrounding cell centres (the
// stencil clamped to the grid); QS = 2
// adds [15..] the c field averaged over the cells of the nx0 x ny0 level-0
// grid, row-major.
struct QoiSpec {
  int set, nq, nx0, ny0;
  double Lx, Ly;
};
__device__ __forceinline__ double cell_c(const double2* xs, int ix, int iy, int nx) { return xs[st_of(ix, iy, nx)].y; }
__global__ void __launch_bounds__(TPB) k_qoi(int B, int nx, int ny, double h, double rho0, double drho,
                                             const Coef* __restrict__ coef, const double2* __restrict__ x,
                                             double* __restrict__ qoi, const double2* __restrict__ cc = nullptr,
                                             QoiSpec Q = QoiSpec{0, 2, 0, 0, 2.0, 1.0}) {
  __shared__ double sh[40];
  const int s = blockIdx.x;
  const int N = nx * ny;
  const double2* xs = x + (int64_t)s * N;
  double* out = qoi + (int64_t)s * Q.nq;
  double acc = 0.0, fresh = 0.0;
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    const double c = xs[i].y;
    const double w = cc ? cc[(int64_t)s * N + i].x : 1.0;
    acc += w * (rho0 + drho * c) * c;
    fresh += (c <= 0.012178) ? 1.0 : 0.0;
  }
  acc = block_reduce(acc, sh);
  if (Q.set >= 1) fresh = block_reduce(fresh, sh);
  if (threadIdx.x == 0) {
    const int ix0 = (3 * ny) / 2 - 1, iy0 = ny / 4 - 1;
    const double c00 = xs[st_of(ix0, iy0, nx)].y, c10 = xs[st_of(ix0 + 1, iy0, nx)].y;
    const double c01 = xs[st_of(ix0, iy0 + 1, nx)].y, c11 = xs[st_of(ix0 + 1, iy0 + 1, nx)].y;
    out[0] = (cc ? 1.0 : coef[s].phi) * acc * h * h;
    out[1] = 0.25 * (((c00 + c10) + c01) + c11);
    if (Q.set >= 1) out[2] = fresh * h * h;
  }
  if (Q.set < 1) return;
  if (threadIdx.x < 12) {
    const double px = 1.10 + 0.25 * (threadIdx.x & 3);
    const int row = threadIdx.x >> 2;
    const double py = (row == 0 ? -0.95 : (row == 1 ? -0.75 : -0.50)) + Q.Ly;
    const double tx = px * nx / Q.Lx - 0.5, ty = py * ny / Q.Ly - 0.5;
    // the 2 x 2 stencil is kept on the grid (linear extrapolation for a point
    // outside the hull of the cell centres, which only coarse user grids have)
    const int ix = min(max((int)floor(tx), 0), nx - 2), iy = min(max((int)floor(ty), 0), ny - 2);
    const double fx = tx - ix, fy = ty - iy;
    out[3 + threadIdx.x] = (1 - fy) * ((1 - fx) * cell_c(xs, ix, iy, nx) + fx * cell_c(xs, ix + 1, iy, nx)) +
                           fy * ((1 - fx) * cell_c(xs, ix, iy + 1, nx) + fx * cell_c(xs, ix + 1, iy + 1, nx));
  }
  if (Q.set != 2) return;
  const int f = nx / Q.nx0;
  for (int c0 = threadIdx.x; c0 < Q.nx0 * Q.ny0; c0 += blockDim.x) {
    const int IY = c0 / Q.nx0, IX = c0 - IY * Q.nx0;
    double a = 0.0;
    for (int jy = 0; jy < f; ++jy)
      for (int jx = 0; jx < f; ++jx) a += cell_c(xs, IX * f + jx, IY * f + jy, nx);
    out[15 + c0] = a / (double)(f * f);
  }
}

// The freshwater integral of Eq. (integral_fw) of the current state, one CTA
// per sample, into out[s * stride] (the Q_FW(t) series of QoI set 3).
__global__ void __launch_bounds__(TPB) k_qfw(int B, int N, double h, const double2* __restrict__ x,
                                             double* __restrict__ out, int stride, const int* __restrict__ status) {
  __shared__ double sh[40];
  const int s = blockIdx.x;
  const double2* xs = x + (int64_t)s * N;
  double fresh = 0.0;
  for (int i = threadIdx.x; i < N; i += blockDim.x) fresh += (xs[i].y <= 0.012178) ? 1.0 : 0.0;
  fresh = block_reduce(fresh, sh);
  if (threadIdx.x == 0) out[(int64_t)s * stride] = status[s] == 0 ? fresh * h * h : 0.0;
}

// Natural layout [B][ny][nx] <-> storage layout (colour-split rows).
__device__ __forceinline__ int64_t storage_of(int64_t e, int nx, int N) {  // of the natural entry e
  const int64_t s = sample_of(e, N);
  const int nat = (int)(e - s * N), iy = nat >> lg2(nx);
  return s * N + st_of(nat - iy * nx, iy, nx);
}
template <typename V2>
__global__ void __launch_bounds__(TPB) k_to_storage(int B, int nx, int ny, const double2* in,
                                                    V2* __restrict__ out) {
  grid_enter();
  const int N = nx * ny;
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  if (e >= (int64_t)B * N) return;
  const double2 v = in[e];
  V2 o;
  o.x = v.x;
  o.y = v.y;
  out[storage_of(e, nx, N)] = o;
}
// Both states of a per-step call, and its samples' flags from their status.
__global__ void __launch_bounds__(TPB) k_states_in(int B, int nx, int ny, const double2* __restrict__ in,
                                                   const double2* __restrict__ in_old, double2* __restrict__ x,
                                                   double2* __restrict__ xo, const int* status,
                                                   int* __restrict__ newton_active, int* __restrict__ lin_active,
                                                   int* __restrict__ newton_it) {
  grid_enter();
  const int N = nx * ny;
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  if (e >= (int64_t)B * N) return;
  const int64_t i = storage_of(e, nx, N);
  x[i] = in[e];
  xo[i] = in_old[e];
  if (e < B) {
    newton_active[e] = lin_active[e] = status[e] == 0 ? 1 : 0;
    newton_it[e] = 0;
  }
}
template <typename V2>
__global__ void __launch_bounds__(TPB) k_from_storage(int B, int nx, int ny, const V2* in,
                                                      double2* __restrict__ out) {
  grid_enter();
  const int N = nx * ny;
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  if (e >= (int64_t)B * N) return;
  const V2 v = in[storage_of(e, nx, N)];
  out[e] = make_double2((double)v.x, (double)v.y);
}
// Jacobian planes -> natural [B][ny][nx][5][2][2] FP64.  One thread per block
// row (two values): a warp writes 512 contiguous bytes and reads whole 32-byte
// blocks; with one thread per cell (20 stores 160 bytes apart) and
// a launch per conversion henry_assemble of 8 samples of 512 x 256 cells took 434 us,
// now 314 us (160 us of it the assembly).
template <typename V2>
__global__ void __launch_bounds__(TPB) k_blocks_out(int B, int nx, int ny, const V2* J, int64_t plane,
                                                    double2* __restrict__ out) {
  grid_enter();
  const int N = nx * ny;
  const int64_t t = (int64_t)blockIdx.x * TPB + threadIdx.x;
  if (t >= (int64_t)B * N * 10) return;
  const int64_t e = t / 10;
  const int q = (int)(t - e * 10);
  const V2 v = J[2 * ((q >> 1) * plane + storage_of(e, nx, N)) + (q & 1)];
  out[t] = make_double2((double)v.x, (double)v.y);
}

// Row permutation of a [n][w] array (uneven mixed-level batches): gather
// dst[i] = src[perm[i]] or scatter dst[perm[i]] = src[i].
template <typename E, bool SCATTER>
__global__ void k_permute_rows(int n, int w, const int* __restrict__ perm, const E* __restrict__ src,
                               E* __restrict__ dst) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)n * w) return;
  const int i = (int)(t / w), k = (int)(t % w);
  const int64_t j = perm[i];
  if (SCATTER) dst[j * w + k] = src[t];
  else dst[t] = src[j * w + k];
}

__global__ void __launch_bounds__(TPB) k_scale_d2(int64_t n, double a, double2* x) {
  grid_enter();
  const int64_t e = (int64_t)blockIdx.x * TPB + threadIdx.x;
  if (e < n) {
    double2 v = x[e];
    x[e] = make_double2(a * v.x, a * v.y);
  }
}

// ---------------------------------------------------------------------------
// a12: MLMC accumulation.  Per QoI and quantity (Y and the fine QoI): the
// batch's count, mean and centred sum of squares M2, merged by Chan's pairwise
// update into the running (count, mean, M2).
//
// The rows are read once, coalesced over CW neighbouring QoIs, by a cluster
// of CTAs per group of CW columns: each CTA sums (y - k) and (y - k)^2 over
// its rows about a pivot k, and the cluster's first CTA merges the CTAs'
// moments through distributed shared memory - no workspace.  The pivot is the
// mean of the used ones among the first 8 rows of the CTA's first step that
// has any there (0 if none has).  M2 = s2 - s1^2 / n keeps its digits while k
// lies within a standard deviation or so of the mean; where it does not
// (those rows failed, or lie far from the rest) a column's M2 comes out below
// s2 / 4 and the CTA goes over its rows once more about the mean it then knows.
// On normally distributed values that takes a mean of 8 more than 4.9 of its
// own deviations off, one CTA and column in a million.  Bound by the FP64 pipe: 7 operations per row and QoI (the
// difference Y, and a subtraction, an addition and a multiply-add for each
// quantity), which at 17-19 cycles a warp instruction and SM is 145 us for
// 20000 rows of 527 QoIs with their partners.  Measured there 187 us, against
// 314 us for one CTA of 1024 threads per QoI and quantity with two strided
// passes; 20000 x 15: 54 -> 27 us, 81675 x 2: 160 -> 44 us, 500 x 527: 68 -> 27
// us, 50 x 2: 15 -> 17 us (event timer around the call, L2 flushed before it).
// A CTA takes columns in groups of CW (1 .. 16); few QoIs take narrow groups
// so that the rows still spread over many CTAs.
constexpr int ACC_THREADS = 256, ACC_MAX_CLUSTER = 8;

constexpr int ACC_WARPS = ACC_THREADS / 32, ACC_R = 8;  // ACC_R: rows a lane holds at a time
template <int CW>
struct AccShared {
  double part[4][ACC_WARPS][CW];
  int cpart[ACC_WARPS][CW];
  double mom[2][CW][4];  // of Y and the fine QoI: count, pivot, mean less the pivot, M2
};
// A CTA's share of the batch: its steps of ACC_THREADS / CW rows of CW columns.
struct AccRows {
  int n, n_qoi, rank, ncta, qq;
  const double *qf, *qc;
  const int32_t* status;
  // ACC_R rows from r0 on, `inc` apart: every load is issued before the first use,
  // the status decides afterwards (a failed sample's NaN is dropped by it)
  __device__ __forceinline__ void load(int64_t r0, int64_t inc, double* f, double* c, bool* ok) const {
#pragma unroll
    for (int j = 0; j < ACC_R; ++j) {
      const int64_t i = r0 + j * inc;
      ok[j] = i < n;
      const int64_t at = (ok[j] ? i : 0) * n_qoi + qq;
      f[j] = qf[at];
      c[j] = qc ? qc[at] : 0.0;
      if (status) ok[j] = ok[j] && status[ok[j] ? i : 0] == 0;
    }
  }
};
// The CTA's moments about the pivots ky and kf into S.mom; true in a thread
// whose column's pivot lies too far from its mean (infinite values have no
// better one).
template <int CW>
__device__ __forceinline__ bool acc_moments(const AccRows& A, double ky, double kf, AccShared<CW>& S) {
  constexpr int NW = ACC_WARPS, RPW = 32 / CW, R = ACC_R;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, col = lane % CW;
  const int64_t step = (int64_t)A.ncta * NW * RPW;
  int cnt = 0;
  double s1y = 0.0, s2y = 0.0, s1f = 0.0, s2f = 0.0;
  for (int64_t r0 = (A.rank * NW + w) * RPW; r0 < A.n; r0 += R * step) {
    double f[R], c[R];
    bool ok[R];
    A.load(r0 + lane / CW, step, f, c, ok);
#pragma unroll
    for (int j = 0; j < R; ++j) {
      if (r0 + j * step >= A.n) break;  // uniform over the warp
      const double df = ok[j] ? f[j] - kf : 0.0, dy = ok[j] ? (f[j] - c[j]) - ky : 0.0;
      cnt += ok[j];
      s1f += df;
      s2f = fma(df, df, s2f);
      s1y += dy;
      s2y = fma(dy, dy, s2y);
    }
  }
#pragma unroll
  for (int o = 16; o >= CW; o >>= 1) {
    cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    s1y += __shfl_xor_sync(0xffffffffu, s1y, o);
    s2y += __shfl_xor_sync(0xffffffffu, s2y, o);
    s1f += __shfl_xor_sync(0xffffffffu, s1f, o);
    s2f += __shfl_xor_sync(0xffffffffu, s2f, o);
  }
  if (lane < CW) {
    S.cpart[w][col] = cnt;
    S.part[0][w][col] = s1y;
    S.part[1][w][col] = s2y;
    S.part[2][w][col] = s1f;
    S.part[3][w][col] = s2f;
  }
  __syncthreads();
  if (w >= 2 || lane >= CW) return false;
  int m = 0;  // warps 0 and 1: Y and the fine QoI
  double s1 = 0.0, s2 = 0.0;
  for (int k = 0; k < NW; ++k) {
    m += S.cpart[k][col];
    s1 += S.part[2 * w][k][col];
    s2 += S.part[2 * w + 1][k][col];
  }
  const double nn = (double)m;
  const double d = m > 0 ? s1 / nn : 0.0;
  const double m2 = s2 - s1 * d;
  S.mom[w][col][0] = nn;
  S.mom[w][col][1] = w == 0 ? ky : kf;
  S.mom[w][col][2] = d;
  S.mom[w][col][3] = m2 < 0.0 ? 0.0 : m2;
  return !(m2 >= 0.25 * s2) && fabs(d) <= 1.0e300;
}
// The second pass, out of line: as a second turn of one loop it slowed the first
// pass down (81675 x 2: 56 us, 44 in this form and without any second pass).
template <int CW>
__device__ __noinline__ void acc_moments_again(const AccRows& A, double ky, double kf, AccShared<CW>& S) {
  acc_moments<CW>(A, ky, kf, S);
}

template <int CW>
__global__ void __launch_bounds__(ACC_THREADS, 4) k_mlmc_accumulate(int n, int n_qoi, const double* __restrict__ qf,
                                                                 const double* __restrict__ qc,
                                                                 const int32_t* __restrict__ status,
                                                                 double* __restrict__ sums) {
  namespace cg = cooperative_groups;
  constexpr int per_cta = ACC_THREADS / CW;
  __shared__ AccShared<CW> S;
  const int lane = threadIdx.x & 31, which = threadIdx.x >> 5;  // warps 0 and 1 merge: Y and the fine QoI
  const int col = lane % CW, q = blockIdx.x * CW + col;
  const int rank = blockIdx.y, ncta = gridDim.y;
  const bool on = q < n_qoi;
  // lanes beyond the last QoI read along
  const AccRows A = {n, n_qoi, rank, ncta, on ? q : n_qoi - 1, qf, qc, status};
  // pivot: the mean of the CTA's first used rows
  double ky = 0.0, kf = 0.0;
  {
    double f[ACC_R], c[ACC_R];
    bool ok[ACC_R];
    int m = 0;
    for (int64_t b = rank * per_cta; b < n && m == 0; b += (int64_t)ncta * per_cta) {
      A.load(b, 1, f, c, ok);
#pragma unroll
      for (int j = 0; j < ACC_R; ++j)
        if (ok[j] && j < per_cta) {
          kf += f[j];
          ky += f[j] - c[j];
          ++m;
        }
    }
    kf = (m > 0 && fabs(kf) <= 1.0e300) ? kf / (double)m : 0.0;  // infinite or NaN values: pivot 0
    ky = (m > 0 && fabs(ky) <= 1.0e300) ? ky / (double)m : 0.0;
  }
  if (__syncthreads_or(acc_moments<CW>(A, ky, kf, S))) {
    const double dy = S.mom[0][col][2], df = S.mom[1][col][2];
    acc_moments_again<CW>(A, fabs(dy) <= 1.0e300 ? ky + dy : ky, fabs(df) <= 1.0e300 ? kf + df : kf, S);
  }
  cg::cluster_group cl = cg::this_cluster();
  cl.sync();
  if (rank == 0 && which < 2 && lane < CW && on) {
    // the batch's moments from the CTAs', then Chan's merge into the sums.
    // The CTAs' means enter as distances from one CTA's pivot, (k - k0) + d:
    // rounded to k + d they would put an error of eps |mean| sd into M2.
    double cb = 0.0, sb = 0.0, k0 = 0.0;
    for (int k = 0; k < ncta; ++k) {
      const double* b = cl.map_shared_rank(&S.mom[which][col][0], k);
      if (b[0] == 0.0) continue;
      if (cb == 0.0) k0 = b[1];
      cb += b[0];
      sb = fma(b[0], (b[1] - k0) + b[2], sb);
    }
    if (cb > 0.0) {
      const double off = sb / cb, mb = k0 + off;
      double m2 = 0.0;
      for (int k = 0; k < ncta; ++k) {
        const double* b = cl.map_shared_rank(&S.mom[which][col][0], k);
        if (b[0] == 0.0) continue;
        const double d = ((b[1] - k0) + b[2]) - off;
        m2 += fma(b[0] * d, d, b[3]);
      }
      double* out = sums + ((int64_t)which * n_qoi + q) * 3;
      const double na = out[0], ma = out[1], m2a = out[2];
      const double nn = na + cb;
      const double d = mb - ma;
      out[0] = nn;
      out[1] = ma + d * (cb / nn);
      out[2] = m2a + m2 + d * d * (na * cb / nn);
    }
  }
  cl.sync();  // the other CTAs' shared memory stays until it has been read
}

}  // namespace hk
