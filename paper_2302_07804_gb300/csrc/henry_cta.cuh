// Fused per-sample solver for the 32 x 16 grid (sm_103a), MLMC level 0 of the
// default configuration.
//
// One CTA runs the complete scenario - every implicit-Euler step, Newton
// iteration, BiCGStab iteration and V-cycle - in a single launch; only the old
// states (read and written once per step and by the assembly) and the QoIs
// touch global memory.  256 threads: thread t has child c = t & 1 of coarse cell
// Q = t / 2, one cell of either colour, and keeps for both cells the Jacobian
// blocks and every Krylov vector in registers.  Shared memory holds what
// neighbours read: the Newton iterate, one vector with a halo of zeros (the
// V-cycle's result, which the matvec reads), and the coarse levels, which
// run as the multigrid tail's phases (TailLevel, henry_tail.cuh: two threads per
// cell, block rows in shared memory).  A matvec forms the product on the red
// cells only: the V-cycle ends with a black half-sweep, which leaves A x = b on
// the black ones (nu2 > 0; otherwise both).
// Bound by latency (dependent phases between barriers) and, in the assembly,
// by the FP64 pipe.  With FP32 linear algebra, 1000 samples of 20 steps: 27.3
// ms with all blocks and vectors in 111 KB of shared memory and one thread per
// cell on the coarse levels, 17.0 ms in this form (41 KB; two CTAs per SM by
// registers either way).
// The per-cell arithmetic is the multi-kernel path's and the steps follow the
// same order, so both paths compute the same iterates up to the summation
// order of the dot products and maxima.
#pragma once
#include "henry_kernels.cuh"
#include "henry_misc.cuh"
#include "henry_tail.cuh"

namespace hk {

constexpr int CTA_THREADS = 256;
constexpr int CTA_NX = 32, CTA_NY = 16, CTA_N = CTA_NX * CTA_NY;
constexpr int CTA_LEVELS = 5;                           // 32 x 16 .. 2 x 1
constexpr int CTA_COARSE = CTA_N / 4 + CTA_N / 16 + CTA_N / 64 + CTA_N / 256;  // cells of the coarse levels

struct CtaParams {
  Phys ph;
  int steps, nu1, nu2, newton_maxit, lin_maxit;
  double h0, tau, inv_s, inv_pref, atol, dxtol, rtol2, predictor, dc_limit;
  int predictor_order;  // 1: linear, 2: quadratic from step 2 on (xoo_g holds x^{n-2})
  double rho0g, Ly;
};

// Shared memory (bytes): the iterate, restricted states and old states of the
// coarse levels, reductions, then (V2) x with halo, the tail's levels.
template <typename T>
struct CtaShared {
  typedef typename VT<T>::v2 V2;
  double2 x[CTA_N], xc[CTA_COARSE], xoc[CTA_COARSE];
  double red[2 * CTA_THREADS], bc[4];
  LevelCoef lc[CTA_LEVELS];
  typename VT<T>::b4 Jk[12];  // the coarsest level's planes (6 x 2 blocks)
  T ainv[16];
  V2 X[tail_x_size(CTA_NX)];
  V2 tail[tail_smem_v2(16) + 16 * 8 + 11 * 16 * 8];  // 16 x 8 down: its b and block rows included
};

template <typename T>
__global__ void __launch_bounds__(CTA_THREADS, sizeof(T) == 4 ? 2 : 1)
    k_cta_solve(const __grid_constant__ CtaParams P, int B, const Coef* __restrict__ coef,
                double2* __restrict__ xo_g, double2* __restrict__ xoo_g, double* __restrict__ qoi,
                int* __restrict__ status, unsigned long long* __restrict__ totals) {
  typedef typename VT<T>::v2 V2;
  typedef typename VT<T>::b4 B4;
  extern __shared__ __align__(32) unsigned char cta_smem[];
  CtaShared<T>& S = *reinterpret_cast<CtaShared<T>*>(cta_smem);
  const int s = blockIdx.x;
  if (s >= B) return;
  const int t = threadIdx.x;
  if (status[s] != 0) {
    if (t < 2) qoi[2 * (int64_t)s + t] = NAN;
    return;
  }
  constexpr int P2 = CTA_NX + 2;
  // the thread's cells: colour col, child c of coarse cell Q
  const int Q = t >> 1, c = t & 1, IY = Q >> 4, IX = Q & 15;
  int ix[2], iy, st[2], xi[2];
  iy = 2 * IY + c;
#pragma unroll
  for (int col = 0; col < 2; ++col) {
    ix[col] = 2 * IX + (c ^ col);
    st[col] = st_of(ix[col], iy, CTA_NX);
    xi[col] = (iy + 1) * P2 + ix[col] + 1;
  }
  const Coef cf = coef[s];
  double2* xo = xo_g + (int64_t)s * CTA_N;
  const bool quad = P.predictor_order == 2 && xoo_g;
  double2* xoo = quad ? xoo_g + (int64_t)s * CTA_N : nullptr;
  const double inv_tau = 1.0 / P.tau;
  if (t < CTA_LEVELS) {
    const double hk = P.h0 * (double)(1 << t);
    S.lc[t] = level_coef(P.ph, cf, hk, hk * hk * inv_tau * P.inv_s, P.inv_s);
  }
  for (int i = t; i < tail_x_size(CTA_NX); i += CTA_THREADS) S.X[i] = mk2<V2>((T)0, (T)0);
  for (int i = t; i < (int)(sizeof(S.tail) / sizeof(V2)); i += CTA_THREADS) S.tail[i] = mk2<V2>((T)0, (T)0);
  // a3: initial state, fresh-water hydrostatic pressure, c = 0
  const double2 v0 = make_double2(P.rho0g * (P.Ly - (iy + 0.5) * P.h0), 0.0);
#pragma unroll
  for (int col = 0; col < 2; ++col) {
    S.x[st[col]] = v0;
    xo[st[col]] = v0;
    if (quad) xoo[st[col]] = v0;
  }
  __syncthreads();
  CellCoefs<double, false> K0;
  K0.load(P.ph, S.lc, nullptr, 0, 0.0, 0.0, 0.0, nullptr, 0);
  TailLevel<T, 16, false> tl;
  tl.place(S.tail);
  const TailRows<T> no_rows{};
  TailArgs ta;
  ta.nu1 = P.nu1;
  ta.nu2 = P.nu2;
  const bool black_known = P.nu2 > 0;

  unsigned long long newton_total = 0, lin_total = 0;
  int fail = 0;
  // blocks of the thread's cells (W, E, S, N; centre; inverse)
  B4 nb[2][4], ce[2], ci[2];
  V2 r[2], rh[2], p[2], v[2], dx[2];

  // mean of the 2x2 children of every coarse level (xf: the fine states)
  auto restrict_all = [&](const double2* xf, double2* out) {
    const double2* f = xf;
    int off = 0;
#pragma unroll
    for (int k = 1; k < CTA_LEVELS; ++k) {
      const int ncx = CTA_NX >> k, Nc = CTA_N >> (2 * k), nxf = 2 * ncx;
      if (t < Nc) {
        int X, Y;
        xy_of(t, ncx, X, Y);
        const double2 a = f[st_of(2 * X, 2 * Y, nxf)], b = f[st_of(2 * X + 1, 2 * Y, nxf)];
        const double2 d = f[st_of(2 * X, 2 * Y + 1, nxf)], e = f[st_of(2 * X + 1, 2 * Y + 1, nxf)];
        out[off + t] = make_double2(0.25 * (((a.x + b.x) + d.x) + e.x), 0.25 * (((a.y + b.y) + d.y) + e.y));
      }
      __syncthreads();
      f = out + off;
      off += Nc;
    }
  };
  // A nb-product of the thread's cell of colour col with the vector in S.X
  auto offdiag = [&](int col, T& r0, T& r1) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const V2 xn = S.X[xi[col] + (k == 0 ? -1 : (k == 1 ? 1 : (k == 2 ? -P2 : P2)))];
      bmv_sub(nb[col][k], xn.x, xn.y, r0, r1);
    }
  };
  auto sweep = [&](int col, const V2 b, bool zero) {
    T r0 = b.x, r1 = b.y, y0, y1;
    if (!zero) offdiag(col, r0, r1);
    bmv(ci[col], r0, r1, y0, y1);
    S.X[xi[col]] = mk2<V2>(y0, y1);
    __syncthreads();
  };
  // One V(nu1, nu2) cycle: S.X = M^{-1} b
  auto vcycle = [&](const V2* b) {
    V2 sum;
    if (P.nu1 > 0) {
      sweep(0, b[0], true);
      sweep(1, b[1], false);
      for (int i = 1; i < P.nu1; ++i) {
        sweep(0, b[0], false);
        sweep(1, b[1], false);
      }
      T r0 = b[0].x, r1 = b[0].y;
      const V2 xx = S.X[xi[0]];
      bmv_sub(ce[0], xx.x, xx.y, r0, r1);
      offdiag(0, r0, r1);
      sum = mk2<V2>(r0 + __shfl_xor_sync(0xffffffffu, r0, 1), r1 + __shfl_xor_sync(0xffffffffu, r1, 1));
    } else {
      S.X[xi[0]] = S.X[xi[1]] = mk2<V2>((T)0, (T)0);
      const T a0 = __shfl_xor_sync(0xffffffffu, b[0].x, 1), a1 = __shfl_xor_sync(0xffffffffu, b[0].y, 1);
      const T d0 = __shfl_xor_sync(0xffffffffu, b[1].x, 1), d1 = __shfl_xor_sync(0xffffffffu, b[1].y, 1);
      sum = mk2<V2>(((b[0].x + b[1].x) + d0) + a0, ((b[0].y + b[1].y) + d1) + a1);  // stored by child 0
    }
    if (c == 0) tl.Bs[Q] = sum;  // natural order of the 16 x 8 grid
    __syncthreads();
    if (t < 128) tl.run(ta, 0, t, no_rows, S.ainv + 4 * (t & 3));
    __syncthreads();
    const V2 pc = tl.X[(IY + 1) * (16 + 2) + IX + 1];
#pragma unroll
    for (int col = 0; col < 2; ++col) {
      if (col == 0 && P.nu2 > 0) continue;
      V2 w = S.X[xi[col]];
      w.x += pc.x;
      w.y += pc.y;
      S.X[xi[col]] = w;
    }
    __syncthreads();
    for (int i = 0; i < P.nu2; ++i) {
      sweep(0, b[0], false);
      sweep(1, b[1], false);
    }
  };
  // A x for the vector in S.X, the result of a cycle for b
  auto matvec = [&](const V2* b, V2* y) {
#pragma unroll
    for (int col = 0; col < 2; ++col) {
      if (col == 1 && black_known) {
        y[1] = b[1];
        continue;
      }
      const V2 xx = S.X[xi[col]];
      T r0, r1;
      bmv(ce[col], xx.x, xx.y, r0, r1);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const V2 xn = S.X[xi[col] + (k == 0 ? -1 : (k == 1 ? 1 : (k == 2 ? -P2 : P2)))];
        bmv_add(nb[col][k], xn.x, xn.y, r0, r1);
      }
      y[col] = mk2<V2>(r0, r1);
    }
  };
  auto dot = [](const V2* a, const V2* b) {
    return (double)fma_(a[0].x, b[0].x, fma_(a[0].y, b[0].y, fma_(a[1].x, b[1].x, a[1].y * b[1].y)));
  };

  for (int step = 0; step < P.steps && !fail; ++step) {
    // a10: x_old <- x (and Newton's first iterate by the predictor)
#pragma unroll
    for (int col = 0; col < 2; ++col) {
      const int i = st[col];
      const double2 a = S.x[i], b = xo[i];
      double2 o = b;
      if (quad) {
        o = xoo[i];
        xoo[i] = b;
      }
      xo[i] = a;
      if (quad && step > 1 && P.predictor > 0.0) {  // as k_step_begin_predict2
        const double ex = 2.0 * (a.x - b.x) - (b.x - o.x), ey = 2.0 * (a.y - b.y) - (b.y - o.y);
        S.x[i] = make_double2(fma(P.predictor, ex, a.x), fma(P.predictor, ey, a.y));
      } else if (step > 0 && P.predictor > 0.0) {
        S.x[i] = make_double2(fma(P.predictor, a.x - b.x, a.x), fma(P.predictor, a.y - b.y, a.y));
      }
    }
    __syncthreads();
    restrict_all(xo, S.xoc);

    for (int it = 0;; ++it) {
      // a4: fine residual and Jacobian; r = r_hat = -F
      double rloc = 0.0;
#pragma unroll
      for (int col = 0; col < 2; ++col) {
        CellSum<T, double> o;
        assemble_cell<T, double>(P.ph, K0, CTA_NX, CTA_NY, P.h0, S.x, xo, st[col], ix[col], iy, o);
#pragma unroll
        for (int k = 0; k < 4; ++k) nb[col][k] = mkblk<B4>(o.Nb[k][0], o.Nb[k][1], o.Nb[k][2], o.Nb[k][3]);
        ce[col] = mkblk<B4>(o.C[0], o.C[1], o.C[2], o.C[3]);
        const T idet = (T)1 / fma_(o.C[0], o.C[3], neg_(mul_(o.C[1], o.C[2]))), nd = neg_(idet);
        ci[col] = mkblk<B4>(mul_(o.C[3], idet), mul_(o.C[1], nd), mul_(o.C[2], nd), mul_(o.C[0], idet));
        r[col] = rh[col] = mk2<V2>((T)(-o.Rm), (T)(-o.Rs));
        rloc = abs_max_or_inf(rloc, abs_max_or_inf(o.Rm, o.Rs));
      }
      const double rmax = block_max_nonneg(rloc, S.red);
      if (!(rmax <= 1.0e300)) {
        fail = 3;
        break;
      }
      if (rmax <= P.atol) break;
      if (it >= P.newton_maxit) {
        fail = 1;
        break;
      }
      ++newton_total;
      // a5: restricted states and rediscretised coarse operators, the block
      // rows straight into the tail's slots
      restrict_all(S.x, S.xc);
      if (t < CTA_COARSE) {
        int k = 1, off = 0, Nc = CTA_N / 4;
        while (t >= off + Nc) {
          off += Nc;
          Nc >>= 2;
          ++k;
        }
        const int ncx = CTA_NX >> k, e = t - off;
        int X, Y;
        xy_of(e, ncx, X, Y);
        CellCoefs<T, false> Kk;
        Kk.load(P.ph, S.lc + k, nullptr, 0, 0.0, 0.0, 0.0, nullptr, 0);
        CellSum<T, T> o;
        assemble_cell<T, T>(P.ph, Kk, ncx, CTA_NY >> k, P.h0 * (double)(1 << k), S.xc + off, S.xoc + off, e, X, Y, o);
        if (k == CTA_LEVELS - 1) {
          store_blocks<T>(S.Jk, 2, e, o.C, o.Nb);
        } else {
          const int col = (X + Y) & 1, items = ncx * ncx / 2;
          V2* base = S.tail;
          for (int w = 16; w > ncx; w >>= 1) base += tail_size(w, false);
          V2* op = base + tail_x_size(ncx) + ncx * ncx / 2;  // past the level's x and b
          const int q = 4 * ((Y >> 1) * (ncx >> 1) + (X >> 1)) + 2 * (Y & 1);
          const T idet = (T)1 / fma_(o.C[0], o.C[3], neg_(mul_(o.C[1], o.C[2]))), nd = neg_(idet);
          const T inv[4] = {mul_(o.C[3], idet), mul_(o.C[1], nd), mul_(o.C[2], nd), mul_(o.C[0], idet)};
#pragma unroll
          for (int row = 0; row < 2; ++row) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              op[(5 * col + j) * items + q + row] = mk2<V2>(o.Nb[j][2 * row], o.Nb[j][2 * row + 1]);
            op[(5 * col + 4) * items + q + row] = mk2<V2>(inv[2 * row], inv[2 * row + 1]);
            if (col == 0) op[10 * items + q + row] = mk2<V2>(o.C[2 * row], o.C[2 * row + 1]);
          }
        }
      }
      __syncthreads();
      if (t < 32) {  // coarsest 4 x 4 inverse
        double M[4];
        coarse_inverse_lanes(S.Jk, 2, t & 7, M);
        if (t >= 4 && t < 8)
          for (int i = 0; i < 4; ++i) S.ainv[i * 4 + t - 4] = (T)M[i];
      }
      // a6: BiCGStab, right-preconditioned by the V-cycle (a7), matvec (a8).
      // The scalars are formed by one thread and broadcast (S.bc).
      const double bn2 = block_sum_tree(dot(r, r), S.red);
      double rho = bn2, rn2 = bn2, beta = 0.0, omega = 1.0;
#pragma unroll
      for (int col = 0; col < 2; ++col) dx[col] = mk2<V2>((T)0, (T)0);
      int lit = 0;
      for (; lit < P.lin_maxit; ++lit) {
        if (!(rn2 <= 1.0e300) || !(rho == rho)) {
          fail = 3;
          break;
        }
        if (rn2 <= P.rtol2 * bn2) break;
        const T bt = (T)beta, om = (T)omega;
#pragma unroll
        for (int col = 0; col < 2; ++col)
          p[col] = lit == 0 ? r[col]
                            : mk2<V2>(r[col].x + bt * (p[col].x - om * v[col].x),
                                      r[col].y + bt * (p[col].y - om * v[col].y));
        vcycle(p);
        matvec(p, v);
        const double rv = block_sum_tree(dot(rh, v), S.red);
        if (t == 0) S.bc[0] = rho / rv;
        __syncthreads();
        const double alpha = S.bc[0];
        const T a = (T)alpha;
#pragma unroll
        for (int col = 0; col < 2; ++col) {
          const V2 pp = S.X[xi[col]];
          r[col] = mk2<V2>(r[col].x - a * v[col].x, r[col].y - a * v[col].y);  // s
          dx[col] = mk2<V2>(dx[col].x + a * pp.x, dx[col].y + a * pp.y);
        }
        __syncthreads();
        vcycle(r);  // s_hat in S.X
        V2 tv[2];
        matvec(r, tv);
        double d = block_sum_pair(dot(tv, r), dot(tv, tv), S.red);
        if (t == CTA_THREADS / 2) S.bc[1] = d;
        __syncthreads();
        if (t == 0) S.bc[0] = S.bc[1] > 0.0 ? d / S.bc[1] : 0.0;
        __syncthreads();
        omega = S.bc[0];
        const T w = (T)omega;
#pragma unroll
        for (int col = 0; col < 2; ++col) {
          const V2 sv = S.X[xi[col]];
          dx[col] = mk2<V2>(dx[col].x + w * sv.x, dx[col].y + w * sv.y);
          r[col] = mk2<V2>(r[col].x - w * tv[col].x, r[col].y - w * tv[col].y);
        }
        d = block_sum_pair(dot(rh, r), dot(r, r), S.red);
        if (t == 0) {
          S.bc[2] = d;
          S.bc[0] = (d / rho) * (alpha / omega);
        }
        if (t == CTA_THREADS / 2) S.bc[3] = d;
        __syncthreads();
        beta = S.bc[0];
        rho = S.bc[2];
        rn2 = S.bc[3];
      }
      lin_total += lit;
      if (fail) break;
      // a9: Newton update (step limited to max |dc| <= dc_limit) and the update test
      double dloc = 0.0, cloc = 0.0;
#pragma unroll
      for (int col = 0; col < 2; ++col) {
        const double dc = abs_max_or_inf((double)dx[col].y, 0.0);
        dloc = abs_max_or_inf(dloc, abs_max_or_inf((double)dx[col].x * P.inv_pref, dc));
        cloc = abs_max_or_inf(cloc, dc);
      }
      const double dmax = block_max_nonneg(dloc, S.red);
      const double cmax = block_max_nonneg(cloc, S.red);
      const double th = (P.dc_limit > 0.0 && cmax > P.dc_limit) ? P.dc_limit / cmax : 1.0;
#pragma unroll
      for (int col = 0; col < 2; ++col) {
        double2 xx = S.x[st[col]];
        xx.x = fma(th, (double)dx[col].x, xx.x);
        xx.y = fma(th, (double)dx[col].y, xx.y);
        S.x[st[col]] = xx;
      }
      __syncthreads();
      if (!(dmax <= 1.0e300)) {
        fail = 3;
        break;
      }
      if (dmax <= P.dxtol) break;
    }
  }
  __syncthreads();
  // a11: QoIs
  double acc = 0.0;
#pragma unroll
  for (int col = 0; col < 2; ++col) {
    const double cc = S.x[st[col]].y;
    acc += (P.ph.rho0 + P.ph.drho * cc) * cc;
  }
  acc = block_sum_tree(acc, S.red);
  if (t == 0) {
    const int ix0 = (3 * CTA_NY) / 2 - 1, iy0 = CTA_NY / 4 - 1;
    const double c00 = S.x[st_of(ix0, iy0, CTA_NX)].y, c10 = S.x[st_of(ix0 + 1, iy0, CTA_NX)].y;
    const double c01 = S.x[st_of(ix0, iy0 + 1, CTA_NX)].y, c11 = S.x[st_of(ix0 + 1, iy0 + 1, CTA_NX)].y;
    qoi[2 * (int64_t)s] = cf.phi * acc * P.h0 * P.h0;
    qoi[2 * (int64_t)s + 1] = 0.25 * (((c00 + c10) + c01) + c11);
    if (fail) status[s] = fail;
    atomicAdd(&totals[0], newton_total);
    atomicAdd(&totals[1], lin_total);
  }
}

}  // namespace hk
