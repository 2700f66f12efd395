// Fused multigrid tail (sm_103a): the part of a V-cycle below a coarse level
// of NX0 x NX0/2 cells, i.e. the V(nu1, nu2) cycle that solves A x = b
// approximately from x = 0 on that level, run by one CTA per sample.
//
// What bounds it, and why it looks like this.  Every phase (half-sweep,
// restriction, prolongation) depends on the one before, and a warp's FP64
// instruction occupies its SM sub-partition's pipe for 64 cycles on GB300
// however many lanes are active (measured: 64.6 cycles with 32, 8 or 1
// lanes; all four sub-partitions together 19), so the time of a phase is the
// number of FP64 instructions on a warp's path, not the number of cells.
//  * Two threads per cell, one per row (equation) of its 2x2 blocks: a
//    half-sweep is 10 dependent FP64 instructions instead of 20, with the two
//    row residuals exchanged by a shuffle.
//  * The four lanes of a coarse cell Q hold the two children of either
//    colour ((0,0), (1,1) and (1,0), (0,1)) times two rows, so the restriction
//    is one shuffle and the prolongation needs the own parent only.
//  * Prolongation first adds x_c to the black cells in place (one addition),
//    instead of adding it to all four neighbours of every red cell (eight).
//  * x lives in shared memory with a halo of zeros and natural row order:
//    the blocks across the domain boundary are zero, so no phase tests for it
//    or divides an index.
//  * A thread reads each block row it will need once per launch, the first
//    level's into registers, the coarser levels' into its own slots of shared
//    memory, all before the first phase and before the wait for the kernel
//    that writes b; levels of one warp (8 x 4 and below)
//    synchronise by __syncwarp, the 16 x 8 level by a barrier of its own four
//    warps.
// The times before and after stand at tail_level (henry_engine.cu).
// The arithmetic per cell and its order are sweep_cell's, residual_cell's and
// coarse_row's, so the result is bit-identical to the level-by-level kernels'.
#pragma once
#include "henry_kernels.cuh"

namespace hk {

constexpr int TAIL_MAX_LEVELS = 6;  // 64 x 32 .. 2 x 1

// Operands of the tail: per level the 6 block planes (plane stride plane[k],
// a sample's N_k blocks at s N_k), the right-hand side b and result x of the
// first level ([B][N_0]), and the coarsest inverses ([B][16]).
struct TailArgs {
  const void* J[TAIL_MAX_LEVELS];
  int64_t plane[TAIL_MAX_LEVELS];
  const void* b;
  void* x;
  const void* ainv;
  const int* active;
  int late;  // the kernel before sets the flags (a tail from the fine grid): read them after the wait
  int nu1, nu2;
};

// CTA size: two threads per cell of one colour up to 32 x 16 cells, one
// thread per coarse cell on 64 x 32.
__host__ __device__ constexpr int tail_threads(int nx0) { return nx0 >= 64 ? 512 : (nx0 * nx0 / 2 < 32 ? 32 : nx0 * nx0 / 2); }

// Shared memory of one level in units of V2: x with its halo, and on every
// level but the first b and the block rows of its threads (11 pairs each: 4
// neighbours and the inverse for either colour, the red cells' centre).
__host__ __device__ constexpr int tail_x_size(int nx) { return (nx / 2 + 2) * (nx + 2); }
__host__ __device__ constexpr int tail_size(int nx, bool first) {
  return tail_x_size(nx) + (first ? 0 : nx * nx / 2 + 11 * (nx * nx / 2));
}
__host__ __device__ constexpr int tail_smem_v2(int nx0) {
  int o = 0;
  for (int nx = nx0; nx >= 4; nx /= 2) o += tail_size(nx, nx == nx0);
  return o + tail_x_size(2) + 2;  // the coarsest level's x (with halo) and b
}

template <int N>
__device__ __forceinline__ void tail_sync(int id) {
  if constexpr (N <= 32) {
    __syncwarp();
  } else {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(N) : "memory");
  }
}

// The block rows of one thread on one level.  Row-split levels: row `row` of
// the children c of colours 0 and 1.
template <typename T>
struct TailRows {
  typedef typename VT<T>::v2 V2;
  V2 nb[2][4], ci[2], ce;
};

// One level of the tail and everything below it.  Called by the threads t <
// NTL of the CTA; the level's x is written to shared memory (X).  FIRST: b
// comes from (and x goes to) global memory.
template <typename T, int NX, bool FIRST>
struct TailLevel {
  typedef typename VT<T>::v2 V2;
  typedef typename VT<T>::b4 B4;
  static constexpr int NY = NX / 2, NC = NX * NX / 8, P = NX + 2;  // cells of the next level, row pitch of x
  static constexpr bool ROWS = NX <= 32;                            // two threads per cell
  static constexpr int NTL = ROWS ? (4 * NC < 32 ? 32 : 4 * NC) : NC;
  static constexpr int ITEMS = 4 * NC;                              // (coarse cell, child, row)
  static constexpr int PC = NX / 2 + 2;                             // row pitch of the next level's x

  // Shared memory of this level (base in V2 units) and the next one's.
  V2* X;
  V2* Bs;   // b in natural order (not FIRST)
  V2* Op;   // block rows [11][ITEMS] (not FIRST)
  V2* Xc;   // next level's x (with halo) and b
  V2* Bc;

  __device__ __forceinline__ void place(V2* base) {
    X = base;
    Bs = base + tail_x_size(NX);
    Op = Bs + NX * NY;
    Xc = base + tail_size(NX, FIRST);
    Bc = Xc + tail_x_size(NX / 2);
  }
  // Cell of coarse cell Q's child c of colour col.
  static __device__ __forceinline__ void cell(int Q, int c, int col, int& ix, int& iy) {
    const int IY = Q / (NX / 2), IX = Q - IY * (NX / 2);
    ix = 2 * IX + (c ^ col);
    iy = 2 * IY + c;
  }
  static __device__ __forceinline__ int xi(int ix, int iy) { return (iy + 1) * P + ix + 1; }

  // Load the thread's block rows from global memory: the sample's blocks Jg
  // with plane stride ps.
  static __device__ __forceinline__ void load_rows(TailRows<T>& R, const B4* Jg, int64_t ps, int t) {
    const int Q = t >> 2, c = (t >> 1) & 1, row = t & 1;
#pragma unroll
    for (int col = 0; col < 2; ++col) {
      int ix, iy;
      cell(Q, c, col, ix, iy);
      const V2* p = reinterpret_cast<const V2*>(Jg + st_of(ix, iy, NX)) + row;
#pragma unroll
      for (int k = 0; k < 4; ++k) R.nb[col][k] = p[2 * (k + 1) * ps];
      R.ci[col] = p[10 * ps];
      if (col == 0) R.ce = p[0];
    }
  }
  __device__ __forceinline__ void park_rows(const TailRows<T>& R, int t) const {
#pragma unroll
    for (int col = 0; col < 2; ++col) {
#pragma unroll
      for (int k = 0; k < 4; ++k) Op[(5 * col + k) * ITEMS + t] = R.nb[col][k];
      Op[(5 * col + 4) * ITEMS + t] = R.ci[col];
    }
    Op[10 * ITEMS + t] = R.ce;
  }
  __device__ __forceinline__ V2 nb(const TailRows<T>& R, int col, int k, int t) const {
    if constexpr (FIRST) return R.nb[col][k];
    else return Op[(5 * col + k) * ITEMS + t];
  }
  __device__ __forceinline__ V2 ci(const TailRows<T>& R, int col, int t) const {
    if constexpr (FIRST) return R.ci[col];
    else return Op[(5 * col + 4) * ITEMS + t];
  }
  __device__ __forceinline__ V2 ce(const TailRows<T>& R, int t) const {
    if constexpr (FIRST) return R.ce;
    else return Op[10 * ITEMS + t];
  }
  // Level barrier; a one-warp level's shuffles and __syncwarp need all 32
  // lanes, so lanes beyond ITEMS run along with t clamped and store nothing.
  static __device__ __forceinline__ void sync() { tail_sync<NTL>(NX == 16 ? 1 : (NX == 32 ? 2 : 3)); }

  // r - sum_nb A_nb x_nb, the thread's row, in sweep_cell's order.
  __device__ __forceinline__ T offdiag(const TailRows<T>& R, int col, int t, int xo, T r) const {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const V2 a = nb(R, col, k, t);
      const V2 xn = X[xo + (k == 0 ? -1 : (k == 1 ? 1 : (k == 2 ? -P : P)))];
      r = fma_(-a.x, xn.x, fma_(-a.y, xn.y, r));
    }
    return r;
  }
  // One half-sweep of colour col (ZERO: from x = 0).
  template <bool ZERO>
  __device__ __forceinline__ void sweep(const TailRows<T>& R, int col, int t, int row, int xo, T b, bool on) const {
    T r = b;
    if (!ZERO) r = offdiag(R, col, t, xo, r);
    const T o = __shfl_xor_sync(0xffffffffu, r, 1);
    const V2 m = ci(R, col, t);
    const T y = fma_(m.x, row ? o : r, m.y * (row ? r : o));
    if (on) reinterpret_cast<T*>(X + xo)[row] = y;
    sync();
  }

  __device__ __forceinline__ void run(const TailArgs& A, int s, int t, const TailRows<T>& R, const T* ainv) const {
    const bool on = ITEMS >= 32 || t < ITEMS;
    const int tt = on ? t : ITEMS - 1;
    const int Q = tt >> 2, c = (tt >> 1) & 1, row = tt & 1;
    int ix0, iy0, ix1, iy1;
    cell(Q, c, 0, ix0, iy0);
    cell(Q, c, 1, ix1, iy1);
    const int x0 = xi(ix0, iy0), x1 = xi(ix1, iy1);
    T b0, b1;
    if constexpr (FIRST) {
      grid_enter();
      if (A.late && !A.active[s]) return;
      const T* bg = reinterpret_cast<const T*>(reinterpret_cast<const V2*>(A.b) + (int64_t)s * (NX * NY));
      b0 = bg[2 * st_of(ix0, iy0, NX) + row];
      b1 = bg[2 * st_of(ix1, iy1, NX) + row];
    } else {
      b0 = reinterpret_cast<const T*>(Bs)[2 * (iy0 * NX + ix0) + row];
      b1 = reinterpret_cast<const T*>(Bs)[2 * (iy1 * NX + ix1) + row];
    }
    const int IY = Q / (NX / 2), IX = Q - IY * (NX / 2);
    T sum;
    if (A.nu1 > 0) {
      sweep<true>(R, 0, tt, row, x0, b0, on);
      sweep<false>(R, 1, tt, row, x1, b1, on);
      for (int i = 1; i < A.nu1; ++i) {
        sweep<false>(R, 0, tt, row, x0, b0, on);
        sweep<false>(R, 1, tt, row, x1, b1, on);
      }
      // residual of the red cells, summed over the coarse cell's two (the
      // black cells' residuals vanish)
      const V2 a = ce(R, tt), xx = X[x0];
      T r = fma_(-a.x, xx.x, fma_(-a.y, xx.y, b0));
      r = offdiag(R, 0, tt, x0, r);
      sum = r + __shfl_xor_sync(0xffffffffu, r, 2);
    } else {  // x = 0: restrict b itself, children in the order (0,0), (1,0), (0,1), (1,1)
      if (on) {
        reinterpret_cast<T*>(X + x0)[row] = (T)0;
        reinterpret_cast<T*>(X + x1)[row] = (T)0;
      }
      const T r1 = __shfl_xor_sync(0xffffffffu, b0, 2), k1 = __shfl_xor_sync(0xffffffffu, b1, 2);
      sum = c ? ((r1 + k1) + b1) + b0 : ((b0 + b1) + k1) + r1;
    }
    if (on && c == 0) reinterpret_cast<T*>(Bc)[2 * (IY * (NX / 2) + IX) + row] = sum;
    sync();
    if constexpr (NX == 4) {  // the 2 x 1 grid: one row of the explicit inverse per thread
      if (t < 4) {
        const T* v = reinterpret_cast<const T*>(Bc);
        reinterpret_cast<T*>(Xc + PC + 1)[t] = coarse_row(ainv, v[0], v[1], v[2], v[3]);
      }
      sync();
    } else {
      typedef TailLevel<T, NX / 2, false> Next;
      if (t < Next::NTL) {
        Next n;
        n.place(Xc);
        TailRows<T> unused;
        n.run(A, s, t, unused, ainv);
      }
      sync();
    }
    // x += P x_c: before a red half-sweep the black cells' values only (the
    // red ones are overwritten)
    if (on) {
      const T pc = reinterpret_cast<const T*>(Xc + (IY + 1) * PC + IX + 1)[row];
      reinterpret_cast<T*>(X + x1)[row] += pc;
      if (A.nu2 == 0) reinterpret_cast<T*>(X + x0)[row] += pc;
    }
    sync();
    for (int i = 0; i < A.nu2; ++i) {
      sweep<false>(R, 0, tt, row, x0, b0, on);
      sweep<false>(R, 1, tt, row, x1, b1, on);
    }
    if constexpr (FIRST) {
      if (on) {
        T* xg = reinterpret_cast<T*>(reinterpret_cast<V2*>(A.x) + (int64_t)s * (NX * NY));
        xg[2 * st_of(ix0, iy0, NX) + row] = reinterpret_cast<const T*>(X + x0)[row];
        xg[2 * st_of(ix1, iy1, NX) + row] = reinterpret_cast<const T*>(X + x1)[row];
      }
    }
  }
};

// The 64 x 32 level, one thread per coarse cell (both children of either
// colour): the same phases with whole cells.  FP32 keeps the blocks of its
// four cells in registers; in FP64 they do not fit and are read through L2
// at every use.
template <typename T>
struct TailWide {
  typedef typename VT<T>::v2 V2;
  typedef typename VT<T>::b4 B4;
  static constexpr int NX = 64, NY = 32, P = NX + 2, PC = NX / 2 + 2;
  static constexpr bool KEEP = sizeof(T) == 4;
  V2 *X, *Xc, *Bc;
  const B4* Jg;
  int64_t ps;
  int st[2][2], xo[2][2];  // [colour][child]: storage index, place in X
  B4 nbk[KEEP ? 2 : 1][2][4], cik[KEEP ? 2 : 1][2], cek[2];
  V2 b[2][2];

  __device__ __forceinline__ void load(const B4* J, int64_t plane, int Q) {
    Jg = J;
    ps = plane;
    const int IY = Q >> 5, IX = Q & 31;
#pragma unroll
    for (int col = 0; col < 2; ++col)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int ix = 2 * IX + (c ^ col), iy = 2 * IY + c;
        st[col][c] = st_of(ix, iy, NX);
        xo[col][c] = (iy + 1) * P + ix + 1;
        if constexpr (KEEP) {
#pragma unroll
          for (int k = 0; k < 4; ++k) nbk[col][c][k] = Jg[(k + 1) * ps + st[col][c]];
          cik[col][c] = Jg[5 * ps + st[col][c]];
          if (col == 0) cek[c] = Jg[st[0][c]];
        }
      }
  }
  __device__ __forceinline__ B4 blk(int col, int c, int k) const {
    if constexpr (KEEP) return nbk[col][c][k];
    else return Jg[(k + 1) * ps + st[col][c]];
  }
  __device__ __forceinline__ B4 inv(int col, int c) const {
    if constexpr (KEEP) return cik[col][c];
    else return Jg[5 * ps + st[col][c]];
  }
  __device__ __forceinline__ B4 cen(int c) const {
    if constexpr (KEEP) return cek[c];
    else return Jg[st[0][c]];
  }
  __device__ __forceinline__ void offdiag(int col, int c, T& r0, T& r1) const {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const V2 xn = X[xo[col][c] + (k == 0 ? -1 : (k == 1 ? 1 : (k == 2 ? -P : P)))];
      bmv_sub(blk(col, c, k), xn.x, xn.y, r0, r1);
    }
  }
  template <bool ZERO>
  __device__ __forceinline__ void sweep(int col) const {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      T r0 = b[col][c].x, r1 = b[col][c].y, y0, y1;
      if (!ZERO) offdiag(col, c, r0, r1);
      bmv(inv(col, c), r0, r1, y0, y1);
      X[xo[col][c]] = mk2<V2>(y0, y1);
    }
    __syncthreads();
  }
  __device__ __forceinline__ void run(const TailArgs& A, int s, int Q, const T* ainv) {
    grid_enter();
    if (A.late && !A.active[s]) return;
    const V2* bg = reinterpret_cast<const V2*>(A.b) + (int64_t)s * (NX * NY);
#pragma unroll
    for (int col = 0; col < 2; ++col)
#pragma unroll
      for (int c = 0; c < 2; ++c) b[col][c] = bg[st[col][c]];
    V2 sum = mk2<V2>((T)0, (T)0);
    if (A.nu1 > 0) {
      sweep<true>(0);
      sweep<false>(1);
      for (int i = 1; i < A.nu1; ++i) {
        sweep<false>(0);
        sweep<false>(1);
      }
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        T r0 = b[0][c].x, r1 = b[0][c].y;
        const V2 xx = X[xo[0][c]];
        bmv_sub(cen(c), xx.x, xx.y, r0, r1);
        offdiag(0, c, r0, r1);
        sum.x += r0;
        sum.y += r1;
      }
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {  // children (0,0), (1,0), (0,1), (1,1)
        const int col = q == 1 || q == 2 ? 1 : 0, c = q >> 1;
        X[xo[col][c]] = mk2<V2>((T)0, (T)0);
        sum.x += b[col][c].x;
        sum.y += b[col][c].y;
      }
    }
    Bc[Q] = sum;  // natural order of the 32 x 16 grid
    __syncthreads();
    {
      TailLevel<T, 32, false> n;
      n.place(Xc);
      TailRows<T> unused;
      n.run(A, s, Q, unused, ainv);
    }
    __syncthreads();
    const V2 pc = Xc[((Q >> 5) + 1) * PC + (Q & 31) + 1];
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int col = 0; col < 2; ++col) {
        if (col == 0 && A.nu2 > 0) continue;
        V2 v = X[xo[col][c]];
        v.x += pc.x;
        v.y += pc.y;
        X[xo[col][c]] = v;
      }
    __syncthreads();
    for (int i = 0; i < A.nu2; ++i) {
      sweep<false>(0);
      sweep<false>(1);
    }
    V2* xg = reinterpret_cast<V2*>(A.x) + (int64_t)s * (NX * NY);
#pragma unroll
    for (int col = 0; col < 2; ++col)
#pragma unroll
      for (int c = 0; c < 2; ++c) xg[st[col][c]] = X[xo[col][c]];
  }
};

// Read the block rows of the levels from NX down (level k of A) into their
// shared-memory slots.
template <typename T, int NX>
__device__ __forceinline__ void tail_park(const TailArgs& A, int k, int s, int t, typename VT<T>::v2* base) {
  if constexpr (NX >= 4) {
    typedef TailLevel<T, NX, false> L;
    if (t < L::ITEMS) {
      L n;
      n.place(base);
      TailRows<T> R;
      L::load_rows(R, reinterpret_cast<const typename VT<T>::b4*>(A.J[k]) + (int64_t)s * (NX * NX / 2), A.plane[k], t);
      n.park_rows(R, t);
    }
    tail_park<T, NX / 2>(A, k + 1, s, t, base + tail_size(NX, false));
  }
}

template <typename T, int NX0>
__global__ void __launch_bounds__(tail_threads(NX0)) k_vcycle_tail(const __grid_constant__ TailArgs A, int B) {
  typedef typename VT<T>::v2 V2;
  typedef typename VT<T>::b4 B4;
  constexpr int NT = tail_threads(NX0);
  extern __shared__ __align__(16) unsigned char tail_smem[];
  V2* sm = reinterpret_cast<V2*>(tail_smem);
  const int s = blockIdx.x;
  if (s >= B || (!A.late && !A.active[s])) {
    grid_enter();
    return;
  }
  // The one- and four-warp levels run in the logical warps 0 and 0-3: rotate
  // those over the sub-partitions from CTA to CTA.
  const int t = (threadIdx.x + 32 * (blockIdx.x & 3)) & (NT - 1);
  for (int i = threadIdx.x; i < tail_smem_v2(NX0); i += NT) sm[i] = mk2<V2>((T)0, (T)0);
  T ainv[4] = {(T)0, (T)0, (T)0, (T)0};
  if (t < 4) {
    const T* ai = reinterpret_cast<const T*>(A.ainv) + (int64_t)s * 16 + 4 * t;
#pragma unroll
    for (int j = 0; j < 4; ++j) ainv[j] = ai[j];
  }
  const B4* J0 = reinterpret_cast<const B4*>(A.J[0]) + (int64_t)s * (NX0 * NX0 / 2);
  if constexpr (NX0 >= 64) {
    TailWide<T> W;
    W.X = sm;
    W.Xc = sm + tail_size(NX0, true);
    W.Bc = W.Xc + tail_x_size(NX0 / 2);
    W.load(J0, A.plane[0], t);
    __syncthreads();  // zeroed before the slots below are filled
    tail_park<T, NX0 / 2>(A, 1, s, t, W.Xc);
    W.run(A, s, t, ainv);
  } else {
    typedef TailLevel<T, NX0, true> L;
    L n;
    n.place(sm);
    TailRows<T> R;
    L::load_rows(R, J0, A.plane[0], t < L::ITEMS ? t : L::ITEMS - 1);
    __syncthreads();
    tail_park<T, NX0 / 2>(A, 1, s, t, n.Xc);
    n.run(A, s, t, R, ainv);
  }
}

}  // namespace hk
