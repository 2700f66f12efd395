// Fused multigrid tail of the vertex-centred scheme (sm_103a): the V(nu1, nu2)
// cycle on a coarse vertex grid of NX0 x NX0/2 elements (32, 16 or 8 wide) and
// everything below it, one CTA per sample.
//
// A vertex level costs 4 colours x (nu1 + nu2) half-steps and four grid
// transfers, each dependent on the one before: 19 launches a level for V(2,2),
// most of them of a few hundred vertices.  Here they are phases between
// barriers, built like henry_tail.cuh: two threads per vertex (one per row of
// its blocks; thread t has vertex t/2 of each of the four colours, so the
// restriction and prolongation use the same map), x with a halo of zeros in
// shared memory, every block row read once per launch into the thread's own
// shared-memory slots - except on the 32 x 16 grid, whose rows (196 KB in
// FP64) do not fit and are read through L2 at each use.  A phase is 18 dependent
// operations (36 with one thread per vertex), which in FP64 take 64 cycles
// each.  The arithmetic and its order are vc_offdiag's, k_vc_restrict's,
// k_vc_prolong_add's and k_vc_coarse_solve's: bit-identical to the
// level-by-level kernels.  Level 1, 64 samples, FP64: 188 ms, 322 ms with the
// same levels as separate kernels.
#pragma once
#include "henry_tail.cuh"
#include "henry_vc_solve.cuh"

namespace hk {

constexpr int VC_TAIL_MAX_LEVELS = 5;  // 32 x 16 .. 2 x 1 elements
struct VcTailArgs {
  const void* J[VC_TAIL_MAX_LEVELS];  // 10 block planes of plane[k]; a sample's at s stride[k]
  int64_t plane[VC_TAIL_MAX_LEVELS];
  int stride[VC_TAIL_MAX_LEVELS];
  const void* b;  // right-hand side and result of the first level
  void* x;
  const void* ainv;
  const int* active;
  int nu1, nu2;
};

// Threads of a level: two per vertex of its largest colour.
__host__ __device__ constexpr int vc_tail_items(int nx) { return 2 * (nx / 2 + 1) * (nx / 4 + 1); }
__host__ __device__ constexpr int vc_tail_threads(int nx) { return (vc_tail_items(nx) + 31) / 32 * 32; }
__host__ __device__ constexpr bool vc_tail_slots(int nx) { return nx <= 16; }  // block rows in shared memory
__host__ __device__ constexpr int vc_tail_x(int nx) { return (nx / 2 + 3) * (nx + 3); }  // with halo
__host__ __device__ constexpr int vc_tail_nv(int nx) { return (nx / 2 + 1) * (nx + 1); }
__host__ __device__ constexpr int vc_tail_size(int nx) {  // x, residual, b, slots
  return 2 * vc_tail_x(nx) + vc_tail_nv(nx) + (vc_tail_slots(nx) ? 40 * vc_tail_items(nx) : 0);
}
__host__ __device__ constexpr int vc_tail_smem_v2(int nx0) {
  int o = 0;
  for (int nx = nx0; nx >= 4; nx /= 2) o += vc_tail_size(nx);
  return o + vc_tail_x(2) + vc_tail_nv(2);
}

template <typename T, int NX, bool FIRST>
struct VcTailLevel {
  typedef typename VT<T>::v2 V2;
  typedef typename VT<T>::b4 B4;
  static constexpr int NXV = NX + 1, NYV = NX / 2 + 1, P = NX + 3, PC = NX / 2 + 3;
  static constexpr int ITEMS = vc_tail_items(NX), NTL = vc_tail_threads(NX);
  static constexpr bool SLOTS = vc_tail_slots(NX);
  V2 *X, *R, *Bs, *Op, *Xc, *Bc;

  __device__ __forceinline__ void place(V2* base) {
    X = base;
    R = X + vc_tail_x(NX);
    Bs = R + vc_tail_x(NX);
    Op = Bs + vc_tail_nv(NX);
    Xc = base + vc_tail_size(NX);
    Bc = Xc + (NX == 4 ? vc_tail_x(2) : 2 * vc_tail_x(NX / 2));
  }
  // Vertex u of colour col: (i, j); false if the colour has fewer.
  static __device__ __forceinline__ bool vertex(int col, int u, int& i, int& j) {
    const int ci = col & 1, cj = col >> 1;
    const int nc = ci ? NX / 2 : NX / 2 + 1, nr = cj ? NX / 4 : NX / 4 + 1;
    const int r = u / nc;
    i = ci + 2 * (u - r * nc);
    j = cj + 2 * r;
    return r < nr;
  }
  static __device__ __forceinline__ int xi(int i, int j) { return (j + 1) * P + i + 1; }
  static __device__ __forceinline__ void sync() { tail_sync<NTL>(NX == 16 ? 1 : 2); }

  // Block rows of the thread's four vertices: slots q = 0..8 the neighbours
  // (4: the centre), 9 the inverse.
  static __device__ __forceinline__ const V2* rows(const VcTailArgs& A, int k, int s, int i, int j, int row) {
    const B4* J = reinterpret_cast<const B4*>(A.J[k]) + (int64_t)s * A.stride[k] + vst(j, i, NXV);
    return reinterpret_cast<const V2*>(J) + row;
  }
  __device__ __forceinline__ void fill_slots(const VcTailArgs& A, int k, int s, int t) const {
    if constexpr (SLOTS) {
      if (t >= ITEMS) return;
#pragma unroll
      for (int col = 0; col < 4; ++col) {
        int i, j;
        if (!vertex(col, t >> 1, i, j)) continue;
        const V2* p = rows(A, k, s, i, j, t & 1);
#pragma unroll
        for (int q = 0; q < 10; ++q) Op[(10 * col + q) * ITEMS + t] = p[2 * q * A.plane[k]];
      }
    }
  }

  struct My {  // the thread's vertices
    int i[4], j[4];
    bool on[4];
    T b[4];
  };
  __device__ __forceinline__ V2 blk(const VcTailArgs& A, int k, int s, int t, int row, const My& m, int col,
                                    int q) const {
    if constexpr (SLOTS) return Op[(10 * col + q) * ITEMS + t];
    else return rows(A, k, s, m.i[col], m.j[col], row)[2 * q * A.plane[k]];
  }
  template <bool CENTRE>
  __device__ __forceinline__ T offdiag(const VcTailArgs& A, int k, int s, int t, int row, const My& m, int col,
                                       T r) const {
    const V2* x = X + xi(m.i[col], m.j[col]);
    V2 a[9];
#pragma unroll
    for (int q = 0; q < 9; ++q)
      if (CENTRE || q != 4) a[q] = blk(A, k, s, t, row, m, col, q);
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      if (!CENTRE && q == 4) continue;
      const V2 xn = x[(q / 3 - 1) * P + q % 3 - 1];
      r = fma_(-a[q].x, xn.x, fma_(-a[q].y, xn.y, r));
    }
    return r;
  }
  __device__ __forceinline__ void sweep(const VcTailArgs& A, int k, int s, int t, int row, const My& m,
                                        int col) const {
    const T r = offdiag<false>(A, k, s, t, row, m, col, m.b[col]);
    const T o = __shfl_xor_sync(0xffffffffu, r, 1);
    const V2 c = blk(A, k, s, t, row, m, col, 9);
    const T y = fma_(c.x, row ? o : r, c.y * (row ? r : o));
    if (m.on[col]) reinterpret_cast<T*>(X + xi(m.i[col], m.j[col]))[row] = y;
    sync();
  }

  // Level k of A; threads t < NTL.  mrow: the thread's row of the coarsest inverse.
  __device__ __forceinline__ void run(const VcTailArgs& A, int k, int s, int t, const T* mrow) const {
    const int tt = t < ITEMS ? t : ITEMS - 1, row = tt & 1;
    My m;
#pragma unroll
    for (int col = 0; col < 4; ++col) {
      m.on[col] = vertex(col, tt >> 1, m.i[col], m.j[col]) && t < ITEMS;
      if (!m.on[col]) vertex(col, 0, m.i[col], m.j[col]);  // read along with the first vertex
    }
    // (the slots of vertices the thread does not have hold the zeros of the initial
    // clear, and nothing is stored for them)
    const V2* bg = reinterpret_cast<const V2*>(A.b) + (int64_t)s * A.stride[0];
    if constexpr (FIRST) grid_enter();
#pragma unroll
    for (int col = 0; col < 4; ++col) {
      if constexpr (FIRST) m.b[col] = reinterpret_cast<const T*>(bg + vst(m.j[col], m.i[col], NXV))[row];
      else m.b[col] = reinterpret_cast<const T*>(Bs + m.j[col] * NXV + m.i[col])[row];
    }
    for (int it = 0; it < A.nu1; ++it)
#pragma unroll
      for (int col = 0; col < 4; ++col) sweep(A, k, s, tt, row, m, col);
    // residual of every vertex, then full weighting onto the coarse ones
#pragma unroll
    for (int col = 0; col < 4; ++col) {
      const T r = offdiag<true>(A, k, s, tt, row, m, col, m.b[col]);
      if (m.on[col]) reinterpret_cast<T*>(R + xi(m.i[col], m.j[col]))[row] = r;
    }
    sync();
    constexpr int NCV = NX / 2 + 1, NVC = NCV * (NX / 4 + 1);  // coarse vertices: those of colour 0
    if (t < 2 * NVC) {
      const int v = t >> 1, Jc = v / NCV, Ic = v - Jc * NCV;
      T sum = (T)0;
#pragma unroll
      for (int a = -1; a <= 1; ++a)
#pragma unroll
        for (int b = -1; b <= 1; ++b) {
          const T w = (T)((a == 0 ? 1.0 : 0.5) * (b == 0 ? 1.0 : 0.5));
          sum = fma_(w, reinterpret_cast<const T*>(R + xi(2 * Ic + b, 2 * Jc + a))[t & 1], sum);
        }
      if (Ic == NX / 2 || (Ic == 0 && (t & 1))) sum = (T)0;  // Dirichlet equations
      reinterpret_cast<T*>(Bc + Jc * NCV + Ic)[t & 1] = sum;
    }
    sync();
    if constexpr (NX == 4) {  // the 2 x 1 element grid: one row of the dense inverse per thread
      if (t < VC_COARSE_N) {
        const T* v = reinterpret_cast<const T*>(Bc);
        T acc = (T)0;
#pragma unroll
        for (int c = 0; c < VC_COARSE_N; ++c) acc = fma_(mrow[c], v[c], acc);
        const int u = t >> 1, j = u / 3, i = u - 3 * j;
        reinterpret_cast<T*>(Xc + (j + 1) * PC + i + 1)[t & 1] = acc;
      }
    } else {
      typedef VcTailLevel<T, NX / 2, false> Next;
      if (t < Next::NTL) {
        Next n;
        n.place(Xc);
        n.run(A, k + 1, s, t, mrow);
      }
    }
    sync();
    // x += P x_c
#pragma unroll
    for (int col = 0; col < 4; ++col) {
      if (!m.on[col]) continue;
      const T* c = reinterpret_cast<const T*>(Xc + ((m.j[col] >> 1) + 1) * PC + (m.i[col] >> 1) + 1) + row;
      T sum = c[0];
      if (col & 1) sum += c[2];
      if (col >> 1) {
        sum += c[2 * PC];
        if (col & 1) sum += c[2 * PC + 2];
      }
      const T w = (T)(((col >> 1) ? 0.5 : 1.0) * ((col & 1) ? 0.5 : 1.0));
      T* xp = reinterpret_cast<T*>(X + xi(m.i[col], m.j[col])) + row;
      *xp = fma_(w, sum, *xp);
    }
    sync();
    for (int it = 0; it < A.nu2; ++it)
#pragma unroll
      for (int col = 3; col >= 0; --col) sweep(A, k, s, tt, row, m, col);
    if constexpr (FIRST) {
      V2* xg = reinterpret_cast<V2*>(A.x) + (int64_t)s * A.stride[0];
#pragma unroll
      for (int col = 0; col < 4; ++col)
        if (m.on[col])
          reinterpret_cast<T*>(xg + vst(m.j[col], m.i[col], NXV))[row] =
              reinterpret_cast<const T*>(X + xi(m.i[col], m.j[col]))[row];
    }
  }
};

template <typename T, int NX>
__device__ __forceinline__ void vc_tail_fill(const VcTailArgs& A, int k, int s, int t, typename VT<T>::v2* base) {
  if constexpr (NX >= 4) {
    VcTailLevel<T, NX, false> n;
    n.place(base);
    n.fill_slots(A, k, s, t);
    vc_tail_fill<T, NX / 2>(A, k + 1, s, t, base + vc_tail_size(NX));
  }
}

template <typename T, int NX0>
__global__ void __launch_bounds__(vc_tail_threads(NX0)) k_vc_tail(const __grid_constant__ VcTailArgs A, int B) {
  typedef typename VT<T>::v2 V2;
  constexpr int NT = vc_tail_threads(NX0);
  extern __shared__ __align__(16) unsigned char vc_tail_mem[];
  V2* sm = reinterpret_cast<V2*>(vc_tail_mem);
  const int s = blockIdx.x, t = threadIdx.x;
  if (s >= B || !A.active[s]) {
    grid_enter();
    return;
  }
  for (int i = t; i < vc_tail_smem_v2(NX0); i += NT) sm[i] = mk2<V2>((T)0, (T)0);
  T mrow[VC_COARSE_N];
#pragma unroll
  for (int c = 0; c < VC_COARSE_N; ++c)
    mrow[c] = t < VC_COARSE_N
                  ? reinterpret_cast<const T*>(A.ainv)[(int64_t)s * VC_COARSE_N * VC_COARSE_N + t * VC_COARSE_N + c]
                  : (T)0;
  __syncthreads();
  vc_tail_fill<T, NX0>(A, 0, s, t, sm);
  VcTailLevel<T, NX0, true> L;
  L.place(sm);
  L.run(A, 0, s, t, mrow);
}

}  // namespace hk
