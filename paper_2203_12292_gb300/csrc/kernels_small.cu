// The operator of levels with few cells: one warp per cell (several cells per
// warp at low degree) writes the cell's result vector, and one thread per DoF
// adds the entries of its cells in a fixed order, in the same pass as what
// follows the operator in the cycle (a Chebyshev step, the residual, the start
// of presmoothing on a restricted right-hand side).
//   Such a level was bound by the chain of latencies inside its kernels: tile
// record, index lists, values, five sweeps with block barriers, up to eight
// sub-colours with a barrier each, then the halo pass and the vector update as
// two more launches.  Here a kernel has one dependent load behind the
// predecessor's completion (its index lists and constants are loaded before
// it), the sweeps need warp synchronisation only, and the accumulation, the
// halo pass and the update are one launch.  The price is memory traffic: every
// cell vector is written and read once ((k+1)^3 values per cell, 2 to 8 per DoF)
// through a list of its own, which is why large levels keep their tiles.
// Q2 octant mesh (6,407 DoFs, 960 cells), fp64: the operator 17.5 -> 7.4 us, the
// solve 1.68 -> 1.09 ms; where the line lies: cell_vectors_pay.
#include <algorithm>

#include "device.cuh"
#include "kernels.h"
#include "lanes.cuh"
#include "zline.cuh"

namespace gcmg {

GCMG_DEFINE_UPLOAD(upload_tables_small_1d)

namespace {

constexpr int SWPB = 4;  // warps per block

// the z-line coefficients again: a lane reads its own line's, which constant memory would serialise
__device__ ZLines g_zl;

template <typename T>
struct CellVecArgs {
  const int32_t* gstart;
  const CellMeta* meta;
  const double* coef;
  double dom;
  int n_cells;
  const T* src;
  T* cv;  // cell vectors: node n of cell c at c (k+1)^3 + n
};

// one direction of C_e (TRANS: C_e^T) on the lane's line
template <int K, int D, bool TRANS, typename V>
__device__ __forceinline__ void cell_hang(V* cb, uint16_t m, int r, bool on) {
  constexpr int N = K + 1;
  if (on) {
    int base, u, v;
    line_geom<N, D>(r, base, u, v);
    if (line_hangs<K, D>(m, u, v)) {
      constexpr int S = line_stride<N, D>();
      V x[N];
#pragma unroll
      for (int a = 0; a < N; ++a) x[a] = cb[base + a * S];
      hang_line<K, TRANS>(x, (m >> D) & 1);
#pragma unroll
      for (int a = 0; a < N; ++a) cb[base + a * S] = x[a];
    }
  }
  __syncwarp();
}

template <int K, int D, bool FWD, typename V>
__device__ __forceinline__ void cell_sweep(V* cb, int r, bool on) {
  constexpr int N = K + 1, S = line_stride<N, D>();
  if (on) {
    int base, u, v;
    line_geom<N, D>(r, base, u, v);
    V x[N];
#pragma unroll
    for (int a = 0; a < N; ++a) x[a] = cb[base + a * S];
    eo_line<K, FWD, (K >= 3)>(x);  // normalised pairs at k >= 3: df_add_step
#pragma unroll
    for (int a = 0; a < N; ++a) cb[base + a * S] = x[a];
  }
  __syncwarp();
}

template <int K, typename T>
__global__ void __launch_bounds__(SWPB * 32) cell_vectors(CellVecArgs<T> A) {
  using AR = Arith<T>;
  using V = typename AR::V;
  constexpr int N = K + 1, N2 = N * N, N3 = N2 * N;
  constexpr int CPW = 32 / N2;                    // cells per warp: 8, 3, 2, 1
  constexpr int NJ = (CPW * N3 + 31) / 32;        // nodes per lane
  __shared__ V s_cb[SWPB][CPW * N3];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int c0 = (blockIdx.x * SWPB + w) * CPW;   // the warp's first cell
  const int nc = min(CPW, A.n_cells - c0);        // <= 0: an idle warp
  V* cb = s_cb[w];
  int idx[NJ];
#pragma unroll
  for (int i = 0; i < NJ; ++i) {
    const int t = lane + 32 * i, q = t / N3, n = t - q * N3;
    idx[i] = -1;
    if (q < nc) {
      int slot, off;
      node_slot<K>(n % N, (n / N) % N, n / N2, slot, off);
      const int32_t g = A.gstart[(size_t)(c0 + q) * NSLOT + slot];
      if (g >= 0) idx[i] = g + off;
    }
  }
  const int q = lane / N2, r = lane - q * N2;     // the lane's cell and line
  const bool on = q < nc;
  uint16_t m = 0;
  constexpr int NC = zline_count(K) + 1;
  // K + (lam_a + lam_b) M on the z-line (a, b) = r
  float zh[NC], zl[sizeof(T) == 8 ? NC : 1];
  V h = V(0);
  if (on) {
    const CellMeta& cm = A.meta[c0 + q];
    m = cm.mask;
    double hd = ldexp(A.dom, -(int)cm.level);
    if (A.coef) hd *= A.coef[c0 + q];
    h = V(hd);
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      zh[i] = g_zl.h[zline_row(K) + r][i];
      if (sizeof(T) == 8) zl[i] = g_zl.l[zline_row(K) + r][i];
    }
  }
  const bool hang = __any_sync(0xffffffffu, (m & MASK_HANG) != 0);
  pdl_wait();
  {
    T x[NJ];
#pragma unroll
    for (int i = 0; i < NJ; ++i) x[i] = idx[i] >= 0 ? A.src[idx[i]] : T(0);
#pragma unroll
    for (int i = 0; i < NJ; ++i)
      if (lane + 32 * i < CPW * N3) cb[lane + 32 * i] = AR::in(x[i]);
  }
  __syncwarp();
  V* cl = cb + (on ? q : 0) * N3;
  if (hang) {
    cell_hang<K, 0, false>(cl, m, r, on);
    cell_hang<K, 1, false>(cl, m, r, on);
    cell_hang<K, 2, false>(cl, m, r, on);
  }
  cell_sweep<K, 0, true>(cl, r, on);
  cell_sweep<K, 1, true>(cl, r, on);
  if (on) {
    V x[N];
#pragma unroll
    for (int c = 0; c < N; ++c) x[c] = cl[r + N2 * c];
    if constexpr (sizeof(T) == 8)
      zline<K, (K >= 3)>(x, zh, zl, r == 0);
    else
      zline<K>(x, zh, true);
#pragma unroll
    for (int c = 0; c < N; ++c) x[c] = x[c] * h;
#pragma unroll
    for (int c = 0; c < N; ++c) cl[r + N2 * c] = x[c];
  }
  __syncwarp();
  cell_sweep<K, 1, false>(cl, r, on);
  cell_sweep<K, 0, false>(cl, r, on);
  if (hang) {
    cell_hang<K, 2, true>(cl, m, r, on);
    cell_hang<K, 1, true>(cl, m, r, on);
    cell_hang<K, 0, true>(cl, m, r, on);
  }
#pragma unroll
  for (int i = 0; i < NJ; ++i)
    if (lane + 32 * i < nc * N3) A.cv[(size_t)c0 * N3 + lane + 32 * i] = AR::out(cb[lane + 32 * i]);
}

// the pass over the DoFs: s = the sum of DoF i's cell-vector entries, then
enum SumOp {
  SUM_STORE,  // y = s
  SUM_ADD,    // y += s
  SUM_RESIDUAL,  // y = b - s
  SUM_CHEB,      // d = c1 d + c2 dinv (b - s), x += d
  SUM_CHEB_X,    // the same with d = x on entry (the step after the start from zero)
  SUM_CHEB_1,    // d = c2 dinv (b - s), x += d
  SUM_START      // b = s, x = c2 dinv b
};
template <typename T>
struct SumArgs {
  const int32_t* ptr;
  const int32_t* pos;
  int n;
  const T* cv;
  T* y;
  const T* b;
  T* x;
  const T* d;
  T* dw;  // d's new value (null: the last step of a smoother, not needed again)
  const T* dinv;
  T c1, c2;
};

template <typename T, int OP>
__global__ void __launch_bounds__(128) cell_sum(SumArgs<T> A) {
  constexpr int PRE = 4;  // list entries loaded ahead of the predecessor's completion
  const int i = blockIdx.x * 128 + threadIdx.x;
  const bool in = i < A.n;
  int e0 = 0, e1 = 0, p[PRE];
  T di = T(0);
  if (in) {
    e0 = A.ptr[i];
    e1 = A.ptr[i + 1];
    if (OP >= SUM_CHEB) di = A.dinv[i];
  }
#pragma unroll
  for (int u = 0; u < PRE; ++u) p[u] = e0 + u < e1 ? A.pos[e0 + u] : -1;
  pdl_wait();
  if (!in) return;
  T v[PRE];
#pragma unroll
  for (int u = 0; u < PRE; ++u) v[u] = p[u] >= 0 ? A.cv[p[u]] : T(0);
  T b = T(0), x = T(0), d = T(0);
  if (OP == SUM_RESIDUAL || OP == SUM_CHEB || OP == SUM_CHEB_X || OP == SUM_CHEB_1) b = A.b[i];
  if (OP == SUM_CHEB || OP == SUM_CHEB_X || OP == SUM_CHEB_1) x = A.x[i];
  if (OP == SUM_CHEB) d = A.d[i];
  if (OP == SUM_ADD) x = A.y[i];
  T s = v[0];
#pragma unroll
  for (int u = 1; u < PRE; ++u)
    if (p[u] >= 0) s += v[u];
  for (int e = e0 + PRE; e < e1; ++e) s += A.cv[A.pos[e]];
  if (OP == SUM_STORE) {
    A.y[i] = s;
  } else if (OP == SUM_ADD) {
    A.y[i] = x + s;
  } else if (OP == SUM_RESIDUAL) {
    A.y[i] = b - s;
  } else if (OP == SUM_START) {
    A.y[i] = s;
    A.x[i] = A.c2 * di * s;
  } else {
    if (OP == SUM_CHEB_X) d = x;
    const T r = b - s;
    const T dn = OP == SUM_CHEB_1 ? A.c2 * di * r : A.c1 * d + A.c2 * di * r;
    if (A.dw) A.dw[i] = dn;
    A.x[i] = x + dn;
  }
}

template <typename T>
void run_cells(const CellLaunch& L, const T* src, cudaStream_t s) {
  CellVecArgs<T> A{L.gstart, L.meta, L.coef, L.dom, L.n_cells, src, static_cast<T*>(L.cell_vec)};
#define GCMG_RUN(K)                                                                                         \
  case K: {                                                                                                 \
    constexpr int CPB = SWPB * (32 / ((K + 1) * (K + 1)));                                                  \
    launch_pdl(cell_vectors<K, T>, (L.n_cells + CPB - 1) / CPB, SWPB * 32, 0, s, A);                        \
  } break;
  switch (L.k) { GCMG_RUN(1) GCMG_RUN(2) GCMG_RUN(3) GCMG_RUN(4) }
#undef GCMG_RUN
  note_launches(1);
}

template <typename T>
SumArgs<T> sum_args(const CellLaunch& L) {
  SumArgs<T> A{};
  A.ptr = L.sum_ptr;
  A.pos = L.sum_pos;
  A.n = L.n_dofs;
  A.cv = static_cast<const T*>(L.cell_vec);
  return A;
}

template <int OP, typename T>
void run_sum(const SumArgs<T>& A, cudaStream_t s) {
  launch_pdl(cell_sum<T, OP>, (A.n + 127) / 128, 128, 0, s, A);
  note_launches(1);
}

template <typename T>
void run_store(const CellLaunch& L, T* dst, bool add, cudaStream_t s) {
  SumArgs<T> A = sum_args<T>(L);
  A.y = dst;
  if (add)
    run_sum<SUM_ADD>(A, s);
  else
    run_sum<SUM_STORE>(A, s);
}

template <typename T>
void run_residual(const CellLaunch& L, const T* b, T* r, cudaStream_t s) {
  SumArgs<T> A = sum_args<T>(L);
  A.y = r;
  A.b = b;
  run_sum<SUM_RESIDUAL>(A, s);
}

template <typename T>
void run_cheb(const CellLaunch& L, int step, bool last, T* x, T* d, const T* b, const T* dinv, double c1, double c2,
              cudaStream_t s) {
  SumArgs<T> A = sum_args<T>(L);
  A.x = x;
  A.d = d;
  A.b = b;
  A.dinv = dinv;
  A.c1 = (T)c1;
  A.c2 = (T)c2;
  A.dw = last ? nullptr : d;
  if (step == CHEB_NEXT)
    run_sum<SUM_CHEB>(A, s);
  else if (step == CHEB_AFTER_ZERO)
    run_sum<SUM_CHEB_X>(A, s);
  else
    run_sum<SUM_CHEB_1>(A, s);
}

template <typename T>
void run_start(const CellLaunch& L, T* b, T* x, const T* dinv, double c2, cudaStream_t s) {
  SumArgs<T> A = sum_args<T>(L);
  A.y = b;
  A.x = x;
  A.dinv = dinv;
  A.c2 = (T)c2;
  run_sum<SUM_START>(A, s);
}

}  // namespace

void upload_tables_small() {
  upload_tables_small_1d();
  static LaneLines ll;
  fill_lane_lines(ll);
  cudaMemcpyToSymbol(c_ll, &ll, sizeof(ll));
  upload_zlines();
  static ZLines z;
  cudaMemcpyFromSymbol(&z, c_zl, sizeof(z));
  cudaMemcpyToSymbol(g_zl, &z, sizeof(z));
}

// recorded launch lists (the persistent batch) keep the tile kernels
bool cells_ok(const CellLaunch& L) { return L.sum_ptr && !L.geom && !dwl_recording(); }

void launch_cell_vectors(const CellLaunch& L, bool fp64, const void* src, cudaStream_t s) {
  if (fp64)
    run_cells(L, static_cast<const double*>(src), s);
  else
    run_cells(L, static_cast<const float*>(src), s);
}

void launch_cell_sum(const CellLaunch& L, bool fp64, void* dst, bool add, cudaStream_t s) {
  if (fp64)
    run_store(L, static_cast<double*>(dst), add, s);
  else
    run_store(L, static_cast<float*>(dst), add, s);
}

void launch_cell_sum_residual(const CellLaunch& L, bool fp64, const void* b, void* r, cudaStream_t s) {
  if (fp64)
    run_residual(L, static_cast<const double*>(b), static_cast<double*>(r), s);
  else
    run_residual(L, static_cast<const float*>(b), static_cast<float*>(r), s);
}

void launch_cell_sum_cheb(const CellLaunch& L, bool fp64, int step, bool last, void* x, void* d, const void* b,
                          const void* dinv, double c1, double c2, cudaStream_t s) {
  if (fp64)
    run_cheb(L, step, last, static_cast<double*>(x), static_cast<double*>(d), static_cast<const double*>(b),
             static_cast<const double*>(dinv), c1, c2, s);
  else
    run_cheb(L, step, last, static_cast<float*>(x), static_cast<float*>(d), static_cast<const float*>(b),
             static_cast<const float*>(dinv), c1, c2, s);
}

void launch_cell_sum_start(const CellLaunch& L, bool fp64, void* b, void* x, const void* dinv, double c2,
                           cudaStream_t s) {
  if (fp64)
    run_start(L, static_cast<double*>(b), static_cast<double*>(x), static_cast<const double*>(dinv), c2, s);
  else
    run_start(L, static_cast<float*>(b), static_cast<float*>(x), static_cast<const float*>(dinv), c2, s);
}

}  // namespace gcmg
