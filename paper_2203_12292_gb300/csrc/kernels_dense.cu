// The V-cycle of the smallest levels as one dense matrix.
//
// With the Chebyshev smoother the V-cycle of level l is a fixed linear map
// x = M_l b (Algorithm 2 with the exact solve M_0 = A_0^{-1}).  On levels of at
// most DENSE_MAX DoFs it was bound by latency alone: 21 launches per level and
// cycle, each a chain of dependent loads on a handful of blocks.  The set-up
// builds M_l once, in fp64 and in a fixed order, from the level operators,
// their Jacobi diagonals, the Chebyshev coefficients and the prolongations:
//   X = p_pre(A) b, X += P M_{l-1} P^T (1 - A X), postsmoothing,  b = identity
// and a cycle applies it as one matrix-vector product.  The matrix and the sums
// are fp64 for fp32 levels too, rounded once into x: the exact solve on level 0
// in it was fp64 level by level, and an fp32 matrix with fp32 sums lost that.
// Q2 octant mesh (6,407 DoFs; the levels up to 659 DoFs in the matrix), solve
// with fp64 V-cycle: 3.36 -> 1.69 ms; batch of 16 problems 14.9 -> 11.2 ms.  The
// matrix of 659 DoFs costs 0.9 ms of set-up.  DENSE_MAX: at 927 DoFs the
// product takes 7.1 us for an fp32 level (3.5 with an fp32 matrix and sums) and 5.8
// for an fp64 one, against 50 to 110 us level by level; beyond it the set-up's
// products (n^2 row lengths) grow faster than the gain.
#include <algorithm>

#include "device.cuh"
#include "kernels.h"

namespace gcmg {

GCMG_DEFINE_UPLOAD(upload_tables_dense_1d)

namespace {

constexpr int DCB = 8;  // cells per pass of the pipeline

template <int K>
__device__ __forceinline__ int slot_dofs(int s) {
  int n = 1;
  if (s % 3 == 1) n *= K - 1;
  if ((s / 3) % 3 == 1) n *= K - 1;
  if (s / 9 == 1) n *= K - 1;
  return n;
}

// local node of offset `off` in slot s
template <int K>
__device__ __forceinline__ int slot_node(int s, int off) {
  constexpr int N = K + 1;
  int x[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int c = d == 0 ? s % 3 : (d == 1 ? (s / 3) % 3 : s / 9);
    x[d] = c == 0 ? 0 : K;
    if (c == 1) {
      x[d] = 1 + off % (K > 1 ? K - 1 : 1);
      off /= (K > 1 ? K - 1 : 1);
    }
  }
  return x[0] + N * (x[1] + N * x[2]);
}

// node of cell c at which it holds DoF j (own: only where it owns it), or -1
template <int K>
__device__ __forceinline__ int find_node(const int32_t* gs, uint32_t allowed, int j) {
  for (int s = 0; s < NSLOT; ++s) {
    const int g = gs[s];
    if (g < 0 || j < g || !((allowed >> s) & 1u)) continue;
    const int nd = slot_dofs<K>(s);
    if (j < g + nd) return slot_node<K>(s, j - g);
  }
  return -1;
}

// row j of A (block j): the cells that hold DoF j, in cell order, DCB at a time
// through the cell pipeline on the unit vector of their node
template <int K>
__global__ void __launch_bounds__(BLOCK) dense_operator(int n, int nc, const int32_t* gstart, const CellMeta* meta,
                                                        const double* coef, double dom, double* A) {
  pdl_begin();
  constexpr int N = K + 1, N3 = N * N * N;
  __shared__ double cb[DCB * N3], sm_h[DCB];
  __shared__ uint16_t sm_mask[DCB];
  __shared__ int s_node[BLOCK], s_list[BLOCK], s_n;
  __shared__ unsigned s_ball[BLOCK / 32];
  const int j = blockIdx.x, tid = threadIdx.x;
  double* row = A + (size_t)j * n;
  for (int i = tid; i < n; i += BLOCK) row[i] = 0.0;
  for (int c0 = 0; c0 < nc; c0 += BLOCK) {
    const int c = c0 + tid;
    const int node = c < nc ? find_node<K>(gstart + (size_t)c * NSLOT, 0x7ffffffu, j) : -1;
    s_node[tid] = node;
    const unsigned ball = __ballot_sync(0xffffffffu, node >= 0);
    if ((tid & 31) == 0) s_ball[tid >> 5] = ball;
    __syncthreads();
    if (tid == 0) {
      int k = 0;
      for (int w = 0; w < BLOCK / 32; ++w)
        for (unsigned m = s_ball[w]; m; m &= m - 1) s_list[k++] = 32 * w + __ffs(m) - 1;
      s_n = k;
    }
    __syncthreads();
    for (int b = 0; b < s_n; b += DCB) {
      const int nb = min(DCB, s_n - b);
      for (int t = tid; t < nb * N3; t += BLOCK) cb[t] = (t % N3 == s_node[s_list[b + t / N3]]) ? 1.0 : 0.0;
      if (tid < nb) {
        const int cc = c0 + s_list[b + tid];
        sm_mask[tid] = meta[cc].mask;
        const double h = ldexp(dom, -(int)meta[cc].level);
        sm_h[tid] = coef ? h * coef[cc] : h;
      }
      __syncthreads();
      hanging_all<K, false>(cb, sm_mask, nb);
      cell_laplace<K>(cb, sm_h, nb);
      hanging_all<K, true>(cb, sm_mask, nb);
      for (int q = 0; q < nb; ++q) {  // one cell after another: a fixed order of additions
        const int32_t* gs = gstart + (size_t)(c0 + s_list[b + q]) * NSLOT;
        for (int t = tid; t < N3; t += BLOCK) {
          int slot, off;
          node_slot<K>(t % N, (t / N) % N, t / (N * N), slot, off);
          const int g = gs[slot];
          if (g >= 0) row[g + off] += cb[q * N3 + t];
        }
        __syncthreads();
      }
    }
    __syncthreads();
  }
}

// row i of the prolongation (block i, n_c columns): the owner of fine DoF i and
// its coarse cell; weights of the coarse nodes, then C^T
template <int KF, int KC>
__global__ void __launch_bounds__(BLOCK) dense_prolongation(int n_c, int ncf, const int32_t* gstart_f,
                                                            const uint32_t* own_f, int ncc, const int32_t* fine_of,
                                                            const uint8_t* refined, const int32_t* gstart_c,
                                                            const uint16_t* mask_c, double* P) {
  pdl_begin();
  constexpr int NF = KF + 1, N = KC + 1, N3 = N * N * N;
  __shared__ double cb[N3];
  __shared__ uint16_t sm_mask[1];
  __shared__ int s_f, s_node, s_c;
  const int i = blockIdx.x, tid = threadIdx.x;
  double* row = P + (size_t)i * n_c;
  for (int t = tid; t < n_c; t += BLOCK) row[t] = 0.0;
  for (int f = tid; f < ncf; f += BLOCK) {
    const int node = find_node<KF>(gstart_f + (size_t)f * NSLOT, own_f[f], i);
    if (node >= 0) {  // exactly one cell owns it
      s_f = f;
      s_node = node;
    }
  }
  __syncthreads();
  for (int c = tid; c < ncc; c += BLOCK) {
    const int f0 = KF == KC ? fine_of[c] : c;
    const int nf = KF == KC && refined[c] ? 8 : 1;
    if (f0 >= 0 && s_f >= f0 && s_f < f0 + nf) s_c = c;
  }
  __syncthreads();
  const int c = s_c;
  const int a = s_node % NF, b = (s_node / NF) % NF, d = s_node / (NF * NF);
  for (int t = tid; t < N3; t += BLOCK) {
    const int x = t % N, y = (t / N) % N, z = t / (N * N);
    const DevTables<double>& tb = tab<double>(KF);
    if (KF != KC) {
      cb[t] = tb.Pp[a][x] * tb.Pp[b][y] * tb.Pp[d][z];
    } else if (refined[c]) {
      const int q = s_f - fine_of[c];
      cb[t] = tb.Ph[(q & 1) * KF + a][x] * tb.Ph[((q >> 1) & 1) * KF + b][y] * tb.Ph[(q >> 2) * KF + d][z];
    } else {
      cb[t] = t == s_node ? 1.0 : 0.0;
    }
  }
  if (tid == 0) sm_mask[0] = mask_c[c];
  __syncthreads();
  hanging_all<KC, true>(cb, sm_mask, 1);
  for (int t = tid; t < N3; t += BLOCK) {
    int slot, off;
    node_slot<KC>(t % N, (t / N) % N, t / (N * N), slot, off);
    const int g = gstart_c[(size_t)c * NSLOT + slot];
    if (g >= 0) row[g + off] = cb[t];
  }
}

__global__ void __launch_bounds__(BLOCK) dense_init(int n, const double* dinv, double c2, double* X, double* D) {
  pdl_begin();
  const int64_t t = blockIdx.x * (int64_t)BLOCK + threadIdx.x;
  if (t >= (int64_t)n * n) return;
  const int i = (int)(t / n), c = (int)(t % n);
  const double v = i == c ? c2 * dinv[i] : 0.0;
  X[t] = v;
  D[t] = v;
}

enum DenseMode { DENSE_PRODUCT, DENSE_ADD, DENSE_RESIDUAL, DENSE_CHEB };
struct DenseProduct {
  const double* A;  // A(i, k) at A[i si + k sk], zeros skipped
  int64_t si, sk;
  int nk;
  const double* B;  // nk x n
  int n;            // columns
  // PRODUCT: C = A B; ADD: C = C + A B; RESIDUAL: C = 1 - A B; CHEB:
  // D = c1 D + c2 dinv (1 - A B), C = B + D (first: c1 = 0, D not read)
  int mode, first;
  double* C;
  double* D;
  const double* dinv;
  double c1, c2;
};

// row i (blockIdx.x), BLOCK columns (blockIdx.y): the row's nonzeros are listed
// in shared memory, BLOCK at a time, in increasing k
__global__ void __launch_bounds__(BLOCK) dense_product(DenseProduct G) {
  pdl_begin();
  __shared__ double s_v[BLOCK];
  __shared__ int s_k[BLOCK];
  __shared__ int s_cnt[BLOCK / 32];
  const int i = blockIdx.x, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int c = blockIdx.y * BLOCK + tid;
  const bool in = c < G.n;
  double s = 0.0;
  for (int k0 = 0; k0 < G.nk; k0 += BLOCK) {
    const int k = k0 + tid;
    const double a = k < G.nk ? G.A[i * G.si + k * G.sk] : 0.0;
    const unsigned ball = __ballot_sync(0xffffffffu, a != 0.0);
    if (lane == 0) s_cnt[w] = __popc(ball);
    __syncthreads();
    int at = 0, total = 0;
    for (int q = 0; q < BLOCK / 32; ++q) {
      if (q < w) at += s_cnt[q];
      total += s_cnt[q];
    }
    if (a != 0.0) {
      at += __popc(ball & ((1u << lane) - 1u));
      s_v[at] = a;
      s_k[at] = k;
    }
    __syncthreads();
    if (in) {
#pragma unroll 4
      for (int e = 0; e < total; ++e) s += s_v[e] * G.B[(size_t)s_k[e] * G.n + c];
    }
    __syncthreads();
  }
  if (!in) return;
  const size_t t = (size_t)i * G.n + c;
  const double r = (i == c ? 1.0 : 0.0) - s;
  if (G.mode == DENSE_PRODUCT) {
    G.C[t] = s;
  } else if (G.mode == DENSE_ADD) {
    G.C[t] += s;
  } else if (G.mode == DENSE_RESIDUAL) {
    G.C[t] = r;
  } else {
    const double d = G.first ? G.c2 * G.dinv[i] * r : G.c1 * G.D[t] + G.c2 * G.dinv[i] * r;
    G.D[t] = d;
    G.C[t] = G.B[t] + d;
  }
}

// x = M b, one warp per row, a lane's partial sums and the lanes in a fixed order.
// The first 256 entries of the rows are loaded before the predecessor's completion
// (the matrix is set-up data); an fp32 b is widened once per block, since a
// conversion costs as much as a product on the FP64 pipe.
constexpr int DROWS = 4;  // rows (warps) per block
template <typename T>
__global__ void __launch_bounds__(DROWS * 32) dense_apply(const double* __restrict__ M, int n,
                                                          const T* __restrict__ b, T* __restrict__ x) {
  constexpr bool WIDEN = sizeof(T) == 4;
  __shared__ double sb[WIDEN ? DENSE_MAX : 1];
  const int i = blockIdx.x * DROWS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const double* row = M + (size_t)min(i, n - 1) * n;
  double m[8], s[8] = {};
#pragma unroll
  for (int u = 0; u < 8; ++u) m[u] = lane + 32 * u < n ? row[lane + 32 * u] : 0.0;
  pdl_wait();
  if constexpr (WIDEN) {
    for (int k = threadIdx.x; k < n; k += DROWS * 32) sb[k] = (double)b[k];
    __syncthreads();
  }
  auto in = [&](int k) -> double {
    if constexpr (WIDEN)
      return sb[k];
    else
      return b[k];
  };
  for (int k = lane; k < n; k += 8 * 32) {
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (k + 32 * u < n) s[u] += m[u] * in(k + 32 * u);
#pragma unroll
    for (int u = 0; u < 8; ++u) m[u] = k + 32 * (u + 8) < n ? row[k + 32 * (u + 8)] : 0.0;
  }
  double v = ((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]));
#pragma unroll
  for (int h = 16; h > 0; h >>= 1) v += __shfl_down_sync(0xffffffffu, v, h);
  if (lane == 0 && i < n) x[i] = (T)v;
}

void product(const DenseProduct& G, int rows, cudaStream_t s) {
  launch_pdl(dense_product, dim3(rows, (G.n + BLOCK - 1) / BLOCK), BLOCK, 0, s, G);
  note_launches(1);
}

}  // namespace

void upload_tables_dense() { upload_tables_dense_1d(); }

void launch_dense_operator(const CellLaunch& L, int n, int n_cells, const int32_t* gstart, double* A, cudaStream_t s) {
#define GCMG_RUN(K) \
  case K: launch_pdl(dense_operator<K>, n, BLOCK, 0, s, n, n_cells, gstart, L.meta, L.coef, L.dom, A); break;
  switch (L.k) { GCMG_RUN(1) GCMG_RUN(2) GCMG_RUN(3) GCMG_RUN(4) }
#undef GCMG_RUN
  note_launches(1);
}

void launch_dense_prolongation(const TransferLaunch& T, int n_f, int n_c, int cells_f, double* P, cudaStream_t s) {
#define GCMG_RUN(KF, KC)                                                                                           \
  launch_pdl(dense_prolongation<KF, KC>, n_f, BLOCK, 0, s, n_c, cells_f, T.gstart_f, T.own_f, T.n_coarse, T.fine_of, \
             T.refined, T.gstart_c, T.mask_c, P)
  if (T.kind == 0) {
    switch (T.kf) {
      case 1: GCMG_RUN(1, 1); break;
      case 2: GCMG_RUN(2, 2); break;
      case 3: GCMG_RUN(3, 3); break;
      case 4: GCMG_RUN(4, 4); break;
    }
  } else {
    switch (T.kf) {
      case 2: GCMG_RUN(2, 1); break;
      case 3: GCMG_RUN(3, 1); break;
      case 4: GCMG_RUN(4, 2); break;
    }
  }
#undef GCMG_RUN
  note_launches(1);
}

size_t dense_scratch_bytes(int n) { return (size_t)5 * n * n * sizeof(double); }

// M (n x n) of one level: coef pairs (c1, c2) of the Chebyshev steps; P, Mc of
// the coarser level (n_c = 0: no correction); work: dense_scratch_bytes(max(n, n_c))
double* dense_vcycle_matrix(int n, const double* A, const double* dinv, int steps, const double* coef, int n_c,
                            const double* P, const double* Mc, double* work, cudaStream_t s) {
  const size_t q = (size_t)std::max(n, n_c) * std::max(n, n_c);
  double *X = work, *Y = work + q, *D = work + 2 * q, *R = work + 3 * q, *Z = work + 4 * q;
  launch_pdl(dense_init, (unsigned)(((size_t)n * n + BLOCK - 1) / BLOCK), BLOCK, 0, s, n, dinv, coef[1], X, D);
  note_launches(1);
  DenseProduct G{};
  G.A = A;
  G.si = n;
  G.sk = 1;
  G.nk = n;
  G.n = n;
  G.D = D;
  G.dinv = dinv;
  auto smooth = [&](int first) {
    for (int it = first; it < steps; ++it) {
      G.mode = DENSE_CHEB;
      G.first = it == 0;
      G.c1 = coef[2 * it];
      G.c2 = coef[2 * it + 1];
      G.B = X;
      G.C = Y;
      product(G, n, s);
      std::swap(X, Y);
    }
  };
  smooth(1);
  if (n_c > 0) {
    DenseProduct r = G;  // Y = 1 - A X
    r.mode = DENSE_RESIDUAL;
    r.B = X;
    r.C = Y;
    product(r, n, s);
    DenseProduct p{};  // R = P^T Y
    p.A = P;
    p.si = 1;
    p.sk = n_c;
    p.nk = n;
    p.B = Y;
    p.n = n;
    p.mode = DENSE_PRODUCT;
    p.C = R;
    product(p, n_c, s);
    p.A = Mc;  // Z = M_c R
    p.si = n_c;
    p.sk = 1;
    p.nk = n_c;
    p.B = R;
    p.C = Z;
    product(p, n_c, s);
    p.A = P;  // X += P Z
    p.B = Z;
    p.mode = DENSE_ADD;
    p.C = X;
    product(p, n, s);
  }
  smooth(0);
  return X;
}

void launch_dense_apply(bool fp64, const double* M, int n, const void* b, void* x, cudaStream_t s) {
  if (fp64)
    launch_pdl(dense_apply<double>, (n + DROWS - 1) / DROWS, DROWS * 32, 0, s, M, n, static_cast<const double*>(b),
               static_cast<double*>(x));
  else
    launch_pdl(dense_apply<float>, (n + DROWS - 1) / DROWS, DROWS * 32, 0, s, M, n, static_cast<const float*>(b),
               static_cast<float*>(x));
  note_launches(1);
}

}  // namespace gcmg
