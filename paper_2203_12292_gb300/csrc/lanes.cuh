// Lane-per-cell steps shared by the operator (kernels_lanes.cu) and the level
// transfer (kernels_lattice.cu): x-line tables with their class partition,
// hanging-line interpolation in registers (fp32 and double-float), ordered
// additions into a tile's DoF buffer.
#pragma once

#include <algorithm>
#include <map>
#include <stdexcept>
#include <vector>

#include "device.cuh"
#include "turns.cuh"

namespace gcmg {

constexpr int LW = 8;  // table entries of x-lines per warp

// x-line r = b + N c of degree K: slot of node (0, b, c) | byte offset of the
// node in its entity << 8 | byte offset of node (1, b, c) in the slot after it
// << 16; per warp the x-lines it gathers and scatters (-1: none),
// class-partitioned
struct LaneLines {
  uint32_t line[KMAX + 1][NMAX * NMAX];
  int8_t xw[KMAX + 1][NMAX][LW];
  int32_t nx[KMAX + 1][NMAX];  // x-lines of each warp
  // lines q = u + N v (the other two coordinates, in increasing axis order) of
  // warp w in the passes of tiles with hanging cells: N lines each, the boundary
  // ones (16 of 25 at k = 4, the only ones that can hang) dealt evenly
  uint8_t bl[KMAX + 1][NMAX][NMAX];
};
static __constant__ LaneLines c_ll;  // one copy per translation unit (filled by its upload function)

// child-side interpolation I_p (TRANS: its transpose) on one line in
// registers.  I_1[a][b] = I_0[k-a][k-b] (Gauss-Lobatto points and Lagrange
// basis are symmetric under x -> 1 - x), so p = 1 reverses the line, applies
// I_0 and reverses back: one set of constant-operand multiply-adds
template <int K, bool TRANS, typename T>
__device__ __forceinline__ void interp_line_reg(T* v, int p) {
  constexpr int N = K + 1;
  const DevTables<T>& tb = tab<T>(K);
  T x[N], y[N];
#pragma unroll
  for (int a = 0; a < N; ++a) x[a] = p ? v[K - a] : v[a];
#pragma unroll
  for (int r = 0; r < N; ++r) {
    T s = T(0);
#pragma unroll
    for (int a = 0; a < N; ++a) s += (TRANS ? tb.I[0][a][r] : tb.I[0][r][a]) * x[a];
    y[r] = s;
  }
#pragma unroll
  for (int a = 0; a < N; ++a) v[a] = p ? y[K - a] : y[a];
}

__device__ __forceinline__ df df_sel(bool p, df a, df b) { return df{p ? a.hi : b.hi, p ? a.lo : b.lo}; }

// sum_j x_j c_j over T double-float values and double-float constants
// (ch + cl) with one normalisation: the high products p_j = x_j.hi ch_j carry
// their exact rounding errors (fused multiply-add), the p_j are summed by
// error-free two-sums, and the low-order terms (product errors, cross terms
// x.hi cl and x.lo ch, two-sum errors) go into one fp32 sum; 12 T - 5
// operations instead of 18 T - 11 for a chain of df_fma.  df_dot_raw leaves the
// normalisation out (3 of them; see df_add_raw)
template <int T>
__device__ __forceinline__ df df_dot_raw(const df* x, const float* ch, const float* cl) {
  float S = __fmul_rn(x[0].hi, ch[0]);
  float L = __fmaf_rn(x[0].hi, cl[0], __fmaf_rn(x[0].lo, ch[0], __fmaf_rn(x[0].hi, ch[0], -S)));
#pragma unroll
  for (int j = 1; j < T; ++j) {
    const float p = __fmul_rn(x[j].hi, ch[j]);
    const float l = __fmaf_rn(x[j].hi, cl[j], __fmaf_rn(x[j].lo, ch[j], __fmaf_rn(x[j].hi, ch[j], -p)));
    const float s = __fadd_rn(S, p);
    const float z = __fsub_rn(s, S);
    const float t = __fadd_rn(__fsub_rn(S, __fsub_rn(s, z)), __fsub_rn(p, z));
    S = s;
    L = __fadd_rn(L, __fadd_rn(l, t));
  }
  return df{S, L};
}
template <int T>
__device__ __forceinline__ df df_dot(const df* x, const float* ch, const float* cl) {
  const df s = df_dot_raw<T>(x, ch, cl);
  return df_norm(s.hi, s.lo);
}

// pairs between two steps of a line: normalised (NORM), or as they come.  Error of
// the fp64 operator on random vectors (uniform cube, 4,096 cells), as they come /
// normalised / of the line-parallel kernel: k = 1 2.4 / 2.4 / 2.9e-15, k = 2 4.2 / 4.1 /
// 4.4e-15, k = 3 6.3 / 5.6 / 6.1e-15, k = 4 6.1 / 5.7 / 5.7e-15; of vmult_lanes_df with
// a forward sweep, the scaling and a backward sweep, all normalised, in place of the
// z-line: k = 2 4.4, k = 3 6.4, k = 4 6.4e-15.  So whole tiles take them as they come
// (Q4 octant 438 us, normalised 488), the cell vectors at k >= 3 normalised (4,096
// cells, k = 4: 16.2 -> 16.3 us).
template <bool NORM>
__device__ __forceinline__ df df_add_step(df a, df b) {
  return NORM ? df_add(a, b) : df_add_raw(a, b);
}
template <int T, bool NORM>
__device__ __forceinline__ df df_dot_step(const df* x, const float* ch, const float* cl) {
  return NORM ? df_dot<T>(x, ch, cl) : df_dot_raw<T>(x, ch, cl);
}

// even-odd forward transform with B (nodal -> modes in mode order) and its
// backward transform, in double-float, rows as df_dot
template <int K, bool NORM = false>
__device__ __forceinline__ void df_eo_fwd_fast(df* u) {
  constexpr int N = K + 1, NH = N / 2, NE = (N + 1) / 2;
  const float(&Bh)[NMAX][NMAX] = c_tf[K].Be;
  const float(&Bl)[NMAX][NMAX] = c_tflo[K].Be;
  df e[NE], o[NH > 0 ? NH : 1];
#pragma unroll
  for (int j = 0; j < NH; ++j) {
    e[j] = df_add_step<NORM>(u[j], u[N - 1 - j]);
    o[j] = df_add_step<NORM>(u[j], df_neg(u[N - 1 - j]));
  }
  if (N % 2) e[NH] = u[NH];
#pragma unroll
  for (int r = 0; r < NE; ++r) u[r] = df_dot<NE>(e, Bh[r], Bl[r]);
#pragma unroll
  for (int r = 0; r < NH; ++r) u[NE + r] = df_dot<NH>(o, Bh[NE + r], Bl[NE + r]);
}

template <int K, bool NORM = false>
__device__ __forceinline__ void df_eo_bwd_fast(df* u) {
  constexpr int N = K + 1, NH = N / 2, NE = (N + 1) / 2;
  df E[NE], O[NH > 0 ? NH : 1];
  float ch[NMAX], cl[NMAX];
#pragma unroll
  for (int j = 0; j < NE; ++j) {
#pragma unroll
    for (int r = 0; r < NE; ++r) {
      ch[r] = c_tf[K].Be[r][j];
      cl[r] = c_tflo[K].Be[r][j];
    }
    E[j] = df_dot_step<NE, NORM>(u, ch, cl);
  }
#pragma unroll
  for (int j = 0; j < NH; ++j) {
#pragma unroll
    for (int r = 0; r < NH; ++r) {
      ch[r] = c_tf[K].Be[NE + r][j];
      cl[r] = c_tflo[K].Be[NE + r][j];
    }
    O[j] = df_dot_step<NH, NORM>(u + NE, ch, cl);
  }
#pragma unroll
  for (int j = 0; j < NH; ++j) {
    u[j] = df_add(E[j], O[j]);
    u[N - 1 - j] = df_sub(E[j], O[j]);
  }
  if (N % 2) u[NH] = df_norm(E[NH].hi, E[NH].lo);
}

// I_p (TRANS: transposed) on one df line, by the mirror identity of interp_line_reg
template <int K, bool TRANS>
__device__ __forceinline__ void interp_line_df(df* v, int p) {
  constexpr int N = K + 1;
  const float(&Ih)[NMAX][NMAX] = c_tf[K].I[0];
  const float(&Il)[NMAX][NMAX] = c_tflo[K].I[0];
  df x[N], y[N];
#pragma unroll
  for (int a = 0; a < N; ++a) x[a] = df_sel(p, v[K - a], v[a]);
  float ch[NMAX], cl[NMAX];
#pragma unroll
  for (int r = 0; r < N; ++r) {
#pragma unroll
    for (int a = 0; a < N; ++a) {
      ch[a] = TRANS ? Ih[a][r] : Ih[r][a];
      cl[a] = TRANS ? Il[a][r] : Il[r][a];
    }
    y[r] = df_dot<N>(x, ch, cl);
  }
#pragma unroll
  for (int a = 0; a < N; ++a) v[a] = df_sel(p, y[K - a], y[a]);
}

// arithmetic of the cell pipeline: fp32, or double-float on fp64 vectors
template <typename T>
struct Arith;
template <>
struct Arith<float> {
  using V = float;
  static __device__ __forceinline__ V in(float x) { return x; }
  static __device__ __forceinline__ float out(V x) { return x; }
};
template <>
struct Arith<double> {
  using V = df;
  static __device__ __forceinline__ V in(double x) { return df_from(x); }
  static __device__ __forceinline__ double out(V x) { return df_to(x); }
};

template <int K, bool FWD, bool NORM = false>
__device__ __forceinline__ void eo_line(float* v) {
  if (FWD)
    eo_forward<K + 1, 0, 1>(v, tab<float>(K).Be);
  else
    eo_backward<K + 1, 0, 1>(v, tab<float>(K).Be);
}
template <int K, bool FWD, bool NORM = false>
__device__ __forceinline__ void eo_line(df* v) {
  if (FWD)
    df_eo_fwd_fast<K, NORM>(v);
  else
    df_eo_bwd_fast<K, NORM>(v);
}
template <int K, bool TRANS>
__device__ __forceinline__ void hang_line(float* v, int p) {
  interp_line_reg<K, TRANS>(v, p);
}
template <int K, bool TRANS>
__device__ __forceinline__ void hang_line(df* v, int p) {
  interp_line_df<K, TRANS>(v, p);
}

// x-line tables: slots and offsets per line; the line classes (lines whose
// nodes can share DoFs between cells) dealt to the k+1 warps, largest class
// first to the least loaded warp
inline void fill_lane_lines(LaneLines& t) {
  t = LaneLines{};
  for (int k = 0; k <= KMAX; ++k)
    for (int w = 0; w < NMAX; ++w)
      for (int i = 0; i < LW; ++i) t.xw[k][w][i] = -1;
  for (int k = 1; k <= KMAX; ++k) {
    const int n = k + 1;
    for (int c = 0; c < n; ++c)
      for (int b = 0; b < n; ++b) {
        int s0, o0, s1, o1 = 0;
        host_node_slot(k, 0, b, c, s0, o0);
        if (k > 1) host_node_slot(k, 1, b, c, s1, o1);
        t.line[k][b + n * c] = (uint32_t)s0 | ((uint32_t)(4 * o0) << 8) | ((uint32_t)(4 * o1) << 16);
      }
    auto cls = [&](int x) { return (x == 0 || x == k) ? -1 : x; };
    std::map<std::pair<int, int>, std::vector<int>> classes;
    for (int c = 0; c < n; ++c)
      for (int b = 0; b < n; ++b) classes[{cls(b), cls(c)}].push_back(b + n * c);
    std::vector<std::vector<int>> cl;
    for (auto& kv : classes) cl.push_back(kv.second);
    std::stable_sort(cl.begin(), cl.end(), [](const std::vector<int>& x, const std::vector<int>& y) {
      return x.size() > y.size();
    });
    std::vector<int> load(n, 0);
    for (const auto& c : cl) {
      int w = 0;
      for (int u = 1; u < n; ++u)
        if (load[u] < load[w]) w = u;
      for (int r : c) {
        if (load[w] >= LW) throw std::runtime_error("lane line table overflow");
        t.xw[k][w][load[w]++] = (int8_t)r;
      }
    }
    for (int w = 0; w < n; ++w) t.nx[k][w] = load[w];
    std::vector<int> bal(n, 0);
    int w = 0;
    for (int pass = 0; pass < 2; ++pass)
      for (int q = 0; q < n * n; ++q) {
        const bool boundary = cls(q % n) < 0 || cls(q / n) < 0;
        if (boundary != (pass == 0)) continue;
        t.bl[k][w][bal[w]++] = (uint8_t)q;
        w = (w + 1) % n;
      }
  }
}

}  // namespace gcmg
