// The innermost direction of the cell operator on lines that are modes in the
// other two directions.
//
// With the x and y directions diagonalised, the operator on the z-line of modes
// (a, b) is h (K + (lam_a + lam_b) M), M and K the 1D mass and stiffness
// matrices.  That is one (k+1) x (k+1) matrix per pair of modes, symmetric under
// reversal: in even-odd form 13 coefficients at k = 4.  Applying it costs half of
// what the forward transform, the scaling by h (lam_a + lam_b + lam_c) and the
// backward transform cost (28 instead of 44 operations per line in fp32, about
// 235 instead of 470 in double-float).
//   The matrix of the constant pair (lam_a + lam_b = 0, the stiffness matrix alone)
// is applied to differences: its rows sum to zero, and rows rounded entry by entry
// do not (-4.8e-7 at k = 4 in fp32), which acts as a reaction term of one sign in
// every cell.  With e_j - t e_mid in place of e_j (t = 2, without a middle node 1)
// the middle column is the row sum, zero, and constants along the line give zero
// whatever the rounding.  x^T A x on sin sin sin, 32^3 cells, relative error of the
// sweeps and scaling, the matrix rounded entry by entry (growing with h^-2), the
// differences: fp32, degree 4: 1.7e-7, 1.5e-5, 2.4e-7; fp64, degree 3: 5.8e-13,
// 1.9e-12, 6.7e-14.
// fp32 operator of the octant meshes: Q3 84 -> 73 us (269,998 cells), Q4 115 -> 111
// us (296,535 cells); a level of few cells (Q4, 4,712 cells) 14.5 -> 9.3 us in fp32,
// 34 -> 24.5 us in fp64.
#pragma once

#include "device.cuh"
#include "lanes.cuh"

namespace gcmg {

// first row of degree k's lines, one row per line of modes i + (k+1) j (mode order
// of DevTables::lame); a row: the even block, rows of (k+2)/2, then the odd block
__host__ __device__ constexpr int zline_row(int k) { return k * (k + 1) * (2 * k + 1) / 6 - 1; }
struct ZLines {
  alignas(16) float h[zline_row(KMAX + 1)][16];  // then t
  alignas(16) float l[zline_row(KMAX + 1)][16];  // low parts: h + l to about 2^-48
};
static __constant__ ZLines c_zl;  // one copy per translation unit (upload_zlines)

__host__ __device__ constexpr int zline_count(int k) { return ((k + 2) / 2) * ((k + 2) / 2) + ((k + 1) / 2) * ((k + 1) / 2); }

// v <- (K + lam M) v with the coefficients c; constants: the line may be that of the
// modes (0, 0) (differences on every line of the Q4 octant operator: 109.3 us, on those
// of the first mode only 108.4 us, as without)
template <int K>
__device__ __forceinline__ void zline(float* v, const float* c, bool constants) {
  constexpr int N = K + 1, NH = N / 2, NE = (N + 1) / 2;
  float e[NE], o[NH];
#pragma unroll
  for (int j = 0; j < NH; ++j) {
    e[j] = v[j] + v[K - j];
    o[j] = v[j] - v[K - j];
  }
  if (N % 2) e[NH] = v[NH];
  if (constants) {
#pragma unroll
    for (int j = 0; j < NE - 1; ++j) e[j] = fmaf(-c[zline_count(K)], e[NE - 1], e[j]);
  }
#pragma unroll
  for (int i = 0; i < NE; ++i) {
    float E = c[NE * i] * e[0];
#pragma unroll
    for (int j = 1; j < NE; ++j) E = fmaf(c[NE * i + j], e[j], E);
    if (i < NH) {
      float O = c[NE * NE + NH * i] * o[0];
#pragma unroll
      for (int j = 1; j < NH; ++j) O = fmaf(c[NE * NE + NH * i + j], o[j], O);
      v[i] = E + O;
      v[K - i] = E - O;
    } else {
      v[i] = E;
    }
  }
}

template <int K, bool NORM = false>
__device__ __forceinline__ void zline(df* v, const float* ch, const float* cl, bool constants) {
  constexpr int N = K + 1, NH = N / 2, NE = (N + 1) / 2;
  df e[NE], o[NH];
#pragma unroll
  for (int j = 0; j < NH; ++j) {
    e[j] = df_add_step<NORM>(v[j], v[K - j]);
    o[j] = df_add_step<NORM>(v[j], df_neg(v[K - j]));
  }
  if (N % 2) e[NH] = v[NH];
  if (constants) {
    const float t = ch[zline_count(K)];
#pragma unroll
    for (int j = 0; j < NE - 1; ++j) e[j] = df_add_step<NORM>(e[j], df{-t * e[NE - 1].hi, -t * e[NE - 1].lo});
  }
#pragma unroll
  for (int i = 0; i < NE; ++i) {
    const df E = df_dot_step<NE, NORM>(e, ch + NE * i, cl + NE * i);
    if (i < NH) {
      const df O = df_dot_step<NH, NORM>(o, ch + NE * NE + NH * i, cl + NE * NE + NH * i);
      v[i] = df_add(E, O);
      v[K - i] = df_sub(E, O);
    } else {
      v[i] = df_norm(E.hi, E.lo);
    }
  }
}

// the coefficients of K + lam M in fp64
inline void zline_coefficients(const Basis1D& b, double lam, double* c) {
  const int n = b.k + 1, nh = n / 2, ne = (n + 1) / 2;
  auto C = [&](int i, int j) { return b.K[i][j] + lam * b.M[i][j]; };
  for (int i = 0; i < ne; ++i)
    for (int j = 0; j < ne; ++j)
      c[ne * i + j] = (i >= nh || j >= nh) ? C(i, j) : 0.5 * (C(i, j) + C(i, n - 1 - j));
  for (int i = 0; i < nh; ++i)
    for (int j = 0; j < nh; ++j) c[ne * ne + nh * i + j] = 0.5 * (C(i, j) - C(i, n - 1 - j));
}

static inline void upload_zlines() {
  static DevTables<double> td[KMAX + 1];
  static DevTables<float> tf[KMAX + 1];
  static ZLines z;
  fill_tables(td, tf);
  for (int k = 1; k <= KMAX; ++k)
    for (int q = 0; q < (k + 1) * (k + 1); ++q) {
      const int nc = zline_count(k), nh = (k + 1) / 2, ne = (k + 2) / 2;
      double c[13] = {};
      zline_coefficients(basis(k), td[k].lame[q % (k + 1)] + td[k].lame[q / (k + 1)], c);
      for (int i = 0; i < 13; ++i) {
        z.h[zline_row(k) + q][i] = (float)c[i];
        z.l[zline_row(k) + q][i] = (float)(c[i] - (double)z.h[zline_row(k) + q][i]);
      }
      if (q == 0 && ne > 1) {  // modes (0, 0): constants; lam = 0
        for (int i = 0; i < ne; ++i) z.h[zline_row(k)][ne * i + ne - 1] = z.l[zline_row(k)][ne * i + ne - 1] = 0.f;
        z.h[zline_row(k)][nc] = ne > nh ? 2.f : 1.f;
      }
    }
  cudaMemcpyToSymbol(c_zl, &z, sizeof(z));
}

}  // namespace gcmg
