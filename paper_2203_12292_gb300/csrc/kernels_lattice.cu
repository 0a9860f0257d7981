// Level transfer (Sec. 3.5, Eqs. 5-7) with one warp per coarse cell.
//
// The eight children of a refined coarse cell carry a lattice of (2k+1)^3
// support points on 5 x 5 x 5 geometric entities (per axis: low vertex, low
// child's interior, middle vertex, high child's interior, high vertex).  Every
// point of the lattice is visited once, through the lowest child that holds
// it: siblings are consecutive in Morton order, so if one of them owns the
// entity for the transfer it is that one.  A table per coarse cell, built once
// per transfer, holds the 125 entity starts (-1: owned elsewhere or
// constrained), and a table per degree lists the lattice points entity by
// entity, so consecutive lanes touch consecutive DoFs (27, 9, 3, 1 at k = 4).
//   What bounded the kernels of kernels_transfer.cu was index arithmetic: the
// 8 (k+1)^3 child nodes of a coarse cell (1,000 at k = 4, of which at most 729
// are distinct) each with two divisions by (k+1)^3, an ownership bit and a slot
// start, and block barriers after every sweep of a few cells.  Here a point
// costs one table word, one entity start and the value; a warp owns its cells,
// so the sweeps need warp synchronisation only.
//   Sweeps run in place on the lattice: a line is read and written by one lane.
// P is symmetric under x -> 1 - x, so a 1D line takes the even-odd form, and
// its rows at the coarse cell's own end (and, k even, middle) points are unit
// vectors: 28 instead of 45 operations per line at k = 4.
//   Restriction: the tile's cell results go to a cell buffer with one lane per
// cell; C^T and the fixed-order accumulation into the tile's DoFs are those of
// the lane-per-cell operator.
// Finest Q4 transfer of the octant mesh (18.7 M fine DoFs), fp32:
// restriction 188 -> 67 us, prolongation 135 -> 44 us (3.7 TB/s of the bytes
// it needs, 54 % of the copy rate; the entity table adds 19 MB).
//   The p transfer (one mesh, degree k to floor(k / 2)) is the same with the cell's
// own nodes as the lattice and its owned slots as the entities: Q4 sphere, fine
// level, restriction with its halo pass 111 -> 57 us, prolongation 61 -> 43 us.
#include <algorithm>
#include <cstring>

#include "device.cuh"
#include "kernels.h"
#include "lanes.cuh"

namespace gcmg {

GCMG_DEFINE_UPLOAD(upload_tables_lattice_1d)

namespace {

constexpr int WPB = 8;             // warps (coarse cells in flight) per block
constexpr int CBS = 33;            // cell buffer: node n of cell j at n * CBS + j
constexpr int PT_MAX = 23 * 32;    // lattice points of k = 4, whole warps
constexpr int ND_MAX = 4 * 32;     // nodes of a cell, whole warps

// words per coarse cell of the entity table: the entity starts, then -1s; the
// last word is 1 for refined cells
__host__ __device__ constexpr int lat_words(int k) { return k == 1 ? 32 : 128; }

struct LatTables {
  uint32_t pt[KMAX + 1][PT_MAX];  // lattice points: entity | offset << 7 | position << 12
  uint32_t nd[KMAX + 1][ND_MAX];  // cell nodes: slot | offset << 7 | lattice position of the coarse node << 12
  // p transfer from degree k: the cell's fine nodes entity by entity, its coarse
  // nodes, positions in the (k+1)^3 lattice
  uint32_t pf[KMAX + 1][ND_MAX];
  uint32_t pc[KMAX + 1][32];
};
__device__ LatTables g_lat;

// even-odd form of the 1D prolongation rows i = 1 .. k (see fill_sweeps)
template <typename T>
struct LatSweeps {
  T e[KMAX + 1][KMAX + 1][3];
  T o[KMAX + 1][KMAX + 1][2];
};
__constant__ LatSweeps<float> c_swf;
__constant__ LatSweeps<double> c_swd;
template <typename T>
__device__ __forceinline__ const LatSweeps<T>& sweeps();
template <>
__device__ __forceinline__ const LatSweeps<float>& sweeps<float>() {
  return c_swf;
}
template <>
__device__ __forceinline__ const LatSweeps<double>& sweeps<double>() {
  return c_swd;
}

template <typename T>
struct LatArgs {
  const int32_t* ent;  // per coarse cell lat_words(k) words
  const int32_t* gstart_f;  // p: fine slots and owned slots per cell
  const uint32_t* own_f;
  const int32_t* gstart_c;
  const uint16_t* mask_c;
  int n_coarse;
  const T* src;
  T* dst;
  const T* rhs;   // restriction: set: restrict rhs - src
  int overwrite;  // restriction: dst = R r instead of dst += R r
  const TileInfo* tiles;
  const LaneTile* lt;
  const LaneHang* lh;
  T* halo;
  const int32_t* halo_pos;
};

// prolongation of one line: v[0..k] -> v[0..2k]
template <int K, typename T>
__device__ __forceinline__ void line_prolong(T* v) {
  constexpr int N = K + 1, NH = N / 2, NE = (N + 1) / 2;
  const LatSweeps<T>& S = sweeps<T>();
  T e[NE], o[NH];
#pragma unroll
  for (int a = 0; a < NH; ++a) {
    e[a] = v[a] + v[K - a];
    o[a] = v[a] - v[K - a];
  }
  if (N % 2) e[NH] = v[NH];
  const T first = v[0], last = v[K];
  T mid;
  if (K % 2 == 0) {
    mid = v[K / 2];
  } else {
    mid = S.e[K][K][0] * e[0];
#pragma unroll
    for (int a = 1; a < NE; ++a) mid += S.e[K][K][a] * e[a];
  }
#pragma unroll
  for (int i = 1; i < K; ++i) {
    T E = S.e[K][i][0] * e[0], O = S.o[K][i][0] * o[0];
#pragma unroll
    for (int a = 1; a < NE; ++a) E += S.e[K][i][a] * e[a];
#pragma unroll
    for (int a = 1; a < NH; ++a) O += S.o[K][i][a] * o[a];
    v[i] = E + O;
    v[2 * K - i] = E - O;
  }
  v[0] = first;
  v[K] = mid;
  v[2 * K] = last;
}

// its transpose: v[0..2k] -> v[0..k]
template <int K, typename T>
__device__ __forceinline__ void line_restrict(T* v) {
  constexpr int N = K + 1, NH = N / 2, NE = (N + 1) / 2;
  const LatSweeps<T>& S = sweeps<T>();
  T s[K + 1], d[K + 1];
#pragma unroll
  for (int i = 1; i < K; ++i) {
    s[i] = v[i] + v[2 * K - i];
    d[i] = v[i] - v[2 * K - i];
  }
  const T first = v[0], mid = v[K], last = v[2 * K];
#pragma unroll
  for (int a = 0; a < NE; ++a) {
    T E = T(0), O = T(0);
    if (K % 2) E = S.e[K][K][a] * mid;
#pragma unroll
    for (int i = 1; i < K; ++i) E += S.e[K][i][a] * s[i];
    if (a < NH) {
#pragma unroll
      for (int i = 1; i < K; ++i) O += S.o[K][i][a] * d[i];
      v[a] = E + O;
      v[K - a] = E - O;
    } else {
      v[a] = E + mid;  // k even: the middle point is a coarse node
    }
  }
  v[0] += first;
  v[K] += last;
}

// lattice of one coarse cell of degree K: the children's (KF = 0, h transfer) or
// the same cell's nodes of degree KF (p transfer)
template <int K, int KF = 0>
struct Lat {
  static constexpr int N = K + 1, N2 = N * N, N3 = N2 * N;
  static constexpr int M = KF ? KF + 1 : 2 * K + 1, M2 = M * M, M3 = M2 * M;
  static constexpr int ES = KF ? 32 : lat_words(K), EPL = ES / 32;
  static constexpr int NI = (M3 + 31) / 32, NJ = (N3 + 31) / 32;
  static constexpr int LS = (M3 + 2) & ~1;  // lattice of a warp; position M3 takes the padding points
  static __device__ __forceinline__ const uint32_t* points() { return KF ? g_lat.pf[KF] : g_lat.pt[K]; }
  static __device__ __forceinline__ const uint32_t* nodes() { return KF ? g_lat.pc[KF] : g_lat.nd[K]; }
  // lane's entity words of coarse cell c (p: the cell's owned slots)
  template <typename T>
  static __device__ __forceinline__ void words(const LatArgs<T>& A, int c, int lane, int32_t* en) {
    if constexpr (KF == 0) {
#pragma unroll
      for (int i = 0; i < EPL; ++i) en[i] = A.ent[(size_t)c * ES + lane + 32 * i];
    } else {
      en[0] = -1;
      if (lane < NSLOT && ((A.own_f[c] >> lane) & 1u)) en[0] = A.gstart_f[(size_t)c * NSLOT + lane];
    }
  }
  // one line down (M -> N values) and up
  template <typename T>
  static __device__ __forceinline__ void down(T* v) {
    if constexpr (KF == 0) {
      line_restrict<K>(v);
    } else {
      T o[N];
#pragma unroll
      for (int a = 0; a < N; ++a) {
        o[a] = tab<T>(KF).Pp[0][a] * v[0];
#pragma unroll
        for (int i = 1; i < M; ++i) o[a] += tab<T>(KF).Pp[i][a] * v[i];
      }
#pragma unroll
      for (int a = 0; a < N; ++a) v[a] = o[a];
    }
  }
  template <typename T>
  static __device__ __forceinline__ void up(T* v) {
    if constexpr (KF == 0) {
      line_prolong<K>(v);
    } else {
      T o[M];
#pragma unroll
      for (int i = 0; i < M; ++i) {
        o[i] = tab<T>(KF).Pp[i][0] * v[0];
#pragma unroll
        for (int a = 1; a < N; ++a) o[i] += tab<T>(KF).Pp[i][a] * v[a];
      }
#pragma unroll
      for (int i = 0; i < M; ++i) v[i] = o[i];
    }
  }
};

// the three sweeps down on a warp's lattice: M^3 -> N^3 values, value i of the x-line
// that starts at p to out(p, i, value)
template <typename L, typename T, typename F>
__device__ __forceinline__ void lattice_down(T* lat, int lane, F&& out) {
  constexpr int N = L::N, M = L::M, M2 = L::M2;
#pragma unroll 1
  for (int q = lane; q < M2; q += 32) {  // z-lines
    T v[M];
#pragma unroll
    for (int i = 0; i < M; ++i) v[i] = lat[q + M2 * i];
    L::down(v);
#pragma unroll
    for (int i = 0; i < N; ++i) lat[q + M2 * i] = v[i];
  }
  __syncwarp();
#pragma unroll 1
  for (int q = lane; q < M * N; q += 32) {  // y-lines (x, c)
    T* p = lat + q % M + M2 * (q / M);
    T v[M];
#pragma unroll
    for (int i = 0; i < M; ++i) v[i] = p[M * i];
    L::down(v);
#pragma unroll
    for (int i = 0; i < N; ++i) p[M * i] = v[i];
  }
  __syncwarp();
  if (lane < N * N) {  // x-lines (b, c)
    T* p = lat + M * (lane % N) + M2 * (lane / N);
    T v[M];
#pragma unroll
    for (int i = 0; i < M; ++i) v[i] = p[i];
    L::down(v);
#pragma unroll
    for (int i = 0; i < N; ++i) out(p, i, v[i]);
  }
}

// shared memory: lane records, point tables, entity starts, then the cell
// buffer, then the warps' lattices; the tile's accumulator takes the lattices'
// place once every cell of the tile has been reduced
template <int K, typename T, int KF>
struct RestrictSmem {
  using L = Lat<K, KF>;
  static constexpr size_t pt = sizeof(LaneTile) + sizeof(LaneHang);
  static constexpr size_t nd = pt + (size_t)L::NI * 32 * 4;
  static constexpr size_t ent = nd + (size_t)L::NJ * 32 * 4;
  static constexpr size_t cb = ent + (size_t)WPB * L::ES * 4;
  static constexpr size_t lat = (cb + (size_t)L::N3 * CBS * sizeof(T) + 15) & ~(size_t)15;
  static size_t total(int max_local) {
    return lat + std::max((size_t)WPB * L::LS, (size_t)max_local + LANE_ZERO + 4) * sizeof(T);
  }
};

template <int K, typename T, int KF>
__global__ void __launch_bounds__(WPB * 32) restrict_lattice(LatArgs<T> A) {
  using L = Lat<K, KF>;
  using SM = RestrictSmem<K, T, KF>;
  constexpr int N = L::N, N2 = L::N2, N3 = L::N3;
  constexpr int NT = WPB * 32;
  extern __shared__ __align__(16) unsigned char smem[];
  LaneTile* st = reinterpret_cast<LaneTile*>(smem);
  LaneHang* hg = reinterpret_cast<LaneHang*>(smem + sizeof(LaneTile));
  uint32_t* s_pt = reinterpret_cast<uint32_t*>(smem + SM::pt);
  uint32_t* s_nd = reinterpret_cast<uint32_t*>(smem + SM::nd);
  T* cb = reinterpret_cast<T*>(smem + SM::cb);
  T* ys = reinterpret_cast<T*>(smem + SM::lat);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t* ent = reinterpret_cast<int32_t*>(smem + SM::ent) + w * L::ES;
  T* lat = ys + w * L::LS;
  const TileInfo ti = A.tiles[blockIdx.x];
  const int nc = ti.n_cells, nloc = ti.n_owned + ti.n_foreign;
  {
    const uint4* g = reinterpret_cast<const uint4*>(A.lt + blockIdx.x);
    uint4* s = reinterpret_cast<uint4*>(st);
    for (int i = threadIdx.x; i < (int)(sizeof(LaneTile) / 16); i += NT) cp_async16(s + i, g + i);
    const uint4* gh = reinterpret_cast<const uint4*>(A.lh + blockIdx.x);
    uint4* sh = reinterpret_cast<uint4*>(hg);
    for (int i = threadIdx.x; i < (int)(sizeof(LaneHang) / 16); i += NT) cp_async16(sh + i, gh + i);
    for (int i = threadIdx.x; i < L::NI * 32; i += NT) cp_async(s_pt + i, L::points() + i);
    for (int i = threadIdx.x; i < L::NJ * 32; i += NT) cp_async(s_nd + i, L::nodes() + i);
  }
  int32_t en[L::EPL];  // the next cell's entity words
  if (w < nc) L::words(A, ti.cell_begin + w, lane, en);
  cp_async_wait_all();
  pdl_wait();
  __syncthreads();
  const T* __restrict__ src = A.src;
  const T* __restrict__ rhs = A.rhs;
  for (int j = w; j < nc; j += WPB) {
#pragma unroll
    for (int i = 0; i < L::EPL; ++i) ent[lane + 32 * i] = en[i];
    if (j + WPB < nc) L::words(A, ti.cell_begin + j + WPB, lane, en);
    __syncwarp();
    if (KF || ent[L::ES - 1] > 0) {
      // the owned fine values, UB points in flight per lane
      constexpr int UB = sizeof(T) == 4 ? 12 : 8;
#pragma unroll
      for (int b = 0; b < L::NI; b += UB) {
        T v[UB];
        int pos[UB];
#pragma unroll
        for (int u = 0; u < UB; ++u)
          if (b + u < L::NI) {
            const uint32_t p = s_pt[lane + 32 * (b + u)];
            const int32_t g = ent[p & 127];
            pos[u] = p >> 12;
            v[u] = T(0);
            if (g >= 0) {
              const int gi = g + (int)((p >> 7) & 31);
              v[u] = rhs ? rhs[gi] - src[gi] : src[gi];
            }
          }
#pragma unroll
        for (int u = 0; u < UB; ++u)
          if (b + u < L::NI) lat[pos[u]] = v[u];
      }
      __syncwarp();
      // the x-lines' results into the cell buffer
      lattice_down<L>(lat, lane, [&](T*, int i, T v) { cb[(N * lane + i) * CBS + j] = v; });
    } else {  // identity category (no fine cells: no owned slots, zeros)
#pragma unroll
      for (int i = 0; i < L::NJ; ++i) {
        const int n = lane + 32 * i;
        const uint32_t p = s_nd[n];
        const int32_t g = ent[p & 127];
        T v = T(0);
        if (g >= 0) {
          const int gi = g + (int)((p >> 7) & 31);
          v = rhs ? rhs[gi] - src[gi] : src[gi];
        }
        if (n < N3) cb[n * CBS + j] = v;
      }
    }
    __syncwarp();
  }
  __syncthreads();
  // C^T (z, y here; x with the scatter), the accumulator cleared meanwhile
  const uint16_t m = st->mask[lane];
  const bool hang = st->hang != 0;
  for (int i = threadIdx.x; i < nloc; i += NT) ys[i] = T(0);
  if (hang) {
    const bool cell = lane < nc;
#pragma unroll 1
    for (int q = w; q < N2; q += WPB)
      if (cell && ((hg->hl[2][lane] >> q) & 1u)) {
        T* p = cb + q * CBS + lane;
        T v[N];
#pragma unroll
        for (int a = 0; a < N; ++a) v[a] = p[a * N2 * CBS];
        interp_line_reg<K, true>(v, (m >> 2) & 1);
#pragma unroll
        for (int a = 0; a < N; ++a) p[a * N2 * CBS] = v[a];
      }
    __syncthreads();
#pragma unroll 1
    for (int q = w; q < N2; q += WPB)
      if (cell && ((hg->hl[1][lane] >> q) & 1u)) {
        T* p = cb + (q % N + N2 * (q / N)) * CBS + lane;
        T v[N];
#pragma unroll
        for (int a = 0; a < N; ++a) v[a] = p[a * N * CBS];
        interp_line_reg<K, true>(v, (m >> 1) & 1);
#pragma unroll
        for (int a = 0; a < N; ++a) p[a * N * CBS] = v[a];
      }
  }
  __syncthreads();
  if (w < N) {  // the warp's class of x-lines: no two warps add to one DoF
    const int nxl = c_ll.nx[K][w];
    char* xb = reinterpret_cast<char*>(ys);
    constexpr int SC = sizeof(T) / 4;
#pragma unroll 1
    for (int i = 0; i < nxl; ++i) {
      const int r = c_ll.xw[K][w][i];
      T v[N];
#pragma unroll
      for (int a = 0; a < N; ++a) v[a] = cb[(N * r + a) * CBS + lane];
      if (hang && ((hg->hl[0][lane] >> r) & 1u)) interp_line_reg<K, true>(v, m & 1);
      const uint32_t li = c_ll.line[K][r];
      const int s0 = li & 0xff, o0 = (li >> 8) & 0xff, o1 = li >> 16;
      T* p0 = reinterpret_cast<T*>(xb + SC * (st->ls[s0][lane] + o0));
      T* p1 = reinterpret_cast<T*>(xb + SC * (st->ls[s0 + 1][lane] + o1));
      T* p2 = reinterpret_cast<T*>(xb + SC * (st->ls[s0 + 2][lane] + o0));
      add_turns<1>(p0, v, hang ? hg->rank[s0][lane] : 0, hang ? hg->most[s0] : 1);
      if constexpr (K > 1)
        add_turns<K - 1>(p1, v + 1, hang ? hg->rank[s0 + 1][lane] : 0, hang ? hg->most[s0 + 1] : 1);
      add_turns<1>(p2, v + K, hang ? hg->rank[s0 + 2][lane] : 0, hang ? hg->most[s0 + 2] : 1);
    }
  }
  __syncthreads();
  T* dst = A.dst + ti.dof_begin;
  if (A.overwrite)
    for (int i = threadIdx.x; i < ti.n_owned; i += NT) dst[i] = ys[i];
  else
    for (int i = threadIdx.x; i < ti.n_owned; i += NT) dst[i] += ys[i];
  const int32_t* hp = A.halo_pos + ti.foreign_begin;
  for (int i = threadIdx.x; i < ti.n_foreign; i += NT) A.halo[hp[i]] = ys[ti.n_owned + i];
}

// one direction of C (TRANS: C^T) on the coarse values of a warp's lattice
// (node (a, b, c) at a + M b + M^2 c)
template <int K, int KF, int D, bool TRANS, typename T>
__device__ __forceinline__ void lattice_hang(T* lat, uint16_t m, int lane) {
  using L = Lat<K, KF>;
  if (lane >= L::N2) return;
  const int u = lane % L::N, v = lane / L::N;
  if (!line_hangs<K, D>(m, u, v)) return;
  constexpr int S = D == 0 ? 1 : (D == 1 ? L::M : L::M2);
  T* p = lat + (D == 0 ? L::M * u + L::M2 * v : (D == 1 ? u + L::M2 * v : u + L::M * v));
  T x[L::N];
#pragma unroll
  for (int a = 0; a < L::N; ++a) x[a] = p[a * S];
  interp_line_reg<K, TRANS>(x, (m >> D) & 1);
#pragma unroll
  for (int a = 0; a < L::N; ++a) p[a * S] = x[a];
}

template <int K, typename T, int KF>
constexpr size_t prolong_smem() {
  using L = Lat<K, KF>;
  return ((size_t)(L::NI + L::NJ) * 32 + (size_t)WPB * (L::ES + 32)) * 4 + (size_t)WPB * L::LS * sizeof(T);
}

template <int K, typename T, int KF>
__global__ void __launch_bounds__(WPB * 32) prolong_lattice(LatArgs<T> A) {
  using L = Lat<K, KF>;
  constexpr int N = L::N, N3 = L::N3, M = L::M, M2 = L::M2;
  constexpr int NT = WPB * 32;
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  T* lat = reinterpret_cast<T*>(smem) + w * L::LS;
  uint32_t* s_pt = reinterpret_cast<uint32_t*>(smem + (size_t)WPB * L::LS * sizeof(T));
  uint32_t* s_nd = s_pt + L::NI * 32;
  int32_t* ent = reinterpret_cast<int32_t*>(s_nd + L::NJ * 32) + w * (L::ES + 32);
  int32_t* gsc = ent + L::ES;
  const int c = blockIdx.x * WPB + w;
  for (int i = threadIdx.x; i < L::NI * 32; i += NT) cp_async(s_pt + i, L::points() + i);
  for (int i = threadIdx.x; i < L::NJ * 32; i += NT) cp_async(s_nd + i, L::nodes() + i);
  uint16_t m = 0;
  if (c < A.n_coarse) {
    int32_t en[L::EPL];
    L::words(A, c, lane, en);
#pragma unroll
    for (int i = 0; i < L::EPL; ++i) ent[lane + 32 * i] = en[i];
    if (lane < NSLOT) cp_async(gsc + lane, A.gstart_c + (size_t)c * NSLOT + lane);
    m = A.mask_c[c];
  }
  cp_async_wait_all();
  pdl_wait();
  __syncthreads();
  if (c >= A.n_coarse) return;
  {  // G^(c)
    T v[L::NJ];
    int pos[L::NJ];
#pragma unroll
    for (int i = 0; i < L::NJ; ++i) {
      const int n = lane + 32 * i;
      const uint32_t p = s_nd[n];
      pos[i] = p >> 12;
      v[i] = T(0);
      if (n < N3) {
        const int32_t g = gsc[p & 127];
        if (g >= 0) v[i] = A.src[g + (int)((p >> 7) & 31)];
      }
    }
#pragma unroll
    for (int i = 0; i < L::NJ; ++i)
      if (lane + 32 * i < N3) lat[pos[i]] = v[i];
  }
  __syncwarp();
  if (m & MASK_HANG) {  // C^(c) (uniform over the warp)
    lattice_hang<K, KF, 0, false>(lat, m, lane);
    __syncwarp();
    lattice_hang<K, KF, 1, false>(lat, m, lane);
    __syncwarp();
    lattice_hang<K, KF, 2, false>(lat, m, lane);
    __syncwarp();
  }
  if (KF || ent[L::ES - 1] > 0) {
    if (lane < N * N) {  // x-lines (b, c)
      T* p = lat + M * (lane % N) + M2 * (lane / N);
      T v[M];
#pragma unroll
      for (int i = 0; i < N; ++i) v[i] = p[i];
      L::up(v);
#pragma unroll
      for (int i = 0; i < M; ++i) p[i] = v[i];
    }
    __syncwarp();
#pragma unroll 1
    for (int q = lane; q < M * N; q += 32) {  // y-lines (x, c)
      T* p = lat + q % M + M2 * (q / M);
      T v[M];
#pragma unroll
      for (int i = 0; i < N; ++i) v[i] = p[M * i];
      L::up(v);
#pragma unroll
      for (int i = 0; i < M; ++i) p[M * i] = v[i];
    }
    __syncwarp();
#pragma unroll 1
    for (int q = lane; q < M2; q += 32) {  // z-lines
      T v[M];
#pragma unroll
      for (int i = 0; i < N; ++i) v[i] = lat[q + M2 * i];
      L::up(v);
#pragma unroll
      for (int i = 0; i < M; ++i) lat[q + M2 * i] = v[i];
    }
    __syncwarp();
    // owner-selected additions (each fine DoF once: red.add gives the read-modify-write's sum)
#pragma unroll
    for (int i = 0; i < L::NI; ++i) {
      const uint32_t p = s_pt[lane + 32 * i];
      const int32_t g = ent[p & 127];
      if (g >= 0) atomicAdd(A.dst + g + (int)((p >> 7) & 31), lat[p >> 12]);
    }
  } else {
#pragma unroll
    for (int i = 0; i < L::NJ; ++i) {
      const int n = lane + 32 * i;
      const uint32_t p = s_nd[n];
      const int32_t g = ent[p & 127];
      if (n < N3 && g >= 0) atomicAdd(A.dst + g + (int)((p >> 7) & 31), lat[p >> 12]);
    }
  }
}

// restriction onto a level of few cells: the coarse cell's result to its cell
// vector (kernels_small.cu adds them up)
template <int K, typename T, int KF>
__global__ void __launch_bounds__(WPB * 32) restrict_cells(LatArgs<T> A) {
  using L = Lat<K, KF>;
  constexpr int N3 = L::N3;
  constexpr int NT = WPB * 32;
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  T* lat = reinterpret_cast<T*>(smem) + w * L::LS;
  uint32_t* s_pt = reinterpret_cast<uint32_t*>(smem + (size_t)WPB * L::LS * sizeof(T));
  uint32_t* s_nd = s_pt + L::NI * 32;
  int32_t* ent = reinterpret_cast<int32_t*>(s_nd + L::NJ * 32) + w * (L::ES + 32);
  const int c = blockIdx.x * WPB + w;
  for (int i = threadIdx.x; i < L::NI * 32; i += NT) cp_async(s_pt + i, L::points() + i);
  for (int i = threadIdx.x; i < L::NJ * 32; i += NT) cp_async(s_nd + i, L::nodes() + i);
  uint16_t m = 0;
  if (c < A.n_coarse) {
    int32_t en[L::EPL];
    L::words(A, c, lane, en);
#pragma unroll
    for (int i = 0; i < L::EPL; ++i) ent[lane + 32 * i] = en[i];
    m = A.mask_c[c];
  }
  cp_async_wait_all();
  pdl_wait();
  __syncthreads();
  if (c >= A.n_coarse) return;
  const T* __restrict__ src = A.src;
  const T* __restrict__ rhs = A.rhs;
  if (KF || ent[L::ES - 1] > 0) {
    T v[L::NI];
#pragma unroll
    for (int i = 0; i < L::NI; ++i) {
      const uint32_t p = s_pt[lane + 32 * i];
      const int32_t g = ent[p & 127];
      v[i] = T(0);
      if (g >= 0) {
        const int gi = g + (int)((p >> 7) & 31);
        v[i] = rhs ? rhs[gi] - src[gi] : src[gi];
      }
    }
#pragma unroll
    for (int i = 0; i < L::NI; ++i) lat[s_pt[lane + 32 * i] >> 12] = v[i];
    __syncwarp();
    lattice_down<L>(lat, lane, [](T* p, int i, T x) { p[i] = x; });
  } else {  // identity category (no fine cells: no owned slots, zeros)
#pragma unroll
    for (int i = 0; i < L::NJ; ++i) {
      const uint32_t p = s_nd[lane + 32 * i];
      const int32_t g = ent[p & 127];
      T v = T(0);
      if (g >= 0) {
        const int gi = g + (int)((p >> 7) & 31);
        v = rhs ? rhs[gi] - src[gi] : src[gi];
      }
      lat[p >> 12] = v;
    }
  }
  __syncwarp();
  if (m & MASK_HANG) {  // C^(c)T
    lattice_hang<K, KF, 2, true>(lat, m, lane);
    __syncwarp();
    lattice_hang<K, KF, 1, true>(lat, m, lane);
    __syncwarp();
    lattice_hang<K, KF, 0, true>(lat, m, lane);
    __syncwarp();
  }
#pragma unroll
  for (int i = 0; i < L::NJ; ++i) {
    const int n = lane + 32 * i;
    if (n < N3) A.dst[(size_t)c * N3 + n] = lat[s_nd[n] >> 12];
  }
}

// entity table: word e of coarse cell c; one thread per word
__global__ void __launch_bounds__(BLOCK) lattice_entities(int k, int n_coarse, const int32_t* __restrict__ fine_of,
                                                          const uint8_t* __restrict__ refined,
                                                          const int32_t* __restrict__ gstart_f,
                                                          const uint32_t* __restrict__ own_f,
                                                          int32_t* __restrict__ ent) {
  const int es = lat_words(k);
  const int64_t t = blockIdx.x * (int64_t)BLOCK + threadIdx.x;
  const int c = (int)(t / es), e = (int)(t % es);
  if (c >= n_coarse) return;
  int32_t out = -1;
  const int f = fine_of[c];
  if (e == es - 1) {
    out = refined[c] ? 1 : 0;
  } else if (f >= 0) {
    int q = 0, slot = -1;
    if (!refined[c]) {
      if (e < NSLOT) slot = e;
    } else {
      const int ne = k == 1 ? 3 : 5;  // entities per axis (k = 1: the three vertices)
      if (e < ne * ne * ne) {
        int x[3] = {e % ne, (e / ne) % ne, e / (ne * ne)}, mul = 1;
        slot = 0;
        for (int d = 0; d < 3; ++d) {
          const int p = k == 1 ? 2 * x[d] : x[d];     // 0, 2, 4: vertices; 1, 3: interiors
          q |= (p > 2 ? 1 : 0) << d;                   // the lowest child that holds it
          slot += mul * (p > 2 ? p - 2 : p);
          mul *= 3;
        }
      }
    }
    if (slot >= 0 && ((own_f[f + q] >> slot) & 1u)) out = gstart_f[(size_t)(f + q) * NSLOT + slot];
  }
  ent[t] = out;
}

void fill_lattice(LatTables& t) {
  std::memset(&t, 0, sizeof(t));
  for (int k = 1; k <= KMAX; ++k) {
    const int n = k + 1, m = 2 * k + 1, ne = k == 1 ? 3 : 5;
    // lattice points of entity (x, y, z), its interior lexicographic
    auto range = [&](int x, int& i0, int& i1) {
      const int p = k == 1 ? 2 * x : x;
      i0 = p == 0 ? 0 : (p == 1 ? 1 : (p == 2 ? k : (p == 3 ? k + 1 : 2 * k)));
      i1 = (p & 1) ? i0 + k - 1 : i0 + 1;
    };
    std::vector<std::vector<uint32_t>> by_dim(4);
    for (int e = 0; e < ne * ne * ne; ++e) {
      int a0, a1, b0, b1, c0, c1, off = 0;
      range(e % ne, a0, a1);
      range((e / ne) % ne, b0, b1);
      range(e / (ne * ne), c0, c1);
      const int dim = (a1 - a0 > 1 || (k == 2 && (e % ne) % 2)) + (b1 - b0 > 1 || (k == 2 && ((e / ne) % ne) % 2)) +
                      (c1 - c0 > 1 || (k == 2 && (e / (ne * ne)) % 2));
      for (int c = c0; c < c1; ++c)
        for (int b = b0; b < b1; ++b)
          for (int a = a0; a < a1; ++a)
            by_dim[dim].push_back((uint32_t)e | ((uint32_t)off++ << 7) | ((uint32_t)(a + m * (b + m * c)) << 12));
    }
    int i = 0;
    for (int d = 3; d >= 0; --d)  // interiors first, as the DoFs of a tile are numbered
      for (uint32_t p : by_dim[d]) t.pt[k][i++] = p;
    const uint32_t pad = (uint32_t)(lat_words(k) - 2) | ((uint32_t)(m * m * m) << 12);  // a word that is -1
    for (; i < PT_MAX; ++i) t.pt[k][i] = pad;
    i = 0;
    for (int c = 0; c < n; ++c)
      for (int b = 0; b < n; ++b)
        for (int a = 0; a < n; ++a) {
          int slot, off;
          host_node_slot(k, a, b, c, slot, off);
          t.nd[k][i++] = (uint32_t)slot | ((uint32_t)off << 7) | ((uint32_t)(a + m * (b + m * c)) << 12);
        }
    for (; i < ND_MAX; ++i) t.nd[k][i] = pad;
    if (k < 2) continue;
    // p: slots by dimension (interior, faces, edges, vertices); a word beyond the slots is -1
    i = 0;
    for (int d = 3; d >= 0; --d)
      for (int s = 0; s < NSLOT; ++s) {
        const int x[3] = {s % 3, (s / 3) % 3, s / 9};
        if ((x[0] == 1) + (x[1] == 1) + (x[2] == 1) != d) continue;
        int lo[3], hi[3], off = 0;
        for (int e = 0; e < 3; ++e) {
          lo[e] = x[e] == 0 ? 0 : (x[e] == 1 ? 1 : k);
          hi[e] = x[e] == 1 ? k : lo[e] + 1;
        }
        for (int c = lo[2]; c < hi[2]; ++c)
          for (int b = lo[1]; b < hi[1]; ++b)
            for (int a = lo[0]; a < hi[0]; ++a)
              t.pf[k][i++] = (uint32_t)s | ((uint32_t)off++ << 7) | ((uint32_t)(a + n * (b + n * c)) << 12);
      }
    for (; i < ND_MAX; ++i) t.pf[k][i] = (uint32_t)NSLOT | ((uint32_t)(n * n * n) << 12);
    i = 0;
    const int kc = k / 2;
    for (int c = 0; c <= kc; ++c)
      for (int b = 0; b <= kc; ++b)
        for (int a = 0; a <= kc; ++a) {
          int slot, off;
          host_node_slot(kc, a, b, c, slot, off);
          t.pc[k][i++] = (uint32_t)slot | ((uint32_t)off << 7) | ((uint32_t)(a + n * (b + n * c)) << 12);
        }
    for (; i < 32; ++i) t.pc[k][i] = (uint32_t)NSLOT | ((uint32_t)(n * n * n) << 12);
  }
}

// E_ia = (P_ia + P_i,k-a) / 2, O_ia = (P_ia - P_i,k-a) / 2 for rows 1 <= i < k;
// the middle column (k even) and the middle row i = k (k odd) undivided
void fill_sweeps(LatSweeps<double>& d, LatSweeps<float>& f) {
  std::memset(&d, 0, sizeof(d));
  for (int k = 1; k <= KMAX; ++k) {
    const Basis1D& b = basis(k);
    for (int i = 1; i <= k; ++i)
      for (int a = 0; a < (k + 2) / 2; ++a) {
        const double p = b.Ph[i][a], q = b.Ph[i][k - a];
        d.e[k][i][a] = (2 * a == k || i == k) ? p : 0.5 * (p + q);
        if (2 * a < k && i < k) d.o[k][i][a] = 0.5 * (p - q);
      }
  }
  const double* s = reinterpret_cast<const double*>(&d);
  float* o = reinterpret_cast<float*>(&f);
  for (size_t i = 0; i < sizeof(d) / sizeof(double); ++i) o[i] = (float)s[i];
}

template <typename T>
LatArgs<T> lat_args(const TransferLaunch& L, const T* src, T* dst) {
  LatArgs<T> A{};
  A.ent = L.lattice;
  A.gstart_f = L.gstart_f;
  A.own_f = L.own_f;
  A.gstart_c = L.gstart_c;
  A.mask_c = L.mask_c;
  A.n_coarse = L.n_coarse;
  A.src = src;
  A.dst = dst;
  A.tiles = L.coarse.tiles;
  A.lt = static_cast<const LaneTile*>(L.coarse.lane_tiles);
  A.lh = static_cast<const LaneHang*>(L.coarse.lane_hang);
  A.halo = static_cast<T*>(L.coarse.halo);
  A.halo_pos = L.coarse.halo_pos;
  return A;
}

template <int K, typename T, int KF = 0>
void run_prolong(const TransferLaunch& L, const T* src, T* dst, cudaStream_t s) {
  const LatArgs<T> A = lat_args(L, src, dst);
  constexpr size_t sm = prolong_smem<K, T, KF>();
  smem_allow(prolong_lattice<K, T, KF>, sm);
  launch_pdl(prolong_lattice<K, T, KF>, (L.n_coarse + WPB - 1) / WPB, WPB * 32, sm, s, A);
  note_launches(1);
}

template <int K, typename T, int KF = 0>
void run_restrict(const TransferLaunch& L, const T* src, T* dst, const T* rhs, bool ow, cudaStream_t s) {
  LatArgs<T> A = lat_args(L, src, dst);
  A.rhs = rhs;
  A.overwrite = ow;
  const size_t sm = RestrictSmem<K, T, KF>::total(L.coarse.max_local);
  smem_allow(restrict_lattice<K, T, KF>, sm);
  launch_pdl(restrict_lattice<K, T, KF>, L.coarse.n_tiles, WPB * 32, sm, s, A);
  note_launches(1);
  launch_halo_add(L.coarse, sizeof(T) == 8, dst, s);
}

template <int K, typename T, int KF = 0>
void run_restrict_cells(const TransferLaunch& L, const T* src, const T* rhs, cudaStream_t s) {
  LatArgs<T> A = lat_args(L, src, static_cast<T*>(L.coarse.cell_vec));
  A.rhs = rhs;
  constexpr size_t sm = prolong_smem<K, T, KF>();
  smem_allow(restrict_cells<K, T, KF>, sm);
  launch_pdl(restrict_cells<K, T, KF>, (L.n_coarse + WPB - 1) / WPB, WPB * 32, sm, s, A);
  note_launches(1);
}

// run F<coarse degree, T, fine degree of a p transfer> for the transfer L
#define GCMG_BY_DEGREE(F, T, ...)                                 \
  if (L.kind == 0) switch (L.kf) {                                \
      case 1: F<1, T>(__VA_ARGS__); break;                        \
      case 2: F<2, T>(__VA_ARGS__); break;                        \
      case 3: F<3, T>(__VA_ARGS__); break;                        \
      case 4: F<4, T>(__VA_ARGS__); break;                        \
    }                                                             \
  else switch (L.kf) {                                            \
      case 2: F<1, T, 2>(__VA_ARGS__); break;                     \
      case 3: F<1, T, 3>(__VA_ARGS__); break;                     \
      case 4: F<2, T, 4>(__VA_ARGS__); break;                     \
    }

template <typename T>
void prolong_any(const TransferLaunch& L, const T* src, T* dst, cudaStream_t s) {
  GCMG_BY_DEGREE(run_prolong, T, L, src, dst, s)
}

template <typename T>
void restrict_any(const TransferLaunch& L, const T* src, T* dst, const T* rhs, bool ow, cudaStream_t s) {
  GCMG_BY_DEGREE(run_restrict, T, L, src, dst, rhs, ow, s)
}

template <typename T>
void restrict_cells_any(const TransferLaunch& L, const T* src, const T* rhs, cudaStream_t s) {
  GCMG_BY_DEGREE(run_restrict_cells, T, L, src, rhs, s)
}
#undef GCMG_BY_DEGREE

}  // namespace

void upload_tables_lattice() {
  upload_tables_lattice_1d();
  static LaneLines ll;
  fill_lane_lines(ll);
  cudaMemcpyToSymbol(c_ll, &ll, sizeof(ll));
  static LatTables t;
  fill_lattice(t);
  cudaMemcpyToSymbol(g_lat, &t, sizeof(t));
  static LatSweeps<double> sd;
  static LatSweeps<float> sf;
  fill_sweeps(sd, sf);
  cudaMemcpyToSymbol(c_swd, &sd, sizeof(sd));
  cudaMemcpyToSymbol(c_swf, &sf, sizeof(sf));
}

size_t lattice_table_words(int k, int n_coarse) { return (size_t)n_coarse * lat_words(k); }

void launch_lattice_entities(const TransferLaunch& L, int32_t* ent, cudaStream_t s) {
  const int64_t n = (int64_t)lattice_table_words(L.kf, L.n_coarse);
  if (n == 0) return;
  launch_pdl(lattice_entities, (unsigned)((n + BLOCK - 1) / BLOCK), BLOCK, 0, s, L.kf, L.n_coarse, L.fine_of, L.refined,
             L.gstart_f, L.own_f, ent);
  note_launches(1);
}

// The restriction accumulates through the coarse level's lane records, which
// exist for tiles of at most 32 cells, and reads its record per tile: larger
// tiles keep restrict_h.
bool lattice_restrict_ok(const TransferLaunch& L) { return L.coarse.lane_tiles && L.coarse.tc <= 32; }

void launch_prolong_lattice(const TransferLaunch& L, bool fp64, const void* coarse, void* fine, cudaStream_t s) {
  if (fp64)
    prolong_any(L, static_cast<const double*>(coarse), static_cast<double*>(fine), s);
  else
    prolong_any(L, static_cast<const float*>(coarse), static_cast<float*>(fine), s);
}

void launch_restrict_cells(const TransferLaunch& L, bool fp64, const void* fine, const void* rhs, cudaStream_t s) {
  if (fp64)
    restrict_cells_any(L, static_cast<const double*>(fine), static_cast<const double*>(rhs), s);
  else
    restrict_cells_any(L, static_cast<const float*>(fine), static_cast<const float*>(rhs), s);
}

void launch_restrict_lattice(const TransferLaunch& L, bool fp64, const void* fine, const void* rhs, void* coarse,
                             bool overwrite, cudaStream_t s) {
  if (fp64)
    restrict_any(L, static_cast<const double*>(fine), static_cast<double*>(coarse), static_cast<const double*>(rhs),
                 overwrite, s);
  else
    restrict_any(L, static_cast<const float*>(fine), static_cast<float*>(coarse), static_cast<const float*>(rhs),
                 overwrite, s);
}

}  // namespace gcmg
