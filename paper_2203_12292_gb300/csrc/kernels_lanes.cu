// fp32 tile kernel of the cell loop of Eq. 2 with one lane per cell:
//   v = sum_e G_e^T C_e^T S_e^T Q_e S_e C_e G_e x
//
// A tile holds at most 32 consecutive (Morton-ordered) cells; lane j of every
// warp works on cell j, and the k+1 warps of the CTA share the (k+1)^2 1D
// lines of each direction.  All lanes of a warp therefore touch the same
// local node of 32 different cells at once, so
//   * the cell buffer is node-major (node n of cell j at n * 32 + j): every
//     access to it, in every direction, reads or writes 32 consecutive words
//     (no bank conflicts), and all indexing except the DoF gather/scatter is
//     uniform across the warp;
//   * the entity starts of the tile are stored transposed (slot s of cell j
//     at s * 32 + j), read conflict-free.
// The sweeps apply the fast-diagonalisation form of the Cartesian cell matrix
// h (K x M x M + M x K x M + M x M x K) in two directions, with the even-odd
// split of B (rows of B are symmetric or antisymmetric under x -> 1 - x), and
// K + (lam + lam') M in the innermost one (zline.cuh).
//
// Accumulation without atomics and in a fixed order.  Two local nodes of
// different cells can be the same DoF only if, along every axis, their
// coordinates are equal or both lie on the cell boundary (0 or k); the same
// holds through hanging faces and edges, whose slots point to the coarse
// entity with the same local offsets.
//   * fp32, tiles without hanging cells: warp w keeps the z-plane c = w of
//     its lane's cell in registers (gather, x and y sweeps forward; the z
//     phase through the cell buffer; y and x sweeps backward and the scatter).
//     The cell buffer and the tile's DoF buffer share one shared-memory
//     region (gathers finish before the cell buffer is written, the
//     accumulator is cleared after its last read; the tiles with hanging
//     cells hold their x-lines in registers across those points), so 8
//     blocks of 48 registers fit an SM at k = 4.
//     Planes c = 0 and c = k are the only ones that meet, so warp k adds after
//     warp 0 (a named barrier); a warp adds its nodes in program order.
//   * tiles with hanging cells, and the double-float kernel: the x-lines
//     (b, c) are grouped into classes by (b or "boundary", c or "boundary");
//     each class is given to one warp, so two warps never add to the same
//     DoF.  Within one instruction two lanes add to the same DoF only through
//     hanging slots (siblings behind one coarse face or edge); they take turns
//     in lane order, with ranks from the set-up (LaneHang).  These tiles apply C_e and C_e^T (Sec. 3.2,
//     direction by direction) between separate passes.
// The sums are therefore reproducible bit for bit.
#include <algorithm>

#include "device.cuh"
#include "kernels.h"
#include "lanes.cuh"
#include "zline.cuh"

namespace gcmg {

GCMG_DEFINE_UPLOAD(upload_tables_lanes_1d)

namespace {

template <typename T>
struct LaneArgsT {
  const TileInfo* tiles;
  const LaneTile* lt;
  const LaneHang* lh;    // per tile: hanging lines and slots of every lane
  const int32_t* order;  // tile of block b: order[b] (null: tile0 + b)
  const TileInfo* tiles_lo;  // with order: block b's TileInfo, LaneTile, LaneHang at [b]
  const LaneTile* lt_lo;
  const LaneHang* lh_lo;
  int n_hang;            // with order: blocks below n_hang have tiles with hanging cells
  const int32_t* foreign;
  const int32_t* halo_pos;
  const T* src;
  T* dst;
  T* halo;
  const double* coef;  // per cell nu_e, null: 1
  double dom;
  int add;
  int tile0;
};
using LaneArgs = LaneArgsT<float>;

// base node of line q = u + N v along D
template <int K, int D>
__device__ __forceinline__ int line_base(int q) {
  constexpr int N = K + 1, N2 = N * N;
  return D == 0 ? N * q : (D == 1 ? q % N + N2 * (q / N) : q);
}

// one direction D of C_e (TRANS: C_e^T) on the lines of warp w; lane j
// interpolates when the line lies on a hanging face or edge of its cell.  SWEEP
// (D = 2 only): the z sweep follows (forward after C_z) or precedes (backward
// before C_z^T) the interpolation on the same lines.
template <int K, int D, bool TRANS, bool SWEEP = false>
__device__ __forceinline__ void hang_pass(float* cb, uint16_t m, uint32_t hlD, int w, int lane) {
  constexpr int N = K + 1, N2 = N * N;
  constexpr int S = (D == 0 ? 1 : (D == 1 ? N : N2)) * 32;
  const DevTables<float>& tb = tab<float>(K);
  const int p = (m >> D) & 1;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const int q = c_ll.bl[K][w][i];
    const bool hl = (hlD >> q) & 1u;
    if (!SWEEP && !hl) continue;
    float* ptr = cb + line_base<K, D>(q) * 32 + lane;
    float x[N];
#pragma unroll
    for (int a = 0; a < N; ++a) x[a] = ptr[a * S];
    if (SWEEP && TRANS) eo_backward<N, 0, 1>(x, tb.Be);
    if (hl) interp_line_reg<K, TRANS>(x, p);
    if (SWEEP && !TRANS) eo_forward<N, 0, 1>(x, tb.Be);
#pragma unroll
    for (int a = 0; a < N; ++a) ptr[a * S] = x[a];
  }
}

// zero the accumulator (n floats from the 16-byte aligned x0)
__device__ __forceinline__ void clear_acc(float* x0, int n, int nt) {
  float4* z4 = reinterpret_cast<float4*>(x0);
  for (int i = threadIdx.x; i < (n + 3) / 4; i += nt) z4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// named barrier `id` of n threads: producers arrive, consumers wait
__device__ __forceinline__ void named_bar_sync(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void named_bar_arrive(int id, int n) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// the three gather/scatter addresses of x-line r of the cell in this lane:
// node (0, b, c), first interior node (1, b, c), node (k, b, c)
template <int K>
__device__ __forceinline__ void xline_ptrs(const LaneTile* st, char* xb, int r, int lane, float*& p0, float*& p1,
                                           float*& p2) {
  const uint32_t li = c_ll.line[K][r];
  const int s0 = li & 0xff, o0 = (li >> 8) & 0xff, o1 = li >> 16;
  p0 = reinterpret_cast<float*>(xb + st->ls[s0][lane] + o0);
  p1 = reinterpret_cast<float*>(xb + st->ls[s0 + 1][lane] + o1);
  p2 = reinterpret_cast<float*>(xb + st->ls[s0 + 2][lane] + o0);
}

// y sweep on the lines (a, c) = (i, w) of warp w
template <int K, bool FWD>
__device__ __forceinline__ void sweep_y(float* cb, int w, int lane) {
  constexpr int N = K + 1, N2 = N * N;
  const DevTables<float>& tb = tab<float>(K);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    float* p = cb + (i + N2 * w) * 32 + lane;
    float v[N];
#pragma unroll
    for (int b = 0; b < N; ++b) v[b] = p[b * N * 32];
    if (FWD)
      eo_forward<N, 0, 1>(v, tb.Be);
    else
      eo_backward<N, 0, 1>(v, tb.Be);
#pragma unroll
    for (int b = 0; b < N; ++b) p[b * N * 32] = v[b];
  }
}

// Blocks per SM that the registers are limited for: dense (many regular tiles: more
// warps hide the block start's chain of loads, at the price of a few spills) or
// roomy (what the code of hanging cells and a level of one wave prefer).  fp32, dense
// against roomy: Q4 octant 108 / 112 us, Q3 octant 71 / 76.5 us, Q2 octant 30.1 / 31.5
// us; Q4 sphere (hanging cells in most tiles) 60 / 56.4 us, Q4 cube of 32,768 cells
// (one wave) 15.2 / 14.4 us, Q3 octant of 34,903 cells 16.8 / 15.8 us.  fp64: Q4 octant
// 447 / 451 us, Q3 octant 233 / 242 us, Q2 octant 82.5 / 84.6 us (438, 233, 84.2 with the
// differences of zline.cuh); Q4 sphere 227 / 220
// us, Q2 sphere 53.3 / 52.6 us.
constexpr int lanes_blocks(int K, bool dense) { return K == 4 ? (dense ? 8 : 7) : !dense ? 1 : K == 3 ? 10 : 14; }
constexpr int lanes_df_blocks(int K, bool dense) { return K == 4 ? (dense ? 6 : 5) : !dense ? 1 : K == 3 ? 8 : 10; }
// blocks per SM of the roomy variants as built
constexpr int lanes_roomy(int K) { return K == 4 ? 7 : K == 3 ? 8 : 12; }
constexpr int lanes_df_roomy(int K) { return K == 4 ? 5 : K == 3 ? 6 : 10; }
// by the level, not by the launch: every range of a level's tiles takes the same code
bool lanes_dense(const CellLaunch& L, int roomy_blocks) {
  return 2 * L.n_hang_tiles <= L.n_tiles && L.n_tiles > roomy_blocks * L.n_sm;
}

template <int K, bool DENSE>
__global__ void __launch_bounds__((K + 1) * 32, lanes_blocks(K, DENSE)) vmult_lanes(LaneArgs A) {
  pdl_begin();
  constexpr int N = K + 1, N2 = N * N, NT = N * 32;
  extern __shared__ __align__(16) unsigned char smem[];
  LaneTile* st = reinterpret_cast<LaneTile*>(smem);
  LaneHang* hg = reinterpret_cast<LaneHang*>(smem + sizeof(LaneTile));
  // the cell buffer and the tile's DoF buffer (input, then accumulator) share one region: the
  // DoFs are gathered into registers before the cell buffer is written, and the accumulator
  // is cleared after the cell buffer's last read (8 instead of 7 blocks per SM at k = 4)
  float* cb = reinterpret_cast<float*>(smem + sizeof(LaneTile) + sizeof(LaneHang));
  float* xs0 = cb;  // 16-byte aligned
  const int lane = threadIdx.x & 31, w = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);  // w: uniform
  // block b's tile: records in launch order at [b] (no dependent load of the tile index) or tile0 + b
  const int bx = blockIdx.x, tl = A.tile0 + bx;
  const LaneTile* ltp = A.order ? A.lt_lo + bx : A.lt + tl;
  const LaneHang* lhp = A.order ? A.lh_lo + bx : A.lh + tl;
  const TileInfo ti = A.order ? A.tiles_lo[bx] : A.tiles[tl];
  const int nloc = ti.n_owned + ti.n_foreign;
  // tile DoF i at xs[i] (then the zero region; later the accumulator): xs + i is 16-byte aligned
  // exactly where src + dof_begin + i is, so the owned range moves in 16-byte pieces
  const float* so = A.src + ti.dof_begin;
  const int sh = (int)((reinterpret_cast<uintptr_t>(so) >> 2) & 3);
  float* xs = xs0 + sh;
  const int h0 = min((4 - sh) & 3, ti.n_owned), nv = (ti.n_owned - h0) >> 2;
  {  // asynchronous copies of the lane metadata and the tile's DoFs, all in flight at once
    const uint4* g = reinterpret_cast<const uint4*>(ltp);
    uint4* s = reinterpret_cast<uint4*>(st);
    for (int i = threadIdx.x; i < (int)(sizeof(LaneTile) / 16); i += NT) cp_async16(s + i, g + i);
    if (!A.order || (int)blockIdx.x < A.n_hang) {  // the tile has hanging cells (or may have)
      const uint4* gh = reinterpret_cast<const uint4*>(lhp);
      uint4* shh = reinterpret_cast<uint4*>(hg);
      for (int i = threadIdx.x; i < (int)(sizeof(LaneHang) / 16); i += NT) cp_async16(shh + i, gh + i);
    }
    if (threadIdx.x < h0) cp_async(xs + threadIdx.x, so + threadIdx.x);
#pragma unroll 4
    for (int j = threadIdx.x; j < nv; j += NT) cp_async16(xs + h0 + 4 * j, so + h0 + 4 * j);
    for (int i = h0 + 4 * nv + threadIdx.x; i < ti.n_owned; i += NT) cp_async(xs + i, so + i);
    const int32_t* fl = A.foreign + ti.foreign_begin;
    float* xf = xs + ti.n_owned;
    for (int i0 = threadIdx.x; i0 < ti.n_foreign; i0 += 4 * NT) {
      int idx[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) idx[u] = (i0 + u * NT < ti.n_foreign) ? fl[i0 + u * NT] : -1;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (idx[u] >= 0) cp_async(xf + i0 + u * NT, A.src + idx[u]);
    }
  }
  if (threadIdx.x < LANE_ZERO) xs[nloc + threadIdx.x] = 0.f;
  cp_async_wait_all();
  __syncthreads();

  const DevTables<float>& tb = tab<float>(K);
  const uint16_t m = st->mask[lane];
  const bool hang = st->hang != 0;  // uniform over the CTA
  float h;
  {
    const int c = ti.cell_begin + min(lane, ti.n_cells - 1);
    const double hd = ldexp(A.dom, -(int)st->level[lane]);
    h = (float)(A.coef ? hd * A.coef[c] : hd);
  }
  char* xb = reinterpret_cast<char*>(xs);
  const int nxl = c_ll.nx[K][w];

  if (!hang) {
    // Warp w holds the plane c = w of its cell in registers: G_e, the x and y
    // sweeps forward; the z phase through the cell buffer; the y and x sweeps
    // backward and G_e^T, again on the plane in registers.
    //   Plane x-lines (b, w): node (0, b, w) lies in slot 9 cls(w) + 3 cls(b),
    // nodes (1..k-1, b, w) in the slot after it, node (k, b, w) two after it;
    // their offsets in the entities are the same for b = 0 and b = k and grow
    // by one x-step (node (0, .)) or one x-line of the entity (node (1, .)) per
    // interior b (entity DoFs lexicographic over the interior axes).
    const uint32_t l0 = c_ll.line[K][N * w], l1 = c_ll.line[K][(K > 1 ? 1 : 0) + N * w];
    const uint16_t* lsw = &st->ls[l0 & 0xff][lane];
    const char* xA0 = xb + ((l0 >> 8) & 0xff);  // node (0, b, w), b = 0 or k
    const char* xA1 = xb + (l0 >> 16);          // node (1, b, w), b = 0 or k
    const char* xB0 = xb + ((l1 >> 8) & 0xff);  // node (0, 1, w)
    const char* xB1 = xb + (l1 >> 16);          // node (1, 1, w)
    float u[N2];
#pragma unroll
    for (int b = 0; b < N; ++b) {
      const bool in = b > 0 && b < K;
      const int sb = b == 0 ? 0 : (b == K ? 6 : 3);
      const int q0 = lsw[(sb + 0) * 32], q1 = lsw[(sb + 1) * 32], q2 = lsw[(sb + 2) * 32];
      const float* p0 = reinterpret_cast<const float*>((in ? xB0 : xA0) + q0) + (in ? b - 1 : 0);
      const float* p1 = reinterpret_cast<const float*>((in ? xB1 : xA1) + q1) + (in ? (b - 1) * (K - 1) : 0);
      const float* p2 = reinterpret_cast<const float*>((in ? xB0 : xA0) + q2) + (in ? b - 1 : 0);
      u[N * b] = *p0;
#pragma unroll
      for (int a = 1; a < K; ++a) u[N * b + a] = p1[a - 1];
      u[N * b + K] = *p2;
    }
    __syncthreads();  // every plane gathered: the DoF buffer is dead
#pragma unroll
    for (int b = 0; b < N; ++b) eo_forward<N, 0, 1>(u + N * b, tb.Be);  // x-lines of the plane
#pragma unroll
    for (int a = 0; a < N; ++a) eo_forward<N, 0, N>(u + a, tb.Be);  // y-lines
    {
      float* p = cb + (N2 * w) * 32 + lane;
#pragma unroll
      for (int n = 0; n < N2; ++n) p[n * 32] = u[n];
    }
    __syncthreads();
    // z: h (K + (lam_a + lam_b) M) on the lines of modes (a, b) = (i, w)
#pragma unroll
    for (int i = 0; i < N; ++i) {
      float* p = cb + (i + N * w) * 32 + lane;
      float v[N];
#pragma unroll
      for (int c = 0; c < N; ++c) v[c] = p[c * N2 * 32];
      zline<K>(v, c_zl.h[zline_row(K) + i + N * w], i == 0);
#pragma unroll
      for (int c = 0; c < N; ++c) p[c * N2 * 32] = h * v[c];
    }
    __syncthreads();
    {
      const float* p = cb + (N2 * w) * 32 + lane;
#pragma unroll
      for (int n = 0; n < N2; ++n) u[n] = p[n * 32];
    }
#pragma unroll
    for (int a = 0; a < N; ++a) eo_backward<N, 0, N>(u + a, tb.Be);
#pragma unroll
    for (int b = 0; b < N; ++b) eo_backward<N, 0, 1>(u + N * b, tb.Be);
    __syncthreads();  // every plane loaded: the cell buffer is dead
    clear_acc(xs0, sh + nloc, NT);
    __syncthreads();
    // G_e^T.  Nodes of two cells are one DoF only where every coordinate is
    // equal or both lie on the cell boundary: between planes only c = 0 and
    // c = k meet, so warp k adds after warp 0 (named barrier 1); within a
    // plane the x-lines and their nodes add in program order (add_turns keeps the
    // lanes together from one slot to the next).
    if (w == K) named_bar_sync(1, 64);
#pragma unroll
    for (int b = 0; b < N; ++b) {
      const bool in = b > 0 && b < K;
      const int sb = b == 0 ? 0 : (b == K ? 6 : 3);
      const int q0 = lsw[(sb + 0) * 32], q1 = lsw[(sb + 1) * 32], q2 = lsw[(sb + 2) * 32];
      float* p0 = reinterpret_cast<float*>(const_cast<char*>(in ? xB0 : xA0) + q0) + (in ? b - 1 : 0);
      float* p1 = reinterpret_cast<float*>(const_cast<char*>(in ? xB1 : xA1) + q1) + (in ? (b - 1) * (K - 1) : 0);
      float* p2 = reinterpret_cast<float*>(const_cast<char*>(in ? xB0 : xA0) + q2) + (in ? b - 1 : 0);
      add_turns<1>(p0, u + N * b, 0, 1);
      if constexpr (K > 1) add_turns<K - 1>(p1, u + N * b + 1, 0, 1);
      add_turns<1>(p2, u + N * b + K, 0, 1);
    }
    if (w == 0) named_bar_arrive(1, 64);
  } else {
    // G_e and C_x on the warp's lines, all gathered before the cell buffer is written
    constexpr int NXW = K <= 2 ? 4 : N;  // x-lines per warp at most (its class in the scatter)
    float v[NXW][N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int r = c_ll.bl[K][w][i];
      float *p0, *p1, *p2;
      xline_ptrs<K>(st, xb, r, lane, p0, p1, p2);
      v[i][0] = *p0;
#pragma unroll
      for (int a = 1; a < K; ++a) v[i][a] = p1[a - 1];
      v[i][K] = *p2;
      if ((hg->hl[0][lane] >> r) & 1u) interp_line_reg<K, false>(v[i], m & 1);
    }
    __syncthreads();  // the DoF buffer is dead
#pragma unroll
    for (int i = 0; i < N; ++i) {
      float* p = cb + N * c_ll.bl[K][w][i] * 32 + lane;
#pragma unroll
      for (int a = 0; a < N; ++a) p[a * 32] = v[i][a];
    }
    __syncthreads();
    hang_pass<K, 1, false>(cb, m, hg->hl[1][lane], w, lane);  // C_y
    __syncthreads();
    hang_pass<K, 2, false, true>(cb, m, hg->hl[2][lane], w, lane);  // C_z, forward z sweep
    __syncthreads();
    sweep_y<K, true>(cb, w, lane);
    __syncthreads();
    // x: h (K + (lam_b + lam_c) M) on the lines of modes (b, c) = (i, w)
#pragma unroll
    for (int i = 0; i < N; ++i) {
      float* p = cb + N * (i + N * w) * 32 + lane;
      float x[N];
#pragma unroll
      for (int a = 0; a < N; ++a) x[a] = p[a * 32];
      zline<K>(x, c_zl.h[zline_row(K) + i + N * w], i == 0);
#pragma unroll
      for (int a = 0; a < N; ++a) p[a * 32] = h * x[a];
    }
    __syncthreads();
    sweep_y<K, false>(cb, w, lane);
    __syncthreads();
    hang_pass<K, 2, true, true>(cb, m, hg->hl[2][lane], w, lane);  // backward z sweep, C_z^T
    __syncthreads();
    hang_pass<K, 1, true>(cb, m, hg->hl[1][lane], w, lane);  // C_y^T
    __syncthreads();
    // C_x^T and G_e^T on the warp's class of x-lines: all lines read before the accumulator
    // (the same region) is cleared
#pragma unroll
    for (int i = 0; i < NXW; ++i)
      if (i < nxl) {
        const float* p = cb + N * c_ll.xw[K][w][i] * 32 + lane;
#pragma unroll
        for (int a = 0; a < N; ++a) v[i][a] = p[a * 32];
      }
    __syncthreads();  // the cell buffer is dead
    clear_acc(xs0, sh + nloc, NT);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NXW; ++i) {
      if (i >= nxl) break;
      const int r = c_ll.xw[K][w][i];
      if ((hg->hl[0][lane] >> r) & 1u) interp_line_reg<K, true>(v[i], m & 1);
      const int s0 = c_ll.line[K][r] & 0xff;
      float *p0, *p1, *p2;
      xline_ptrs<K>(st, xb, r, lane, p0, p1, p2);
      add_turns<1>(p0, v[i], hg->rank[s0][lane], hg->most[s0]);
      if constexpr (K > 1) add_turns<K - 1>(p1, v[i] + 1, hg->rank[s0 + 1][lane], hg->most[s0 + 1]);
      add_turns<1>(p2, v[i] + K, hg->rank[s0 + 2][lane], hg->most[s0 + 2]);
    }
  }
  __syncthreads();
  // owned DoFs: plain stores (or additions), 16 bytes at a time where src and dst are aligned
  // alike; foreign DoFs: into their halo slots
  float* d = A.dst + ti.dof_begin;
  if ((int)((reinterpret_cast<uintptr_t>(d) >> 2) & 3) == sh) {
    if (threadIdx.x < h0) d[threadIdx.x] = A.add ? d[threadIdx.x] + xs[threadIdx.x] : xs[threadIdx.x];
    for (int j = threadIdx.x; j < nv; j += NT) {
      float4 x4 = *reinterpret_cast<const float4*>(xs + h0 + 4 * j);
      float4* d4 = reinterpret_cast<float4*>(d + h0 + 4 * j);
      if (A.add) {
        const float4 o = *d4;
        x4 = make_float4(o.x + x4.x, o.y + x4.y, o.z + x4.z, o.w + x4.w);
      }
      *d4 = x4;
    }
    for (int i = h0 + 4 * nv + threadIdx.x; i < ti.n_owned; i += NT) d[i] = A.add ? d[i] + xs[i] : xs[i];
  } else {
    for (int i = threadIdx.x; i < ti.n_owned; i += NT) d[i] = A.add ? d[i] + xs[i] : xs[i];
  }
  const int32_t* hp = A.halo_pos + ti.foreign_begin;
  for (int i = threadIdx.x; i < ti.n_foreign; i += NT) A.halo[hp[i]] = xs[ti.n_owned + i];
}

// ---------------------------------------------------------------------------
// fp64 operator (the CG operator of the mixed solve and every level of the
// fp64 multigrid) with the same lane-per-cell structure: fp64 vectors in and
// out, all arithmetic in double-float (hi + lo floats, about 48 significand
// bits: error-free two-sum and fused product error, the fp64 tables split
// into high and low parts), on the FP32 pipe, which GB300 has many times
// wider than its FP64 pipe.  Values are converted once on entry to and once
// on exit from the tile; the cell buffer and the accumulator hold df pairs.
// ---------------------------------------------------------------------------
// The passes over the 1D lines as one loop, so that each transform is one piece
// of code: written out pass by pass, the kernel's instructions did not fit the
// instruction caches (the largest stall was "no instruction", 57 % issue
// active).  A pass is one operation on the lines along direction D; its loop over
// the warp's lines holds that operation alone, with the lines' first nodes from a
// table: tests of the operation and divisions in every line's iteration cost 7 to 14
// % (Q4 octant 479 -> 448 us, Q2 octant 98 -> 85 us).  Leaving out the barriers that a
// plane per warp makes unnecessary was no faster (451 us), nor was one quarter of
// the tiles in native fp64 (615 us) or five blocks per SM (451 us).
enum : uint8_t { DF_C = 0, DF_FWD = 4, DF_Z = 8, DF_BWD = 12, DF_CT = 16 };  // bits 0-1: D
__constant__ uint8_t c_df_pass[2][11] = {
    // tiles without hanging cells: x, y forward, z, y, x backward
    {0 | DF_FWD, 1 | DF_FWD, 2 | DF_Z, 1 | DF_BWD, 0 | DF_BWD, 0, 0, 0, 0, 0, 0},
    // with hanging cells: C_x, C_y, C_z and the sweeps in the order z, y, x, and back
    {0 | DF_C, 1 | DF_C, 2 | DF_C, 2 | DF_FWD, 1 | DF_FWD, 0 | DF_Z, 1 | DF_BWD, 2 | DF_BWD, 2 | DF_CT, 1 | DF_CT,
     0 | DF_CT}};
// first node of the warp's i-th line along D, times 32: [k][D][w][i]
__constant__ uint16_t c_df_node[KMAX + 1][3][NMAX][8];

// op(v, i) on the warp's lines, first node ptr + node[i], node stride S * 32
template <int N, typename F>
__device__ __forceinline__ void df_lines(df* cb, const uint16_t* node, int S, F&& op) {
#pragma unroll 1
  for (int i = 0; i < N; ++i) {
    df* ptr = cb + node[i];
    df v[N];
#pragma unroll
    for (int a = 0; a < N; ++a) v[a] = ptr[a * S];
    op(v, i);
#pragma unroll
    for (int a = 0; a < N; ++a) ptr[a * S] = v[a];
  }
}

template <int K, bool DENSE>
__global__ void __launch_bounds__((K + 1) * 32, lanes_df_blocks(K, DENSE)) vmult_lanes_df(LaneArgsT<double> A) {
  constexpr int N = K + 1, N2 = N * N, NT = N * 32;
  extern __shared__ __align__(16) unsigned char smem[];
  LaneTile* st = reinterpret_cast<LaneTile*>(smem);
  LaneHang* hg = reinterpret_cast<LaneHang*>(smem + sizeof(LaneTile));
  // the cell buffer and the tile's DoF buffer (input, then accumulator) share one region, as in
  // vmult_lanes: 6 instead of 4 blocks per SM at k = 4
  df* cb = reinterpret_cast<df*>(smem + sizeof(LaneTile) + sizeof(LaneHang));
  double* xd0 = reinterpret_cast<double*>(cb);  // 16-byte aligned
  const int lane = threadIdx.x & 31, w = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);  // w: uniform
  // block b's tile: records in launch order at [b] (no dependent load of the tile index) or tile0 + b
  const int bx = blockIdx.x, tl = A.tile0 + bx;
  const LaneTile* ltp = A.order ? A.lt_lo + bx : A.lt + tl;
  const LaneHang* lhp = A.order ? A.lh_lo + bx : A.lh + tl;
  const TileInfo ti = A.order ? A.tiles_lo[bx] : A.tiles[tl];
  const int nloc = ti.n_owned + ti.n_foreign;
  {
    const uint4* g = reinterpret_cast<const uint4*>(ltp);
    uint4* s = reinterpret_cast<uint4*>(st);
    for (int i = threadIdx.x; i < (int)(sizeof(LaneTile) / 16); i += NT) cp_async16(s + i, g + i);
    if (!A.order || (int)blockIdx.x < A.n_hang) {  // the tile has hanging cells (or may have)
      const uint4* gh = reinterpret_cast<const uint4*>(lhp);
      uint4* shh = reinterpret_cast<uint4*>(hg);
      for (int i = threadIdx.x; i < (int)(sizeof(LaneHang) / 16); i += NT) cp_async16(shh + i, gh + i);
    }
  }
  pdl_wait();
  // tile DoF i at xd[i] (fp64 on arrival, then df in place; the zero region after it)
  const double* so = A.src + ti.dof_begin;
  const int sh = (int)((reinterpret_cast<uintptr_t>(so) >> 3) & 1);
  double* xd = xd0 + sh;
  df* xs = reinterpret_cast<df*>(xd);
  const int h0 = min(sh, ti.n_owned), nv = (ti.n_owned - h0) >> 1;
  {
    if (threadIdx.x < h0) cp_async(xd + threadIdx.x, so + threadIdx.x);
#pragma unroll 4
    for (int j = threadIdx.x; j < nv; j += NT) cp_async16(xd + h0 + 2 * j, so + h0 + 2 * j);
    for (int i = h0 + 2 * nv + threadIdx.x; i < ti.n_owned; i += NT) cp_async(xd + i, so + i);
    const int32_t* fl = A.foreign + ti.foreign_begin;
    double* xf = xd + ti.n_owned;
    for (int i0 = threadIdx.x; i0 < ti.n_foreign; i0 += 4 * NT) {
      int idx[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) idx[u] = (i0 + u * NT < ti.n_foreign) ? fl[i0 + u * NT] : -1;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (idx[u] >= 0) cp_async(xf + i0 + u * NT, A.src + idx[u]);
    }
  }
  if (threadIdx.x < LANE_ZERO) xs[nloc + threadIdx.x] = df{0.f, 0.f};
  cp_async_wait_all();
  __syncthreads();
  for (int i = threadIdx.x; i < nloc; i += NT) xs[i] = df_from_bits(xd[i]);  // one thread per element: in place
  const uint16_t m = st->mask[lane];
  const bool hang = st->hang != 0;
  df h;
  {
    const int c = ti.cell_begin + min(lane, ti.n_cells - 1);
    const double hd = ldexp(A.dom, -(int)st->level[lane]);
    h = df_from(A.coef ? hd * A.coef[c] : hd);
  }
  const bool h_pow2 = __all_sync(0xffffffffu, h.lo == 0.f && (__float_as_uint(h.hi) & 0x7fffffu) == 0u);
  char* xb = reinterpret_cast<char*>(xs);
  __syncthreads();
  {  // G_e: the warp's x-lines, all gathered before the cell buffer is written
    df v[N][N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const uint32_t li = c_ll.line[K][c_ll.bl[K][w][i]];
      const int s0 = li & 0xff, o0 = (li >> 8) & 0xff, o1 = li >> 16;
      const df* p0 = reinterpret_cast<const df*>(xb + 2 * (st->ls[s0][lane] + o0));
      const df* p1 = reinterpret_cast<const df*>(xb + 2 * (st->ls[s0 + 1][lane] + o1));
      const df* p2 = reinterpret_cast<const df*>(xb + 2 * (st->ls[s0 + 2][lane] + o0));
      v[i][0] = *p0;
#pragma unroll
      for (int a = 1; a < K; ++a) v[i][a] = p1[a - 1];
      v[i][K] = *p2;
    }
    __syncthreads();  // the DoF buffer is dead
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
      for (int a = 0; a < N; ++a) cb[(N * c_ll.bl[K][w][i] + a) * 32 + lane] = v[i][a];
  }
  // the first pass takes the warp's own lines
  const int npass = hang ? 11 : 5;
#pragma unroll 1
  for (int ps = 0; ps < npass; ++ps) {
    const int f = c_df_pass[hang][ps], D = f & 3;
    const int S = 32 * (D == 0 ? 1 : (D == 1 ? N : N2));
    const uint16_t* node = c_df_node[K][D][w];
    df* cl = cb + lane;
    if ((f & ~3) == DF_FWD) {
      df_lines<N>(cl, node, S, [&](df* v, int) { df_eo_fwd_fast<K>(v); });
    } else if ((f & ~3) == DF_BWD) {
      df_lines<N>(cl, node, S, [&](df* v, int) { df_eo_bwd_fast<K>(v); });
    } else if ((f & ~3) == DF_Z) {  // h (K + (lam + lam') M) on the line of modes r
      df_lines<N>(cl, node, S, [&](df* v, int i) {
        const int r = c_ll.bl[K][w][i];
        zline<K>(v, c_zl.h[zline_row(K) + r], c_zl.l[zline_row(K) + r], r == 0);
        if (h_pow2) {  // 2 operations per value instead of 7, the same result
#pragma unroll
          for (int c = 0; c < N; ++c) v[c] = df{v[c].hi * h.hi, v[c].lo * h.hi};
        } else {
#pragma unroll
          for (int c = 0; c < N; ++c) v[c] = df_mul(v[c], h);
        }
      });
    } else {  // the hanging lines only
      const uint32_t hl = hg->hl[D][lane];
      const int p = (m >> D) & 1;
#pragma unroll 1
      for (int i = 0; i < N; ++i) {
        if (!((hl >> c_ll.bl[K][w][i]) & 1u)) continue;
        df* ptr = cl + node[i];
        df v[N];
#pragma unroll
        for (int a = 0; a < N; ++a) v[a] = ptr[a * S];
        if ((f & ~3) == DF_C)
          interp_line_df<K, false>(v, p);
        else
          interp_line_df<K, true>(v, p);
#pragma unroll
        for (int a = 0; a < N; ++a) ptr[a * S] = v[a];
      }
    }
    __syncthreads();
  }
  // G_e^T on the warp's class of x-lines: all lines read before the accumulator (the same
  // region) is cleared
  {
    constexpr int NXW = K <= 2 ? 4 : N;  // x-lines per warp at most
    const int nxl = c_ll.nx[K][w];
    df v[NXW][N];
#pragma unroll
    for (int i = 0; i < NXW; ++i)
      if (i < nxl) {
        const df* p = cb + N * c_ll.xw[K][w][i] * 32 + lane;
#pragma unroll
        for (int a = 0; a < N; ++a) v[i][a] = p[a * 32];
      }
    __syncthreads();  // the cell buffer is dead
    {
      float4* z4 = reinterpret_cast<float4*>(xd0);
      for (int i = threadIdx.x; i < (sh + nloc + 1) / 2; i += NT) z4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NXW; ++i) {
      if (i >= nxl) break;
      const uint32_t li = c_ll.line[K][c_ll.xw[K][w][i]];
      const int s0 = li & 0xff, o0 = (li >> 8) & 0xff, o1 = li >> 16;
      df* q0 = reinterpret_cast<df*>(xb + 2 * (st->ls[s0][lane] + o0));
      df* q1 = reinterpret_cast<df*>(xb + 2 * (st->ls[s0 + 1][lane] + o1));
      df* q2 = reinterpret_cast<df*>(xb + 2 * (st->ls[s0 + 2][lane] + o0));
      add_turns<1>(q0, v[i], hang ? hg->rank[s0][lane] : 0, hang ? hg->most[s0] : 1);
      if constexpr (K > 1)
        add_turns<K - 1>(q1, v[i] + 1, hang ? hg->rank[s0 + 1][lane] : 0, hang ? hg->most[s0 + 1] : 1);
      add_turns<1>(q2, v[i] + K, hang ? hg->rank[s0 + 2][lane] : 0, hang ? hg->most[s0 + 2] : 1);
    }
  }
  __syncthreads();
  double* d = A.dst + ti.dof_begin;
  if (A.add)
    for (int i = threadIdx.x; i < ti.n_owned; i += NT) d[i] += df_to_bits(xs[i]);
  else
    for (int i = threadIdx.x; i < ti.n_owned; i += NT) d[i] = df_to_bits(xs[i]);
  const int32_t* hp = A.halo_pos + ti.foreign_begin;
  for (int i = threadIdx.x; i < ti.n_foreign; i += NT) A.halo[hp[i]] = df_to_bits(xs[ti.n_owned + i]);
}

// ---------------------------------------------------------------------------
// degree 1: one warp per tile, the lane's cell (8 values) in registers.  The
// sweeps need neither a cell buffer nor a barrier, and a tile is one chain of its
// metadata, its DoFs and about 300 instructions: four tiles per block, each on
// its own, hide one another's latencies, and only the vertex rows of the lane
// record are copied (512 of 1,856 B).  Octant mesh, 269,998 cells: fp32 19.9 ->
// 14.4 us, fp64 45 -> 34 us.  At k = 2 (27 values, 64 or 96 registers) the same
// kernel was slower than vmult_lanes: 34,903 cells 14 -> 21 us in fp32, 31 -> 44 us
// in fp64.
// ---------------------------------------------------------------------------
constexpr int RWPB = 4;  // tiles (warps) per block

template <int K>
__device__ __forceinline__ void reg_z(float* v, int q) {
  zline<K>(v, c_zl.h[zline_row(K) + q], q == 0);
}
template <int K>
__device__ __forceinline__ void reg_z(df* v, int q) {
  zline<K>(v, c_zl.h[zline_row(K) + q], c_zl.l[zline_row(K) + q], q == 0);
}

template <int K, int D, bool FWD, typename V>
__device__ __forceinline__ void reg_sweep(V* u) {
  constexpr int N = K + 1, S = line_stride<N, D>();
#pragma unroll
  for (int q = 0; q < N * N; ++q) {
    const int base = line_base<K, D>(q);
    V v[N];
#pragma unroll
    for (int a = 0; a < N; ++a) v[a] = u[base + a * S];
    eo_line<K, FWD>(v);
#pragma unroll
    for (int a = 0; a < N; ++a) u[base + a * S] = v[a];
  }
}

template <int K, int D, bool TRANS, typename V>
__device__ __forceinline__ void reg_hang(V* u, uint16_t m, uint32_t hl) {
  constexpr int N = K + 1, S = line_stride<N, D>();
  const int p = (m >> D) & 1;
#pragma unroll
  for (int q = 0; q < N * N; ++q) {
    const int x = q % N, y = q / N;
    if (x > 0 && x < K && y > 0 && y < K) continue;  // inside the cell
    if (!((hl >> q) & 1u)) continue;
    const int base = line_base<K, D>(q);
    V v[N];
#pragma unroll
    for (int a = 0; a < N; ++a) v[a] = u[base + a * S];
    hang_line<K, TRANS>(v, p);
#pragma unroll
    for (int a = 0; a < N; ++a) u[base + a * S] = v[a];
  }
}

// rows of the lane record in shared memory: the 8 vertex slots
constexpr int REG_ROWS = 8;
__device__ __forceinline__ int vertex_slot(int r) { return 2 * (r & 1) + 6 * ((r >> 1) & 1) + 18 * (r >> 2); }
template <typename V>
size_t reg_smem(int max_local) {
  return RWPB * ((size_t)REG_ROWS * 64 + ((((size_t)max_local + LANE_ZERO) * sizeof(V) + 15) & ~(size_t)15));
}

template <typename T>
__global__ void __launch_bounds__(RWPB * 32) vmult_q1(LaneArgsT<T> A, int n_tiles, int warp_bytes) {
  using AR = Arith<T>;
  using V = typename AR::V;
  constexpr int K = 1, N = 2, N2 = 4, N3 = 8, NR = REG_ROWS;
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int bx = blockIdx.x * RWPB + w, tl = A.tile0 + bx;
  if (bx >= n_tiles) return;
  uint16_t(*ls)[32] = reinterpret_cast<uint16_t(*)[32]>(smem + (size_t)w * warp_bytes);
  V* xs = reinterpret_cast<V*>(smem + (size_t)w * warp_bytes + NR * 64);
  T* xt = reinterpret_cast<T*>(xs);  // the values as they arrive; converted in place
  const LaneTile* lt = A.order ? A.lt_lo + bx : A.lt + tl;
  const LaneHang* lh = A.order ? A.lh_lo + bx : A.lh + tl;
  const TileInfo ti = A.order ? A.tiles_lo[bx] : A.tiles[tl];
  const int nloc = ti.n_owned + ti.n_foreign;
  for (int i = lane; i < NR * 4; i += 32)
    cp_async16(reinterpret_cast<unsigned char*>(ls) + 16 * i,
               reinterpret_cast<const unsigned char*>(lt->ls[vertex_slot(i >> 2)]) + 16 * (i & 3));
  const uint16_t m = lt->mask[lane];
  const bool hang = lt->hang != 0;
  uint32_t hl[3] = {0u, 0u, 0u};
  if (hang)
#pragma unroll
    for (int d = 0; d < 3; ++d) hl[d] = lh->hl[d][lane];
  const int32_t* fl = A.foreign + ti.foreign_begin;
  constexpr int FU = 4;  // foreign indices loaded ahead of the predecessor's completion
  int idx[FU];
#pragma unroll
  for (int u = 0; u < FU; ++u) idx[u] = lane + 32 * u < ti.n_foreign ? fl[lane + 32 * u] : -1;
  double h = ldexp(A.dom, -(int)lt->level[lane]);
  if (A.coef) h *= A.coef[ti.cell_begin + min(lane, ti.n_cells - 1)];
  pdl_wait();
  const T* so = A.src + ti.dof_begin;
  for (int i = lane; i < ti.n_owned; i += 32) cp_async(xt + i, so + i);
#pragma unroll
  for (int u = 0; u < FU; ++u)
    if (idx[u] >= 0) cp_async(xt + ti.n_owned + lane + 32 * u, A.src + idx[u]);
  for (int i = lane + 32 * FU; i < ti.n_foreign; i += 32) cp_async(xt + ti.n_owned + i, A.src + fl[i]);
  cp_async_wait_all();
  __syncwarp();
  if constexpr (sizeof(T) == 8)
    for (int i = lane; i < nloc; i += 32) xs[i] = AR::in(xt[i]);  // one lane per element: in place
  for (int i = lane; i < LANE_ZERO; i += 32) xs[nloc + i] = V(0);
  __syncwarp();
  // G_e
  V u[N3];
#pragma unroll
  for (int n = 0; n < N3; ++n) u[n] = xs[ls[n][lane] >> 2];
  __syncwarp();
  for (int i = lane; i < nloc; i += 32) xs[i] = V(0);  // the accumulator
  if (hang) {
    reg_hang<K, 0, false>(u, m, hl[0]);
    reg_hang<K, 1, false>(u, m, hl[1]);
    reg_hang<K, 2, false>(u, m, hl[2]);
  }
  reg_sweep<K, 0, true>(u);
  reg_sweep<K, 1, true>(u);
  {  // z: h (K + (lam_a + lam_b) M)
    const V hv = V(h);
#pragma unroll
    for (int q = 0; q < N2; ++q) {
      V v[N];
#pragma unroll
      for (int a = 0; a < N; ++a) v[a] = u[q + a * N2];
      reg_z<K>(v, q);
#pragma unroll
      for (int a = 0; a < N; ++a) u[q + a * N2] = v[a] * hv;
    }
  }
  reg_sweep<K, 1, false>(u);
  reg_sweep<K, 0, false>(u);
  if (hang) {
    reg_hang<K, 2, true>(u, m, hl[2]);
    reg_hang<K, 1, true>(u, m, hl[1]);
    reg_hang<K, 0, true>(u, m, hl[0]);
  }
  __syncwarp();
  // G_e^T, node by node: the lanes of one node meet only behind hanging faces and edges (turns)
#pragma unroll
  for (int n = 0; n < N3; ++n) {
    const int slot = vertex_slot(n);
    add_turns<1>(xs + (ls[n][lane] >> 2), &u[n], hang ? lh->rank[slot][lane] : 0, hang ? lh->most[slot] : 1);
  }
  T* d = A.dst + ti.dof_begin;
  for (int i = lane; i < ti.n_owned; i += 32) {
    const T v = AR::out(xs[i]);
    d[i] = A.add ? d[i] + v : v;
  }
  const int32_t* hp = A.halo_pos + ti.foreign_begin;
  for (int i = lane; i < ti.n_foreign; i += 32) A.halo[hp[i]] = AR::out(xs[ti.n_owned + i]);
}

template <typename T>
cudaError_t run_q1(const CellLaunch& L, const LaneArgsT<T>& A, int n_tiles, cudaStream_t s) {
  const size_t sm = reg_smem<typename Arith<T>::V>(L.max_local);
  cudaError_t e = smem_allow(vmult_q1<T>, sm);
  if (e != cudaSuccess) return e;
  e = launch_pdl(vmult_q1<T>, (n_tiles + RWPB - 1) / RWPB, RWPB * 32, sm, s, A, n_tiles, (int)(sm / RWPB));
  note_launches(1);
  return e;
}

template <int K>
size_t lanes_smem(int max_local) {
  constexpr int N3 = (K + 1) * (K + 1) * (K + 1);
  // one region for the cell buffer and the tile DoFs (shifted by up to 3 for the 16-byte
  // copies, the zero region, and the float4 clearing)
  return sizeof(LaneTile) + sizeof(LaneHang) +
         std::max((size_t)N3 * 32, (size_t)max_local + LANE_ZERO + 8) * sizeof(float);
}

template <int K>
size_t lanes_df_smem(int max_local) {
  constexpr int N3 = (K + 1) * (K + 1) * (K + 1);
  // one region for the cell buffer and the tile DoFs, as in lanes_smem
  return sizeof(LaneTile) + sizeof(LaneHang) +
         std::max((size_t)N3 * 32, (size_t)max_local + LANE_ZERO + 4) * sizeof(double);
}

template <int K>
cudaError_t run_lanes_df(const CellLaunch& L, const LaneArgsT<double>& A, int n_tiles, cudaStream_t s) {
  const size_t sm = lanes_df_smem<K>(L.max_local);
  const auto kernel = lanes_dense(L, lanes_df_roomy(K)) ? vmult_lanes_df<K, true> : vmult_lanes_df<K, false>;
  cudaError_t e = smem_allow(kernel, sm);
  if (e != cudaSuccess) return e;
  e = launch_pdl(kernel, n_tiles, (K + 1) * 32, sm, s, A);
  note_launches(1);
  return e;
}

template <int K>
cudaError_t run_lanes(const CellLaunch& L, const LaneArgs& A, int n_tiles, cudaStream_t s) {
  const size_t sm = lanes_smem<K>(L.max_local);
  const auto kernel = lanes_dense(L, lanes_roomy(K)) ? vmult_lanes<K, true> : vmult_lanes<K, false>;
  cudaError_t e = smem_allow(kernel, sm);
  if (e != cudaSuccess) return e;
  e = launch_pdl(kernel, n_tiles, (K + 1) * 32, sm, s, A);
  note_launches(1);
  return e;
}

}  // namespace

void upload_tables_lanes() {
  upload_tables_lanes_1d();
  static LaneLines t;
  fill_lane_lines(t);
  cudaMemcpyToSymbol(c_ll, &t, sizeof(t));
  upload_zlines();
  static uint16_t node[KMAX + 1][3][NMAX][8];
  for (int k = 1; k <= KMAX; ++k)
    for (int D = 0; D < 3; ++D)
      for (int w = 0; w <= k; ++w)
        for (int i = 0; i <= k; ++i) {
          const int n = k + 1, r = t.bl[k][w][i];
          node[k][D][w][i] = (uint16_t)(32 * (D == 0 ? n * r : (D == 1 ? r % n + n * n * (r / n) : r)));
        }
  cudaMemcpyToSymbol(c_df_node, node, sizeof(node));
}

bool lanes_ok(const CellLaunch& L) { return L.lane_tiles && L.tc <= 32 && !L.geom && L.k >= 1 && L.k <= KMAX; }

void launch_vmult_lanes_df(const CellLaunch& L, const double* src, double* dst, int add, int t0, int t1,
                           cudaStream_t s) {
  if (t1 <= t0 || !lanes_ok(L)) return;
  LaneArgsT<double> A{};
  A.tiles = L.tiles;
  A.lt = static_cast<const LaneTile*>(L.lane_tiles);
  A.lh = static_cast<const LaneHang*>(L.lane_hang);
  A.n_hang = L.n_hang_tiles;
  A.order = (t0 == 0 && t1 == L.n_tiles) ? L.lane_order : nullptr;
  A.tiles_lo = L.tiles_lo;
  A.lt_lo = static_cast<const LaneTile*>(L.lane_tiles_lo);
  A.lh_lo = static_cast<const LaneHang*>(L.lane_hang_lo);
  A.foreign = L.foreign;
  A.halo_pos = L.halo_pos;
  A.src = src;
  A.dst = dst;
  A.halo = static_cast<double*>(L.halo);
  A.coef = L.coef;
  A.dom = L.dom;
  A.add = add;
  A.tile0 = t0;
  switch (L.k) {
    case 1: run_q1(L, A, t1 - t0, s); break;
    case 2: run_lanes_df<2>(L, A, t1 - t0, s); break;
    case 3: run_lanes_df<3>(L, A, t1 - t0, s); break;
    case 4: run_lanes_df<4>(L, A, t1 - t0, s); break;
    default: break;
  }
}

void launch_vmult_lanes(const CellLaunch& L, const void* src, void* dst, int add, int t0, int t1, cudaStream_t s) {
  if (t1 <= t0 || !lanes_ok(L)) return;
  LaneArgs A{};
  A.tiles = L.tiles;
  A.lt = static_cast<const LaneTile*>(L.lane_tiles);
  A.lh = static_cast<const LaneHang*>(L.lane_hang);
  A.n_hang = L.n_hang_tiles;
  // a whole level: tiles with hanging cells first (their longer code path then
  // runs mostly on its own instead of interleaved with the regular tiles')
  A.order = (t0 == 0 && t1 == L.n_tiles) ? L.lane_order : nullptr;
  A.tiles_lo = L.tiles_lo;
  A.lt_lo = static_cast<const LaneTile*>(L.lane_tiles_lo);
  A.lh_lo = static_cast<const LaneHang*>(L.lane_hang_lo);
  A.foreign = L.foreign;
  A.halo_pos = L.halo_pos;
  A.src = static_cast<const float*>(src);
  A.dst = static_cast<float*>(dst);
  A.halo = static_cast<float*>(L.halo);
  A.coef = L.coef;
  A.dom = L.dom;
  A.add = add;
  A.tile0 = t0;
  switch (L.k) {
    case 1: run_q1(L, A, t1 - t0, s); break;
    case 2: run_lanes<2>(L, A, t1 - t0, s); break;
    case 3: run_lanes<3>(L, A, t1 - t0, s); break;
    case 4: run_lanes<4>(L, A, t1 - t0, s); break;
    default: break;
  }
}

}  // namespace gcmg
