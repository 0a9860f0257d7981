// Launch interface of the CUDA kernels of libgcmg (internal).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "internal.h"

namespace gcmg {

// count of kernel launches issued by the library (all host threads)
void note_launches(int n);

enum CellMode { MODE_VMULT = 0, MODE_RHS = 1, MODE_DIAG = 2, MODE_LIFT = 3 };

// arguments of the tile kernels (operator, right-hand side, diagonal)
struct CellLaunch {
  const TileInfo* tiles;
  int n_tiles;
  const CellMeta* meta;
  const int32_t* foreign;
  const uint16_t* subptr;
  const uint8_t* perm;
  const int32_t* cell_ijk;  // per cell i, j, k (right-hand side only)
  // halo: one slot per (tile, foreign DoF), in the order of the halo pass
  void* halo;  // n_foreign_total values of the launch precision
  const int32_t* halo_ents;       // first DoF of every halo entity
  const HaloBlock* halo_blocks;
  const int32_t* halo_pos;  // per foreign slot: position in the halo buffer
  int n_halo;                     // blocks of the halo pass
  int k;
  int tc;
  int max_local;
  int use_lines;  // 1: fp32 operator with the line-parallel kernel
  int threads;    // threads per CTA of the line-parallel operator kernel (128, 256, 384 or 512)
  int n_sm;       // multiprocessors of the device (grid sizes, chunk choices)
  int chunk;      // coarse cells per restriction chunk (0: from the level size)
  int use_lanes;  // 1: fp32 operator with the lane-per-cell kernel (tiles of at most 32 cells)
  const void* lane_tiles;  // per tile LaneTile (null: level without them)
  const int32_t* lane_order;  // launch order of the tiles: those with hanging cells first
  const void* lane_hang;      // per tile LaneHang
  // the same in launch order (block b runs tile lane_order[b]): TileInfo and
  // LaneTile of every tile, LaneHang of the first n_hang_tiles
  const TileInfo* tiles_lo;
  const void* lane_tiles_lo;
  const void* lane_hang_lo;
  int n_hang_tiles;           // tiles with hanging cells
  // levels of few cells (kernels_small.cu): per DoF its entries in the cell
  // vectors (null: the level has none)
  const int32_t* sum_ptr;
  const int32_t* sum_pos;
  void* cell_vec;             // n_cells (k+1)^3 values of the launch precision
  const int32_t* gstart;
  int n_cells;
  int n_dofs;
  double lo, dom;
  const double* coef;  // per cell coefficient nu_e (element matrix nu_e h A_ref); null: 1
  int geom;            // 0: Cartesian cells; GEOM_WARP: the cells mapped by the warp below
  double geps;         // its eps
};

// non-Cartesian geometry: the octree cells (parameter space) mapped by
// Phi(x) = x + eps (x1 x2, 2 x2 x0, x0 x1 / 2), the Jacobian evaluated at every
// Gauss point
constexpr int GEOM_WARP = 1;

// analytic function of a right-hand side or of Dirichlet data
enum FuncKind { FUNC_ONE = 0, FUNC_FOURIER = 1, FUNC_GAUSSIAN = 2, FUNC_POLYNOMIAL = 3 };
struct RhsDesc {
  int kind;               // FuncKind
  const double* params;   // FOURIER: per mode kx, ky, kz, phi; GAUSSIAN: alpha, x0, y0, z0;
                          // POLYNOMIAL: per term c, a, b, e (u = sum c x^a y^b z^e)
  int n;                  // modes or terms
  double amp;             // FOURIER: amplitude
};

// dst = A src (add = 0) or dst += A src (add = 1), precision by `fp64`
void launch_vmult(const CellLaunch& L, bool fp64, const void* src, void* dst, int add, cudaStream_t s);
// the tile kernel of the operator for tiles [t0, t1) only (the halo pass is
// launch_halo_add, after all tiles); a tile reads x only below the end of its
// owned range (first-touch ownership), so tile groups can start as the input
// arrives in DoF order.  vmult_tiles_ok: the level's kernels allow it.
bool vmult_tiles_ok(const CellLaunch& L, bool fp64);
void launch_vmult_tiles(const CellLaunch& L, bool fp64, const void* src, void* dst, int t0, int t1, cudaStream_t s);
// the lane-per-cell fp32 operator (tile kernel only, tiles [t0, t1)); lanes_ok:
// the level has its metadata (tiles of at most 32 cells, Cartesian cells)
bool lanes_ok(const CellLaunch& L);
void launch_vmult_lanes(const CellLaunch& L, const void* src, void* dst, int add, int t0, int t1, cudaStream_t s);
// the fp64 operator (double-float arithmetic) with the same structure
void launch_vmult_lanes_df(const CellLaunch& L, const double* src, double* dst, int add, int t0, int t1,
                           cudaStream_t s);
void upload_tables_lanes();
// dst = C^T F: Gauss quadrature of f against the basis (FOURIER, ONE: f
// itself; GAUSSIAN, POLYNOMIAL: f = -Lap u of the manufactured solution u)
void launch_rhs(const CellLaunch& L, const RhsDesc& f, double* dst, cudaStream_t s);
// dst -= C^T A_all u_g: the lifting u_g of the Dirichlet data g = u (u at
// boundary support points, interpolated at hanging points, zero elsewhere)
void launch_rhs_lift(const CellLaunch& L, const RhsDesc& u, double* dst, cudaStream_t s);

// variable coefficient: nu_e = (sum_q w_q) / (sum_q w_q / nu_q) from the
// (k+1)^3 Gauss-point values of every cell; coarse cells from the fine level
// (the fine cell's value, or the mean of the eight children of a refined
// cell); Gauss points of every cell (n_cells x (k+1)^3 x 3, x fastest)
void launch_coef_harmonic(int k, int64_t n_cells, const double* nu_q, double* nu, cudaStream_t s);
void launch_coef_coarsen(int n_coarse, const int32_t* fine_of, const uint8_t* refined, const double* nu_f,
                         double* nu_c, cudaStream_t s);
void launch_quadrature_points(const CellLaunch& L, int64_t n_cells, double* xyz, cudaStream_t s);
// *bad = 1 if any of v[0..n) is not positive and finite (*bad unchanged otherwise)
void launch_check_positive(const double* v, int64_t n, int* bad, cudaStream_t s);
void launch_diag(const CellLaunch& L, const double* diag_tab, double* dst, cudaStream_t s);
// diag_tab[m * (k+1)^3 + j] = (C_m^T A_ref C_m)_{jj} for all 512 masks m
void launch_diag_table(int k, double* diag_tab, cudaStream_t s);
// second pass of every tile loop: dst[g] += halo slots of g, fixed order
void launch_halo_add(const CellLaunch& L, bool fp64, void* dst, cudaStream_t s);
size_t cell_smem_bytes(int k, bool fp64, int tc, int max_local, bool mapped = false);

// transfer between levels; fine_of/refined per coarse cell
struct TransferLaunch {
  int kind;  // 0 = h, 1 = p
  int kf, kc;
  int n_coarse;
  const int32_t* fine_of;
  const uint8_t* refined;
  const int32_t* gstart_f;  // fine cells x 27
  const uint32_t* own_f;    // fine cells
  const int32_t* gstart_c;  // coarse cells x 27
  const uint16_t* mask_c;   // coarse cells
  const int32_t* lattice;   // h: entity table of the lattice kernels
  CellLaunch coarse;        // coarse level tiles (restriction scatter)
};
void launch_prolongate_add(const TransferLaunch& T, bool fp64, const void* coarse, void* fine, cudaStream_t s);
void launch_restrict_add(const TransferLaunch& T, bool fp64, const void* fine, void* coarse, cudaStream_t s);
// coarse (+)= R (b - Ax): the residual formed inside the restriction's gather
// (the same subtraction as launch_residual, so the same values); overwrite:
// coarse = R (b - Ax), no zeroing of coarse needed
void launch_restrict_residual(const TransferLaunch& T, bool fp64, const void* b, const void* Ax, void* coarse,
                              bool overwrite, cudaStream_t s);

// the h transfer with one warp per coarse cell (kernels_lattice.cu); the table
// (lattice_table_words words) is built once per transfer from the other members
size_t lattice_table_words(int k, int n_coarse);
void launch_lattice_entities(const TransferLaunch& T, int32_t* table, cudaStream_t s);
bool lattice_restrict_ok(const TransferLaunch& T);
void launch_prolong_lattice(const TransferLaunch& T, bool fp64, const void* coarse, void* fine, cudaStream_t s);
// coarse (+)= R fine, or R (rhs - fine) with rhs set
void launch_restrict_lattice(const TransferLaunch& T, bool fp64, const void* fine, const void* rhs, void* coarse,
                             bool overwrite, cudaStream_t s);
// the restriction of fine (rhs - fine with rhs set) to the coarse level's cell vectors
void launch_restrict_cells(const TransferLaunch& T, bool fp64, const void* fine, const void* rhs, cudaStream_t s);
void upload_tables_lattice();

// the operator of a level of few cells: cell vectors, then one pass over the
// DoFs that adds them up and goes on (kernels_small.cu)
// Levels that take them: those too small for 32-cell tiles (fewer than two tiles
// per SM), and larger ones of low degree up to CELL_VEC_MAX entries.  Postsmoothing,
// lane kernels -> cell vectors, fp32 / fp64 in us: Q1 61,440 cells (0.49 M entries)
// 31.6 -> 21.7 / 53.8 -> 55.6, 82,776 cells (0.66 M) 42.0 -> 32.9 / 80.5 -> 71.5, but
// 113,688 (0.91 M) 43.9 -> 39.2 / 89.6 -> 91.8; Q2 28,400 cells (0.77 M) 45.9 -> 39.4 /
// 96.4 -> 98.6, but 34,903 (0.94 M) 39.7 -> 39.0 / 84.1 -> 98.0; Q3 12,608 cells (0.81 M)
// 43.0 -> 29.4 / 94.4 -> 76.2, but 28,400 (1.8 M) 64.4 -> 62.1 / 164 -> 194; Q4 9,024
// cells 56.0 -> 43.5 / 148 -> 125, but 9,864 (1.2 M) 63.3 -> 54.6 / 175 -> 185.
constexpr int64_t CELL_VEC_MAX = 850000;
inline bool cell_vectors_pay(int64_t cells, int k, int n_sm) {
  return cells < 2 * (int64_t)n_sm * 32 || cells * (k + 1) * (k + 1) * (k + 1) <= CELL_VEC_MAX;
}
bool cells_ok(const CellLaunch& L);
// The operator on its own has no update to go on with.  fp64 at degrees 1 and 2: the
// lane kernels from fewer entries on.  Lane kernels / cell vectors: Q1 28,400 cells (0.23
// M) 14.2 / 11.9 us, 32,768 (0.26 M) 7.7 / 15.2, 37,871 (0.30 M) 13.4 / 13.2, 61,440
// 13.6 / 16.7; Q2 9,864 (0.27 M) 18.7 / 15.5, 11,096 (0.30 M) 15.5 / 15.7, 28,400 27.4 /
// 31.2.  fp32 and degrees 3 and 4 keep the level's choice (Q1 80,781 cells 9.2 / 8.0,
// Q2 28,400 12.9 / 12.5; fp64 Q3 12,608 26.4 / 22.9, Q4 9,024 40.9 / 37.3).
bool cells_operator_ok(const CellLaunch& L, bool fp64);
void launch_cell_vectors(const CellLaunch& L, bool fp64, const void* src, cudaStream_t s);
void launch_cell_sum(const CellLaunch& L, bool fp64, void* dst, bool add, cudaStream_t s);
void launch_cell_sum_residual(const CellLaunch& L, bool fp64, const void* b, void* r, cudaStream_t s);
// a Chebyshev step on b - sum: the first of a smoother, the one after the start
// from zero (d = x on entry), or a later one; last: d is not written
enum ChebStep { CHEB_FIRST, CHEB_AFTER_ZERO, CHEB_NEXT };
void launch_cell_sum_cheb(const CellLaunch& L, bool fp64, int step, bool last, void* x, void* d, const void* b,
                          const void* dinv, double c1, double c2, cudaStream_t s);
// b = sum (a restricted residual), x = c2 dinv b
void launch_cell_sum_start(const CellLaunch& L, bool fp64, void* b, void* x, const void* dinv, double c2,
                           cudaStream_t s);
void upload_tables_small();

// the V-cycle of the smallest levels as one dense matrix (kernels_dense.cu),
// on levels of at most DENSE_MAX DoFs
constexpr int DENSE_MAX = 1024;
void upload_tables_dense();
// A of a level (n x n, rows) and P of a transfer (n_f x n_c, rows), fp64
void launch_dense_operator(const CellLaunch& L, int n, int n_cells, const int32_t* gstart, double* A, cudaStream_t s);
void launch_dense_prolongation(const TransferLaunch& T, int n_f, int n_c, int cells_f, double* P, cudaStream_t s);
size_t dense_scratch_bytes(int n);
double* dense_vcycle_matrix(int n, const double* A, const double* dinv, int steps, const double* coef, int n_c,
                            const double* P, const double* Mc, double* work, cudaStream_t s);
// x = M b, sums in fp64; fp64: of b and x
void launch_dense_apply(bool fp64, const double* M, int n, const void* b, void* x, cudaStream_t s);

// vector kernels
void upload_tables();
void launch_cast(bool to64, const void* src, void* dst, int64_t n, cudaStream_t s);
void launch_zero(bool fp64, void* x, int64_t n, cudaStream_t s);
// x += om c with om = (r.c) / (c.w) (0 when c.w <= 0), w = A c; the two inner
// products in fp64, deterministic; scratch: 2 DOT_BLOCKS + 2 doubles
void launch_galerkin_step(bool fp64, const void* r, const void* c, const void* w, void* x, int64_t n,
                          double* scratch, cudaStream_t s);
// local smoothing, Algorithm 1: dst[idx[i]] = src[g[i]] (to a level, in its
// precision) and dst[g[i]] = src[idx[i]] (back to the fp64 active vector)
void launch_copy_to_level(bool fp64, const double* src, const int32_t* g, const int32_t* idx, int64_t n, void* dst,
                          cudaStream_t s);
void launch_copy_from_level(bool fp64, const void* src, const int32_t* g, const int32_t* idx, int64_t n, double* dst,
                            cudaStream_t s);
// a[idx[i]] = b[idx[i]] = 0 (Jacobi inverse on refinement-edge DoFs)
void launch_zero_at(const int32_t* idx, int64_t n, double* a, float* b, cudaStream_t s);
void launch_invert(const double* d, double* inv64, float* inv32, int64_t n, cudaStream_t s);
void launch_cheb_init(bool fp64, void* x, const void* b, const void* dinv, double c2, int64_t n, cudaStream_t s);
void launch_cheb_step(bool fp64, int step, bool last, void* x, void* d, const void* b, const void* Ax, const void* dinv,
                      double c1, double c2, int64_t n, cudaStream_t s);
void launch_residual(bool fp64, void* r, const void* b, const void* Ax, int64_t n, cudaStream_t s);
void launch_axpy(bool fp64, void* y, const void* x, double a, int64_t n, cudaStream_t s);
void launch_fill(double* x, double v, int64_t n, cudaStream_t s);
void launch_pmul(double* z, const double* a, const double* b, int64_t n, cudaStream_t s);
// p = z + beta p (host scalar)
void launch_xpby(double* p, const double* z, double beta, int64_t n, cudaStream_t s);
void launch_coarse_solve(bool fp64, const double* Ainv, int n, const void* b, void* x, cudaStream_t s);

// deterministic fp64 dot products: partial sums into `scratch` (DOT_BLOCKS
// doubles and a counter, zero between launches), combined in fixed order
constexpr int DOT_BLOCKS = 304;
constexpr size_t DOT_SCRATCH_BYTES = (DOT_BLOCKS + 1) * sizeof(double);
enum DotOp { DOT_STORE = 0, DOT_ALPHA = 1, DOT_BETA = 2, DOT_BETA_FLEX = 3, DOT_BETA_FIRST = 4 };
void launch_dot(const double* x, const double* y, int64_t n, double* scratch, double* scal, int slot, int op,
                cudaStream_t s);
// the same with y in fp32 (widened exactly: equal to the sums over an fp64 copy of y)
void launch_dot(const double* x, const float* y, int64_t n, double* scratch, double* scal, int slot, int op,
                cudaStream_t s);
// inner product with the partial sums in a fixed device array (no allocation);
// n <= dot_noalloc_max_n()
int64_t dot_noalloc_max_n();
cudaError_t launch_dot_noalloc(const double* x, const double* y, int64_t n, double* result, cudaStream_t s);
// CG updates with device scalars: scal[0] = rz, [1] = pq, [2] = rr, [3] = alpha, [4] = beta, [5] = rz_new,
// [6] = r_{k+1}.z_k of flexible CG
// rb != null: r is also written into the V-cycle's right-hand side, rounded to fp32
void launch_cg_update_xr(double* x, double* r, const double* p, const double* q, double* scal, int64_t n,
                         double* scratch, cudaStream_t s, float* rb = nullptr);
// CG as a loop inside a graph: further scalars.  cg_limits sets the limits of the
// next solve, cg_start begins it (|b|^2 in scal[7]), the update of x and r ends
// an iteration (it sets the WHILE node's condition h), cg_result writes
// (iterations, rr, |b|^2, status)
constexpr int CG_ITERATIONS = 8, CG_MAXIT = 9, CG_RTOL = 10, CG_RR = 12;
void launch_cg_limits(double* scal, int maxit, double rtol, cudaStream_t s);
void launch_cg_start(cudaGraphConditionalHandle h, double* scal, cudaStream_t s);
void launch_cg_update_xr_loop(double* x, double* r, const double* p, const double* q, double* scal, int64_t n,
                              double* scratch, cudaStream_t s, void* rb, bool rb64, cudaGraphConditionalHandle h);
void launch_cg_result(const double* scal, double* out, cudaStream_t s);
void launch_cg_update_p(double* p, const double* z, const double* scal, int64_t n, cudaStream_t s);
void launch_cg_update_p(double* p, const float* z, const double* scal, int64_t n, cudaStream_t s);
// CG inside a graph: scal[7] = |b|^2, scal[8] = iterations; the check kernel
// counts an iteration and sets the while-node condition h; the stats kernel
// writes (iterations, rr, |b|^2, status) to out
void launch_cg_check(cudaGraphConditionalHandle h, double* scal, int maxit, double rtol2, cudaStream_t s);
void launch_cg_stats(const double* scal, double rtol2, double* out, cudaStream_t s);
void launch_scalar_set(double* scal, int slot, double v, cudaStream_t s);
void launch_copy(const double* src, double* dst, int64_t n, cudaStream_t s);

// ---------------------------------------------------------------------------
// learned per-cell smoother
// ---------------------------------------------------------------------------
constexpr int MLP_DF = 128;  // bf16 diagonal features stored per cell (Q4: 125 + 3 zeros)
constexpr float MLP_BETA1 = 0.9f, MLP_BETA2 = 0.999f, MLP_EPS = 1e-8f;

// out[c][j] = (C_e G_e v)_j for the cells `cells` (null: 0..n-1), fp64
void launch_cell_gather(int k, const double* v, const int32_t* cells, int64_t n, const int32_t* gstart,
                        const CellMeta* meta, double* out, cudaStream_t s);
// training rows from gathered cell values R (residual), E (error, may be
// null), D (diagonal): X = [R / |R|, D / (h a)], T = E h a / |R|,
// W = (|R| / (h a))^2 (T, W may be null)
void launch_mlp_samples(const double* R, const double* E, const double* D, const int32_t* cells, int64_t n, int n3,
                        const CellMeta* meta, double dom, double abar, float* X, float* T, float* W, cudaStream_t s);
// bf16 rows of MLP_DF diagonal features per cell (all cells of a level)
void launch_mlp_dfeat(const double* D, int64_t n, int n3, const CellMeta* meta, double dom, double abar, void* out,
                      cudaStream_t s);

// C[m][n] = sum_k A(m, k) B(k, n) (+ bias[n]) with bf16 operands and fp32
// accumulation; A(m, k) = A[m sam + k sak], B(k, n) = B[k sbk + n sbn]
struct GemmArgs {
  const float* A;
  int64_t sam, sak;
  const float* B;
  int64_t sbk, sbn;
  float* C;
  int64_t ldc;
  const float* bias;
  int M, N, K;
  const uint16_t* Ab = nullptr;  // bf16 A (row stride sam, k contiguous) in place of A
};
void launch_gemm_bf16(const GemmArgs& g, cudaStream_t s);
void launch_gelu(const float* Z, float* H, int64_t n, cudaStream_t s);
void launch_gelu_bwd(const float* dH, const float* Z, float* dZ, int64_t n, cudaStream_t s);
// B rows of m outputs, weights W (null: 1): dY = w (Y - T) / sum w,
// *loss = sum w |Y - T|^2 / (2 sum w)
void launch_mse(const float* Y, const float* T, const float* W, float* dY, int B, int m, float* loss,
                cudaStream_t s);
void launch_colsum(const float* X, int M, int N, float* out, cudaStream_t s);
void launch_gather_rows(const float* X, int64_t ld, const int32_t* idx, int B, float* out, cudaStream_t s);
// Adam with bias corrections bc1 = 1 - beta1^t, bc2 = 1 - beta2^t
void launch_adam(float* p, const float* g, float* m, float* v, int64_t n, float lr, float bc1, float bc2,
                 cudaStream_t s);

// fused per-cell correction x += owner-selected MLP(r) for Q4 (250-128-128-125)
struct MlpFused {
  const void* wimg;        // packed bf16 weight image (launch_mlp_prepare), 16-byte aligned
  const float* dproj;      // per cell: b1 + the diagonal features times their W1 columns (128)
  const int32_t* gstart;   // cells x 27
  const uint32_t* own;     // per cell: owned slots
  const CellMeta* meta;
  int64_t n_cells;
  double dom;              // edge length of the domain
  double abar;             // mean diagonal entry of the unit-cell matrix
};
size_t mlp_fused_smem_bytes();
size_t mlp_image_bytes();
// weight image of a 250-128-128-125 network from its packed fp32 parameters,
// and the diagonal part of its first layer for every cell of a level (dproj:
// n_cells x 128 fp32, from the bf16 diagonal features dfeat)
void launch_mlp_prepare(const float* params, const uint16_t* dfeat, int64_t n_cells, void* image, float* dproj,
                        cudaStream_t s);
// bounded tensor-core waits that gave up since the last reset (synchronous)
unsigned int wait_timeouts(bool reset);
// multiprocessors of the current device (152 without a usable device)
int device_sm_count();
cudaError_t launch_mlp_correct(const MlpFused& P, bool fp64, const void* r, void* x, cudaStream_t s);

}  // namespace gcmg
