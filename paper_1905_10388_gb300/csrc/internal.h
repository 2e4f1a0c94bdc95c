// Internal declarations shared by the spectau translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <map>
#include <string>
#include <vector>

#include "common.cuh"

namespace spectau {

constexpr int GPU_SMS = 152;           // GB300

// Column chunk streamed per bulk copy by the pencil-solve kernel, and the
// ring depth.  Factor arrays are padded to a multiple of SOLVE_CHUNK columns.
constexpr int SOLVE_CHUNK = 32;
constexpr int SOLVE_RING = 2;

// Pencils per warp in the lane-per-right-hand-side substitution (two lanes
// each: real and imaginary part).
constexpr int LANE_GROUP = 16;
// Its right-hand sides are stored by group, [G][npad][16] complex: element (p, r).
__host__ __device__ inline size_t lane_index(int p, int r, int npad) {
  return ((size_t)(p / LANE_GROUP) * npad + r) * LANE_GROUP + p % LANE_GROUP;
}

// A factor's entries listed for the lane substitution (lanes.cu), by groups of
// LANE_GROUP pencils (G of them), 16 values per entry.
struct LaneList {
  // records of two entries: [16 pencils][2] values, the byte offsets of their
  // rows in the shared-memory ring (bit 0 of the second: the row's last record)
  double* Lv = nullptr;         // [G][lcap]  multipliers, rows rising, band offset rising
  double* Uv = nullptr;         // [G][ucap]  scaled U entries, rows falling, offset falling
  uint32_t* lmask = nullptr;    // [G][npad] bit t: L_{j+t,j} listed
  unsigned long long* umask = nullptr;   // [G][npad] bit t: U_{j,j+t} listed
  int32_t* lco = nullptr;       // [G][npad/4 + 1] first record of each four-row chunk
  int32_t* uco = nullptr;
  uint16_t* pg = nullptr;       // [G][npad][16] the pivot row's byte offset in the ring
  int32_t* tot = nullptr;       // [G][4] record counts (lane_list_build's scratch)
  int lcap = 0, ucap = 0;       // records allocated per group
  int lrecs = 0, urecs = 0;     // most records of a four-row chunk
  double l_listed = 0, u_listed = 0;     // mean entries per row, pads included
};

// Banded LU factors of one matrix a*M~ + b*L~ for all pencils.
struct BandFactor {
  double alpha = 0, beta = 0;   // A = alpha M~ + beta L~
  double* L = nullptr;          // [P][npad][lpad]  multipliers of column j (rows j+1..j+kl)
  uint8_t* piv = nullptr;       // [P][npad]        pivot row offset (piv - j) in [0, kl]
  double* U = nullptr;          // [P][npad][upad]  t=0: 1/U_jj, t>=1: U_{j-t,j}/U_jj
  double* rd = nullptr;         // [P][npad]        1/U_jj (0 on padding columns)
  // partitioned substitution (spike.cu): coupling matrices of the row blocks
  double* spD = nullptr;        // [P][nblk_f][7][8]   forward window after a block from the window before
  double* spE = nullptr;        // [P][nblk][kuu][32]  back-substitution outflow from the inflow
  LaneList ll;                  // lists of the lane substitution (whole or partitioned)
};

// Substitution of one problem's pencils in launches of their own: by lanes,
// whole (nblk = nblk_f = 1) or in row blocks (lanes.cu), or row blocks of a warp's
// window (spike.cu).
struct LaneArgs {
  int P, n, npad, kl, kuu;
  int nblk, m, nblk_f, m_f;     // blocks per pencil and their rows, back and forward
  int lcap, ucap, lrecs, urecs;
  const double* Lv; const double* Uv;
  const int32_t* lco; const int32_t* uco;
  const uint16_t* pg;
  const double* L; const uint8_t* piv; const double* U; int lpad, upad;   // spike.cu: the factor itself
  // right-hand sides by group, [G][npad][16 pencils] complex, zero beyond n
  // (spike.cu: by pencil, [p][n])
  int by_pencil;
  const double2* bg;            // B~
  double* yg;                   // y = L^-1 P B~
  double2* xg;                  // b = U_jj x~
  double* s0; double* sst;      // forward outflows / inflows [p][nblk_f][2][8]
  double* o0; double* uin;      // backward outflows / inflows [p][nblk][2][32]
  int cold;                     // 1: pass 1 starts from zero inflows instead of uin
  DevStatus* status;
};
// pass 0: whole pencils; 1: blocks from zero / guessed inflows; 2: from the true ones
cudaError_t launch_lane_forward(cudaStream_t s, const LaneArgs& a, int pass);
cudaError_t launch_lane_backward(cudaStream_t s, const LaneArgs& a, int pass);
cudaError_t lane_list_build(cudaStream_t s, int P, int n, int npad, int kl, int kuu, int lpad, int upad,
                            const double* L, const uint8_t* piv, const double* U, LaneList& f);
void lane_list_free(LaneList& f);

// Problems with fewer pencils than this, of at least SPIKE_MIN_ROWS rows with kl
// <= 7 and kl + ku <= 31, use a partitioned substitution by default: from
// LANE_SPLIT_PENCILS pencils on in its lane form (Fisher-KPP 2048 x 1024, 1024
// pencils: 0.41 ms per solve against 0.78 ms with the window kernel), below
// that one CTA per pencil where split_serves says so, else passes over the
// blocks in launches of their own.
constexpr int SPIKE_MAX_PENCILS = 4096;
constexpr int LANE_SPLIT_PENCILS = 4 * GPU_SMS;
constexpr int SPIKE_MIN_ROWS = 512;
// Problems that have at most two CTAs per SM take one CTA per pencil from fewer
// rows on (us per RK222 step, window kernel and one CTA: 48 x 24, 192 rows, 108 and
// 102; 384 x 24 155 and 147; 64 x 32, 224 rows, 16 steps 2.27 and 2.10 ms).  Below
// it gains nothing and the coupling matrices cost (32 x 16, 128 rows: a step 84 and
// 85, a factorization 163 and 188), but for narrow bands, whose back recurrence
// is short, while every pencil has an SM of its own (Fisher-KPP, 128 rows: 32
// pencils 65 and 63, 128 pencils 68 and 66, 256 pencils 72 and 74; 96 rows 82 and 86).
constexpr int SPLIT_MAX_PENCILS = 2 * GPU_SMS;
inline int split_min_rows(int P, int kuu) { return kuu <= 16 && P <= GPU_SMS ? 128 : 192; }
// Whether one CTA of `smem` bytes per pencil beats passes in separate launches
// (us per solve, one CTA against passes).  All pencils have to be on the GPU at
// once (512 x 512: 592 against 373 with one CTA on each SM at a time).  Its time
// is that of the fullest SM, the passes' goes with the pencils, so it wins with
// most SMs' places taken (256 x 128, 128 pencils: 65 against 110; 512 x 256, 256
// pencils: 186 against 209; 256 x 512: 217 against 223), and with fewer pencils
// as long as their chains are short (64 x 256, 1792 rows: faster; 64 x 384, 2688
// rows: 166 against 136; 192 pencils of 1344 rows 167 against 159).  A wide lower
// band has no such passes forward: there one CTA wins wherever all fit (adjoint
// step at 128 x 512: 1.83 ms against 2.12) from the rows on at which its 32-lane
// windows repay the second pass (us per eigenvalue iteration, one CTA against the
// window kernel: 128 pencils of 224 rows 50 against 44, 448 rows 69 against 79; 256
// pencils of 448 rows 100 against 86, 896 rows 154 against 155).
inline bool split_serves(int P, int npad, bool wide, size_t smem) {
  const int per_sm = (P + GPU_SMS - 1) / GPU_SMS;
  if (P > SPLIT_MAX_PENCILS || smem > 227 * 1024 || per_sm * (smem + 1024) > 228 * 1024) return false;
  if (wide) return npad >= (per_sm == 1 ? 384 : 512);
  return 4 * P >= 3 * per_sm * GPU_SMS || npad * per_sm <= 2048;
}
bool spike_supported(int kl, int kuu, int npad, int nblk);
bool spike_bwd_supported(int kuu, int npad, int nblk);
cudaError_t launch_spike_coupling(cudaStream_t s, int P, int npad, int nblk_f, int nblk, int kl, int kuu, int lpad,
                                  int upad, const BandFactor& f, bool by_row);
// the passes over row blocks of a warp's window: 1 from zero / guessed inflows, 2 from the true ones
cudaError_t launch_spike_forward(cudaStream_t s, const LaneArgs& a, int pass);
cudaError_t launch_spike_backward(cudaStream_t s, const LaneArgs& a, int pass);
cudaError_t launch_spike_forward_rec(cudaStream_t s, const LaneArgs& a, const double* D);
cudaError_t launch_spike_backward_rec(cudaStream_t s, const LaneArgs& a, const double* E);

// Problems with at least this many pencils use the lane substitution on whole
// pencils.  Its time is the chain's (about 0.93 us per row and solve) up to
// 608 groups, the whole-row-order kernel's (pair.cu) grows with the pencils:
// 288 rows of 3D Rayleigh-Benard take 0.27 ms against 0.14 ms for 1024 pencils.
// Pencils that row blocks serve take those first (2048 pencils of Fisher-KPP, per
// solve: 512 rows 0.28 ms whole, 0.17 ms in blocks; 2048 rows 1.13 and 0.55).
constexpr int LANE_MIN_PENCILS = 2048;

// Chebyshev backward transform on the tensor cores (chebmma.cu): the split
// FP32 copy of the coefficients it reads, the transform matrix halves, and
// the TMA tensor maps (opaque CUtensorMap storage, 64-byte aligned).
struct ChebMMA {
  bool ready = false;
  int P = 0, Nz = 0, Ng = 0, S = 0;
  float* xs32 = nullptr;        // [S][2P][Nz]: real part (column 2p) and imaginary part (2p + 1)
  float* Thi = nullptr;         // [Ng][Nz] T_m(x_zg) truncated to TF32
  float* Tlo = nullptr;         // [Ng][Nz] the FP32 remainder
  alignas(64) unsigned char tmA[128];
  alignas(64) unsigned char tmThi[128];
  alignas(64) unsigned char tmTlo[128];
};
bool cheb_mma_supported(int Nz, int Ng);
cudaError_t cheb_mma_setup(ChebMMA& c, int P, int Nz, int Ng, int S, cudaStream_t s);
void cheb_mma_free(ChebMMA& c);
// grid fields f (variable f_var[f], operator f_op[f]; host arrays) of the
// FP32 coefficients in c.xs32 to gz [f][Ng][P] complex FP32
cudaError_t launch_cheb_backward_mma(cudaStream_t s, const ChebMMA& c, int nf, const int* f_var, const int* f_op,
                                     const float* kx32, void* gz, DevStatus* st);
cudaError_t launch_to_f32_split(cudaStream_t s, const double2* src, float* dst, size_t ncols, int Nz);

// Up to four device vectors with coefficients, passed to kernels by value.
struct VecList4 {
  const double2* p[4];
  double c[4];
  int n;
};

// Adjoint-step helper kernels (band.cu).
cudaError_t launch_adj_gather(cudaStream_t s, int P, int Nz, int Ng, int n, int nslot, const int32_t* nl_eq,
                              const int32_t* row_map, const int32_t* eq_diff, const int32_t* eq_phase,
                              int nvec, const double2* const* vecs, const double* coefs, double2* fbar,
                              float2* fbar32);
cudaError_t launch_adj_combine(cudaStream_t s, int P, int Nz, int S, int n, int nf, const int32_t* f_var,
                               const int32_t* f_op, const double* kx, const double2* xbar,
                               const int32_t* col_map, const int32_t* var_rec, const int32_t* var_phase,
                               int nadd, const double2* const* adds, const double* add_coefs, double2* out);
cudaError_t launch_adj_tinvh(cudaStream_t s, int P, int Nz, int S, int n, const double2* xt_bar,
                             const int32_t* col_map, const int32_t* var_rec, const int32_t* var_phase,
                             double2* out);
cudaError_t launch_dz_adjoint(cudaStream_t s, int P, int Nz, double scale, const double2* dst_bar,
                              double2* src_bar);

// Stored vectors and right-hand sides one stage combines: RK443's fourth
// stage takes M~X~^0 and three L~X~^j, and four F~^j.
constexpr int SP_MAX_TERMS = 4;

// Row items of the right-hand-side assembly: -1 where a mode has no row, else
// row << 3 | differential << 2 | (-phase & 3).
constexpr int ROW_ITEM_BITS = 3;
constexpr int ROW_ITEM_DIF = 4;

// Arguments of the pencil right-hand-side assembly + solve + epilogue kernel.
struct SolveArgs {
  int P, n, Nz, S, nbc;
  int kl, kuu, npad, lpad, upad;
  const double* Lf; const uint8_t* piv; const double* Uf; const double* rd;
  // prologue: B = sum_k vec_coef[k] vec[k] + mv_coef (Mat x) + sum_k fc_coef[k] P^L Fc_k + bc_coef g
  int nvec; const double2* vec[SP_MAX_TERMS]; double vec_coef[SP_MAX_TERMS];
  const double2* mv_x; const double* mv_vals; double mv_coef; double2* mv_store;
  const int32_t* mv_indptr; const int32_t* mv_indices; int mv_nnz;   // pattern of mv_vals
  // + mv2_coef (Mat2 x) on the same x (null mv2_vals: none)
  const double* mv2_vals; double mv2_coef;
  const int32_t* mv2_indptr; const int32_t* mv2_indices; int mv2_nnz;
  int nfc; const double2* fc[SP_MAX_TERMS]; double fc_coef[SP_MAX_TERMS];
  // fc_coef / 2 and -fc_coef / 2 for the T-to-U rows, filled by the launcher
  double fc_half[SP_MAX_TERMS], fc_mhalf[SP_MAX_TERMS];
  double bc_coef;
  // epilogue
  double2* xt_out; double2* xc_out; float2* xc32_out;   // xc32_out: FP32 copy (mixed precision)
  float* xs32_out;                             // split FP32 copy [var][2p + c][m] (tensor-core z transform)
  const double* ep_mv_vals; double2* ep_mv_store;
  // epilogue (mode 2): store (B~ - ep_alpha M~X~) ep_from_b, i.e. L~X~ from the
  // stage's own right-hand side, when ep_from_b != 0 (mixed precision only)
  double ep_from_b, ep_alpha;
  const double2* ep_mv_addvec;                 // epilogue matvec acts on (X~ + addvec) if set
  const int4* ep_list; int ep_nl;              // (row, first entry, entries) of its ep_nl rows with entries
  const int32_t* ep_indices; int ep_nnz;
  // tables (device)
  const int32_t* row_item;               // [equation][mode], see ROW_ITEM_BITS
  const int32_t* col_map;
  const int32_t* var_recombine; const int32_t* var_phase;
  const int32_t* nl_eq; int n_nl;        // equation index of each nonlinear slot
  const int32_t* bc_rows; const double2* bc_values;
  DevStatus* status;
  // mode 0: assembly, substitution and epilogue in one kernel; 1: assembly
  // only, B~ to bg; 2: epilogue only, from xg (the substitution runs in between:
  // bg, xg by group or by pencil, xg holds b = U_jj x~); 3: assembly and
  // whole-row forward substitution, y to yg (by pencil).  The one-CTA partitioned
  // kernel keeps B~ [p][n] in bg for the epilogue's L~X~
  int mode, by_pencil;
  double2* bg; const double2* xg; double2* yg;
  // the factor's lists (host pointer; null: no lane substitution)
  const LaneList* ll;
  // coupling matrices of the partitioned substitution (null: not available)
  const double* spD; const double* spE;
  int sp_passes;                // 1: row blocks in launches of their own (spike.cu), 0: in one (split.cu)
  int sp_nblk, sp_nblk_f;       // back- and forward-substitution blocks per pencil (nblk_f 0: forward whole)
  double* sp_u;                 // back-substitution inflows, the next solve's guesses [p][nblk][2][32]
  // 1: start from zero inflows; 0: from the previous solve's, for right-hand
  // sides that change little from solve to solve (rounding errors scale with the guess)
  int sp_cold;
};

// fc_half / fc_mhalf from fc_coef (exact scalings), before a launch
inline void fill_f_halves(SolveArgs& a) {
  for (int k = 0; k < SP_MAX_TERMS; ++k) {
    a.fc_half[k] = 0.5 * a.fc_coef[k];
    a.fc_mhalf[k] = -0.5 * a.fc_coef[k];
  }
}

// Transform arguments.
struct GridField { int var; int op; };

struct TransformPlan {
  int Nc, Ng;                   // coefficients and grid points along one axis
  int radix3;
  void* tw64 = nullptr;         // double2[Ng]  exp(-2 pi i t / Ng)
  void* tw32 = nullptr;         // float2[Ng]
  void* dct64 = nullptr;        // double2[Ng]  exp(-i pi k / (2 Ng))
  void* dct32 = nullptr;
};

// Per-problem descriptors of the transform kernels (tw / wq / gz / h are
// typed by the precision of the launch).
struct ZDesc {
  int Nc, Ng, radix3, P;
  const void* tw; const void* wq;
  // backward
  const int32_t* f_var; const int32_t* f_op; const double* kx; const double2* xc; int xc_stride; void* gz;
  const float* kx32; const float2* xc32;     // FP32 copies (mixed precision)
  // forward
  const void* h; double2* fc;
  int unweighted;                            // 1: transpose of the backward transform
  int weighted_in;                           // 1: transpose of the forward transform
};
struct XDesc {
  int N, radix3, rows, K, mode, nf;
  const void* tw;
  const void* gz; const double* grid_in; double* grid_out;
  int nterms; const int32_t* t_eq; const double* t_coef; const int32_t* t_fa; const int32_t* t_fb;
  int ne; void* h;
  const float* t_coef32;
  const void* hin; void* gzadj;             // adjoint rows: inputs / outputs
  int xscale;                                // bit 1: transpose of forward x on input; bit 2: of backward x on output
  int pairs;                                 // field pairs per backward FFT round (0: two)
  // rows.cuh: grid field f is input f_src[f], times i k_x where f_dx[f] is set
  const int32_t* f_src; const int32_t* f_dx; const double* kx; const float* kx32;
};

// Complex Fourier y transform of nf x nz planes of N_y slots x K columns.
struct YDesc {
  int Ny, Ng, K, nz, radix3, dir;
  const void* tw;
  const void* src; void* dst;
  // rows.cuh, dir < 0: output f is input f_src[f], times i k_y where f_dy[f] is
  // set (ky, ky32: one value per slot, K apart)
  const int32_t* f_src; const int32_t* f_dy; const double* ky; const float* ky32;
};

// --- launchers (band.cu) ---------------------------------------------------
cudaError_t launch_band_factor(cudaStream_t s, int P, int n, int nnz, int kl, int ku,
                               const int32_t* indptr, const int32_t* indices,
                               const double* Mv, const double* Lv, double alpha, double beta,
                               double* work, const BandFactor& f, int npad, int lpad, int upad,
                               DevStatus* st);
cudaError_t launch_pencil_solve(cudaStream_t s, const SolveArgs& a);
cudaError_t launch_eig_update(cudaStream_t s, int P, int n, double2* x, const double2* y, double2* mu);
cudaError_t launch_eig_residual(cudaStream_t s, int P, int n, int nnz, const int32_t* indptr, const int32_t* indices,
                                const double* Mv, const double* Lv, const double2* x, const double2* sig,
                                double* res);
size_t pencil_solve_smem(int npad, int lpad, int upad);
// the kernel that solves P pencils in whole-row order, one launch
enum WholeRowKernel { WHOLE_WINDOW, WHOLE_NARROW, WHOLE_PAIR };
WholeRowKernel whole_row_kernel(int P, int npad, int lpad, int upad);
cudaError_t launch_pencil_solve_batched(cudaStream_t s, const SolveArgs* args, const int4* work, int nwork, int max_kuu,
                                        size_t smem);
// partitioned pencil solve, one CTA per pencil (split.cu)
cudaError_t launch_pencil_split(cudaStream_t s, const SolveArgs& a);
cudaError_t launch_pencil_split_batched(cudaStream_t s, const SolveArgs* args, const int4* work, int nwork,
                                        size_t smem);
size_t pencil_split_smem(int npad, int nblk, int nblk_f, int kuu, bool wide);
// whole-row-order solves of one or two pencils per CTA (pair.cu); batched: work
// items (problem, first pencil, pencils)
cudaError_t launch_pencil_pair(cudaStream_t s, const SolveArgs& a);
cudaError_t launch_pencil_pair_batched(cudaStream_t s, const SolveArgs* args, const int4* work, int nwork, int max_kl,
                                       int max_kuu, size_t smem);
size_t pencil_pair_smem(int npad, int per);
int pencil_pair_per(int npad, long long pencils);
constexpr int PAIR_MIN_PENCILS = 4 * GPU_SMS;
// assembly and epilogue launches with fewer pencils use 512 threads per pencil
constexpr int STAGE_WIDE_PENCILS = 2 * GPU_SMS;
bool lanes_supported(int kl, int kuu);
cudaError_t launch_coef_to_solve(cudaStream_t s, int P, int S, int Nz, const double2* xc,
                                 double2* xt, const int32_t* col_map, const int32_t* var_recombine,
                                 const int32_t* var_phase);
cudaError_t launch_dz(cudaStream_t s, int P, int Nz, double scale, const double2* src, double2* dst);
cudaError_t launch_to_f32(cudaStream_t s, const double2* src, float2* dst, size_t n);

// --- launchers (transforms.cu) ---------------------------------------------
// precision: 0 = double, 1 = float.  Buffers of the grid stages are typed by
// the precision; coefficient-space inputs/outputs are always double2.
cudaError_t launch_cheb_backward(cudaStream_t s, int prec, const TransformPlan& pz, int P,
                                 int nf, const int32_t* f_var, const int32_t* f_op,
                                 const double* kx, const double2* xc, int xc_field_stride,
                                 void* gz, const float* kx32 = nullptr, const float2* xc32 = nullptr,
                                 int weighted_in = 0);
cudaError_t launch_fourier_rows(cudaStream_t s, int prec, const TransformPlan& px, int rows,
                                int P, int mode, int nf, const void* gz, double* grid_in,
                                double* grid_out, int nterms, const int32_t* t_eq,
                                const double* t_coef, const int32_t* t_fa, const int32_t* t_fb,
                                int ne, void* h, const float* t_coef32 = nullptr, int xscale = 0);
cudaError_t launch_cheb_forward(cudaStream_t s, int prec, const TransformPlan& pz, int P, int ne,
                                const void* h, double2* fc, int unweighted = 0);
cudaError_t launch_fourier_rows_adjoint(cudaStream_t s, int prec, const TransformPlan& px, int rows, int P,
                                        int nf, const void* gz, int ne, const void* hin, int nterms,
                                        const int32_t* t_eq, const double* t_coef, const float* t_coef32,
                                        const int32_t* t_fa, const int32_t* t_fb, void* gzadj);
// dir < 0: slots -> grid, dir > 0: grid -> slots (1/N_gy, Nyquist slot zero);
// py = plan (N_y, N_gy); buffers [f][zg][slot or yg][K] in the precision.
cudaError_t launch_cfl_max(cudaStream_t s, const double* grid, int nvel, const int* axes, int Ngx, int Ngy, int Ngz,
                           double inv_dx, double inv_dy, const double* inv_dz, unsigned long long* out);
cudaError_t launch_fourier_y(cudaStream_t s, int prec, const TransformPlan& py, int dir, int nf, int nz, int K,
                             const void* src, void* dst);
size_t z_smem_bytes(int prec, int Ng, int tile);
size_t x_smem_bytes(int prec, int N, int mode, int nf, int ne, int pairs = 0);
// the right-hand side's transforms on compile-time lengths (rows.cuh), float or
// double; cudaErrorInvalidValue for a length or size they do not take
constexpr size_t ROWS_SMEM_MAX = 226 * 1024;   // dynamic shared memory of a CTA, its static tables beside it
inline bool fft_planned(int N) { return N >= 16 && N <= 4096 && (((N & (N - 1)) == 0) || (N % 3 == 0 && (((N / 3) & (N / 3 - 1)) == 0))); }
inline size_t rows_padded(int prec, int N) { return (size_t)(N + (prec ? N / 16 : N / 8)) * (prec ? 8 : 16); }
inline size_t x_rows_bytes(int prec, int N, int nf, int ne) {
  const int nbi = (nf + 1) / 2, nbo = (ne + 1) / 2;
  return (nbi + (nbi > 2 * nbo ? nbi : 2 * nbo)) * rows_padded(prec, N);
}
// Forward sums leave the FP32 x transform times 2^-rows_shift(2 N), the y
// transform times 2^-rows_shift(N): exact, and no sum grows past its own
// transform's length.  The z transform's table takes the rest of 1 / (2 N_gx N_gy).
__host__ __device__ constexpr int rows_shift(int n) {
  int e = 0;
  while ((1 << e) < n) ++e;
  return e;
}
inline int z_cols_tile(int prec) { return prec ? 8 : 4; }
inline size_t z_cols_bytes(int prec, int N) {   // two buffers of tile columns, each one element over a multiple of 16
  const size_t el = N + (prec ? N / 16 : N / 8);
  return 2 * z_cols_tile(prec) * ((el + 15) / 16 * 16 + 1) * (prec ? 8 : 16);
}
template <typename T> cudaError_t launch_x_rows(cudaStream_t s, const XDesc& d);
template <typename T> cudaError_t launch_y_cols(cudaStream_t s, const YDesc& d, int nf);
template <typename T> cudaError_t launch_z_cols(cudaStream_t s, const ZDesc& d, int nf, bool forward);
template <typename T>
cudaError_t launch_x_rows_batched(cudaStream_t s, const XDesc* ds, const int4* work, int nwork, size_t smem,
                                  int* queue);
template <typename T>
cudaError_t launch_z_cols_batched(cudaStream_t s, bool forward, const ZDesc* ds, const int4* work, int nwork,
                                  size_t smem, int* queue);
// batched transforms: queue null: one CTA per work item; else a persistent
// grid pulling items from the device counter *queue (zero before the launch)
cudaError_t launch_cheb_backward_batched(cudaStream_t s, int prec, int tile, const ZDesc* ds, const int4* work,
                                         int nwork, int max_ng, int* queue = nullptr);
cudaError_t launch_cheb_forward_batched(cudaStream_t s, int prec, int tile, const ZDesc* ds, const int4* work,
                                        int nwork, int max_ng, int* queue = nullptr);
cudaError_t launch_fourier_rows_batched(cudaStream_t s, int prec, const XDesc* ds, const int4* work, int nwork,
                                        size_t smem, int* queue = nullptr);

}  // namespace spectau
