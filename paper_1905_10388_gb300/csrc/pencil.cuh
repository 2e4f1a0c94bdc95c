// Right-hand-side assembly and epilogue of one pencil's solve, shared by the
// solve kernels (sm_103a).  B: the pencil's right-hand side / solution in
// shared memory, one complex entry per row.
#pragma once
#include "internal.h"

namespace spectau {

// acc + the left-preconditioned F~ entry of row (slot sl, mode m): the
// combination sum_k c_k F_k of the stored right-hand sides, through the
// T-to-U conversion P^L for differential equations (Appendix: row m holds
// (1 + delta_m0)/2 F_m - F_{m+2}/2) and the phase i^-q of the equation's
// real-ification.  One FMA per term and component: on GB300 every FP64
// instruction holds the sub-partition's FP64 pipe for 64 cycles, so the
// halves c/2 and -c/2 come precomputed with the arguments and the phase is
// applied to the loaded values (a sign and swap, no arithmetic).
__device__ __forceinline__ double2 add_f_row(const SolveArgs& a, int sl, int m, int p, double2 acc) {
  const int Nz = a.Nz;
  const int e = a.nl_eq[sl];
  const bool dif = a.eq_differential[e] != 0;
  const int ph = -a.eq_phase[e];
#pragma unroll
  for (int k = 0; k < SP_MAX_TERMS; ++k) {
    if (k >= a.nfc) break;
    const double2* F = a.fc[k] + ((size_t)sl * a.P + p) * Nz;
    const double2 v0 = cipow_d(F[m], ph);
    const double c = (dif && m > 0) ? a.fc_half[k] : a.fc_coef[k];
    acc.x = fma(c, v0.x, acc.x);
    acc.y = fma(c, v0.y, acc.y);
    if (dif && m + 2 < Nz) {
      const double2 v2 = cipow_d(F[m + 2], ph);
      acc.x = fma(a.fc_mhalf[k], v2.x, acc.x);
      acc.y = fma(a.fc_mhalf[k], v2.y, acc.y);
    }
  }
  return acc;
}

// c v, exactly v when c = 1 (tested on the bit pattern: no FP64 compare)
__device__ __forceinline__ double2 scale_first(double c, double2 v) {
  if (__double_as_longlong(c) == 0x3FF0000000000000LL) return v;
  return make_double2(c * v.x, c * v.y);
}

// B~ of pencil p = linear combination of stored vectors, one or two matvecs,
// left-preconditioned F~ (T-to-U conversion, tau rows dropped) and boundary
// values, in two passes over the rows, each with every lane on the same kind
// of row, since on GB300 an FP64 warp instruction holds the FP64 pipe for 64
// cycles whatever its active mask: stored vectors and matvec for every row,
// then the F~ entries by (slot, mode), then the boundary rows.  Rows [n, top)
// are zeroed.  Called by all nt threads of the pencil; ends with a barrier.
__device__ __forceinline__ void pencil_assemble(const SolveArgs& a, int p, int tid, int nt, int top, double2* B) {
  const int n = a.n, Nz = a.Nz;
  const size_t prow = (size_t)p * n;
  const float invNz = 1.0f / (float)Nz;
  for (int r = tid; r < n; r += nt) {
    double2 acc = make_double2(0.0, 0.0);
    if (a.nvec > 0) acc = scale_first(a.vec_coef[0], a.vec[0][prow + r]);
    for (int k = 1; k < a.nvec; ++k) {
      const double2 v = a.vec[k][prow + r];
      acc.x = fma(a.vec_coef[k], v.x, acc.x);
      acc.y = fma(a.vec_coef[k], v.y, acc.y);
    }
    if (a.mv_x != nullptr) {
      double2 s = make_double2(0.0, 0.0);
      const double* vals = a.mv_vals + (size_t)p * a.mv_nnz;
      for (int e = a.mv_indptr[r]; e < a.mv_indptr[r + 1]; ++e) {
        const double m = vals[e];
        const double2 x = a.mv_x[prow + a.mv_indices[e]];
        s.x = fma(m, x.x, s.x);
        s.y = fma(m, x.y, s.y);
      }
      if (a.mv_store != nullptr) a.mv_store[prow + r] = s;
      acc.x = fma(a.mv_coef, s.x, acc.x);
      acc.y = fma(a.mv_coef, s.y, acc.y);
    }
    if (a.mv2_vals != nullptr) {                 // a second matrix on the same vector (CNAB: L~ X~^n)
      double2 s = make_double2(0.0, 0.0);
      const double* vals = a.mv2_vals + (size_t)p * a.mv2_nnz;
      for (int e = a.mv2_indptr[r]; e < a.mv2_indptr[r + 1]; ++e) {
        const double m = vals[e];
        const double2 x = a.mv_x[prow + a.mv2_indices[e]];
        s.x = fma(m, x.x, s.x);
        s.y = fma(m, x.y, s.y);
      }
      acc.x = fma(a.mv2_coef, s.x, acc.x);
      acc.y = fma(a.mv2_coef, s.y, acc.y);
    }
    B[r] = acc;
  }
  for (int r = n + tid; r < top; r += nt) B[r] = make_double2(0.0, 0.0);
  __syncthreads();
  for (int idx = tid; idx < a.n_nl * Nz; idx += nt) {
    const int sl = div_idx(idx, invNz), m = idx - sl * Nz;
    const int e = a.nl_eq[sl];
    const int row = a.row_map[e * Nz + m];
    if (row < 0) continue;
    B[row] = add_f_row(a, sl, m, p, B[row]);
  }
  for (int q = tid; q < a.nbc; q += nt) {
    const int row = a.bc_rows[q];
    const double2 g = a.bc_values[(size_t)p * a.nbc + q];
    double2 b = B[row];
    b.x = fma(a.bc_coef, g.x, b.x);
    b.y = fma(a.bc_coef, g.y, b.y);
    B[row] = b;
  }
  __syncthreads();
}

// X~, the T coefficients and the stored matvec of pencil p from its solution
// B (vec(r): element r of the pencil in the substitution kernels' vectors;
// from_b: L~X~ may come from the stored B~).  Called by all nt threads.
template <typename V>
__device__ __forceinline__ void pencil_epilogue(const SolveArgs& a, int p, int tid, int nt, bool from_b, V&& vec,
                                                const double2* B) {
  const int n = a.n, Nz = a.Nz;
  const size_t prow = (size_t)p * n;
  const float invNz = 1.0f / (float)Nz;
  // ---- epilogue: store X~, recombine to T coefficients, optional M~ X~
  bool finite = true;
  for (int r = tid; r < n; r += nt) {
    const double2 x = B[r];
    finite = finite && dfinite(x.x) && dfinite(x.y);
    if (a.xt_out) a.xt_out[prow + r] = x;
  }
  if (a.xc_out) {
    for (int idx = tid; idx < a.S * Nz; idx += nt) {
      const int v = div_idx(idx, invNz), m = idx - v * Nz;
      double2 x = B[a.col_map[idx]];
      if (a.var_recombine[v] && m + 2 < Nz) {
        const double2 x2 = B[a.col_map[idx + 2]];
        x.x -= x2.x;
        x.y -= x2.y;
      }
      const double2 xv = cipow_d(x, a.var_phase[v]);
      a.xc_out[((size_t)v * a.P + p) * Nz + m] = xv;
      if (a.xc32_out) a.xc32_out[((size_t)v * a.P + p) * Nz + m] = make_float2((float)xv.x, (float)xv.y);
      if (a.xs32_out) {
        a.xs32_out[(((size_t)v * a.P + p) * 2) * Nz + m] = (float)xv.x;
        a.xs32_out[(((size_t)v * a.P + p) * 2 + 1) * Nz + m] = (float)xv.y;
      }
    }
  }
  if (a.ep_mv_vals) {
    const double* vals = a.ep_mv_vals + (size_t)p * a.ep_nnz;
    const bool listed = a.ep_rows != nullptr;
    if (listed) {
      // rows without entries first (zero, or B~/beta for L~X~ from the
      // stage right-hand side), then the listed rows with every lane on a
      // row that has entries; the barrier orders the two stores of a row
      for (int r = tid; r < n; r += nt) {
        double2 s = make_double2(0.0, 0.0);
        if (from_b && a.ep_from_b != 0.0) {
          const double2 bb = a.bg[vec(r)];
          s.x = bb.x * a.ep_from_b;
          s.y = bb.y * a.ep_from_b;
        }
        a.ep_mv_store[prow + r] = s;
      }
      __syncthreads();
    }
    const int nrows = listed ? a.ep_nrows : n;
    for (int i = tid; i < nrows; i += nt) {
      const int r = listed ? a.ep_rows[i] : i;
      double2 s = make_double2(0.0, 0.0);
      for (int e = a.ep_indptr[r]; e < a.ep_indptr[r + 1]; ++e) {
        const double m = vals[e];
        double2 x = B[a.ep_indices[e]];
        if (a.ep_mv_addvec) {
          const double2 y = a.ep_mv_addvec[prow + a.ep_indices[e]];
          x.x += y.x;
          x.y += y.y;
        }
        s.x = fma(m, x.x, s.x);
        s.y = fma(m, x.y, s.y);
      }
      if (from_b && a.ep_from_b != 0.0) {
        // L~ X~ = (B~ - alpha M~ X~) / beta for the stage matrix alpha M~ + beta L~
        const double2 bb = a.bg[vec(r)];
        s.x = (bb.x - a.ep_alpha * s.x) * a.ep_from_b;
        s.y = (bb.y - a.ep_alpha * s.y) * a.ep_from_b;
      }
      a.ep_mv_store[prow + r] = s;
    }
  }
  if (!finite) raise_status(a.status, SP_ERR_NONFINITE, p);
}

}  // namespace spectau
