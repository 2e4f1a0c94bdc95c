// Right-hand-side assembly and epilogue of one pencil's solve, shared by the
// solve kernels (sm_103a).  B: the pencil's right-hand side / solution in
// shared memory, one complex entry per row.
#pragma once
#include "internal.h"

namespace spectau {

// U: rows (or entries) a thread takes at once; their loads are issued
// together, then used.  Each is a chain of two or three dependent reads of
// global memory.  Four in the assembly-only and epilogue-only kernels, which do
// nothing else (3D 128 x 128 x 64 mixed, per stage: assembly 120 -> 106 us,
// epilogue 150 -> 132 us, the rest is FP64 issue; Fisher-KPP 2048 x 1024: 76 ->
// 53 us and 112 -> 103 us).  One in the kernels that also substitute: there each
// CTA runs straight through all the code once and the longer code costs more
// than the overlap gives (64 x 32, one solve: 43.0 us with 1, 43.9 with 2, 44.6
// with 4; batched 16-problem solve 586, 597 and 592 us).

// c v, exactly v when c = 1 (tested on the bit pattern: no FP64 compare)
__device__ __forceinline__ double2 scale_first(double c, double2 v) {
  if (__double_as_longlong(c) == 0x3FF0000000000000LL) return v;
  return make_double2(c * v.x, c * v.y);
}

// B~ of pencil p = linear combination of stored vectors, one or two matvecs,
// left-preconditioned F~ (T-to-U conversion, tau rows dropped) and boundary
// values, in passes over the rows, each with every lane on the same kind of
// row, since on GB300 an FP64 warp instruction holds the FP64 pipe for 64
// cycles whatever its active mask: stored vectors and matvecs for every row,
// then the F~ entries by (slot, mode), then the boundary rows.  Rows [n, top)
// are zeroed.  Called by all nt threads of the pencil; ends with a barrier.
template <int U>
__device__ __forceinline__ void pencil_assemble(const SolveArgs& a, int p, int tid, int nt, int top, double2* B) {
  const int n = a.n, Nz = a.Nz;
  const size_t prow = (size_t)p * n;
  const float invNz = 1.0f / (float)Nz;
  const double2 zero = make_double2(0.0, 0.0);
  for (int r0 = tid; r0 < n; r0 += U * nt) {
    double2 acc[U], v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int r = r0 + u * nt;
      acc[u] = (a.nvec > 0 && r < n) ? a.vec[0][prow + r] : zero;
    }
    if (a.nvec > 0) {
#pragma unroll
      for (int u = 0; u < U; ++u) acc[u] = scale_first(a.vec_coef[0], acc[u]);
    }
    for (int k = 1; k < a.nvec; ++k) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int r = r0 + u * nt;
        v[u] = r < n ? a.vec[k][prow + r] : zero;
      }
      const double c = a.vec_coef[k];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (r0 + u * nt >= n) break;
        acc[u].x = fma(c, v[u].x, acc[u].x);
        acc[u].y = fma(c, v[u].y, acc[u].y);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (r0 + u * nt < n) B[r0 + u * nt] = acc[u];
  }
  if (a.mv_x != nullptr) {
    // (every thread adds to the rows it has just written)
    for (int r = tid; r < n; r += nt) {
      double2 acc = B[r], s = zero;
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
      if (a.mv2_vals != nullptr) {               // a second matrix on the same vector (CNAB: L~ X~^n)
        s = zero;
        const double* vals2 = a.mv2_vals + (size_t)p * a.mv2_nnz;
        for (int e = a.mv2_indptr[r]; e < a.mv2_indptr[r + 1]; ++e) {
          const double m = vals2[e];
          const double2 x = a.mv_x[prow + a.mv2_indices[e]];
          s.x = fma(m, x.x, s.x);
          s.y = fma(m, x.y, s.y);
        }
        acc.x = fma(a.mv2_coef, s.x, acc.x);
        acc.y = fma(a.mv2_coef, s.y, acc.y);
      }
      B[r] = acc;
    }
  }
  for (int r = n + tid; r < top; r += nt) B[r] = zero;
  __syncthreads();
  // acc + the left-preconditioned F~ entry of (slot, mode m): the combination
  // sum_k c_k F_k of the stored right-hand sides, through the T-to-U
  // conversion P^L for differential equations (Appendix: row m holds
  // (1 + delta_m0)/2 F_m - F_{m+2}/2) and the phase i^-q of the equation's
  // real-ification.  One FMA per term and component: the halves c/2 and -c/2
  // come precomputed with the arguments and the phase is applied to the
  // loaded values (a sign and swap, no arithmetic).
  const int nf = a.nfc > 0 ? a.n_nl * Nz : 0;
  for (int i0 = tid; i0 < nf; i0 += U * nt) {
    int it[U];
    size_t at[U];
    bool two[U], top_row[U];                     // a second term; half the first one
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int idx = i0 + u * nt;
      const int sl = div_idx(idx, invNz), m = idx - sl * Nz;
      it[u] = idx < nf ? a.row_item[a.nl_eq[sl] * Nz + m] : -1;
      at[u] = ((size_t)sl * a.P + p) * Nz + m;
      two[u] = m + 2 < Nz;
      top_row[u] = m > 0;
    }
    double2 acc[U], v0[U], v2[U];
    for (int k = 0; k < a.nfc; ++k) {
      const double2* F = a.fc[k];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const bool dif = (it[u] & ROW_ITEM_DIF) != 0;
        v0[u] = it[u] >= 0 ? F[at[u]] : zero;
        v2[u] = (it[u] >= 0 && dif && two[u]) ? F[at[u] + 2] : zero;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (it[u] < 0) continue;
        const bool dif = (it[u] & ROW_ITEM_DIF) != 0;
        if (k == 0) acc[u] = B[it[u] >> ROW_ITEM_BITS];
        const double2 f0 = cipow_d(v0[u], it[u]);
        const double c = (dif && top_row[u]) ? a.fc_half[k] : a.fc_coef[k];
        acc[u].x = fma(c, f0.x, acc[u].x);
        acc[u].y = fma(c, f0.y, acc[u].y);
        if (dif && two[u]) {
          const double2 f2 = cipow_d(v2[u], it[u]);
          acc[u].x = fma(a.fc_mhalf[k], f2.x, acc[u].x);
          acc[u].y = fma(a.fc_mhalf[k], f2.y, acc[u].y);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (it[u] >= 0) B[it[u] >> ROW_ITEM_BITS] = acc[u];
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
template <int U, typename V>
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
  const int nx = a.xc_out ? a.S * Nz : 0;
  for (int i0 = tid; i0 < nx; i0 += U * nt) {
    int v[U], m[U], c0[U], c2[U], ph[U];         // columns of the entry's one or two coefficients
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int idx = i0 + u * nt;
      const bool in = idx < nx;
      v[u] = in ? div_idx(idx, invNz) : 0;
      m[u] = idx - v[u] * Nz;
      c0[u] = in ? a.col_map[idx] : -1;
      c2[u] = (in && m[u] + 2 < Nz) ? a.col_map[idx + 2] : -1;
      ph[u] = a.var_phase[v[u]];
      if (!a.var_recombine[v[u]]) c2[u] = -1;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (c0[u] < 0) continue;
      double2 x = B[c0[u]];
      if (c2[u] >= 0) {
        const double2 x2 = B[c2[u]];
        x.x -= x2.x;
        x.y -= x2.y;
      }
      const double2 xv = cipow_d(x, ph[u]);
      const size_t o = (size_t)v[u] * a.P + p;
      a.xc_out[o * Nz + m[u]] = xv;
      if (a.xc32_out) a.xc32_out[o * Nz + m[u]] = make_float2((float)xv.x, (float)xv.y);
      if (a.xs32_out) {
        a.xs32_out[o * 2 * Nz + m[u]] = (float)xv.x;
        a.xs32_out[(o * 2 + 1) * Nz + m[u]] = (float)xv.y;
      }
    }
  }
  if (a.ep_mv_vals) {
    const double* vals = a.ep_mv_vals + (size_t)p * a.ep_nnz;
    const bool listed = a.ep_nl < n;
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
    const int nrows = a.ep_nl;
    for (int i = tid; i < nrows; i += nt) {
      const int4 it = a.ep_list[i];
      const int r = it.x;
      double2 s = make_double2(0.0, 0.0);
      for (int e = it.y; e < it.y + it.z; ++e) {
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
