// Partitioned pencil solve in one kernel (sm_103a): assembly, substitution in
// row blocks and epilogue of one pencil per CTA, for problems with few
// pencils.
//
// Sec. "Matrix solvers": each pencil's banded LU factor is reused for every
// solve while dt is fixed, and the solve is O(n) per pencil.  With few pencils
// the substitutions are too few dependent chains of n rows for GB300's 608
// sub-partitions, and each row costs a shuffle and a dependent DFMA (about 130
// cycles): the chain's latency bounds the whole-row-order solve.  Here every
// pencil's rows are cut into blocks substituted in parallel by the CTA's
// warps, in the manner of the SPIKE family of partitioned banded solvers
// (Polizzi & Sameh): a block's substitution is an affine map of the values
// that flow into it from its neighbour (the forward window's pending rows; the
// back substitution's kuu partial sums), so
//   1. every block runs with zero inflow, giving its outflow o0_k;
//   2. a short recurrence over blocks, inflow_{k+1} = o0_k + C_k inflow_k,
//      with C_k the block's coupling matrix (its response to unit inflows,
//      computed once per factorization, spike.cu), gives the true inflows;
//   3. every block runs again with its true inflow, giving its rows.
// The back substitution starts step 1 from a guess g_k instead of zero
// inflow, the true inflow of the problem's previous solve, and step 2
// becomes inflow_{k-1} = o_k + E_k (inflow_k - g_k): exact for any guess,
// but with zero inflow the velocity rows of a block's top (true values
// ~1e-3 of the buoyancy's early in a run) come out O(1) and the recurrence
// cancels them, so their rounding errors are O(1) too; consecutive solves of
// a time step differ by O(dt), the correction is small and nothing cancels.
// Factorization and setting a field reset the guesses to zero, and a guess
// that is not finite reads as zero.  The block that needs no inflow (the first
// for the forward pass, the last for the back substitution) is exact after
// step 1.  Every row's arithmetic is the whole-row-order substitution's; only
// the inflows are summed in another order.
//
// Forward substitution with kl <= 7 uses 8-lane windows (rows j .. j + 7), four
// chains per warp and FP64 instruction, over blocks of their own; a wider band
// (the adjoint's transposed factor) one 32-lane window per chain.  Back
// substitution: a 32-lane window per chain (kl + ku <= 31), the U columns
// loaded 16 ahead into registers, coalesced.  Right-hand side, y and x share
// one shared-memory vector; the boundary rows that a block's window reads
// ahead are set aside before its neighbour overwrites them.
#include <algorithm>

#include "internal.h"
#include "pencil.cuh"
#include "tma.cuh"

namespace spectau {

constexpr int SPL_W = 32;                        // window of the back and the wide forward substitution

// The back recurrence's coupling matrices (blocks 1 .. nblk - 2), in shared
// memory up to 48 KB (two CTAs per SM fit), else read where they are.
__host__ __device__ inline int split_e_doubles(int nblk, int kuu) {
  const int d = nblk > 2 ? (nblk - 2) * kuu * SPL_W : 0;
  return d * 8 <= 48 * 1024 ? d : 0;
}
// shared-memory doubles of one CTA
struct SplitSmem {
  size_t B, raw, s0, ss, D, E, o0, us, gs, part, ucur, bar, total;
};
__host__ __device__ inline SplitSmem split_smem(int npad, int nblk, int nblk_f, int kuu, bool wide) {
  const int fw = wide ? SPL_W : 8;
  SplitSmem m;
  size_t o = 0;
  m.B = o;    o += 2 * (size_t)(npad + 64);
  m.raw = o;  o += 2 * (size_t)(nblk_f + 1) * fw;
  m.s0 = o;   o += 2 * (size_t)(nblk_f + 1) * fw;
  m.ss = o;   o += 2 * (size_t)(nblk_f + 1) * fw;
  m.D = o;    o += wide ? 0 : (size_t)nblk_f * 56;
  m.E = o;    o += split_e_doubles(nblk, kuu);
  m.o0 = o;   o += 2 * (size_t)nblk * SPL_W;
  m.us = o;   o += 2 * (size_t)nblk * SPL_W;
  m.gs = o;   o += 2 * (size_t)nblk * SPL_W;
  m.part = o; o += 2 * 4 * SPL_W;
  m.ucur = o; o += 2 * SPL_W;
  m.bar = o;  o += 2;
  m.total = o;
  return m;
}

// ---------------------------------------------------------------------------
// forward substitution of block k's part c in an 8-lane segment.  Lane q of
// the segment holds row j + ((q - j) & 7) at step j.  PASS 1: zero inflow (the
// first block: its true rows), writes the outflow s0[k + 1]; PASS 2: the true
// inflow ss[k], writes y over the block's rows.
// ---------------------------------------------------------------------------
template <int PASS>
__device__ __forceinline__ void split_fwd8(const SolveArgs& a, int p, int k, int c, bool act, int m, double* B,
                                           const double* raw, double* s0, const double* ss) {
  const int q = threadIdx.x & 7;
  const int j0 = k * m, j1 = j0 + m;
  double* Bd = B + c;                            // row r at Bd[2 r]
  auto fresh = [&](int r) -> double {
    if (!act) return 0.0;
    return (PASS == 2 && r >= j1) ? raw[2 * ((k + 1) * 8 + r - j1) + c] : Bd[2 * r];
  };
  double v;
  if (PASS == 1)
    v = (k == 0 || q == 7) ? fresh(j0 + q) : 0.0;
  else
    v = (q < 7) ? (act ? ss[(2 * k + c) * 8 + q] : 0.0) : fresh(j0 + q);
  const double* Lp = a.Lf + (size_t)p * a.npad * a.lpad;
  const uint8_t* pv = a.piv + (size_t)p * a.npad;
  const int kl = a.kl, lpad = a.lpad;
  // each 8-row chunk's pivots, multipliers and fresh rows are loaded one
  // chunk ahead (a load consumed in its own chunk would stall the chain)
  unsigned long long pw;
  double lv[8], nv;
  auto load = [&](int j8, unsigned long long& pw_, double* lv_, double& nv_) {
    const bool in = act && j8 < j1;
    pw_ = in ? *reinterpret_cast<const unsigned long long*>(pv + j8) : 0ull;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int d = (q - i) & 7;
      lv_[i] = (in && d >= 1 && d <= kl) ? Lp[(size_t)(j8 + i) * lpad + d - 1] : 0.0;
    }
    nv_ = in ? fresh(j8 + 8 + q) : 0.0;
  };
  load(j0, pw, lv, nv);
  for (int j8 = j0; j8 < j1; j8 += 8) {
    unsigned long long pw2;
    double lv2[8], nv2, yo = 0.0;
    load(j8 + 8, pw2, lv2, nv2);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int off = (int)((pw >> (8 * i)) & 0xff);
      const int pl = (i + off) & 7;
      const double bj = __shfl_sync(0xffffffffu, v, pl, 8);   // pivot row value = y_j
      const double vo = __shfl_sync(0xffffffffu, v, i, 8);    // old row j value moves to the pivot row
      v = (q == pl) ? vo : v;
      v = fma(-lv[i], bj, v);
      yo = (q == i) ? bj : yo;
      v = (q == i) ? nv : v;                                   // row j + 8 enters in row j's slot
    }
    if (PASS == 2 && act) Bd[2 * (j8 + q)] = yo;
    pw = pw2;
    nv = nv2;
#pragma unroll
    for (int i = 0; i < 8; ++i) lv[i] = lv2[i];
  }
  // lane q now holds row j1 + q: the outflow is rows j1 .. j1 + 6
  if (PASS == 1 && act && q < 7) s0[(2 * (k + 1) + c) * 8 + q] = v;
}

// The same in a 32-lane window for kl <= 31 (rows j .. j + 31, outflow 31 rows).
template <int PASS>
__device__ __forceinline__ void split_fwd32(const SolveArgs& a, int p, int k, int c, int m, double* B,
                                            const double* raw, double* s0, const double* ss) {
  const int lane = threadIdx.x & 31;
  const int j0 = k * m, j1 = j0 + m, kl = a.kl, lpad = a.lpad;
  double* Bd = B + c;
  auto fresh = [&](int r) -> double { return (PASS == 2 && r >= j1) ? raw[2 * ((k + 1) * SPL_W + r - j1) + c] : Bd[2 * r]; };
  double v;
  if (PASS == 1)
    v = (k == 0 || lane == 31) ? fresh(j0 + lane) : 0.0;
  else
    v = lane < 31 ? ss[(2 * k + c) * SPL_W + lane] : fresh(j0 + lane);
  const double* Lp = a.Lf + (size_t)p * a.npad * lpad;
  const uint8_t* pv = a.piv + (size_t)p * a.npad;
  double la[16], lb[16];
  auto load = [&](int j, double* l) {            // multipliers of columns j .. j + 15 (j a multiple of 16)
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int d = (lane - j - i) & 31;
      l[i] = (j < j1 && d >= 1 && d <= kl) ? Lp[(size_t)(j + i) * lpad + d - 1] : 0.0;
    }
  };
  load(j0, la);
  load(j0 + 16, lb);
  uint4 pa = *reinterpret_cast<const uint4*>(pv + j0), pb = *reinterpret_cast<const uint4*>(pv + j0 + 16);
  double nv = fresh(j0 + 32 + lane);
  double vs = v;                                 // shuffle source: v before the owner takes its next row
  for (int jc = j0; jc < j1; jc += 32) {
    const bool more = jc + 32 < j1;
    const double nxt = more ? fresh(jc + 64 + lane) : 0.0;
    double yo = 0.0;
    auto half = [&](const double* l, const uint4& pw, int h) {
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int jj = h + i;
        const uint32_t w = i < 4 ? pw.x : (i < 8 ? pw.y : (i < 12 ? pw.z : pw.w));
        const int pl = (jj + (int)((w >> (8 * (i & 3))) & 0xff)) & 31;
        const double bj = __shfl_sync(0xffffffffu, vs, pl);
        const double vo = __shfl_sync(0xffffffffu, vs, jj);
        v = (lane == pl) ? vo : v;
        v = fma(-l[i], bj, v);
        vs = v;
        const bool own = lane == jj;
        yo = own ? bj : yo;
        v = own ? nv : v;
      }
    };
    half(la, pa, 0);
    load(jc + 32, la);
    if (more) pa = *reinterpret_cast<const uint4*>(pv + jc + 32);
    half(lb, pb, 16);
    load(jc + 48, lb);
    if (more) pb = *reinterpret_cast<const uint4*>(pv + jc + 48);
    if (PASS == 2) Bd[2 * (jc + lane)] = yo;
    nv = nxt;
  }
  if (PASS == 1 && lane < 31) s0[(2 * (k + 1) + c) * SPL_W + lane] = v;
}

// ---------------------------------------------------------------------------
// back substitution of block k's part c by one warp.  Lane l holds the row
// congruent to l mod 32 of rows j - 31 .. j.  PASS 1 (blocks 1 .. nblk - 1, or
// the one block): the guessed inflow, writes the outflow (the last block, which
// has no inflow, is final: x over its rows); PASS 2 (blocks 0 .. nblk - 2): the
// true inflow, x = y / U_jj over the block's rows.
// ---------------------------------------------------------------------------
template <int PASS>
__device__ __forceinline__ void split_bwd(const SolveArgs& a, int p, int k, int c, int nblk, int m, double* B,
                                          const double* gs, const double* us, double* o0) {
  const int lane = threadIdx.x & 31;
  const int j0 = k * m, j1 = j0 + m, kuu = a.kuu;
  double* Bd = B + c;
  const double* Up = a.Uf + (size_t)p * a.npad * SPL_W;
  const double* rdp = a.rd + (size_t)p * a.npad;
  double ua[16], ub[16];                         // scaled columns jc + 31 .. jc + 16 and jc + 15 .. jc
  auto load = [&](int j, double* u) {            // columns j + 15 .. j; the owner's entry (t = 0) is not used
#pragma unroll
    for (int i = 0; i < 16; ++i) u[i] = j >= j0 ? Up[(size_t)(j + 15 - i) * SPL_W + ((j + 15 - i - lane) & 31)] : 0.0;
  };
  load(j1 - 16, ua);
  load(j1 - 32, ub);
  auto yv = [&](int r) -> double { return r >= j0 ? Bd[2 * r] : 0.0; };
  double w = yv(j1 - SPL_W + lane);
  const int first_in = SPL_W - kuu;              // lanes first_in .. 31 hold the inflow rows
  if (lane >= first_in && k < nblk - 1) w += (PASS == 2 ? us : gs)[(2 * k + c) * SPL_W + lane - first_in];
  double nw = yv(j1 - 2 * SPL_W + lane);         // lane l takes row jc - 32 + l when it owns column jc + l
  double ws = w;                                 // shuffle source: w before the owner takes its next row
  const bool store = PASS == 2 || k == nblk - 1;
  for (int jc = j1 - 32; jc >= j0; jc -= 32) {
    const double rdl = store ? rdp[jc + lane] : 0.0;
    const double nxt = yv(jc - 2 * SPL_W + lane);
    double xo = 0.0;
    auto half = [&](const double* u, int h) {
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int jj = h + 15 - i;
        const double bj = __shfl_sync(0xffffffffu, ws, jj);
        w = fma(-u[i], bj, w);
        ws = w;
        const bool own = lane == jj;
        xo = own ? bj : xo;
        w = own ? nw : w;
      }
    };
    half(ua, 16);
    load(jc - 16, ua);
    half(ub, 0);
    load(jc - 32, ub);
    nw = nxt;
    if (store) Bd[2 * (jc + lane)] = xo * rdl;
  }
  // lane l holds row j0 - 32 + l: the outflow is rows j0 - kuu .. j0 - 1
  if (PASS == 1 && k > 0 && lane >= first_in) o0[(2 * k + c) * SPL_W + lane - first_in] = w;
}

// Recurrence vec_{q+1} = add_q + M_q (vec_q - g_q), q < steps, of both parts by
// the CTA's first eight warps, four per part: warp wq multiplies columns
// 8 wq .. 8 wq + 7 of row r = lane, the part's first warp adds the four sums.
// mat(q): rows of 32; add, guess (null: none) and store by step; vec_0 comes
// from the caller in `first` (lane r of each part's first warp).
template <typename M, typename A, typename G, typename S>
__device__ __forceinline__ void split_rec(int steps, int dim, double first, double* part, double* ucur, M&& mat,
                                          A&& add, G&& guess, S&& store) {
  const int r = threadIdx.x & 31, w = threadIdx.x >> 5, c = w >> 2, wq = w & 3;
  const bool in = w < 8;
  double en[8];
  auto load = [&](int q) {
    const double* row = mat(q) + (size_t)(r < dim ? r : 0) * SPL_W + wq * 8;
#pragma unroll
    for (int t = 0; t < 8; ++t) en[t] = (r < dim && wq * 8 + t < dim) ? row[t] : 0.0;
  };
  if (in && steps > 0) load(0);
  if (in && wq == 0) ucur[c * SPL_W + r] = r < dim ? first - (steps > 0 ? guess(0, c, r) : 0.0) : 0.0;
  __syncthreads();
  for (int q = 0; q < steps; ++q) {
    if (in) {
      double acc = 0.0;
#pragma unroll
      for (int t = 0; t < 8; ++t) acc = fma(en[t], ucur[c * SPL_W + wq * 8 + t], acc);
      part[(c * 4 + wq) * SPL_W + r] = acc;
      if (q + 1 < steps) load(q + 1);
    }
    __syncthreads();
    if (in && wq == 0) {
      double u = r < dim ? add(q, c, r) : 0.0;
#pragma unroll
      for (int t = 0; t < 4; ++t) u += part[(c * 4 + t) * SPL_W + r];
      if (r < dim) store(q, c, r, u);
      ucur[c * SPL_W + r] = (r < dim && q + 1 < steps) ? u - guess(q + 1, c, r) : 0.0;
    }
    __syncthreads();
  }
}

template <bool WIDE, int NT>
__device__ __forceinline__ void pencil_split_body(const SolveArgs& a, int p, double* sm) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = NT / 32, FW = WIDE ? SPL_W : 8;
  const int n = a.n, npad = a.npad, nblk = a.sp_nblk, nf = a.sp_nblk_f, kuu = a.kuu;
  const int m = npad / nblk, mf = npad / nf;
  const SplitSmem o = split_smem(npad, nblk, nf, kuu, WIDE);
  double *B = sm + o.B, *raw = sm + o.raw, *s0 = sm + o.s0, *ss = sm + o.ss, *Dm = sm + o.D;
  double *o0 = sm + o.o0, *us = sm + o.us, *gs = sm + o.gs, *part = sm + o.part, *ucur = sm + o.ucur;
  double* Em = sm + o.E;
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm + o.bar);
  // the coupling matrices (bulk copies) and the guesses come in while the
  // right-hand side is assembled
  const uint32_t dbytes = WIDE ? 0 : nf * 56 * 8, ebytes = split_e_doubles(nblk, kuu) * 8;
  const double* E1 = a.spE + ((size_t)p * nblk + 1) * kuu * SPL_W;
  if (tid == 0) {
    mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(bar, dbytes + ebytes);
    if (dbytes) bulk_g2s(Dm, a.spD + (size_t)p * nf * 56, dbytes, bar);
    if (ebytes) bulk_g2s(Em, E1, ebytes, bar);
  }
  double* uin = a.sp_u + (size_t)p * nblk * 2 * SPL_W;
  for (int q = tid; q < nblk * 2 * SPL_W; q += NT) {
    const double g = uin[q];
    gs[q] = (!a.sp_cold && dfinite(g)) ? g : 0.0;
  }
  pencil_assemble<1>(a, p, tid, NT, npad + 64, reinterpret_cast<double2*>(B));
  const size_t prow = (size_t)p * n;
  if (a.ep_from_b != 0.0)                        // the epilogue's L~X~ takes B~
    for (int r = tid; r < n; r += NT) a.bg[prow + r] = reinterpret_cast<double2*>(B)[r];
  for (int q = tid; q < (nf + 1) * FW; q += NT) {    // each block's first rows, before y overwrites them
    const int k = q / FW;
    reinterpret_cast<double2*>(raw)[q] = reinterpret_cast<double2*>(B)[k * mf + q - k * FW];
  }
  if (!bounded_wait(bar, 0)) {                   // (latched; the CTA ends as usual, its copies given time to land)
    raise_status(a.status, SP_ERR_TIMEOUT, p);
    bounded_wait(bar, 0);
  }
  __syncthreads();

  // ---- forward
  if (WIDE) {
    for (int t = warp; t < (nf - 1) * 2; t += NW) split_fwd32<1>(a, p, t >> 1, t & 1, mf, B, raw, s0, ss);
  } else {
    for (int t = warp * 4; t < (nf - 1) * 2; t += NW * 4) {
      const int ch = t + (lane >> 3);
      const bool act = ch < (nf - 1) * 2;
      split_fwd8<1>(a, p, act ? ch >> 1 : 0, ch & 1, act, mf, B, raw, s0, ss);
    }
  }
  __syncthreads();
  // inflows: s_1 = s0_1 (block 0 is exact), s_{k+1} = s0_{k+1} + D_k s_k
  if (WIDE) {
    const int c = warp >> 2;
    const bool lead = warp < 8 && (warp & 3) == 0 && lane < 31;
    if (lead) {
      ss[c * SPL_W + lane] = B[2 * lane + c];
      if (nf > 1) ss[(2 + c) * SPL_W + lane] = s0[(2 + c) * SPL_W + lane];
    }
    split_rec(nf - 2, 31, (lead && nf > 1) ? s0[(2 + c) * SPL_W + lane] : 0.0, part, ucur,
              [&](int q) { return a.spD + ((size_t)p * nf + q + 1) * 31 * SPL_W; },
              [&](int q, int cc, int r) { return s0[(2 * (q + 2) + cc) * SPL_W + r]; },
              [&](int, int, int) { return 0.0; },
              [&](int q, int cc, int r, double v) { ss[(2 * (q + 2) + cc) * SPL_W + r] = v; });
  } else if (warp == 0) {
    // lanes 0 .. 15: columns 0 .. 3 of part 0 and 1, lanes 16 .. 31: columns 4 .. 6
    const int c = (lane >> 3) & 1, i = lane & 7, ii = i < 7 ? i : 0, t0 = lane & 16 ? 4 : 0, nt = lane & 16 ? 3 : 4;
    const bool w = lane < 16 && i < 7;
    if (w) ss[c * 8 + i] = B[2 * i + c];
    double st = s0[(2 + c) * 8 + ii];
    if (w && nf > 1) ss[(2 + c) * 8 + i] = st;
    double d[4], add = 0.0;
    auto load = [&](int k) {
#pragma unroll
      for (int t = 0; t < 4; ++t) d[t] = t < nt ? Dm[(size_t)(k * 7 + ii) * 8 + t0 + t] : 0.0;
      add = lane < 16 ? s0[(2 * (k + 1) + c) * 8 + ii] : 0.0;
    };
    if (nf > 2) load(1);
    for (int k = 1; k < nf - 1; ++k) {
      double acc = add;
#pragma unroll
      for (int t = 0; t < 4; ++t) acc = fma(d[t], __shfl_sync(0xffffffffu, st, (t0 + t) & 7, 8), acc);
      if (k + 1 < nf - 1) load(k + 1);
      st = acc + __shfl_xor_sync(0xffffffffu, acc, 16);
      if (w) ss[(2 * (k + 1) + c) * 8 + i] = st;
    }
  }
  __syncthreads();
  if (WIDE) {
    for (int t = warp; t < nf * 2; t += NW) split_fwd32<2>(a, p, t >> 1, t & 1, mf, B, raw, s0, ss);
  } else {
    for (int t = warp * 4; t < nf * 2; t += NW * 4) {
      const int ch = t + (lane >> 3);
      const bool act = ch < nf * 2;
      split_fwd8<2>(a, p, act ? ch >> 1 : 0, ch & 1, act, mf, B, raw, s0, ss);
    }
  }
  __syncthreads();

  // ---- back (block 0's outflow has no use; the last block is final after pass 1)
  const int k0 = nblk > 1 ? 1 : 0;
  for (int t = warp; t < (nblk - k0) * 2; t += NW) split_bwd<1>(a, p, k0 + (t >> 1), t & 1, nblk, m, B, gs, us, o0);
  __syncthreads();
  if (nblk > 1) {
    // u_{nblk-2} = o_{nblk-1} (exact), u_{k-1} = o_k + E_k (u_k - g_k): step q of
    // the recurrence is k = nblk - 2 - q
    const int c = warp >> 2;
    const bool lead = warp < 8 && (warp & 3) == 0 && lane < kuu;
    const double first = lead ? o0[(2 * (nblk - 1) + c) * SPL_W + lane] : 0.0;
    if (lead) {
      us[(2 * (nblk - 2) + c) * SPL_W + lane] = first;
      uin[(2 * (nblk - 2) + c) * SPL_W + lane] = first;
    }
    split_rec(nblk - 2, kuu, first, part, ucur,
              [&](int q) { return (ebytes ? Em : E1) + (size_t)(nblk - 3 - q) * kuu * SPL_W; },
              [&](int q, int cc, int r) { return o0[(2 * (nblk - 2 - q) + cc) * SPL_W + r]; },
              [&](int q, int cc, int r) { return gs[(2 * (nblk - 2 - q) + cc) * SPL_W + r]; },
              [&](int q, int cc, int r, double v) {
                us[(2 * (nblk - 3 - q) + cc) * SPL_W + r] = v;
                uin[(2 * (nblk - 3 - q) + cc) * SPL_W + r] = v;
              });
    __syncthreads();
    for (int t = warp; t < (nblk - 1) * 2; t += NW) split_bwd<2>(a, p, t >> 1, t & 1, nblk, m, B, gs, us, o0);
    __syncthreads();
  }
  pencil_epilogue<1>(a, p, tid, NT, true, [&](int r) { return prow + r; }, reinterpret_cast<const double2*>(B));
}

template <bool WIDE, int NT>
__global__ void __launch_bounds__(NT, 512 / NT) k_pencil_split(SolveArgs a) {
  extern __shared__ __align__(16) double split_sm[];
  pencil_split_body<WIDE, NT>(a, blockIdx.x, split_sm);
}
// a batch of problems: work item (problem, pencil) per CTA
template <int NT>
__global__ void __launch_bounds__(NT, 512 / NT) k_pencil_split_batched(const SolveArgs* __restrict__ args,
                                                                       const int4* __restrict__ work) {
  extern __shared__ __align__(16) double split_sm[];
  const int4 w = work[blockIdx.x];
  pencil_split_body<false, NT>(args[w.x], w.y, split_sm);
}

size_t pencil_split_smem(int npad, int nblk, int nblk_f, int kuu, bool wide) {
  return split_smem(npad, nblk, nblk_f, kuu, wide).total * sizeof(double);
}

// One CTA of 512 threads per SM while every pencil has an SM of its own, two
// of 256 beyond that.
cudaError_t launch_pencil_split(cudaStream_t s, const SolveArgs& args) {
  SolveArgs a = args;
  fill_f_halves(a);
  const bool wide = a.kl > 7;
  if (a.kl > 30 || a.kuu >= SPL_W || a.upad != SPL_W || a.npad % (a.sp_nblk * SOLVE_CHUNK) ||
      a.npad % (a.sp_nblk_f * SOLVE_CHUNK))
    return cudaErrorInvalidValue;
  const size_t smem = pencil_split_smem(a.npad, a.sp_nblk, a.sp_nblk_f, a.kuu, wide);
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  cudaError_t e;
  auto go = [&](auto kernel, int nt) {
    if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) == cudaSuccess) {
      kernel<<<a.P, nt, smem, s>>>(a);
      e = cudaGetLastError();
    }
  };
  if (a.P <= GPU_SMS) {
    if (wide) go(k_pencil_split<true, 512>, 512);
    else go(k_pencil_split<false, 512>, 512);
  } else {
    if (wide) go(k_pencil_split<true, 256>, 256);
    else go(k_pencil_split<false, 256>, 256);
  }
  return e;
}

cudaError_t launch_pencil_split_batched(cudaStream_t s, const SolveArgs* args, const int4* work, int nwork,
                                        size_t smem) {
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  cudaError_t e;
  auto go = [&](auto kernel, int nt) {
    if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) == cudaSuccess) {
      kernel<<<nwork, nt, smem, s>>>(args, work);
      e = cudaGetLastError();
    }
  };
  if (nwork <= GPU_SMS) go(k_pencil_split_batched<512>, 512);
  else go(k_pencil_split_batched<256>, 256);
  return e;
}

}  // namespace spectau
