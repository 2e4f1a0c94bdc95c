// Partitioned substitution in launches of their own (sm_103a): the coupling
// matrices of every partitioned form (split.cu has the method), the recurrences
// over row blocks, and, for pencils that one CTA each does not suit (too many for
// one wave of them, or long and few), passes over the blocks of all pencils.
#include <algorithm>

#include "internal.h"
#include "tma.cuh"

namespace spectau {

constexpr int SPK_FW = 8;             // forward window rows (kl <= 7), 32 for wider bands
constexpr int SPK_FS = SPK_FW - 1;    // forward inflow: the window's first 7 rows
constexpr int SPK_BW = 32;            // backward window rows (kl + ku <= 31)
constexpr int SPK_CHUNK = 32;         // rows of a block: a multiple of this

// ---------------------------------------------------------------------------
// factorization time: the coupling matrices, lane i carrying unit inflow i.
// D_k[r][i]: forward window row r after block k for window row i = 1 before it
// (no fresh right-hand side); E_k[r][t]: backward outflow r (row j0 - kuu + r)
// for unit inflow t (row j1 - kuu + t), or, for the lane substitution (by_row),
// b of row j0 + r for unit b of row j1 + t.  The arithmetic is the
// substitution's own, written per row.  A warp takes a block's E, or its D with
// a 32-row window, or four blocks' D with 8-row windows.
//
// Bound by the FP64 pipe (64 cycles per warp instruction) and, with few
// pencils, by the row chain.  A 32-row window's row has 2 to 9 multipliers that
// are not zero of up to 31: they are loaded one per lane, four rows ahead, and
// a ballot picks the FMAs that are issued; the window stays in registers, the
// shift by a row being the FMA's destination.  One thread per inflow with
// indexed windows in local memory and every multiplier's FMA took 1625 us at
// 512 x 256 (256 pencils, 28 forward and 4 back blocks), 241 us for the
// 256 x 64 eigenvalue problem; this form 206 us and 87 us.
// ---------------------------------------------------------------------------
// window w of the row chain past one row with value y: w[t - 1] = w[t] - l_t y,
// l_t held by lane t (zero where the row has no multiplier)
__device__ __forceinline__ void window_step(double (&w)[SPK_BW], double l, double y) {
  const unsigned on = __ballot_sync(0xffffffffu, (__double_as_longlong(l) << 1) != 0);
#pragma unroll
  for (int t = 1; t < SPK_BW; ++t) {
    if ((on >> t) & 1u)
      w[t - 1] = fma(-__shfl_sync(0xffffffffu, l, t), y, w[t]);
    else
      w[t - 1] = w[t];
  }
  w[SPK_BW - 1] = 0.0;
}

constexpr int SPK_AHEAD = 4;          // rows loaded ahead (a divisor of SPK_CHUNK)

// D of one block, 32-row window
__device__ __forceinline__ void coupling_d32(int j0, int j1, int kl, int lpad, const double* __restrict__ Lp,
                                             const uint8_t* __restrict__ pv, double* __restrict__ Dk) {
  const int lane = threadIdx.x & 31;
  double w[SPK_BW], l[SPK_AHEAD];
#pragma unroll
  for (int t = 0; t < SPK_BW; ++t) w[t] = (t == lane) ? 1.0 : 0.0;
  uint32_t pw;
  auto load = [&](int j, double (&l_)[SPK_AHEAD], uint32_t& pw_) {
    const bool in = j < j1;
    pw_ = in ? *reinterpret_cast<const uint32_t*>(pv + j) : 0u;
#pragma unroll
    for (int i = 0; i < SPK_AHEAD; ++i)
      l_[i] = (in && lane >= 1 && lane <= kl) ? Lp[(size_t)(j + i) * lpad + lane - 1] : 0.0;
  };
  load(j0, l, pw);
  for (int j = j0; j < j1; j += SPK_AHEAD) {
    double ln[SPK_AHEAD];
    uint32_t pn;
    load(j + SPK_AHEAD, ln, pn);
#pragma unroll
    for (int i = 0; i < SPK_AHEAD; ++i) {
      const int off = (pw >> (8 * i)) & 0xff;
      double y = w[0];                  // the pivot row's value is y_j
      if (off != 0) {
#pragma unroll
        for (int t = 1; t < SPK_BW; ++t)
          if (t == off) { y = w[t]; w[t] = w[0]; }   // row j's value moves to the pivot row
      }
      window_step(w, l[i], y);
    }
    pw = pn;
#pragma unroll
    for (int i = 0; i < SPK_AHEAD; ++i) l[i] = ln[i];
  }
  if (lane < SPK_BW - 1) {
#pragma unroll
    for (int r = 0; r < SPK_BW - 1; ++r) Dk[r * SPK_BW + lane] = w[r];
  }
}

// D of one block, 8-row window, by eight lanes
__device__ __forceinline__ void coupling_d8(bool act, int j0, int m, int kl, int lpad, const double* __restrict__ Lp,
                                            const uint8_t* __restrict__ pv, double* __restrict__ Dk) {
  const int i = threadIdx.x & 7;
  double w[SPK_FW], l[SPK_FS];
#pragma unroll
  for (int t = 0; t < SPK_FW; ++t) w[t] = (t == i) ? 1.0 : 0.0;
  int off;
  auto load = [&](int j, double (&l_)[SPK_FS], int& off_) {
    const bool in = act && j < j0 + m;
    off_ = in ? pv[j] : 0;
#pragma unroll
    for (int d = 0; d < SPK_FS; ++d) l_[d] = (in && d < kl) ? Lp[(size_t)j * lpad + d] : 0.0;
  };
  load(j0, l, off);
  for (int j = j0; j < j0 + m; ++j) {
    double ln[SPK_FS];
    int on;
    load(j + 1, ln, on);
    double y = w[0];
#pragma unroll
    for (int t = 1; t < SPK_FW; ++t) {
      const bool at = t == off;
      y = at ? w[t] : y;
      w[t] = at ? w[0] : w[t];
    }
#pragma unroll
    for (int d = 0; d < SPK_FS; ++d) w[d] = fma(-l[d], y, w[d + 1]);
    w[SPK_FW - 1] = 0.0;
    off = on;
#pragma unroll
    for (int d = 0; d < SPK_FS; ++d) l[d] = ln[d];
  }
  if (act && i < SPK_FS) {
#pragma unroll
    for (int r = 0; r < SPK_FS; ++r) Dk[r * SPK_FW + i] = w[r];
  }
}

// E of one block
__device__ __forceinline__ void coupling_e(int j0, int j1, int kuu, int npad, int upad, bool by_row,
                                           const double* __restrict__ Up, double* __restrict__ Ek) {
  const int lane = threadIdx.x & 31;
  double w[SPK_BW], l[SPK_AHEAD];     // w[t]: pending row j - t
  // inflow `lane`: partial sum of row j1 - kuu + lane, or (by_row) b of row j1 + lane
#pragma unroll
  for (int t = 0; t < SPK_BW; ++t) {
    if (by_row)
      w[t] = (lane + 1 + t <= kuu && j1 + lane < npad) ? -Up[(size_t)(j1 + lane) * upad + lane + 1 + t] : 0.0;
    else
      w[t] = t == kuu - 1 - lane ? 1.0 : 0.0;
  }
  auto load = [&](int j, double (&l_)[SPK_AHEAD]) {     // rows j, j - 1, ..
#pragma unroll
    for (int i = 0; i < SPK_AHEAD; ++i)
      l_[i] = (j >= j0 && lane >= 1 && lane <= kuu) ? Up[(size_t)(j - i) * upad + lane] : 0.0;
  };
  load(j1 - 1, l);
  for (int j = j1 - 1; j >= j0; j -= SPK_AHEAD) {
    double ln[SPK_AHEAD];
    load(j - SPK_AHEAD, ln);
#pragma unroll
    for (int i = 0; i < SPK_AHEAD; ++i) {
      const double bj = w[0];
      if (by_row && j - i - j0 < kuu && lane < kuu) Ek[(j - i - j0) * SPK_BW + lane] = bj;
      window_step(w, l[i], bj);
    }
#pragma unroll
    for (int i = 0; i < SPK_AHEAD; ++i) l[i] = ln[i];
  }
  if (!by_row && lane < kuu) {
#pragma unroll
    for (int t = 0; t < SPK_BW; ++t)
      if (t < kuu) Ek[(kuu - 1 - t) * SPK_BW + lane] = w[t];
  }
}

constexpr int SPK_COUPLING_WARPS = 2;   // per CTA: few pencils spread over more SMs
template <int FW>
__global__ void __launch_bounds__(SPK_COUPLING_WARPS * 32)
    k_spike_coupling(int P, int npad, int nblk_f, int nblk, int kl, int kuu, int lpad, int upad,
                     const double* __restrict__ L, const uint8_t* __restrict__ piv, const double* __restrict__ U,
                     double* __restrict__ D, double* __restrict__ E, bool by_row) {
  constexpr int FS = FW - 1, PER = SPK_BW / FW;          // blocks of D per warp
  const int nd = (P * nblk_f + PER - 1) / PER, ne = P * nblk;
  int w = blockIdx.x * SPK_COUPLING_WARPS + (threadIdx.x >> 5);
  // the back blocks, the longer chains, first
  if (w < ne) {
    const int p = w / nblk, k = w - p * nblk, m = npad / nblk;
    coupling_e(k * m, (k + 1) * m, kuu, npad, upad, by_row, U + (size_t)p * npad * upad,
               E + (size_t)w * kuu * SPK_BW);
    return;
  }
  w -= ne;
  if (w >= nd) return;
  const int m = npad / nblk_f;
  const int b = w * PER + (FW == 8 ? (threadIdx.x & 31) >> 3 : 0);
  const bool act = b < P * nblk_f;
  const int p = act ? b / nblk_f : 0, k = act ? b - p * nblk_f : 0;
  const double* Lp = L + (size_t)p * npad * lpad;
  const uint8_t* pv = piv + (size_t)p * npad;
  double* Dk = D + ((size_t)p * nblk_f + k) * FS * FW;
  if constexpr (FW == 8)
    coupling_d8(act, k * m, m, kl, lpad, Lp, pv, Dk);
  else
    coupling_d32(k * m, (k + 1) * m, kl, lpad, Lp, pv, Dk);
}

cudaError_t launch_spike_coupling(cudaStream_t s, int P, int npad, int nblk_f, int nblk, int kl, int kuu, int lpad,
                                  int upad, const BandFactor& f, bool by_row) {
  // (nblk_f 0: E alone)
  if (kl > SPK_BW - 2 || kuu >= SPK_BW || nblk < 1 || nblk_f < 0 || npad % (nblk * SPK_CHUNK) ||
      (nblk_f > 0 && npad % (nblk_f * SPK_CHUNK)))
    return cudaErrorInvalidValue;
  const bool wide = kl > SPK_FS;
  const long long warps = (long long)P * nblk + (wide ? (long long)P * nblk_f : ((long long)P * nblk_f + 3) / 4);
  auto* k = wide ? k_spike_coupling<SPK_BW> : k_spike_coupling<SPK_FW>;
  k<<<(unsigned)((warps + SPK_COUPLING_WARPS - 1) / SPK_COUPLING_WARPS), SPK_COUPLING_WARPS * 32, 0, s>>>(
      P, npad, nblk_f, nblk, kl, kuu, lpad, upad, f.L, f.piv, f.U, f.spD, f.spE, by_row);
  return cudaGetLastError();
}

// forward inflows: s_0 = rows 0..6 of B~, s_1 from block 0 (exact), then
// s_{k+1} = s0_{k+1} + D_k s_k; eight lanes per (pencil, part), four of them per
// warp and FMA (a warp each, at seven FMAs a step, was bound by the FP64 pipe:
// Fisher-KPP 2048 x 1024, 2048 chains, 18.8 us against 13.9 us).  The
// next step's matrix row and outflow are loaded before this step's FMAs.
__global__ void __launch_bounds__(128) k_spike_fwd_rec(LaneArgs s, const double* __restrict__ D) {
  const int chain = (blockIdx.x * blockDim.x + threadIdx.x) >> 3;
  const bool act = chain < s.P * 2;
  const int p = act ? chain >> 1 : 0, c = chain & 1;
  const int q = threadIdx.x & 7, i = q < SPK_FS ? q : 0;
  const bool own = act && q < SPK_FS;
  const int r0 = i < s.n ? i : 0;
  const double* Bp =
      reinterpret_cast<const double*>(s.bg + (s.by_pencil ? (size_t)p * s.n + r0 : lane_index(p, r0, s.npad))) + c;
  auto at = [&](int k) { return (((size_t)p * s.nblk_f + k) * 2 + c) * SPK_FW; };
  double st = i < s.n ? Bp[0] : 0.0;
  if (own) s.sst[at(0) + i] = st;
  if (s.nblk_f < 2) return;
  st = s.s0[at(1) + i];
  if (own) s.sst[at(1) + i] = st;
  double dn[SPK_FS], sn = 0.0;
  auto load = [&](int k) {
    const double* Dk = D + ((size_t)p * s.nblk_f + k) * SPK_FS * SPK_FW + i * SPK_FW;
#pragma unroll
    for (int t = 0; t < SPK_FS; ++t) dn[t] = Dk[t];
    sn = s.s0[at(k + 1) + i];
  };
  if (s.nblk_f > 2) load(1);
  for (int k = 1; k < s.nblk_f - 1; ++k) {
    double dc[SPK_FS];
#pragma unroll
    for (int t = 0; t < SPK_FS; ++t) dc[t] = dn[t];
    double acc = sn, acc2 = 0.0;      // two independent FMA chains per step
    if (k + 1 < s.nblk_f - 1) load(k + 1);
#pragma unroll
    for (int t = 0; t < SPK_FS; t += 2) acc = fma(dc[t], __shfl_sync(0xffffffffu, st, t, 8), acc);
#pragma unroll
    for (int t = 1; t < SPK_FS; t += 2) acc2 = fma(dc[t], __shfl_sync(0xffffffffu, st, t, 8), acc2);
    st = acc + acc2;
    if (own) s.sst[at(k + 1) + i] = st;
  }
}

// the inflow that pass 1 started a block from
__device__ __forceinline__ double spike_guess(const LaneArgs& s, size_t i) {
  const double g = s.uin[i];
  return (!s.cold && dfinite(g)) ? g : 0.0;
}

// backward inflows: u_{nblk-2} = o_{nblk-1} (exact), then
// u_{k-1} = o_k + E_k (u_k - g_k), g_k the guess PASS 1 started block k
// from, which u_k replaces in place; one CTA of four warps per (pencil,
// part): warp q multiplies columns 8q .. 8q + 7 of row r = lane (four
// sub-partitions share each step's FMAs), warp 0 adds the four partial
// sums.  The next step's matrix entries are loaded before this step's FMAs.
constexpr int SPK_REC_WARPS = 4;
constexpr int SPK_REC_COLS = SPK_BW / SPK_REC_WARPS;
__global__ void __launch_bounds__(SPK_REC_WARPS * 32) k_spike_bwd_rec(LaneArgs s, const double* __restrict__ E) {
  __shared__ double part[SPK_REC_WARPS][SPK_BW];
  __shared__ double ucur[SPK_BW];
  const int p = blockIdx.x >> 1, c = blockIdx.x & 1;
  const int r = threadIdx.x & 31, wq = threadIdx.x >> 5;
  const int kuu = s.kuu;
  auto at = [&](int k) { return (((size_t)p * s.nblk + k) * 2 + c) * SPK_BW; };
  if (s.nblk < 2) return;
  if (wq == 0) {
    const double u = r < kuu ? s.o0[at(s.nblk - 1) + r] : 0.0;
    const double g = (r < kuu && s.nblk > 2) ? spike_guess(s, at(s.nblk - 2) + r) : 0.0;
    ucur[r] = u - g;                                 // u_k - g_k for the next step
    if (r < kuu) s.uin[at(s.nblk - 2) + r] = u;
  }
  double en[SPK_REC_COLS];
  auto load = [&](int k) {
    const double* Ek = E + ((size_t)p * s.nblk + k) * kuu * SPK_BW + (size_t)(r < kuu ? r : 0) * SPK_BW;
#pragma unroll
    for (int tt = 0; tt < SPK_REC_COLS; ++tt) {
      const int t = wq * SPK_REC_COLS + tt;
      en[tt] = (r < kuu && t < kuu) ? Ek[t] : 0.0;
    }
  };
  if (s.nblk > 2) load(s.nblk - 2);
  __syncthreads();
  for (int k = s.nblk - 2; k >= 1; --k) {
    double ec[SPK_REC_COLS];
#pragma unroll
    for (int tt = 0; tt < SPK_REC_COLS; ++tt) ec[tt] = en[tt];
    const double o = (wq == 0 && r < kuu) ? s.o0[at(k) + r] : 0.0;
    if (k > 1) load(k - 1);
    double acc = 0.0;
#pragma unroll
    for (int tt = 0; tt < SPK_REC_COLS; ++tt) acc = fma(ec[tt], ucur[wq * SPK_REC_COLS + tt], acc);
    part[wq][r] = acc;
    __syncthreads();
    if (wq == 0) {
      double u = o;
#pragma unroll
      for (int q = 0; q < SPK_REC_WARPS; ++q) u += part[q][r];
      const double g = (r < kuu && k > 1) ? spike_guess(s, at(k - 1) + r) : 0.0;
      ucur[r] = r < kuu ? u - g : 0.0;
      if (r < kuu) s.uin[at(k - 1) + r] = u;
    }
    __syncthreads();
  }
}

// the same for kuu <= W (8 or 16), W lanes per (pencil, part): four or two
// chains share each FMA and nothing waits at a barrier (the four-warp form
// issues its 32 columns' FMAs whatever kuu: Fisher-KPP 2048 x 1024, kuu = 8,
// 75 us against 21 us).
template <int W>
__global__ void __launch_bounds__(128) k_spike_bwd_rec_narrow(LaneArgs s, const double* __restrict__ E) {
  const int chain = (blockIdx.x * blockDim.x + threadIdx.x) / W;
  const bool act = chain < s.P * 2;
  const int p = act ? chain >> 1 : 0, c = chain & 1;
  const int r = threadIdx.x & (W - 1), kuu = s.kuu;
  const bool in = act && r < kuu;
  auto at = [&](int k) { return (((size_t)p * s.nblk + k) * 2 + c) * SPK_BW + r; };
  if (s.nblk < 2) return;
  double en[W], on = 0.0, gn = 0.0;
  auto load = [&](int k) {
    const double* Ek = E + (((size_t)p * s.nblk + k) * kuu + (in ? r : 0)) * SPK_BW;
#pragma unroll
    for (int t = 0; t < W; ++t) en[t] = (in && t < kuu) ? Ek[t] : 0.0;
    on = in ? s.o0[at(k)] : 0.0;
    gn = (in && k > 1) ? spike_guess(s, at(k - 1)) : 0.0;
  };
  double d;                           // u_k - g_k
  {
    const double u = in ? s.o0[at(s.nblk - 1)] : 0.0;
    const double g = (in && s.nblk > 2) ? spike_guess(s, at(s.nblk - 2)) : 0.0;
    d = u - g;
    if (in) s.uin[at(s.nblk - 2)] = u;
  }
  if (s.nblk > 2) load(s.nblk - 2);
  for (int k = s.nblk - 2; k >= 1; --k) {
    double ec[W];
#pragma unroll
    for (int t = 0; t < W; ++t) ec[t] = en[t];
    const double o = on, g = gn;
    if (k > 1) load(k - 1);
    double acc = 0.0, acc2 = 0.0;     // two independent FMA chains per step
#pragma unroll
    for (int t = 0; t < W; t += 2) acc = fma(ec[t], __shfl_sync(0xffffffffu, d, t, W), acc);
#pragma unroll
    for (int t = 1; t < W; t += 2) acc2 = fma(ec[t], __shfl_sync(0xffffffffu, d, t, W), acc2);
    const double u = o + (acc + acc2);
    if (in) s.uin[at(k - 1)] = u;
    d = u - g;
  }
}

// ---------------------------------------------------------------------------
// forward substitution of one block per 8-lane segment, four segments
// (chains: pencil, block, real or imaginary part) per warp.  Lane q of a
// segment holds row j + ((q - j) & 7) at step j.  PASS 1: zero inflow
// (the first block: its true rows 0..7), writes the outflow; PASS 2: the
// true inflow, writes y.
// ---------------------------------------------------------------------------
template <int PASS>
__global__ void __launch_bounds__(128) k_spike_fwd(LaneArgs s) {
  const int gl = blockIdx.x * blockDim.x + threadIdx.x;
  const int q = threadIdx.x & 7;
  const int nk = PASS == 1 ? s.nblk_f - 1 : s.nblk_f;   // PASS 1 skips the last block (no next block)
  const int ch = gl >> 3;
  const bool act = ch < s.P * nk * 2;
  const int chv = act ? ch : 0;
  const int c = chv & 1, k = (chv >> 1) % nk, p = (chv >> 1) / nk;
  const int j0 = k * s.m_f, j1 = j0 + s.m_f, n = s.n;
  const double* Bp = reinterpret_cast<const double*>(s.bg + (size_t)p * n) + c;   // row r at Bp[2 r]
  auto fresh = [&](int r) -> double { return (act && r < n) ? Bp[2 * r] : 0.0; };
  const size_t sidx = (((size_t)p * s.nblk_f + k) * 2 + c) * SPK_FW;
  double v;
  if (PASS == 1)
    v = (k == 0 || q == SPK_FS) ? fresh(j0 + q) : 0.0;
  else
    v = (q < SPK_FS) ? (act ? s.sst[sidx + q] : 0.0) : fresh(j0 + q);
  const double* Lp = s.L + (size_t)p * s.npad * s.lpad;
  const uint8_t* pv = s.piv + (size_t)p * s.npad;
  double* Yp = s.yg + (size_t)p * n * 2 + c;
  const int kl = s.kl, lpad = s.lpad;
  // each 8-row chunk's pivots, multipliers and fresh right-hand side are
  // loaded one chunk ahead (warps issue in order: a load consumed in the
  // same chunk would stall the chain)
  unsigned long long pw;
  double lv[SPK_FW], nv;
  auto load = [&](int j8, unsigned long long& pw_, double* lv_, double& nv_) {
    const bool in = act && j8 < j1;
    pw_ = in ? *reinterpret_cast<const unsigned long long*>(pv + j8) : 0ull;
#pragma unroll
    for (int i = 0; i < SPK_FW; ++i) {
      const int d = (q - i) & 7;
      lv_[i] = (in && d >= 1 && d <= kl) ? Lp[(size_t)(j8 + i) * lpad + d - 1] : 0.0;
    }
    nv_ = in ? fresh(j8 + SPK_FW + q) : 0.0;
  };
  load(j0, pw, lv, nv);
  for (int j8 = j0; j8 < j1; j8 += SPK_FW) {
    unsigned long long pw2;
    double lv2[SPK_FW], nv2;
    load(j8 + SPK_FW, pw2, lv2, nv2);
#pragma unroll
    for (int i = 0; i < SPK_FW; ++i) {
      const int off = (int)((pw >> (8 * i)) & 0xff);
      const int pl = (i + off) & 7;
      const double bj = __shfl_sync(0xffffffffu, v, pl, 8);   // pivot row value = y_j
      const double vo = __shfl_sync(0xffffffffu, v, i, 8);    // old row j value moves to the pivot row
      v = (q == pl) ? vo : v;
      v = fma(-lv[i], bj, v);
      if (PASS == 2 && act && q == i && j8 + i < n) Yp[2 * (j8 + i)] = bj;
      v = (q == i) ? nv : v;                                   // row j + 8 enters in row j's slot
    }
    pw = pw2;
    nv = nv2;
#pragma unroll
    for (int i = 0; i < SPK_FW; ++i) lv[i] = lv2[i];
  }
  // lane q now holds row j1 + q: the outflow is rows j1 .. j1 + 6
  if (PASS == 1 && act && q < SPK_FS) s.s0[(((size_t)p * s.nblk_f + k + 1) * 2 + c) * SPK_FW + q] = v;
}

// ---------------------------------------------------------------------------
// back substitution of one block, one CTA of two warps (real and imaginary
// part) per block, with the scaled U columns (U_{j-t,j} / U_jj) streamed chunk by
// chunk into a shared-memory ring.  Lane l holds the row congruent to l mod 32
// of rows j - 31 .. j.  PASS 1 (blocks 1 .. nblk - 1, or the one block): the
// guessed inflow, zero for the last block, writes the outflow (and b for the
// last block, which has no inflow); PASS 2 (blocks 0 .. nblk - 2): the true
// inflow, writes b = U_jj x for the block's rows.
// ---------------------------------------------------------------------------
constexpr int SPK_RING = 2;           // U chunks in flight per block (16 KB: about 11 blocks per SM)
template <int PASS>
__global__ void __launch_bounds__(64, 10) k_spike_bwd(LaneArgs s) {
  __shared__ __align__(128) double Uring[SPK_RING * SPK_CHUNK * SPK_BW];
  __shared__ __align__(8) uint64_t bar[SPK_RING];
  __shared__ int abort_flag;
  // PASS 1 skips block 0 (its outflow has no use); PASS 2 the last block,
  // final after PASS 1
  const int k0 = (PASS == 1 && s.nblk > 1) ? 1 : 0;
  const int nk = s.nblk > 1 ? s.nblk - 1 : 1;
  const int p = blockIdx.x / nk, k = k0 + (blockIdx.x - p * nk);
  const int lane = threadIdx.x & 31, c = threadIdx.x >> 5;
  const int m = s.m, j0 = k * m, j1 = j0 + m, n = s.n, kuu = s.kuu;
  const int nch = m / SPK_CHUNK, chi = j1 / SPK_CHUNK - 1;     // chunks chi, chi - 1, ..., chi - nch + 1
  const double* Usrc = s.U + (size_t)p * s.npad * s.upad;
  const uint32_t ubytes = SPK_CHUNK * SPK_BW * 8;
  auto issue = [&](int q) {                       // q-th chunk of the block in backward order
    const int sl = q % SPK_RING;
    mbar_expect_tx(&bar[sl], ubytes);
    bulk_g2s(Uring + (size_t)sl * SPK_CHUNK * SPK_BW, Usrc + (size_t)(chi - q) * SPK_CHUNK * s.upad, ubytes,
             &bar[sl]);
  };
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int sl = 0; sl < SPK_RING; ++sl) mbar_init(&bar[sl], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int q = 0; q < min(nch, SPK_RING); ++q) issue(q);
  }
  __syncthreads();
  const double* Yp = s.yg + (size_t)p * n * 2 + c;
  auto yv = [&](int r) -> double { return (r >= j0 && r < n) ? Yp[2 * r] : 0.0; };
  double w = yv(j1 - SPK_BW + lane);
  const int first_in = SPK_BW - kuu;              // lanes first_in .. 31 hold the inflow rows
  const size_t bidx = (((size_t)p * s.nblk + k) * 2 + c) * SPK_BW;
  if (lane >= first_in) {
    if (PASS == 2) w += s.uin[bidx + lane - first_in];
    else if (k < s.nblk - 1) w += spike_guess(s, bidx + lane - first_in);
  }
  // lane l takes row jc - 32 + l when it owns column jc + l of the chunk
  // at jc: nw holds that row, loaded one chunk ahead
  double nw = yv(j1 - 2 * SPK_BW + lane);
  double ws = w;   // shuffle source: w before the owner swaps in its next row (the
                   // next column's owner is another lane, so the swap stays off the chain)
  const bool store = PASS == 2 || k == s.nblk - 1;
  double* Xp = reinterpret_cast<double*>(s.xg + (size_t)p * n) + c;
  int done = 0;
  bool ok = true;
  for (int q = 0; q < nch; ++q) {
    const int sl = q % SPK_RING;
    const bool got = bounded_wait(&bar[sl], (q / SPK_RING) & 1);
    if (!got) atomicOr(&abort_flag, 1);
    __syncthreads();
    if (abort_flag) { ok = false; break; }
    done = q + 1;
    if (threadIdx.x == 0 && q >= 1 && q - 1 + SPK_RING < nch) {
      fence_proxy_async();
      issue(q - 1 + SPK_RING);                    // both warps are past chunk q - 1
    }
    const double* Uc = Uring + (size_t)sl * SPK_CHUNK * SPK_BW;
    const int jc = (chi - q) * SPK_CHUNK;
    const double nxt = yv(jc - 2 * SPK_BW + lane);   // this lane's row of the next chunk
    double xo = 0.0;
#pragma unroll
    for (int jj = SPK_CHUNK - 1; jj >= 0; --jj) {
      const double bj = __shfl_sync(0xffffffffu, ws, jj);
      const int t = (jj - lane) & 31;
      const double u = (t >= 1) ? Uc[jj * SPK_BW + t] : 0.0;
      w = fma(-u, bj, w);
      ws = w;
      const bool own = lane == jj;
      xo = own ? bj : xo;
      w = own ? nw : w;
    }
    nw = nxt;
    if (store && jc + lane < n) Xp[2 * (jc + lane)] = xo;
  }
  if (!ok) {
    if (threadIdx.x == 0) {
      raise_status(s.status, SP_ERR_TIMEOUT, p);
      const int issued = min(nch, done == 0 ? SPK_RING : done - 1 + SPK_RING);
      for (int q = done; q < issued; ++q) bounded_wait(&bar[q % SPK_RING], (q / SPK_RING) & 1);
    }
    return;
  }
  // lane l holds row j0 - 32 + l: the outflow is rows j0 - kuu .. j0 - 1
  if (PASS == 1 && k > 0 && lane >= first_in) s.o0[bidx + lane - first_in] = w;
}

cudaError_t launch_spike_forward(cudaStream_t st, const LaneArgs& s, int pass) {
  if (!spike_supported(s.kl, s.kuu, s.npad, s.nblk) || s.nblk_f < 1 || s.m_f * s.nblk_f != s.npad || s.m_f % SPK_FW)
    return cudaErrorInvalidValue;
  const int T = 128;
  const long long lanes = (long long)s.P * (pass == 1 ? s.nblk_f - 1 : s.nblk_f) * 2 * SPK_FW;
  if (lanes == 0) return cudaSuccess;
  if (pass == 1) k_spike_fwd<1><<<(unsigned)((lanes + T - 1) / T), T, 0, st>>>(s);
  else k_spike_fwd<2><<<(unsigned)((lanes + T - 1) / T), T, 0, st>>>(s);
  return cudaGetLastError();
}

cudaError_t launch_spike_backward(cudaStream_t st, const LaneArgs& s, int pass) {
  if (!spike_bwd_supported(s.kuu, s.npad, s.nblk) || s.m * s.nblk != s.npad || s.upad != SPK_BW)
    return cudaErrorInvalidValue;
  const unsigned grid = s.P * (s.nblk > 1 ? s.nblk - 1 : 1);
  if (pass == 1) k_spike_bwd<1><<<grid, 64, 0, st>>>(s);
  else if (s.nblk > 1) k_spike_bwd<2><<<grid, 64, 0, st>>>(s);
  return cudaGetLastError();
}

bool spike_supported(int kl, int kuu, int npad, int nblk) {
  return kl <= SPK_FS && spike_bwd_supported(kuu, npad, nblk);
}

// (kl' of the adjoint's transposed factor may be wider)
bool spike_bwd_supported(int kuu, int npad, int nblk) {
  return kuu < SPK_BW && nblk >= 1 && npad % (nblk * SPK_CHUNK) == 0;
}

// the recurrences alone, between the passes of the lane substitution
cudaError_t launch_spike_forward_rec(cudaStream_t st, const LaneArgs& s, const double* D) {
  const int T = 128;
  k_spike_fwd_rec<<<(unsigned)(((size_t)s.P * 2 * 8 + T - 1) / T), T, 0, st>>>(s, D);
  return cudaGetLastError();
}

cudaError_t launch_spike_backward_rec(cudaStream_t st, const LaneArgs& s, const double* E) {
  if (s.nblk < 2) return cudaSuccess;
  const int T = 128;
  if (s.kuu <= 8)
    k_spike_bwd_rec_narrow<8><<<(unsigned)(((size_t)s.P * 2 * 8 + T - 1) / T), T, 0, st>>>(s, E);
  else if (s.kuu <= 16)
    k_spike_bwd_rec_narrow<16><<<(unsigned)(((size_t)s.P * 2 * 16 + T - 1) / T), T, 0, st>>>(s, E);
  else
    k_spike_bwd_rec<<<s.P * 2, SPK_REC_WARPS * 32, 0, st>>>(s, E);
  return cudaGetLastError();
}

}  // namespace spectau
