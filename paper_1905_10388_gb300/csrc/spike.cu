// Coupling matrices of the partitioned substitutions (split.cu, lanes.cu) and
// the lane form's recurrences over row blocks (sm_103a).
#include <algorithm>

#include "internal.h"

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
  if (kl > SPK_BW - 2 || kuu >= SPK_BW || nblk < 1 || nblk_f < 1 || npad % (nblk * SPK_CHUNK) ||
      npad % (nblk_f * SPK_CHUNK))
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
  const double* Bp = reinterpret_cast<const double*>(s.bg + lane_index(p, i < s.n ? i : 0, s.npad)) + c;
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
