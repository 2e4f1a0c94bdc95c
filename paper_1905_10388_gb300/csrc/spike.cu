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
// factorization time: the coupling matrices, one thread per (pencil, block,
// unit inflow).  D_k[r][i]: forward window row r after block k for window
// row i = 1 before it (no fresh right-hand side); E_k[r][t]: backward
// outflow r (row j0 - kuu + r) for unit inflow t (row j1 - kuu + t), or, for
// the lane substitution (by_row), b of row j0 + r for unit b of row j1 + t.
// The arithmetic is the substitution's own, written per row.
// ---------------------------------------------------------------------------
template <int FW>
__global__ void k_spike_coupling(int P, int npad, int nblk_f, int nblk, int kl, int kuu, int lpad, int upad,
                                 const double* __restrict__ L, const uint8_t* __restrict__ piv,
                                 const double* __restrict__ U, double* __restrict__ D, double* __restrict__ E,
                                 bool by_row) {
  constexpr int FS = FW - 1;
  const long long nf = (long long)P * nblk_f * FS;
  const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (idx >= nf + (long long)P * nblk * kuu) return;
  if (idx < nf) {
    const int i = (int)(idx % FS);
    const int k = (int)((idx / FS) % nblk_f);
    const int p = (int)(idx / ((long long)FS * nblk_f));
    const int m = npad / nblk_f, j0 = k * m, j1 = j0 + m;
    double win[FW];
    for (int t = 0; t < FW; ++t) win[t] = (t == i) ? 1.0 : 0.0;
    const double* Lp = L + (size_t)p * npad * lpad;
    const uint8_t* pv = piv + (size_t)p * npad;
    for (int j = j0; j < j1; ++j) {
      const int off = pv[j];
      const double y = win[off];        // the pivot row's value is y_j
      win[off] = win[0];                // row j's value moves to the pivot row
      for (int d = 1; d <= kl; ++d) win[d] = fma(-Lp[(size_t)j * lpad + d - 1], y, win[d]);
      for (int t = 0; t < FW - 1; ++t) win[t] = win[t + 1];
      win[FW - 1] = 0.0;
    }
    double* Dk = D + ((size_t)p * nblk_f + k) * FS * FW;
    for (int r = 0; r < FS; ++r) Dk[r * FW + i] = win[r];
  } else {
    const long long jdx = idx - nf;
    const int t0 = (int)(jdx % kuu);
    const int k = (int)((jdx / kuu) % nblk);
    const int p = (int)(jdx / ((long long)kuu * nblk));
    const int m = npad / nblk, j0 = k * m, j1 = j0 + m;
    double w[SPK_BW];                   // w[t]: pending row j - t
    const double* Up = U + (size_t)p * npad * upad;
    double* Ek = E + ((size_t)p * nblk + k) * kuu * SPK_BW;
    // inflow t0: partial sum of row j1 - kuu + t0, or (by_row) b of row j1 + t0
    for (int t = 0; t < SPK_BW; ++t)
      w[t] = by_row ? ((t0 + 1 + t <= kuu && j1 + t0 < npad) ? -Up[(size_t)(j1 + t0) * upad + t0 + 1 + t] : 0.0)
                    : (t == kuu - 1 - t0 ? 1.0 : 0.0);
    for (int j = j1 - 1; j >= j0; --j) {
      const double bj = w[0];
      if (by_row && j - j0 < kuu) Ek[(j - j0) * SPK_BW + t0] = bj;
      for (int t = 1; t <= kuu; ++t) w[t] = fma(-Up[(size_t)j * upad + t], bj, w[t]);
      for (int t = 0; t < SPK_BW - 1; ++t) w[t] = w[t + 1];
      w[SPK_BW - 1] = 0.0;
    }
    for (int r = 0; r < kuu && !by_row; ++r) Ek[r * SPK_BW + t0] = w[kuu - 1 - r];
  }
}

cudaError_t launch_spike_coupling(cudaStream_t s, int P, int npad, int nblk_f, int nblk, int kl, int kuu, int lpad,
                                  int upad, const BandFactor& f, bool by_row) {
  if (kl > SPK_BW - 2 || kuu >= SPK_BW || nblk < 1 || nblk_f < 1 || npad % (nblk * SPK_CHUNK) ||
      npad % (nblk_f * SPK_CHUNK))
    return cudaErrorInvalidValue;
  const bool wide = kl > SPK_FS;
  const long long total = (long long)P * (nblk_f * (wide ? SPK_BW - 1 : SPK_FS) + nblk * kuu);
  auto* k = wide ? k_spike_coupling<SPK_BW> : k_spike_coupling<SPK_FW>;
  k<<<(unsigned)((total + 127) / 128), 128, 0, s>>>(P, npad, nblk_f, nblk, kl, kuu, lpad, upad, f.L, f.piv, f.U,
                                                   f.spD, f.spE, by_row);
  return cudaGetLastError();
}

// forward inflows: s_0 = rows 0..6 of B~, s_1 from block 0 (exact), then
// s_{k+1} = s0_{k+1} + D_k s_k; one warp per (pencil, part), lanes 0..6.
// The next step's matrix row and outflow are loaded before this step's FMAs.
__global__ void __launch_bounds__(128) k_spike_fwd_rec(LaneArgs s, const double* __restrict__ D) {
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= s.P * 2) return;
  const int p = w >> 1, c = w & 1;
  const int i = lane < SPK_FS ? lane : 0;
  const double* Bp = reinterpret_cast<const double*>(s.bg + lane_index(p, i < s.n ? i : 0, s.npad)) + c;
  auto at = [&](int k) { return (((size_t)p * s.nblk_f + k) * 2 + c) * SPK_FW; };
  double st = i < s.n ? Bp[0] : 0.0;
  if (lane < SPK_FS) s.sst[at(0) + i] = st;
  if (s.nblk_f < 2) return;
  st = s.s0[at(1) + i];
  if (lane < SPK_FS) s.sst[at(1) + i] = st;
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
    for (int t = 0; t < SPK_FS; t += 2) acc = fma(dc[t], __shfl_sync(0xffffffffu, st, t), acc);
#pragma unroll
    for (int t = 1; t < SPK_FS; t += 2) acc2 = fma(dc[t], __shfl_sync(0xffffffffu, st, t), acc2);
    st = acc + acc2;
    if (lane < SPK_FS) s.sst[at(k + 1) + i] = st;
  }
}

__device__ __forceinline__ double spike_guess(double g) { return dfinite(g) ? g : 0.0; }

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
    const double g = (r < kuu && s.nblk > 2) ? spike_guess(s.uin[at(s.nblk - 2) + r]) : 0.0;
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
      const double g = (r < kuu && k > 1) ? spike_guess(s.uin[at(k - 1) + r]) : 0.0;
      ucur[r] = r < kuu ? u - g : 0.0;
      if (r < kuu) s.uin[at(k - 1) + r] = u;
    }
    __syncthreads();
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
  k_spike_fwd_rec<<<(unsigned)((s.P * 2 * 32 + T - 1) / T), T, 0, st>>>(s, D);
  return cudaGetLastError();
}

cudaError_t launch_spike_backward_rec(cudaStream_t st, const LaneArgs& s, const double* E) {
  if (s.nblk < 2) return cudaSuccess;
  k_spike_bwd_rec<<<s.P * 2, SPK_REC_WARPS * 32, 0, st>>>(s, E);
  return cudaGetLastError();
}

}  // namespace spectau
