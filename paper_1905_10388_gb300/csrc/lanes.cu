// Lane-per-right-hand-side banded substitution on listed factor entries
// (FP64, sm_103a).
//
// Sec. "Matrix solvers": each pencil's banded LU factor is reused for every
// solve while dt is fixed.  On GB300 the FP64 pipe bounds these solves: a
// warp FP64 instruction holds its sub-partition's pipe for 64 cycles whatever
// its active mask, so the substitution is laid out to issue as few of them as
// possible.  A warp takes a group of 16 pencils, one lane per pencil and
// real / imaginary part, so every lane of every FMA works on a right-hand
// side of its own; and only the factor entries that are nonzero in some
// pencil of the group are stored and multiplied (2D Rayleigh-Benard: 5.2 of 7
// multipliers and 7.5 of 29 superdiagonals per row; 3D: 6.3 of 9 and 7 of
// 38), about 0.4 FP64 instructions per row and right-hand side against 1 to 2
// with a band row across a warp's lanes.
//
// Both directions work on rings in shared memory, so any band width runs
// the same code and the row loop shifts no registers:
//   forward: the window of pending rows j .. j + kl; y_j leaves it through
//     the row interchange and the listed multipliers update it;
//   backward: the row's own sum, b_j = y_j - sum_t U'_{j,j+t} b_{j+t} over the
//     listed entries in order of falling t (the column-oriented
//     substitution's order of every FMA, with b_{j+1}, the newest value, last
//     on the chain), U' the columns scaled by their pivots; the epilogue
//     kernel forms x_j = b_j / U_jj.
// A lone warp issues in order, about one instruction every five cycles, so
// what counts besides the FMAs (64 cycles apart, 80 when dependent) is the
// number of instructions between them: entries come in pairs, a record of 2 x
// 16 values and the two ring offsets (one 16-byte and one 8-byte load, each
// ahead of its use); a row's odd entry is padded with a zero against a
// scratch row; no branch depends on more than the record's last-of-row flag
// (a jump table per entry or row costs more than its FMAs); and records,
// pivots and right-hand-side rows of four-row chunks arrive by bulk copies
// (cp.async.bulk, three chunks in flight, bounded waits), the forward rows
// straight into their window slots.  Right-hand sides are stored by group,
// [G][npad][16 pencils][2]: a row of a group is one 256-byte line.
//
// Measured: 8192 pencils of 576 rows (3D Rayleigh-Benard 128 x 128 x 64, one
// warp on most sub-partitions) 1507 us per solve with the band's U entries
// picked by a jump table and the rows shifted through registers, 534 us here
// (260 forward, 274 backward: 930 to 990 cycles a row); Fisher-KPP 2048 x 1024
// 778 us for the whole window-kernel solve, 410 us here.
#include <algorithm>
#include <vector>

#include "internal.h"
#include "tma.cuh"

namespace spectau {

constexpr int LN_ROWS = 4;                       // rows per staged chunk
constexpr int LN_BUFS = 3;                       // chunks in flight
constexpr int LN_REC = 2 * LANE_GROUP + 2;       // doubles of a record: [16 pencils][2 entries], offsets, pad
constexpr int LN_RECB = LN_REC * 8;

// doubles of shared memory per warp: value ring (rows + the scratch row),
// records and pivots (forward) or y rows (backward) of LN_BUFS chunks, two
// records read ahead of the last chunk's end, barriers
__host__ __device__ inline int lane_fwd_doubles(int wr, int recs) {
  return (wr + 1) * 32 + LN_BUFS * (recs * LN_REC + LN_ROWS * 4) + 2 * LN_REC + 4;
}
__host__ __device__ inline int lane_bwd_doubles(int xr, int recs) {
  return (xr + 1) * 32 + LN_BUFS * (recs * LN_REC + LN_ROWS * 32) + 2 * LN_REC + 4;
}

__device__ __forceinline__ double* ln_at(double* base, int off) {
  return reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(base) + off);
}
__device__ __forceinline__ int2 ln_off(const unsigned char* rec) { return *reinterpret_cast<const int2*>(rec + 256); }
__device__ __forceinline__ double2 ln_val(const unsigned char* rec, int i) {
  return *reinterpret_cast<const double2*>(rec + i * 16);
}
__device__ __forceinline__ void ln_bars(uint64_t* bar, int lane) {
  if (lane == 0) {
    for (int s = 0; s <= LN_BUFS; ++s) mbar_init(bar + s, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
}
// A copy that did not land: latch the error, let the others land.  `from` ..
// `to` the chunks still in flight.
__device__ __forceinline__ void ln_lost(uint64_t* bar, int from, int to, int p, DevStatus* st, int lane) {
  if (lane == 0) {
    raise_status(st, SP_ERR_TIMEOUT, p);
    for (int c = from; c < to; ++c) bounded_wait(bar + c % LN_BUFS, (c / LN_BUFS) & 1);
  }
}

// ---------------------------------------------------------------------------
// forward substitution of block k of group g.  PASS 0: whole pencils; PASS 1:
// from zero inflow (block 0: its true rows), writes the outflow, the pending
// rows j1 .. j1 + 6; PASS 2: from the true inflow, writes y.
// ---------------------------------------------------------------------------
template <int WR, int PASS>
__device__ __forceinline__ void lane_fwd_body(const LaneArgs& a, int g, int blk, double* sm) {
  const int lane = threadIdx.x & 31, i = lane >> 1, comp = lane & 1;
  const int p0 = g * LANE_GROUP;
  const bool act = p0 + i < a.P;
  const int j0 = blk * a.m_f, j1 = j0 + a.m_f;
  double* W = sm;                                // [WR + 1][32] pending rows, scratch row
  unsigned char* S = reinterpret_cast<unsigned char*>(W + (WR + 1) * 32);   // [3][lrecs] records
  unsigned char* V = S + (LN_BUFS * a.lrecs + 2) * LN_RECB;                 // [3][4][16] pivot rows' ring offsets
  uint64_t* bar = reinterpret_cast<uint64_t*>(V + LN_BUFS * LN_ROWS * 32);
  const double* Lv = a.Lv + (size_t)g * a.lcap * LN_REC;
  const double* bg = reinterpret_cast<const double*>(a.bg) + (size_t)g * a.npad * 32;
  const int total = a.npad / LN_ROWS;
  const int32_t* co = a.lco + (size_t)g * (total + 1);
  const uint16_t* pg = a.pg + (size_t)g * a.npad * LANE_GROUP;
  const int c0 = j0 / LN_ROWS, nch = (j1 - j0) / LN_ROWS;
  // chunks of rows that enter the window before their own chunk
  // (partitioned: the outflow's 7 rows at least)
  const int ahead = max((a.kl + LN_ROWS - 1) / LN_ROWS, PASS == 0 ? 1 : 2);
  auto rows = [&](int c, int count, uint64_t* b) {    // rows 4c .. into their window slots; bytes copied
    count = min(count, total - c);
    if (count > 0)
      bulk_g2s(W + ((c * LN_ROWS) & (WR - 1)) * 32, bg + (size_t)c * LN_ROWS * 32, count * LN_ROWS * 256, b);
  };
  int cb = 0, coff = co[min(c0 + lane, total)];  // lane l: first record of chunk c0 + cb + l
  // records and pivots of chunk c0 + c, rows of chunk c0 + c + ahead (by lane
  // 0; every lane takes part in finding the records)
  auto issue = [&](int c) {
    if (c - cb >= 31) {
      cb = c;
      coff = co[min(c0 + cb + lane, total)];
    }
    const int k0 = __shfl_sync(0xffffffffu, coff, c - cb), k1 = __shfl_sync(0xffffffffu, coff, c + 1 - cb);
    if (lane != 0) return;
    uint64_t* b = bar + c % LN_BUFS;
    const uint32_t rb = (k1 - k0) * LN_RECB;
    mbar_expect_tx(b, rb + LN_ROWS * 32 + (c0 + c + ahead < total ? LN_ROWS * 256 : 0));
    bulk_g2s(S + c % LN_BUFS * a.lrecs * LN_RECB, Lv + (size_t)k0 * LN_REC, rb, b);
    bulk_g2s(V + c % LN_BUFS * LN_ROWS * 32, pg + (size_t)(c0 + c) * LN_ROWS * LANE_GROUP, LN_ROWS * 32, b);
    rows(c0 + c + ahead, 1, b);
  };
  W[WR * 32 + lane] = 0.0;
  ln_bars(bar, lane);
  if (lane == 0) {
    mbar_expect_tx(bar + LN_BUFS, min(ahead, total - c0) * LN_ROWS * 256);
    rows(c0, ahead, bar + LN_BUFS);
  }
  for (int c = 0; c < min(LN_BUFS, nch); ++c) issue(c);
  bool ok = bounded_wait(bar + LN_BUFS, 0);
  const size_t sidx = (((size_t)(p0 + (act ? i : 0)) * a.nblk_f + blk) * 2 + comp) * 8;
  if (PASS != 0 && blk > 0 && ok) {              // the inflow stands in rows j0 .. j0 + 6
#pragma unroll
    for (int r = 0; r < 7; ++r)
      W[((j0 + r) & (WR - 1)) * 32 + lane] = (PASS == 2 && act) ? a.sst[sidx + r] : 0.0;
  }
  double* yp = a.yg + ((size_t)g * a.npad + j0) * 32 + lane;
  double* Wl = W + lane;
  int done = 0;
  for (int c = 0, s = 0, ph = 0; c < nch; ++c) {
    ok = ok && bounded_wait(bar + s, ph);
    if (__any_sync(0xffffffffu, !ok)) { ok = false; break; }
    done = c + 1;
    const unsigned char* rec = S + s * a.lrecs * LN_RECB;
    const uint16_t* pv = reinterpret_cast<const uint16_t*>(V + s * LN_ROWS * 32) + i;
    double* wc = Wl + (((c0 + c) * LN_ROWS) & (WR - 1)) * 32;
    int2 o = ln_off(rec), on = ln_off(rec + LN_RECB);
    double2 l = ln_val(rec, i);
#pragma unroll
    for (int r = 0; r < LN_ROWS; ++r) {
      double* wp = ln_at(Wl, pv[r * LANE_GROUP]);
      const double y = *wp, x0 = wc[r * 32];
      *wp = x0;                                  // row j's value moves to the pivot row's place
      if (PASS != 1) yp[r * 32] = y;
      double v0 = *ln_at(Wl, o.x), v1 = *ln_at(Wl, o.y & ~1), r0 = 0.0, r1 = 0.0;
      int px = WR * 256, py = WR * 256;
      while (true) {
        // the next pair's operands before this one's FMAs, the results of the
        // pair before after them: no load or store waits for an FMA in flight
        const int last = o.y & 1;
        double n0 = 0.0, n1 = 0.0;
        rec += LN_RECB;
        if (!last) {
          n0 = *ln_at(Wl, on.x);
          n1 = *ln_at(Wl, on.y & ~1);
        }
        const double2 ln = ln_val(rec, i);
        const int2 o2 = ln_off(rec + LN_RECB);
        const double f0 = fma(-l.x, y, v0), f1 = fma(-l.y, y, v1);
        *ln_at(Wl, px) = r0;
        *ln_at(Wl, py) = r1;
        px = o.x; py = o.y & ~1; r0 = f0; r1 = f1;
        o = on; on = o2; l = ln; v0 = n0; v1 = n1;
        if (last) break;
      }
      *ln_at(Wl, px) = r0;
      *ln_at(Wl, py) = r1;
    }
    yp += LN_ROWS * 32;
    __syncwarp();                                // the chunk's buffers and rows are free
    if (c + LN_BUFS < nch) {
      if (lane == 0) fence_proxy_async();
      issue(c + LN_BUFS);
    }
    if (++s == LN_BUFS) { s = 0; ph ^= 1; }
  }
  if (!ok) {
    ln_lost(bar, done, min(nch, done + LN_BUFS), p0, a.status, lane);
    if (lane == 0) bounded_wait(bar + LN_BUFS, 0);   // the first rows' copy
    return;
  }
  if (PASS == 1 && act) {
    double* o = a.s0 + sidx + 16;                // block blk + 1's inflow before its coupling
#pragma unroll
    for (int r = 0; r < 7; ++r) o[r] = W[((j1 + r) & (WR - 1)) * 32 + lane];
  }
}

// ---------------------------------------------------------------------------
// back substitution of block k of group g.  PASS 0: whole pencils; PASS 1:
// from the guessed inflow (none for the last block, which is final), writes
// the outflow, b of the block's first kuu rows; PASS 2: from the true inflow.
// ---------------------------------------------------------------------------
template <int XR, int PASS>
__device__ __forceinline__ void lane_bwd_body(const LaneArgs& a, int g, int blk, double* sm) {
  const int lane = threadIdx.x & 31, i = lane >> 1, comp = lane & 1;
  const int p0 = g * LANE_GROUP, kuu = a.kuu;
  const bool act = p0 + i < a.P;
  const int j0 = blk * a.m, j1 = j0 + a.m;
  double* X = sm;                                // [XR + 1][32] b of the last XR rows, scratch row
  unsigned char* S = reinterpret_cast<unsigned char*>(X + (XR + 1) * 32);   // [3][urecs] records
  double* Y = reinterpret_cast<double*>(S + (LN_BUFS * a.urecs + 2) * LN_RECB);   // [3][4][32] y rows
  uint64_t* bar = reinterpret_cast<uint64_t*>(Y + LN_BUFS * LN_ROWS * 32);
  const double* Uv = a.Uv + (size_t)g * a.ucap * LN_REC;
  const double* yg = a.yg + (size_t)g * a.npad * 32;
  double* xp = reinterpret_cast<double*>(a.xg) + ((size_t)g * a.npad + j1) * 32 + lane;
  const int total = a.npad / LN_ROWS;
  const int32_t* co = a.uco + (size_t)g * (total + 1);
  const int q0 = total - j1 / LN_ROWS, nch = (j1 - j0) / LN_ROWS;     // chunks q0 .. in falling row order
  int cb = 0, coff = co[min(q0 + lane, total)];  // lane l: first record of chunk q0 + cb + l
  auto issue = [&](int c) {
    if (c - cb >= 31) {
      cb = c;
      coff = co[min(q0 + cb + lane, total)];
    }
    const int k0 = __shfl_sync(0xffffffffu, coff, c - cb), k1 = __shfl_sync(0xffffffffu, coff, c + 1 - cb);
    if (lane != 0) return;
    uint64_t* b = bar + c % LN_BUFS;
    const uint32_t rb = (k1 - k0) * LN_RECB;
    mbar_expect_tx(b, rb + LN_ROWS * 256);
    bulk_g2s(S + c % LN_BUFS * a.urecs * LN_RECB, Uv + (size_t)k0 * LN_REC, rb, b);
    bulk_g2s(Y + c % LN_BUFS * LN_ROWS * 32, yg + (size_t)(j1 - (c + 1) * LN_ROWS) * 32, LN_ROWS * 256, b);
  };
  ln_bars(bar, lane);
  for (int c = 0; c < min(LN_BUFS, nch); ++c) issue(c);
  const size_t bidx = (((size_t)(p0 + (act ? i : 0)) * a.nblk + blk) * 2 + comp) * 32;
  X[XR * 32 + lane] = 0.0;
  if (PASS != 0) {
    const bool in = act && (PASS == 2 || (blk < a.nblk - 1 && !a.cold));
#pragma unroll 8
    for (int r = 0; r < XR; ++r) {
      const double v = (in && r < kuu) ? a.uin[bidx + r] : 0.0;
      X[((j1 + r) & (XR - 1)) * 32 + lane] = (PASS == 1 && !dfinite(v)) ? 0.0 : v;
    }
  }
  const bool store = PASS != 1 || blk == a.nblk - 1;
  double* Xl = X + lane;
  bool ok = true;
  int done = 0;
  for (int c = 0, s = 0, ph = 0; c < nch; ++c) {
    ok = bounded_wait(bar + s, ph);
    if (__any_sync(0xffffffffu, !ok)) { ok = false; break; }
    done = c + 1;
    const unsigned char* rec = S + s * a.urecs * LN_RECB;
    const double* y = Y + s * LN_ROWS * 32 + lane;
    double* xc = Xl + ((j1 - (c + 1) * LN_ROWS) & (XR - 1)) * 32;
    xp -= LN_ROWS * 32;
    int2 o = ln_off(rec), on = ln_off(rec + LN_RECB);
    double2 u = ln_val(rec, i);
#pragma unroll
    for (int r = LN_ROWS - 1; r >= 0; --r) {
      double acc = y[r * 32];
      double v0 = *ln_at(Xl, o.x), v1 = *ln_at(Xl, o.y & ~1);
      while (true) {
        // the next pair's operands before this one's FMAs
        const int last = o.y & 1;
        double n0 = 0.0, n1 = 0.0;
        rec += LN_RECB;
        if (!last) {
          n0 = *ln_at(Xl, on.x);
          n1 = *ln_at(Xl, on.y & ~1);
        }
        const double2 un = ln_val(rec, i);
        const int2 o2 = ln_off(rec + LN_RECB);
        acc = fma(-u.x, v0, acc);
        acc = fma(-u.y, v1, acc);
        o = on; on = o2; u = un; v0 = n0; v1 = n1;
        if (last) break;
      }
      xc[r * 32] = acc;
      if (store) xp[r * 32] = acc;
    }
    __syncwarp();                                // the chunk's buffers are free
    if (c + LN_BUFS < nch) {
      if (lane == 0) fence_proxy_async();
      issue(c + LN_BUFS);
    }
    if (++s == LN_BUFS) { s = 0; ph ^= 1; }
  }
  if (!ok) {
    ln_lost(bar, done, min(nch, done + LN_BUFS), p0, a.status, lane);
    return;
  }
  if (PASS == 1 && blk > 0 && act)
    for (int r = 0; r < kuu; ++r) a.o0[bidx + r] = X[((j0 + r) & (XR - 1)) * 32 + lane];
}

// ---------------------------------------------------------------------------
// kernels: one warp per (group, block) of one problem
// ---------------------------------------------------------------------------
template <int WR, int PASS>
__global__ void __launch_bounds__(128) k_lane_fwd(LaneArgs a, int doubles) {
  extern __shared__ __align__(16) double lane_smem[];
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nk = PASS == 0 ? 1 : (PASS == 1 ? a.nblk_f - 1 : a.nblk_f);   // PASS 1: no block follows the last
  const int g = w / nk;
  if (g * LANE_GROUP >= a.P) return;             // whole warps leave together
  lane_fwd_body<WR, PASS>(a, g, w - g * nk, lane_smem + (threadIdx.x >> 5) * doubles);
}
template <int XR, int PASS>
__global__ void __launch_bounds__(128) k_lane_bwd(LaneArgs a, int doubles) {
  extern __shared__ __align__(16) double lane_smem[];
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  // PASS 1 skips block 0 (its outflow has no use), PASS 2 the last block (final after PASS 1)
  const int nk = (PASS == 0 || a.nblk < 2) ? 1 : a.nblk - 1;
  const int g = w / nk, k0 = (PASS == 1 && a.nblk > 1) ? 1 : 0;
  if (g * LANE_GROUP >= a.P) return;
  lane_bwd_body<XR, PASS>(a, g, k0 + w - g * nk, lane_smem + (threadIdx.x >> 5) * doubles);
}

// warps per CTA: four, fewer when their rings do not fit a CTA's shared memory
template <typename K>
static cudaError_t lane_launch(K kernel, cudaStream_t s, const LaneArgs& a, int warps, int doubles) {
  int wpc = 4;
  while (wpc > 1 && (size_t)wpc * doubles * 8 > 227 * 1024) wpc >>= 1;
  const size_t smem = (size_t)wpc * doubles * 8;
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kernel<<<(warps + wpc - 1) / wpc, wpc * 32, smem, s>>>(a, doubles);
  return cudaGetLastError();
}

// window rows: a chunk, the ceil(kl / 4) (partitioned: two at least) after it
// and two in flight
static int lane_window(int kl) { return std::max(2, (kl + LN_ROWS - 1) / LN_ROWS) + 3 <= 8 ? 32 : 64; }

// back-substitution ring rows: more than kuu
static int lane_ring(int kuu) { return kuu <= 31 ? 32 : 64; }

template <int PASS>
static cudaError_t launch_fwd(cudaStream_t s, const LaneArgs& a) {
  const int G = (a.P + LANE_GROUP - 1) / LANE_GROUP;
  const int warps = G * (PASS == 0 ? 1 : (PASS == 1 ? a.nblk_f - 1 : a.nblk_f));
  const int wr = lane_window(a.kl), d = lane_fwd_doubles(wr, a.lrecs);
  if constexpr (PASS == 0)                        // (row blocks: kl <= 7, 32 rows)
    if (wr == 64) return lane_launch(k_lane_fwd<64, PASS>, s, a, warps, d);
  return lane_launch(k_lane_fwd<32, PASS>, s, a, warps, d);
}
template <int PASS>
static cudaError_t launch_bwd(cudaStream_t s, const LaneArgs& a) {
  const int G = (a.P + LANE_GROUP - 1) / LANE_GROUP;
  const int warps = G * ((PASS == 0 || a.nblk < 2) ? 1 : a.nblk - 1);
  if constexpr (PASS == 0)                        // (row blocks: kuu <= 31, 32 rows)
    if (lane_ring(a.kuu) == 64) return lane_launch(k_lane_bwd<64, PASS>, s, a, warps, lane_bwd_doubles(64, a.urecs));
  return lane_launch(k_lane_bwd<32, PASS>, s, a, warps, lane_bwd_doubles(32, a.urecs));
}

cudaError_t launch_lane_forward(cudaStream_t s, const LaneArgs& a, int pass) {
  if (pass == 0) return launch_fwd<0>(s, a);
  if (a.kl > 7 || a.m_f % 32 || a.m_f * a.nblk_f != a.npad) return cudaErrorInvalidValue;
  if (pass == 1) return a.nblk_f > 1 ? launch_fwd<1>(s, a) : cudaSuccess;
  return launch_fwd<2>(s, a);
}
cudaError_t launch_lane_backward(cudaStream_t s, const LaneArgs& a, int pass) {
  if (pass == 0) return launch_bwd<0>(s, a);
  if (a.kuu > 31 || a.m % 32 || a.m * a.nblk != a.npad) return cudaErrorInvalidValue;
  if (pass == 1) return launch_bwd<1>(s, a);
  return a.nblk > 1 ? launch_bwd<2>(s, a) : cudaSuccess;
}

// ---------------------------------------------------------------------------
// factorization time: the lists.  A multiplier L_{j+t,j} is listed with row j
// (bit t of lmask), a scaled entry U_{j,j+t} / U_{j+t,j+t} with row j (bit t
// of umask), when it is nonzero in some pencil of the group.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_lane_mask(int P, int n, int npad, int kl, int kuu, int lpad, int upad,
                                                   const double* __restrict__ L, const double* __restrict__ U,
                                                   uint32_t* __restrict__ lmask,
                                                   unsigned long long* __restrict__ umask) {
  const size_t w = (blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5;    // (group, column)
  const int lane = threadIdx.x & 31;
  const int g = (int)(w / n), j = (int)(w - (size_t)g * n);
  if (g * LANE_GROUP >= P) return;
  const int p1 = min(P, (g + 1) * LANE_GROUP);
  bool l = false, u0 = false, u1 = false;
  for (int p = g * LANE_GROUP; p < p1; ++p) {
    const size_t col = (size_t)p * npad + j;
    if (lane >= 1 && lane <= kl) l |= L[col * lpad + lane - 1] != 0.0;
    if (lane <= kuu) u0 |= U[col * upad + lane] != 0.0;
    if (lane + 32 <= kuu) u1 |= U[col * upad + lane + 32] != 0.0;
  }
  const uint32_t lb = __ballot_sync(0xffffffffu, l);
  if (lane == 0) lmask[(size_t)g * npad + j] = lb;
  unsigned long long* um = umask + (size_t)g * npad;
  if (lane >= 1 && u0 && j - lane >= 0) atomicOr(um + j - lane, 1ull << lane);
  if (u1 && j - lane - 32 >= 0) atomicOr(um + j - lane - 32, 1ull << (lane + 32));
}

// records of a row: two entries each, one at least
__device__ __forceinline__ int ln_records(unsigned long long m) { return max(1, (__popcll(m) + 1) >> 1); }

// First record of every four-row chunk (multipliers in rising, U entries in
// falling row order), the group's record counts and the most records of a
// chunk: tot[g] = {L, U, L chunk, U chunk}.
__global__ void __launch_bounds__(64) k_lane_scan(int npad, const uint32_t* __restrict__ lmask,
                                                  const unsigned long long* __restrict__ umask,
                                                  int32_t* __restrict__ lco, int32_t* __restrict__ uco,
                                                  int32_t* __restrict__ tot) {
  const int g = blockIdx.x, lane = threadIdx.x & 31, dir = threadIdx.x >> 5;   // warp 0: L, warp 1: U
  const int total = npad / LN_ROWS;
  int32_t* co = (dir ? uco : lco) + (size_t)g * (total + 1);
  int run = 0, most = 0;
  for (int c0 = 0; c0 < total; c0 += 32) {
    const int c = c0 + lane;
    int cnt = 0;
    if (c < total) {
      const size_t r0 = (size_t)g * npad + (dir ? total - 1 - c : c) * LN_ROWS;
      for (int r = 0; r < LN_ROWS; ++r) cnt += ln_records(dir ? umask[r0 + r] : (unsigned long long)lmask[r0 + r]);
    }
    int inc = cnt;
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, d);
      if (lane >= d) inc += v;
    }
    if (c < total) co[c] = run + inc - cnt;
    most = max(most, cnt);
    run += __shfl_sync(0xffffffffu, inc, 31);
  }
  for (int d = 16; d > 0; d >>= 1) most = max(most, __shfl_xor_sync(0xffffffffu, most, d));
  if (lane == 0) {
    co[total] = run;
    tot[g * 4 + dir] = run;
    tot[g * 4 + 2 + dir] = most;
  }
}

// The listed values, their ring offsets and the pivots, one half warp per
// direction of a (group, row); wr, xr the window and ring rows.
__global__ void __launch_bounds__(256) k_lane_pack(int P, int n, int npad, int lpad, int upad, int wr, int xr,
                                                   const double* __restrict__ L, const uint8_t* __restrict__ piv,
                                                   const double* __restrict__ U, LaneList f) {
  const size_t w = (blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31, i = lane & 15;
  const int g = (int)(w / npad), j = (int)(w - (size_t)g * npad);
  const int p = g * LANE_GROUP + i;
  if (g * LANE_GROUP >= P) return;
  const bool act = p < P;
  const int total = npad / LN_ROWS, c = j / LN_ROWS;
  const size_t row = (size_t)g * npad + j;
  const bool fwd = lane < 16;
  if (fwd) f.pg[row * LANE_GROUP + i] = (uint16_t)(((j + ((act && j < n) ? piv[(size_t)p * npad + j] : 0)) & (wr - 1)) * 256);
  const unsigned long long* um = f.umask + (size_t)g * npad;
  const uint32_t* lm = f.lmask + (size_t)g * npad;
  int k = (fwd ? f.lco : f.uco)[(size_t)g * (total + 1) + (fwd ? c : total - 1 - c)];
  if (fwd)
    for (int r = c * LN_ROWS; r < j; ++r) k += ln_records(lm[r]);
  else
    for (int r = (c + 1) * LN_ROWS - 1; r > j; --r) k += ln_records(um[r]);
  unsigned long long m = fwd ? (unsigned long long)lm[j] : um[j];
  const int count = __popcll(m), nr = ln_records(m);
  const int pads = 2 * nr - count, scratch = (fwd ? wr : xr) * 256;
  double* out = fwd ? f.Lv + ((size_t)g * f.lcap + k) * LN_REC : f.Uv + ((size_t)g * f.ucap + k) * LN_REC;
  for (int q = 0; q < nr; ++q, out += LN_REC) {
    double v[2];
    int o[2];
    for (int h = 0; h < 2; ++h) {
      if (2 * q + h < pads) {                    // the pads come first
        v[h] = 0.0;
        o[h] = scratch;
        continue;
      }
      const int t = fwd ? __ffsll((long long)m) - 1 : 63 - __clzll(m);
      m ^= 1ull << t;
      v[h] = !act ? 0.0 : fwd ? L[((size_t)p * npad + j) * lpad + t - 1] : U[((size_t)p * npad + j + t) * upad + t];
      o[h] = ((j + t) & ((fwd ? wr : xr) - 1)) * 256;
    }
    *reinterpret_cast<double2*>(out + i * 2) = make_double2(v[0], v[1]);
    if (i == 0) *reinterpret_cast<int2*>(out + 32) = make_int2(o[0], o[1] | (q == nr - 1 ? 1 : 0));   // bit 0: last of the row
  }
}

void lane_list_free(LaneList& f) {
  for (void* p : {(void*)f.Lv, (void*)f.Uv, (void*)f.lmask, (void*)f.umask, (void*)f.lco, (void*)f.uco, (void*)f.pg,
                  (void*)f.tot})
    if (p) cudaFree(p);
  f = LaneList{};
}

// Lists of the factor (L, piv, U) of P pencils.  Reads the entry counts back
// (synchronous).
cudaError_t lane_list_build(cudaStream_t s, int P, int n, int npad, int kl, int kuu, int lpad, int upad,
                            const double* L, const uint8_t* piv, const double* U, LaneList& f) {
  const int G = (P + LANE_GROUP - 1) / LANE_GROUP, total = npad / LN_ROWS;
  auto alloc = [](auto** p, size_t count) {
    return *p ? cudaSuccess : cudaMalloc((void**)p, count * sizeof(**p));
  };
  cudaError_t e;
  if ((e = alloc(&f.umask, (size_t)G * npad)) != cudaSuccess) return e;
  if ((e = alloc(&f.lmask, (size_t)G * npad)) != cudaSuccess) return e;
  if ((e = alloc(&f.lco, (size_t)G * (total + 1))) != cudaSuccess) return e;
  if ((e = alloc(&f.uco, (size_t)G * (total + 1))) != cudaSuccess) return e;
  if ((e = alloc(&f.pg, (size_t)G * npad * LANE_GROUP)) != cudaSuccess) return e;
  if ((e = alloc(&f.tot, (size_t)G * 4)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(f.umask, 0, (size_t)G * npad * sizeof(*f.umask), s)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(f.lmask, 0, (size_t)G * npad * sizeof(*f.lmask), s)) != cudaSuccess) return e;
  const size_t mt = (size_t)G * n * 32, pt = (size_t)G * npad * 32;
  k_lane_mask<<<(unsigned)((mt + 255) / 256), 256, 0, s>>>(P, n, npad, kl, kuu, lpad, upad, L, U, f.lmask, f.umask);
  k_lane_scan<<<G, 64, 0, s>>>(npad, f.lmask, f.umask, f.lco, f.uco, f.tot);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  std::vector<int32_t> tot((size_t)G * 4);
  e = cudaMemcpyAsync(tot.data(), f.tot, tot.size() * sizeof(int32_t), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return e;
  int lmax = 1, umax = 1, lr = 1, ur = 1;
  double ls = 0, us = 0;
  for (int g = 0; g < G; ++g) {
    lmax = std::max(lmax, tot[g * 4]); umax = std::max(umax, tot[g * 4 + 1]);
    lr = std::max(lr, tot[g * 4 + 2]); ur = std::max(ur, tot[g * 4 + 3]);
    ls += tot[g * 4]; us += tot[g * 4 + 1];
  }
  f.l_listed = 2.0 * ls / G / n;                 // pads included
  f.u_listed = 2.0 * us / G / n;
  f.lrecs = lr;
  f.urecs = ur;
  auto grow = [&](double** v, int* cap, int want) {
    if (want <= *cap) return cudaSuccess;
    if (*v) cudaFree(*v);
    *v = nullptr;
    *cap = 0;
    cudaError_t r = cudaMalloc((void**)v, (size_t)G * want * LN_REC * sizeof(double));
    if (r == cudaSuccess) *cap = want;
    return r;
  };
  if ((e = grow(&f.Lv, &f.lcap, lmax)) != cudaSuccess) return e;
  if ((e = grow(&f.Uv, &f.ucap, umax)) != cudaSuccess) return e;
  k_lane_pack<<<(unsigned)((pt + 255) / 256), 256, 0, s>>>(P, n, npad, lpad, upad, lane_window(kl), lane_ring(kuu), L, piv, U, f);
  return cudaGetLastError();
}

}  // namespace spectau
