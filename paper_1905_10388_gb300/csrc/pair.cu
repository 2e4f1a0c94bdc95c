// Whole-row-order pencil solves of one or two pencils per CTA (sm_103a), for
// problems and batches with more pencils than the GPU holds CTAs of the other
// kernels: assembly, substitution and epilogue.
//
// Sec. "Matrix solvers": each pencil's banded LU factor is reused for every
// solve while dt is fixed.  A row costs a shuffle and a dependent DFMA of one
// warp (about 130 cycles), so many chains have to be in flight, and an FP64 warp
// instruction holds its sub-partition's FP64 pipe for 64 cycles whatever its
// active mask, so chains share instructions where they can:
//   - forward substitution in windows of W = 8 (kl <= 7), 16 (kl <= 15) or 32
//     lanes, 32 / W chains of (pencil, real or imaginary part) per warp and
//     DFMA: with W = 8 one warp carries both parts of both pencils;
//   - back substitution by a warp per chain, a window of 32 RU rows (kl + ku <
//     32 RU), lane l holding the rows congruent to l mod 32.
// Multipliers, pivots and U columns go straight to registers, a chunk of rows
// ahead: shared memory holds the right-hand sides alone (16 KB for two pencils
// of 448 rows), so the 96-register threads set the occupancy: five CTAs, ten
// pencils, per SM.  With the factor streamed through shared memory (46 KB per
// pencil) an SM held four pencils.
// Each entry's arithmetic and order is that of the window kernel (band.cu):
// the same bits.
// Measured per solve against one pencil per CTA with the factor in shared
// memory: 16 problems of 224 to 1792 rows, 2464 pencils, 586 -> 495 us; 3D 32 x
// 64 x 32, 1024 pencils with kl = 9 and kl + ku = 38, 179 -> 141 us.  The FP64
// pipe is then 60 percent busy, the rest is the longest pencils' chains.  Four
// CTAs and 16 columns ahead: 519 us.  Both parts of a pencil in one warp's
// 16-lane windows, skipping the far half of a column where it is zero (a
// quarter of the FMAs): 747 us, half the chains in flight and a branch per row.
#include "internal.h"
#include "pencil.cuh"

namespace spectau {

constexpr int PAIR_THREADS = 128;

// Forward substitution of one chain per W-lane segment over rows [0, npad).
// Lane q of a segment holds row j + ((q - j) mod W) at step j; B2: the chain's
// part of its pencil's vector, row r at B2[2 r].
template <int W>
__device__ __forceinline__ void pair_forward(const SolveArgs& a, int p, bool act, double* B2) {
  constexpr int C = W < 16 ? W : 16;               // rows loaded at a time
  const int q = threadIdx.x & (W - 1);
  const double* Lp = a.Lf + (size_t)p * a.npad * a.lpad;
  const uint8_t* pv = a.piv + (size_t)p * a.npad;
  const int kl = a.kl, lpad = a.lpad, npad = a.npad;
  double v = act ? B2[2 * q] : 0.0;
  double lv[C], nv;
  uint32_t pw[C / 4];
  auto load = [&](int j, uint32_t (&pw_)[C / 4], double (&lv_)[C], double& nv_) {
    const bool in = act && j < npad;
#pragma unroll
    for (int i = 0; i < C / 4; ++i) pw_[i] = in ? *reinterpret_cast<const uint32_t*>(pv + j + 4 * i) : 0u;
#pragma unroll
    for (int i = 0; i < C; ++i) {
      const int d = (q - j - i) & (W - 1);
      lv_[i] = (in && d >= 1 && d <= kl) ? Lp[(size_t)(j + i) * lpad + d - 1] : 0.0;
    }
    // the row that enters this lane's slot when it owns a row of the chunk
    nv_ = in ? B2[2 * (j + W + ((q - j) & (W - 1)))] : 0.0;
  };
  // two chunks ahead with 8-row chunks (a chunk takes ~1000 cycles, a load from
  // HBM under load as long), one with 16-row chunks
  constexpr int AHEAD = C == 8 ? 2 : 1;
  uint32_t pn[AHEAD][C / 4];
  double ln[AHEAD][C], nn[AHEAD];
  load(0, pw, lv, nv);
#pragma unroll
  for (int h = 0; h < AHEAD - 1; ++h) load((h + 1) * C, pn[h], ln[h], nn[h]);
  for (int jc = 0; jc < npad; jc += C) {
    double yo = 0.0;
    load(jc + AHEAD * C, pn[AHEAD - 1], ln[AHEAD - 1], nn[AHEAD - 1]);
    const int base = jc & (W - 1);
    const int mine = (q - base) & (W - 1);         // the chunk's row this lane owns, if < C
#pragma unroll
    for (int i = 0; i < C; ++i) {
      const int off = (int)((pw[i >> 2] >> (8 * (i & 3))) & 0xff);
      const int pl = (base + i + off) & (W - 1);
      const double bj = __shfl_sync(0xffffffffu, v, pl, W);        // pivot row value = y_j
      const double vo = __shfl_sync(0xffffffffu, v, base + i, W);  // old row j value moves to the pivot row
      v = (q == pl) ? vo : v;
      v = fma(-lv[i], bj, v);
      yo = (mine == i) ? bj : yo;
      v = (mine == i) ? nv : v;
    }
    if (act && mine < C) B2[2 * (jc + mine)] = yo;
#pragma unroll
    for (int i = 0; i < C / 4; ++i) pw[i] = pn[0][i];
#pragma unroll
    for (int i = 0; i < C; ++i) lv[i] = ln[0][i];
    nv = nn[0];
#pragma unroll
    for (int h = 0; h < AHEAD - 1; ++h) {
#pragma unroll
      for (int i = 0; i < C / 4; ++i) pn[h][i] = pn[h + 1][i];
#pragma unroll
      for (int i = 0; i < C; ++i) ln[h][i] = ln[h + 1][i];
      nn[h] = nn[h + 1];
    }
  }
}

// Back substitution of one chain by a warp: scaled U columns (U_{j-t,j}/U_jj),
// x_j = b_j / U_jj applied once per 32 rows.
template <int RU>
__device__ __forceinline__ void pair_backward(const SolveArgs& a, int p, double* B2) {
  constexpr int C = 8 / RU, NC = 32 / C;           // rows loaded at a time, chunks per 32 rows
  constexpr int W = 32 * RU;
  const int lane = threadIdx.x & 31;
  const int npad = a.npad, kuu = a.kuu, upad = a.upad;
  const double* Up = a.Uf + (size_t)p * npad * upad;
  const double* rdp = a.rd + (size_t)p * npad;
  double u0[C][RU], u1[C][RU];
  auto load = [&](int j, double (&u)[C][RU]) {     // columns j + C - 1 .. j; an owner's entry is not used
#pragma unroll
    for (int i = 0; i < C; ++i) {
      const int col = j + C - 1 - i;
#pragma unroll
      for (int r = 0; r < RU; ++r) {
        const int t = (col - lane - 32 * r) & (W - 1);
        u[i][r] = (j >= 0 && (RU == 1 || t <= kuu)) ? Up[(size_t)col * upad + t] : 0.0;
      }
    }
  };
  load(npad - C, u0);
  load(npad - 2 * C, u1);
  const int ng = npad >> 5;                        // 32-row groups; group g sits in register g mod RU
  double w[RU];
#pragma unroll
  for (int r = 0; r < RU; ++r) {
    const int g = ng - 1 - ((ng - 1 - r) & (RU - 1));
    w[r] = g >= 0 ? B2[2 * (32 * g + lane)] : 0.0;
  }
  auto group = [&](int g, auto reg) {
    constexpr int O = decltype(reg)::value;        // the group's register
    const double rdl = rdp[32 * g + lane];
    const double nw = g >= RU ? B2[2 * (32 * (g - RU) + lane)] : 0.0;
    double xo = 0.0;
    auto chunk = [&](int h, const double (&u)[C][RU]) {
#pragma unroll
      for (int i = 0; i < C; ++i) {
        const int jj = h * C + C - 1 - i;
        const double bj = __shfl_sync(0xffffffffu, w[O], jj);
#pragma unroll
        for (int r = 0; r < RU; ++r) w[r] = fma(-u[i][r], bj, w[r]);
        const bool own = lane == jj;
        xo = own ? bj : xo;
        w[O] = own ? nw : w[O];
      }
    };
#pragma unroll
    for (int h = NC - 1; h >= 0; h -= 2) {
      chunk(h, u0);
      load(32 * g + (h - 2) * C, u0);
      chunk(h - 1, u1);
      load(32 * g + (h - 3) * C, u1);
    }
    B2[2 * (32 * g + lane)] = xo * rdl;
  };
  for (int g = ng - 1; g >= 0; --g) {
    if (RU == 1 || (g & 1) == 0) group(g, std::integral_constant<int, 0>{});
    else group(g, std::integral_constant<int, RU - 1>{});
  }
}

// np pencils p0 .. p0 + np - 1 (one or two) of a CTA
template <int RU, int W>
__device__ __forceinline__ void pencil_pair_body(const SolveArgs& a, int p0, int np, double2* B) {
  const int tid = threadIdx.x, warp = tid >> 5;
  const int stride = a.npad + 64;
  // assembly and epilogue: half of the threads each
  const int nt = np == 2 ? PAIR_THREADS / 2 : PAIR_THREADS;
  const int own = np == 2 ? tid / (PAIR_THREADS / 2) : 0, ot = tid - own * nt;
  pencil_assemble<1>(a, p0 + own, ot, nt, stride, B + (size_t)own * stride);
  double* Bd = reinterpret_cast<double*>(B);
  auto part = [&](int ch) { return Bd + (size_t)(ch >> 1) * 2 * stride + (ch & 1); };
  constexpr int PER = 32 / W;
  if (warp * PER < 2 * np) {
    const int ch = warp * PER + (tid & 31) / W;
    const bool act = ch < 2 * np;
    pair_forward<W>(a, p0 + (act ? ch >> 1 : 0), act, part(act ? ch : 0));
  }
  __syncthreads();
  if (warp < 2 * np) pair_backward<RU>(a, p0 + (warp >> 1), part(warp));
  __syncthreads();
  pencil_epilogue<1>(a, p0 + own, ot, nt, false, [](int r) { return (size_t)r; }, B + (size_t)own * stride);
}

template <int RU, int W>
__global__ void __launch_bounds__(PAIR_THREADS, 5) k_pencil_pair(SolveArgs a, int per) {
  extern __shared__ __align__(16) double2 pair_sm[];
  const int p0 = blockIdx.x * per;
  pencil_pair_body<RU, W>(a, p0, min(per, a.P - p0), pair_sm);
}
// a batch of problems: work item (problem, first pencil, pencils) per CTA
template <int RU, int W>
__global__ void __launch_bounds__(PAIR_THREADS, 5) k_pencil_pair_batched(const SolveArgs* __restrict__ args,
                                                                         const int4* __restrict__ work) {
  extern __shared__ __align__(16) double2 pair_sm[];
  const int4 w = work[blockIdx.x];
  pencil_pair_body<RU, W>(args[w.x], w.y, w.z, pair_sm);
}

size_t pencil_pair_smem(int npad, int per) { return (size_t)per * (npad + 64) * sizeof(double2); }

// Two pencils per CTA once single-pencil CTAs would not all be resident (four
// per SM), as long as five such CTAs fit an SM's shared memory: longer
// pencils (more than 1344 rows) go one per CTA.
int pencil_pair_per(int npad, long long pencils) {
  return pencils > 4 * GPU_SMS && pencil_pair_smem(npad, 2) <= 44 * 1024 ? 2 : 1;
}

// f(kernel) for the instance that serves bands up to kl, kuu
template <typename F>
static cudaError_t pair_instance(int kl, int kuu, F&& f) {
  if (kl > 31 || kuu > 63) return cudaErrorInvalidValue;
  const std::integral_constant<int, 8> w8;
  const std::integral_constant<int, 16> w16;
  const std::integral_constant<int, 32> w32;
  const std::integral_constant<int, 1> r1;
  const std::integral_constant<int, 2> r2;
  if (kuu <= 31) return kl <= 7 ? f(r1, w8) : kl <= 15 ? f(r1, w16) : f(r1, w32);
  return kl <= 7 ? f(r2, w8) : kl <= 15 ? f(r2, w16) : f(r2, w32);
}

cudaError_t launch_pencil_pair(cudaStream_t s, const SolveArgs& a) {
  const int per = pencil_pair_per(a.npad, a.P);
  const size_t smem = pencil_pair_smem(a.npad, per);
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  return pair_instance(a.kl, a.kuu, [&](auto r, auto w) {
    auto* k = k_pencil_pair<decltype(r)::value, decltype(w)::value>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<(a.P + per - 1) / per, PAIR_THREADS, smem, s>>>(a, per);
    return cudaGetLastError();
  });
}

cudaError_t launch_pencil_pair_batched(cudaStream_t s, const SolveArgs* args, const int4* work, int nwork, int max_kl,
                                       int max_kuu, size_t smem) {
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  return pair_instance(max_kl, max_kuu, [&](auto r, auto w) {
    auto* k = k_pencil_pair_batched<decltype(r)::value, decltype(w)::value>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<nwork, PAIR_THREADS, smem, s>>>(args, work);
    return cudaGetLastError();
  });
}

}  // namespace spectau
