// Spectral transforms on compile-time lengths (fftn.cuh): the right-hand
// side's x rows with the dealiased products, the y transforms and the
// Chebyshev (z) transforms.  Conventions and data layouts as in
// transforms.cu, whose run-time-length kernels serve the other transforms
// (set-up, CFL, adjoint) and lengths.
//
// Derivatives i k_x and i k_y commute with the transforms of the other axes:
// z transforms run once per variable, y transforms once per variable and once
// more where a y derivative is used, and the x rows apply i k_x as they load
// (2D Rayleigh-Benard: 6 z transforms for 8 grid fields; 3D: 8 and 12 y
// transforms for 15).
//
// FP64 is bound by its pipe: the work is counted in FP64 instructions (signs,
// halves and scales live in tables, +-1 coefficients take no multiplication, the
// padded third of a spectrum enters no butterfly).  FP32 is bound by
// instruction issue (57 % active, FMA pipe 20 %): a run-time length, a branch or
// an address per element costs more than the arithmetic.  Per launch, the
// run-time-length kernels before and these now: x rows 512 x 256 FP64 171 ->
// 125 us (three of the 384 rows on some SMs, two on most), FP32 28 -> 17; 3D 128 x
// 128 x 64 FP32 390 -> 163; Fisher-KPP 2048 x 1024 FP32 137 -> 72 (its radix-16
// passes load 15 twiddles each); y of the 3D case 139 and 40 -> 66 and 21; z 512 x
// 256 FP64 76 and 40 -> 43 and 30.
#pragma once
#include <algorithm>
#include <type_traits>

#include "fftn.cuh"
#include "internal.h"

namespace spectau {

constexpr size_t ROWS_SMEM = ROWS_SMEM_MAX;

// -x by the sign bit (off the FP64 pipe)
__device__ __forceinline__ double neg_bits(double x) { return dneg(x); }
__device__ __forceinline__ float neg_bits(float x) { return -x; }

// Factor that a forward transform's results leave with: 1 in FP64; in FP32 an
// exact 2^-rows_shift(N), else the sums over all axes would overflow where each
// product and each axis' sum still fits
template <typename T, int N>
__host__ __device__ constexpr T rows_scale() {
  return sizeof(T) == 4 ? (T)1 / (T)(1 << rows_shift(N)) : (T)1;
}

// threads of a CTA: about the butterflies of four sequences, in whole warps
template <typename T, int N>
constexpr int rows_threads() {
  if (N <= 192) return N < 64 ? 64 : N;
  if (N <= 768) return N / 2 > 256 && sizeof(T) == 4 ? N / 4 : N / 2;
  return 256;
}

// CTAs per SM the register budget is set for (registers, not shared memory,
// limit them at the common lengths)
template <typename T>
constexpr int rows_ctas(int nt) {
  return sizeof(T) == 8 ? (nt <= 96 ? 6 : nt <= 128 ? 4 : nt <= 192 ? 3 : 2) : (nt <= 64 ? 14 : nt <= 96 ? 10 : nt <= 128 ? 8 : nt <= 192 ? 5 : 3);
}

// ---------------------------------------------------------------------------
// x rows: backward transforms of all field pairs, products, forward
// transforms of the products, for row `row`; grid data stay in shared memory.
// ---------------------------------------------------------------------------
template <typename T, int N>
size_t x_rows_smem(int nf, int ne) {
  const int nbi = (nf + 1) / 2, nbo = (ne + 1) / 2;
  return (size_t)(nbi + std::max(nbi, 2 * nbo)) * fft_padded<T>(N) * sizeof(C<T>);
}

template <typename T, int N, int NT, bool PAD>
__device__ __forceinline__ void x_rows_body(const XDesc& d, int row, unsigned char* rows_smem) {
  constexpr int NP = fft_padded<T>(N), MAX_TERMS = 16, MAX_F = 16;
  const int K = d.K, rows = d.rows, nf = d.nf, ne = d.ne, tid = threadIdx.x;
  const int nbi = (nf + 1) / 2, nbo = (ne + 1) / 2;
  C<T>* u = reinterpret_cast<C<T>*>(rows_smem);
  C<T>* v = u + nbi * NP;
  T* G = reinterpret_cast<T*>(u);                // grid fields [f][N], over the first buffer
  __shared__ int fs[MAX_F], fx[MAX_F];
  __shared__ int4 term[MAX_TERMS];               // field offsets, equation offset (last of its equation: | 1), coefficient kind
  __shared__ T tc[MAX_TERMS];
  const int nterms = min(d.nterms, MAX_TERMS);
  const T* tcoef = reinterpret_cast<const T*>(sizeof(T) == 8 ? (const void*)d.t_coef : (const void*)d.t_coef32);
  const T* __restrict__ kx = reinterpret_cast<const T*>(sizeof(T) == 8 ? (const void*)d.kx : (const void*)d.kx32);
  if (tid < nterms) {
    const int e = d.t_eq[tid];
    const bool last = tid + 1 == nterms || d.t_eq[tid + 1] != e;
    const T c = tcoef[tid];
    tc[tid] = c;
    term[tid] = make_int4(d.t_fa[tid] * N, d.t_fb[tid] * N, ((e >> 1) * 4 * NP + (e & 1) * 2) | (last ? 1 : 0),
                          c == (T)1 ? 1 : c == (T)-1 ? -1 : 0);
  }
  if (tid < nf) { fs[tid] = d.f_src[tid]; fx[tid] = d.f_dx[tid]; }
  const C<T>* __restrict__ tw = reinterpret_cast<const C<T>*>(d.tw);
  __syncthreads();
  const C<T>* __restrict__ gz = reinterpret_cast<const C<T>*>(d.gz) + (size_t)row * K;
  const size_t plane = (size_t)rows * K;
  constexpr int Q0 = N / FftPlan<N>::R0;
  fft_run<T, N, +1, NT, PAD>(
      nbi, u, v, tw,
      [&](int b, int j) {
        // two real fields a, b as a + i b: the Hermitian spectrum of the stored k >= 0 modes
        const bool two = 2 * b + 1 < nf;
        const C<T>* pa = gz + fs[2 * b] * plane;
        const C<T>* pb = gz + fs[two ? 2 * b + 1 : 2 * b] * plane;
        const bool xa = fx[2 * b] != 0, xb = two && fx[2 * b + 1] != 0;
        return [=](auto t) -> C<T> {
          constexpr int i0 = decltype(t)::value * Q0;
          const bool mirror = PAD ? 3 * i0 >= 2 * N : j + i0 > N - K;
          const int k = mirror ? N - i0 - j : i0 + j;
          if ((!PAD || 3 * i0 == 2 * N) && (mirror ? k >= K : k >= K)) return mk<T>(0, 0);
          C<T> A = pa[k], B = two ? pb[k] : mk<T>(0, 0);
          if (xa || xb) {
            const T q = kx[k];
            if (xa) A = mk<T>(-q * A.y, q * A.x);
            if (xb) B = mk<T>(-q * B.y, q * B.x);
          }
          if (i0 == 0 && j == 0) A.y = B.y = 0;
          return mirror ? mk<T>(A.x + B.y, B.x - A.y) : mk<T>(A.x - B.y, A.y + B.x);
        };
      },
      [&](int b, int i, C<T> z) {
        G[2 * b * N + i] = z.x;
        if (2 * b + 1 < nf) G[(2 * b + 1) * N + i] = z.y;
      });
  // products: terms are grouped by equation; two equations share a complex
  // sequence.  Coefficients +-1 cost one FMA per term.
  T* O = reinterpret_cast<T*>(v);
  for (int i = tid; i < N; i += NT) {
    const int o = 2 * fft_pad<T>(i);
    T acc = 0;
    for (int t = 0; t < nterms; ++t) {
      const int4 m = term[t];
      T ga = G[m.x + i];
      const T gb = G[m.y + i];
      if (m.w < 0) ga = neg_bits(ga);
      else if (m.w == 0) ga *= tc[t];
      acc = fma(ga, gb, acc);
      if (m.z & 1) {
        O[(m.z >> 1) + o] = acc;
        acc = 0;
      }
    }
    if (ne & 1) O[(ne >> 1) * 2 * NP + o + 1] = 0;
  }
  __syncthreads();
  constexpr bool three = FftPlan<N>::R2 > 1;
  C<T>* u2 = v + nbo * NP;
  C<T>* Z = three ? u2 : v;
  fft_run<T, N, -1, NT, false>(
      nbo, u2, three ? v : u2, tw,
      [&](int b, int j) {
        const C<T>* x = v + b * NP;
        return [=](auto t) -> C<T> { return x[fft_pad<T>(j + decltype(t)::value * Q0)]; };
      },
      [&](int b, int i, C<T> z) { Z[b * NP + fft_pad<T>(i)] = z; });
  C<T>* h = reinterpret_cast<C<T>*>(d.h) + (size_t)row * K;
  // (1 / (2 N), in FP32 what rows_scale leaves of it, is in the z transform's table)
  constexpr T sc = rows_scale<T, 2 * N>();
  for (int b = 0; b < nbo; ++b)
    for (int k = tid; k < K; k += NT) {
      const C<T> z = Z[b * NP + fft_pad<T>(k)], r = Z[b * NP + fft_pad<T>(k == 0 ? 0 : N - k)];
      h[2 * b * plane + k] = mk<T>(sc * (z.x + r.x), sc * (z.y - r.y));
      if (2 * b + 1 < ne) h[(2 * b + 1) * plane + k] = mk<T>(sc * (z.y + r.y), sc * (r.x - z.x));
    }
}

template <typename T, int N, int NT, bool PAD>
__global__ void __launch_bounds__(NT, rows_ctas<T>(NT)) k_x_rows(XDesc d) {
  extern __shared__ __align__(16) unsigned char rows_smem[];
  x_rows_body<T, N, NT, PAD>(d, blockIdx.x, rows_smem);
}

template <typename T>
cudaError_t launch_x_rows(cudaStream_t s, const XDesc& d) {
  return fft_dispatch(d.N, [&](auto n) -> cudaError_t {
    constexpr int N = decltype(n)::value, NT = rows_threads<T, N>();
    const size_t smem = x_rows_smem<T, N>(d.nf, d.ne);
    if (smem > ROWS_SMEM || d.nf > 16 || d.nterms > 16) return cudaErrorInvalidValue;
    auto* k = k_x_rows<T, N, NT, false>;
    if constexpr (N % 3 == 0)
      if (3 * d.K == N) k = k_x_rows<T, N, NT, true>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<d.rows, NT, smem, s>>>(d);
    return cudaGetLastError();
  });
}

// ---------------------------------------------------------------------------
// Column transforms (y and z): TC columns of a plane per CTA, adjacent in
// memory on the grid side.  A butterfly's columns run fastest over the threads
// where its elements go to or come from the column-adjacent layout (64-byte
// pieces), its index where they do not.
// ---------------------------------------------------------------------------
constexpr int COL_TC32 = 8, COL_TC64 = 4;
template <typename T>
constexpr int col_tile() { return sizeof(T) == 4 ? COL_TC32 : COL_TC64; }
// sequence stride: one element more than a multiple of 16, so that adjacent
// columns sit in adjacent banks
template <typename T, int N>
constexpr int col_stride() { return (fft_padded<T>(N) + 15) / 16 * 16 + 1; }
template <typename T, int N>
constexpr size_t col_smem() { return (size_t)2 * col_tile<T>() * col_stride<T, N>() * sizeof(C<T>); }

// One transform of the tile: readers `open(c, j)` (fftn.cuh), `fin(c, i, v)`; IN_COL / OUT_COL:
// columns fastest over the threads in the first / last pass.  Two-pass lengths
// use buffer v alone.  Ends after a barrier.
template <typename T, int N, int SIGN, int NT, bool PAD, bool IN_COL, bool OUT_COL, typename OPEN, typename FIN>
__device__ __forceinline__ void col_run(C<T>* u, C<T>* v, const C<T>* tw, OPEN&& open, FIN&& fin) {
  using P = FftPlan<N>;
  constexpr int TC = col_tile<T>(), NS = col_stride<T, N>();
  C<T>* first = P::R2 > 1 ? u : v;
  {
    constexpr int R = P::R0, Q = N / R;
    for (int id = threadIdx.x; id < TC * Q; id += NT) {
      const int c = IN_COL ? id % TC : id / Q, j = IN_COL ? id / TC : id % Q;
      C<T> a[R], y[R];
      fft_read<T, R, PAD>(open(c, j), a);
      dft_first<T, SIGN, R, PAD>(a, y);
#pragma unroll
      for (int q = 0; q < R; ++q) first[c * NS + fft_pad<T>(j * R + q)] = y[q];
    }
  }
  __syncthreads();
  auto pass = [&](auto r, auto ns, const C<T>* x, auto col, auto&& out) {
    constexpr int R = decltype(r)::value, Ns = decltype(ns)::value, Q = N / R, STEP = N / (R * Ns);
    constexpr bool COL = decltype(col)::value;
    for (int id = threadIdx.x; id < TC * Q; id += NT) {
      const int c = COL ? id % TC : id / Q, j = COL ? id / TC : id % Q;
      const int k = j % Ns;
      const C<T>* xc = x + c * NS;
      C<T> a[R], y[R];
#pragma unroll
      for (int t = 0; t < R; ++t) a[t] = xc[fft_pad<T>(j + t * Q)];
      const unsigned w0 = k * STEP;
      dft_twiddled<T, SIGN, R>(a, y, [&](int t) {
        const C<T> w = fft_tw<T>(tw, t * w0);
        return SIGN > 0 ? mk<T>(w.x, -w.y) : w;
      });
      const int o = j / Ns * (R * Ns) + k;
#pragma unroll
      for (int q = 0; q < R; ++q) out(c, o + q * Ns, y[q]);
    }
    __syncthreads();
  };
  using std::integral_constant;
  if constexpr (P::R2 > 1) {
    pass(integral_constant<int, P::R1>(), integral_constant<int, P::R0>(), u, integral_constant<bool, false>(),
         [&](int c, int i, C<T> z) { v[c * NS + fft_pad<T>(i)] = z; });
    pass(integral_constant<int, P::R2>(), integral_constant<int, P::R0 * P::R1>(), v, integral_constant<bool, OUT_COL>(),
         fin);
  } else {
    pass(integral_constant<int, P::R1>(), integral_constant<int, P::R0>(), v, integral_constant<bool, OUT_COL>(), fin);
  }
}

// y axis (complex): DIR < 0: slots -> grid of output field f, with i k_y where
// f_dy is set; DIR > 0: grid -> slots (unscaled, Nyquist slot zero)
template <typename T, int N, int NT, int DIR, bool PAD>
__global__ void __launch_bounds__(NT, rows_ctas<T>(NT)) k_y_cols(YDesc d) {
  extern __shared__ __align__(16) unsigned char rows_smem[];
  constexpr int TC = col_tile<T>(), Q0 = N / FftPlan<N>::R0;
  const int Ny = d.Ny, K = d.K, half = Ny / 2, zg = blockIdx.y, f = blockIdx.z;
  C<T>* u = reinterpret_cast<C<T>*>(rows_smem);
  C<T>* v = u + col_tile<T>() * col_stride<T, N>();
  const C<T>* __restrict__ tw = reinterpret_cast<const C<T>*>(d.tw);
  const int ix0 = blockIdx.x * TC;
  const size_t skip = (size_t)(N - Ny) * K;      // the padded modes
  if constexpr (DIR < 0) {
    const C<T>* __restrict__ in = reinterpret_cast<const C<T>*>(d.src) + ((size_t)d.f_src[f] * d.nz + zg) * Ny * K + ix0;
    C<T>* out = reinterpret_cast<C<T>*>(d.dst) + ((size_t)f * d.nz + zg) * N * K + ix0;
    const T* __restrict__ ky = reinterpret_cast<const T*>(sizeof(T) == 8 ? (const void*)d.ky : (const void*)d.ky32);
    const bool dy = d.f_dy[f] != 0;
    col_run<T, N, +1, NT, PAD, true, true>(
        u, v, tw,
        [&](int c, int j) {
          // mode n at position n mod N; slots [0, half) and (half, Ny)
          const C<T>* x = in + c + (size_t)j * K;
          const T* q = ky + (size_t)j * K;
          const bool ok = ix0 + c < K;
          return [=](auto t) -> C<T> {
            constexpr int i0 = decltype(t)::value * Q0;
            const int i = i0 + j;
            const bool low = PAD ? 3 * i0 < N : i < half;
            const bool high = PAD ? 3 * i0 > 2 * N || (3 * i0 == 2 * N && j > 0) : i > N - half;
            if (!ok || !(low || high)) return mk<T>(0, 0);
            const size_t at = (size_t)i0 * K - (low ? 0 : skip);
            const C<T> z = x[at];
            if (!dy) return z;
            const T w = q[at];
            return mk<T>(-w * z.y, w * z.x);
          };
        },
        [&](int c, int i, C<T> z) {
          if (ix0 + c < K) out[(size_t)i * K + c] = z;
        });
  } else {
    // (1 / N, in FP32 what rows_scale leaves of it, is in the z transform's table)
    constexpr T sc = rows_scale<T, N>();
    const C<T>* __restrict__ in = reinterpret_cast<const C<T>*>(d.src) + ((size_t)f * d.nz + zg) * N * K + ix0;
    C<T>* out = reinterpret_cast<C<T>*>(d.dst) + ((size_t)f * d.nz + zg) * Ny * K + ix0;
    col_run<T, N, -1, NT, false, true, true>(
        u, v, tw,
        [&](int c, int j) {
          const C<T>* x = in + c + (size_t)j * K;
          const bool ok = ix0 + c < K;
          return [=](auto t) -> C<T> { return ok ? x[(size_t)(decltype(t)::value * Q0) * K] : mk<T>(0, 0); };
        },
        [&](int c, int i, C<T> z) {
          if (ix0 + c >= K) return;
          if (i < half) out[(size_t)i * K + c] = cscale<T>(z, sc);
          else if (i > N - half) out[(size_t)i * K + c - skip] = cscale<T>(z, sc);
          if (i == 0) out[(size_t)half * K + c] = mk<T>(0, 0);
        });
  }
}

template <typename T>
cudaError_t launch_y_cols(cudaStream_t s, const YDesc& d, int nf) {
  if (d.nz > 65535 || nf > 65535) return cudaErrorInvalidValue;
  return fft_dispatch(d.Ng, [&](auto n) -> cudaError_t {
    constexpr int N = decltype(n)::value, NT = rows_threads<T, N>();
    constexpr size_t smem = col_smem<T, N>();
    if constexpr (smem > ROWS_SMEM) {
      return cudaErrorInvalidValue;
    } else {
      dim3 grid((d.K + col_tile<T>() - 1) / col_tile<T>(), d.nz, nf);
      auto* k = d.dir < 0 ? k_y_cols<T, N, NT, -1, false> : k_y_cols<T, N, NT, 1, false>;
      if constexpr (N % 3 == 0)
        if (d.dir < 0 && 3 * d.Ny == 2 * N) k = k_y_cols<T, N, NT, -1, true>;
      cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      k<<<grid, NT, smem, s>>>(d);
      return cudaGetLastError();
    }
  });
}

// Chebyshev backward of variable f_var[f] (no derivative), pencil columns bx TC
// ..: V_k = conj(w_k)(X_k - i X_{N-k}), X_0 = d_0, X_k = d_k / 2, d_n = (-1)^n
// c_n.  X_k and X_{N-k} carry the same sign and half (N is even), so the table
// wq holds (-1)^k w_k / 2 (1 at k = 0) and the coefficients go in as they are.
template <typename T, int N, int NT>
__device__ __forceinline__ void z_backward_body(const ZDesc& d, int bx, int f, unsigned char* rows_smem) {
  constexpr int TC = col_tile<T>(), Q0 = N / FftPlan<N>::R0;
  const int Nc = d.Nc, P = d.P, p0 = bx * TC;
  C<T>* u = reinterpret_cast<C<T>*>(rows_smem);
  C<T>* v = u + col_tile<T>() * col_stride<T, N>();
  const C<T>* __restrict__ tw = reinterpret_cast<const C<T>*>(d.tw);
  const C<T>* __restrict__ wq = reinterpret_cast<const C<T>*>(d.wq);
  const C<T>* __restrict__ src =
      reinterpret_cast<const C<T>*>(sizeof(T) == 8 ? (const void*)d.xc : (const void*)d.xc32) +
      (size_t)d.f_var[f] * d.xc_stride + (size_t)p0 * Nc;
  C<T>* gz = reinterpret_cast<C<T>*>(d.gz) + (size_t)f * N * P + p0;
  col_run<T, N, +1, NT, false, false, true>(
      u, v, tw,
      [&](int c, int j) {
        const C<T>* x = src + (size_t)c * Nc;
        const int top = p0 + c < P ? Nc : 0;     // no pencil: no coefficients
        return [=](auto t) -> C<T> {
          const int k = j + decltype(t)::value * Q0;
          const C<T> a = k < top ? x[k] : mk<T>(0, 0), b = N - k < top ? x[N - k] : mk<T>(0, 0);
          return cmulc<T>(mk<T>(a.x + b.y, a.y - b.x), fft_tw<T>(wq, k));
        };
      },
      [&](int c, int j, C<T> z) {
        const int zg = j < N / 2 ? 2 * j : 2 * (N - 1 - j) + 1;
        if (p0 + c < P) gz[(size_t)zg * P + c] = z;
      });
}

// Chebyshev forward of product f: out_k = w_k V_k + conj(w_k) V_{N-k}, wq the
// w_k with the T coefficients' sign and scale and the part of 1 / (2 N_gx)
// [/ N_gy] that the x [and y] transforms leave out
template <typename T, int N, int NT>
__device__ __forceinline__ void z_forward_body(const ZDesc& d, int bx, int f, unsigned char* rows_smem) {
  constexpr int TC = col_tile<T>(), NS = col_stride<T, N>(), Q0 = N / FftPlan<N>::R0;
  const int Nc = d.Nc, P = d.P, p0 = bx * TC;
  C<T>* u = reinterpret_cast<C<T>*>(rows_smem);
  C<T>* v = u + col_tile<T>() * col_stride<T, N>();
  const C<T>* __restrict__ tw = reinterpret_cast<const C<T>*>(d.tw);
  const C<T>* __restrict__ wq = reinterpret_cast<const C<T>*>(d.wq);
  const C<T>* __restrict__ h = reinterpret_cast<const C<T>*>(d.h) + (size_t)f * N * P + p0;
  col_run<T, N, -1, NT, false, true, false>(
      u, v, tw,
      [&](int c, int j) {
        const bool ok = p0 + c < P;
        return [=](auto t) -> C<T> {
          const int i = j + decltype(t)::value * Q0;
          const int zg = i < N / 2 ? 2 * i : 2 * (N - 1 - i) + 1;
          return ok ? h[(size_t)zg * P + c] : mk<T>(0, 0);
        };
      },
      [&](int c, int i, C<T> z) { u[c * NS + fft_pad<T>(i)] = z; });
  for (int k = threadIdx.x; k < Nc; k += NT) {
    const C<T> w = wq[k];
    for (int c = 0; c < TC && p0 + c < P; ++c) {
      const C<T> a = u[c * NS + fft_pad<T>(k)], b = u[c * NS + fft_pad<T>(k == 0 ? 0 : N - k)];
      const C<T> s = cadd<T>(a, b), m = csub<T>(a, b);
      const T x = fma(-w.y, m.y, w.x * s.x), y = fma(w.y, m.x, w.x * s.y);
      // the k_x = 0 column is the transform of a real function: real coefficients
      d.fc[((size_t)f * P + p0 + c) * Nc + k] = make_double2((double)x, p0 + c == 0 ? 0.0 : (double)y);
    }
  }
}

template <typename T, int N, int NT>
__global__ void __launch_bounds__(NT, rows_ctas<T>(NT)) k_z_backward(ZDesc d) {
  extern __shared__ __align__(16) unsigned char rows_smem[];
  z_backward_body<T, N, NT>(d, blockIdx.x, blockIdx.y, rows_smem);
}
template <typename T, int N, int NT>
__global__ void __launch_bounds__(NT, rows_ctas<T>(NT)) k_z_forward(ZDesc d) {
  extern __shared__ __align__(16) unsigned char rows_smem[];
  z_forward_body<T, N, NT>(d, blockIdx.x, blockIdx.y, rows_smem);
}

template <typename T>
cudaError_t launch_z_cols(cudaStream_t s, const ZDesc& d, int nf, bool forward) {
  return fft_dispatch(d.Ng, [&](auto n) -> cudaError_t {
    constexpr int N = decltype(n)::value, NT = rows_threads<T, N>();
    constexpr size_t smem = col_smem<T, N>();
    if constexpr (smem > ROWS_SMEM || N > 1536) {
      return cudaErrorInvalidValue;
    } else {
      dim3 grid((d.P + col_tile<T>() - 1) / col_tile<T>(), nf);
      auto* k = forward ? k_z_forward<T, N, NT> : k_z_backward<T, N, NT>;
      cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      k<<<grid, NT, smem, s>>>(d);
      return cudaGetLastError();
    }
  });
}

// ---------------------------------------------------------------------------
// batches of uneven problems: one CTA per work item, or a persistent grid on a
// work queue; the item's length picks its code
// ---------------------------------------------------------------------------
constexpr int BATCH_NT = 256;

template <int MOST, typename F>
__device__ __forceinline__ void fft_switch(int N, F&& f) {
  switch (N) {
#define SP_FFT_CASE(n)                                                            \
  case n:                                                                         \
    if constexpr (n <= MOST) f(std::integral_constant<int, n>());                 \
    break;
    SP_FFT_CASE(16) SP_FFT_CASE(24) SP_FFT_CASE(32) SP_FFT_CASE(48) SP_FFT_CASE(64) SP_FFT_CASE(96)
    SP_FFT_CASE(128) SP_FFT_CASE(192) SP_FFT_CASE(256) SP_FFT_CASE(384) SP_FFT_CASE(512) SP_FFT_CASE(768)
    SP_FFT_CASE(1024) SP_FFT_CASE(1536) SP_FFT_CASE(2048) SP_FFT_CASE(3072) SP_FFT_CASE(4096)
#undef SP_FFT_CASE
    default: break;
  }
}

template <typename T>
__global__ void __launch_bounds__(BATCH_NT, sizeof(T) == 8 ? 2 : 3) k_x_rows_batched(const XDesc* __restrict__ ds,
                                                             const int4* __restrict__ work, int nwork, int* queue) {
  extern __shared__ __align__(16) unsigned char rows_smem[];
  for_each_item(nwork, queue, [&](int it) {
    const int4 w = work[it];
    const XDesc& d = ds[w.x];
    fft_switch<4096>(d.N, [&](auto n) {
      constexpr int N = decltype(n)::value;
      if (N % 3 == 0 && 3 * d.K == N) x_rows_body<T, N, BATCH_NT, N % 3 == 0>(d, w.y, rows_smem);
      else x_rows_body<T, N, BATCH_NT, false>(d, w.y, rows_smem);
    });
  });
}
template <typename T, bool FWD>
__global__ void __launch_bounds__(BATCH_NT, sizeof(T) == 8 ? 2 : 3) k_z_cols_batched(const ZDesc* __restrict__ ds,
                                                             const int4* __restrict__ work, int nwork, int* queue) {
  extern __shared__ __align__(16) unsigned char rows_smem[];
  for_each_item(nwork, queue, [&](int it) {
    const int4 w = work[it];
    fft_switch<1536>(ds[w.x].Ng, [&](auto n) {
      constexpr int N = decltype(n)::value;
      if constexpr (FWD) z_forward_body<T, N, BATCH_NT>(ds[w.x], w.y, w.z, rows_smem);
      else z_backward_body<T, N, BATCH_NT>(ds[w.x], w.y, w.z, rows_smem);
    });
  });
}

// persistent (queue set): as many CTAs as fit on the GPU at once
template <typename K>
cudaError_t rows_batched(K kernel, cudaStream_t s, size_t smem, int nwork, const int* queue, int& grid) {
  if (smem > ROWS_SMEM) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  grid = nwork;
  if (e != cudaSuccess || queue == nullptr) return e;
  int dev = 0, sms = 1, per_sm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, BATCH_NT, smem) != cudaSuccess || per_sm < 1)
    per_sm = 1;
  grid = std::max(1, std::min(nwork, sms * per_sm));
  return cudaSuccess;
}

template <typename T>
cudaError_t launch_x_rows_batched(cudaStream_t s, const XDesc* ds, const int4* work, int nwork, size_t smem,
                                  int* queue) {
  int grid;
  cudaError_t e = rows_batched(k_x_rows_batched<T>, s, smem, nwork, queue, grid);
  if (e != cudaSuccess) return e;
  k_x_rows_batched<T><<<grid, BATCH_NT, smem, s>>>(ds, work, nwork, queue);
  return cudaGetLastError();
}
template <typename T>
cudaError_t launch_z_cols_batched(cudaStream_t s, bool forward, const ZDesc* ds, const int4* work, int nwork,
                                  size_t smem, int* queue) {
  auto* k = forward ? k_z_cols_batched<T, true> : k_z_cols_batched<T, false>;
  int grid;
  cudaError_t e = rows_batched(k, s, smem, nwork, queue, grid);
  if (e != cudaSuccess) return e;
  k<<<grid, BATCH_NT, smem, s>>>(ds, work, nwork, queue);
  return cudaGetLastError();
}

}  // namespace spectau
