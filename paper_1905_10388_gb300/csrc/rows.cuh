// Spectral transforms on compile-time lengths (fftn.cuh): the right-hand
// side's x rows with the dealiased products, the y transforms and the
// Chebyshev (z) transforms.  Conventions and data layouts as in
// transforms.cu, whose run-time-length kernels serve the other transforms
// (set-up, batches of uneven problems, adjoint) and lengths.
//
// Derivatives i k_x and i k_y commute with the transforms of the other axes:
// z transforms run once per variable, y transforms once per variable and once
// more where a y derivative is used, and the x rows apply i k_x as they load
// (2D Rayleigh-Benard: 6 z transforms for 8 grid fields; 3D: 8 and 12 y
// transforms for 15).
#pragma once
#include <algorithm>
#include <type_traits>

#include "fftn.cuh"
#include "internal.h"

namespace spectau {

constexpr size_t ROWS_SMEM = ROWS_SMEM_MAX;

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

template <typename T, int N, int NT>
__device__ __forceinline__ void x_rows_body(const XDesc& d, int row, unsigned char* rows_smem) {
  constexpr int NP = fft_padded<T>(N), MAX_TERMS = 16, MAX_F = 16;
  const int K = d.K, rows = d.rows, nf = d.nf, ne = d.ne, tid = threadIdx.x;
  const int nbi = (nf + 1) / 2, nbo = (ne + 1) / 2;
  C<T>* u = reinterpret_cast<C<T>*>(rows_smem);
  C<T>* v = u + nbi * NP;
  T* G = reinterpret_cast<T*>(u);                // grid fields [f][N], over the first buffer
  __shared__ T tc[MAX_TERMS];
  __shared__ int ta[MAX_TERMS], tb[MAX_TERMS], te[MAX_TERMS];
  __shared__ int fs[MAX_F], fx[MAX_F];
  const int nterms = min(d.nterms, MAX_TERMS);
  const T* tcoef = reinterpret_cast<const T*>(sizeof(T) == 8 ? (const void*)d.t_coef : (const void*)d.t_coef32);
  const T* kx = reinterpret_cast<const T*>(sizeof(T) == 8 ? (const void*)d.kx : (const void*)d.kx32);
  if (tid < nterms) {
    tc[tid] = tcoef[tid]; ta[tid] = d.t_fa[tid] * N; tb[tid] = d.t_fb[tid] * N; te[tid] = d.t_eq[tid];
  }
  if (tid < nf) { fs[tid] = d.f_src[tid]; fx[tid] = d.f_dx[tid]; }
  const C<T>* __restrict__ tw = reinterpret_cast<const C<T>*>(d.tw);
  __syncthreads();
  const C<T>* __restrict__ gz = reinterpret_cast<const C<T>*>(d.gz) + (size_t)row * K;
  const size_t plane = (size_t)rows * K;
  auto spec = [&](int f, int k) -> C<T> {
    if (f >= nf) return mk<T>(0, 0);
    const C<T> z = gz[fs[f] * plane + k];
    if (!fx[f]) return z;
    const T q = kx[k];
    return mk<T>(-q * z.y, q * z.x);
  };
  fft_run<T, N, +1, NT>(
      nbi, u, v, tw,
      [&](int b, int i) -> C<T> {
        // two real fields a, b as a + i b: the Hermitian spectrum of the stored k >= 0 modes
        if (i < K) {
          const C<T> A = spec(2 * b, i), B = spec(2 * b + 1, i);
          return i == 0 ? mk<T>(A.x, B.x) : mk<T>(A.x - B.y, A.y + B.x);
        }
        if (i > N - K) {
          const C<T> A = spec(2 * b, N - i), B = spec(2 * b + 1, N - i);
          return mk<T>(A.x + B.y, B.x - A.y);
        }
        return mk<T>(0, 0);
      },
      [&](int b, int i, C<T> z) {
        G[2 * b * N + i] = z.x;
        if (2 * b + 1 < nf) G[(2 * b + 1) * N + i] = z.y;
      });
  // products: terms are grouped by equation; two equations share a complex sequence
  T* O = reinterpret_cast<T*>(v);
  for (int i = tid; i < N; i += NT) {
    const int o = 2 * fft_pad<T>(i);
    T acc = 0;
    for (int t = 0; t < nterms; ++t) {
      acc += tc[t] * G[ta[t] + i] * G[tb[t] + i];
      if (t + 1 == nterms || te[t + 1] != te[t]) {
        O[(te[t] >> 1) * 2 * NP + o + (te[t] & 1)] = acc;
        acc = 0;
      }
    }
    if (ne & 1) O[(ne >> 1) * 2 * NP + o + 1] = 0;
  }
  __syncthreads();
  constexpr bool three = FftPlan<N>::R2 > 1;
  C<T>* u2 = v + nbo * NP;
  C<T>* Z = three ? u2 : v;
  fft_run<T, N, -1, NT>(
      nbo, u2, three ? v : u2, tw, [&](int b, int i) -> C<T> { return v[b * NP + fft_pad<T>(i)]; },
      [&](int b, int i, C<T> z) { Z[b * NP + fft_pad<T>(i)] = z; });
  C<T>* h = reinterpret_cast<C<T>*>(d.h) + (size_t)row * K;
  const T s = (T)1 / (T)(2 * N);
  for (int b = 0; b < nbo; ++b)
    for (int k = tid; k < K; k += NT) {
      const C<T> z = Z[b * NP + fft_pad<T>(k)], r = Z[b * NP + fft_pad<T>(k == 0 ? 0 : N - k)];
      h[2 * b * plane + k] = mk<T>((z.x + r.x) * s, (z.y - r.y) * s);
      if (2 * b + 1 < ne) h[(2 * b + 1) * plane + k] = mk<T>((z.y + r.y) * s, (r.x - z.x) * s);
    }
}

template <typename T, int N, int NT>
__global__ void __launch_bounds__(NT, rows_ctas<T>(NT)) k_x_rows(XDesc d) {
  extern __shared__ __align__(16) unsigned char rows_smem[];
  x_rows_body<T, N, NT>(d, blockIdx.x, rows_smem);
}

template <typename T>
cudaError_t launch_x_rows(cudaStream_t s, const XDesc& d) {
  return fft_dispatch(d.N, [&](auto n) -> cudaError_t {
    constexpr int N = decltype(n)::value, NT = rows_threads<T, N>();
    const size_t smem = x_rows_smem<T, N>(d.nf, d.ne);
    if (smem > ROWS_SMEM || d.nf > 16 || d.nterms > 16) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(k_x_rows<T, N, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_x_rows<T, N, NT><<<d.rows, NT, smem, s>>>(d);
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

// One transform of the tile: `in(c, i)`, `fin(c, i, v)`; IN_COL / OUT_COL:
// columns fastest over the threads in the first / last pass.  Two-pass lengths
// use buffer v alone.  Ends after a barrier.
template <typename T, int N, int SIGN, int NT, bool IN_COL, bool OUT_COL, typename IN, typename FIN>
__device__ __forceinline__ void col_run(C<T>* u, C<T>* v, const C<T>* tw, IN&& in, FIN&& fin) {
  using P = FftPlan<N>;
  constexpr int TC = col_tile<T>(), NS = col_stride<T, N>();
  C<T>* first = P::R2 > 1 ? u : v;
  {
    constexpr int R = P::R0, Q = N / R;
    for (int id = threadIdx.x; id < TC * Q; id += NT) {
      const int c = IN_COL ? id % TC : id / Q, j = IN_COL ? id / TC : id % Q;
      C<T> a[R], y[R];
#pragma unroll
      for (int t = 0; t < R; ++t) a[t] = in(c, j + t * Q);
      dft_first<T, SIGN, R>(a, y);
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
      const int w0 = k * STEP;
      auto at = [&](int m, int q, int rr) {
        const C<T> w = tw[m * w0 + q * (N / rr)];
        return SIGN > 0 ? mk<T>(w.x, -w.y) : w;
      };
      DitTw<T, SIGN, R, 1, 1, decltype(at)>::run(a, y, at);
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
// f_dy is set; DIR > 0: grid -> slots (1/N, Nyquist slot zero)
template <typename T, int N, int NT, int DIR>
__global__ void __launch_bounds__(NT, rows_ctas<T>(NT)) k_y_cols(YDesc d) {
  extern __shared__ __align__(16) unsigned char rows_smem[];
  constexpr int TC = col_tile<T>();
  const int Ny = d.Ny, K = d.K, half = Ny / 2, zg = blockIdx.y, f = blockIdx.z;
  C<T>* u = reinterpret_cast<C<T>*>(rows_smem);
  C<T>* v = u + col_tile<T>() * col_stride<T, N>();
  const C<T>* __restrict__ tw = reinterpret_cast<const C<T>*>(d.tw);
  const int ix0 = blockIdx.x * TC;
  if constexpr (DIR < 0) {
    const C<T>* in = reinterpret_cast<const C<T>*>(d.src) + ((size_t)d.f_src[f] * d.nz + zg) * Ny * K + ix0;
    C<T>* out = reinterpret_cast<C<T>*>(d.dst) + ((size_t)f * d.nz + zg) * N * K + ix0;
    const T* ky = reinterpret_cast<const T*>(sizeof(T) == 8 ? (const void*)d.ky : (const void*)d.ky32);
    const bool dy = d.f_dy[f] != 0;
    col_run<T, N, +1, NT, true, true>(
        u, v, tw,
        [&](int c, int i) -> C<T> {
          // mode n at position n mod N; slots [0, half) and (half, Ny)
          const int sl = i < half ? i : (i > N - half ? i - N + Ny : -1);
          if (sl < 0 || ix0 + c >= K) return mk<T>(0, 0);
          const C<T> z = in[(size_t)sl * K + c];
          if (!dy) return z;
          const T q = ky[(size_t)sl * K];
          return mk<T>(-q * z.y, q * z.x);
        },
        [&](int c, int i, C<T> z) {
          if (ix0 + c < K) out[(size_t)i * K + c] = z;
        });
  } else {
    const C<T>* in = reinterpret_cast<const C<T>*>(d.src) + ((size_t)f * d.nz + zg) * N * K + ix0;
    C<T>* out = reinterpret_cast<C<T>*>(d.dst) + ((size_t)f * d.nz + zg) * Ny * K + ix0;
    const T s = (T)1 / (T)N;
    col_run<T, N, -1, NT, true, true>(
        u, v, tw, [&](int c, int i) -> C<T> { return ix0 + c < K ? in[(size_t)i * K + c] : mk<T>(0, 0); },
        [&](int c, int i, C<T> z) {
          const int sl = i < half ? i : (i > N - half ? i - N + Ny : -1);
          if (ix0 + c >= K) return;
          if (sl >= 0) out[(size_t)sl * K + c] = mk<T>(z.x * s, z.y * s);
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
      auto* k = d.dir < 0 ? k_y_cols<T, N, NT, -1> : k_y_cols<T, N, NT, 1>;
      cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      k<<<grid, NT, smem, s>>>(d);
      return cudaGetLastError();
    }
  });
}

// Chebyshev backward of variable f_var[f] (no derivative), pencil columns bx TC ..: V_k = conj(w_k)(X_k - i X_{N-k}), X_0 = d_0, X_k =
// d_k / 2, d_n = (-1)^n c_n
template <typename T, int N, int NT>
__device__ __forceinline__ void z_backward_body(const ZDesc& d, int bx, int f, unsigned char* rows_smem) {
  constexpr int TC = col_tile<T>();
  const int Nc = d.Nc, P = d.P, p0 = bx * TC;
  C<T>* u = reinterpret_cast<C<T>*>(rows_smem);
  C<T>* v = u + col_tile<T>() * col_stride<T, N>();
  const C<T>* __restrict__ tw = reinterpret_cast<const C<T>*>(d.tw);
  const C<T>* wq = reinterpret_cast<const C<T>*>(d.wq);
  const C<T>* src = reinterpret_cast<const C<T>*>(sizeof(T) == 8 ? (const void*)d.xc : (const void*)d.xc32) +
                    (size_t)d.f_var[f] * d.xc_stride + (size_t)p0 * Nc;
  C<T>* gz = reinterpret_cast<C<T>*>(d.gz) + (size_t)f * N * P + p0;
  col_run<T, N, +1, NT, false, true>(
      u, v, tw,
      [&](int c, int k) -> C<T> {
        if (p0 + c >= P) return mk<T>(0, 0);
        auto coef = [&](int n) -> C<T> {
          if (n >= Nc) return mk<T>(0, 0);
          const C<T> x = src[(size_t)c * Nc + n];
          const T s = ((n & 1) ? (T)-1 : (T)1) * (n == 0 ? (T)1 : (T)0.5);
          return mk<T>(s * x.x, s * x.y);
        };
        const C<T> a = coef(k), b = k == 0 ? mk<T>(0, 0) : coef(N - k);
        return cmulc<T>(mk<T>(a.x + b.y, a.y - b.x), wq[k]);
      },
      [&](int c, int j, C<T> z) {
        const int zg = j < N / 2 ? 2 * j : 2 * (N - 1 - j) + 1;
        if (p0 + c < P) gz[(size_t)zg * P + c] = z;
      });
}

// Chebyshev forward of product f: out_k = (w_k V_k + conj(w_k) V_{N-k})
// scaled to T coefficients
template <typename T, int N, int NT>
__device__ __forceinline__ void z_forward_body(const ZDesc& d, int bx, int f, unsigned char* rows_smem) {
  constexpr int TC = col_tile<T>(), NS = col_stride<T, N>();
  const int Nc = d.Nc, P = d.P, p0 = bx * TC, e = f;
  C<T>* u = reinterpret_cast<C<T>*>(rows_smem);
  C<T>* v = u + col_tile<T>() * col_stride<T, N>();
  const C<T>* __restrict__ tw = reinterpret_cast<const C<T>*>(d.tw);
  const C<T>* wq = reinterpret_cast<const C<T>*>(d.wq);
  const C<T>* h = reinterpret_cast<const C<T>*>(d.h) + (size_t)e * N * P + p0;
  col_run<T, N, -1, NT, true, false>(
      u, v, tw,
      [&](int c, int j) -> C<T> {
        const int zg = j < N / 2 ? 2 * j : 2 * (N - 1 - j) + 1;
        return p0 + c < P ? h[(size_t)zg * P + c] : mk<T>(0, 0);
      },
      [&](int c, int i, C<T> z) { u[c * NS + fft_pad<T>(i)] = z; });
  const T inv = (T)1 / (T)N;
  for (int c = 0; c < TC && p0 + c < P; ++c)
    for (int k = threadIdx.x; k < Nc; k += NT) {
      const C<T> a = u[c * NS + fft_pad<T>(k)], b = u[c * NS + fft_pad<T>(k == 0 ? 0 : N - k)], w = wq[k];
      const C<T> o = cadd<T>(cmul<T>(w, a), cmulc<T>(b, w));
      const T s = ((k & 1) ? (T)-1 : (T)1) * (k == 0 ? inv * (T)0.5 : inv);
      // the k_x = 0 column is the transform of a real function: real coefficients
      d.fc[((size_t)e * P + p0 + c) * Nc + k] = make_double2((double)(o.x * s), p0 + c == 0 ? 0.0 : (double)(o.y * s));
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
    fft_switch<4096>(ds[w.x].N, [&](auto n) { x_rows_body<T, decltype(n)::value, BATCH_NT>(ds[w.x], w.y, rows_smem); });
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
