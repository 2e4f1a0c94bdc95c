// Shared-memory Stockham FFT passes of compile-time length N = 2^k or 3 * 2^k,
// two or three per transform, each butterfly in one thread's registers.
//
// A pass of radix R over sub-transforms of length Ns: butterfly j < N / R reads
// the R elements j + t N / R, twiddles element t by W_N^{t k N / (R Ns)}, k = j
// mod Ns, and writes the R outputs (j / Ns) R Ns + k + q Ns; the first pass has
// Ns = 1 and no twiddles and takes the factor 3, and the result is in natural
// order.  With N a template constant every index is a shift, a mask or an
// immediate: at run-time lengths the index arithmetic alone was most of the
// FP32 kernels' instructions.
//
// A twiddled butterfly multiplies each input once.  In FP64, whose pipe is the
// bound, half of the products sit in the first two-point steps, E + w O in four
// FMAs and E - w O = 2 E - (E + w O) in two: 72 instructions for radix 8 instead of
// 80.  FP32 has no fewer instructions that way.  Error of the right-hand side
// against extended precision, geometric means over lengths of 48 to 768, and an
// FP64 512 x 256 RK222 step: FP64 here 1.37e-15 (770 us), products first 1.33e-15
// (796 us), a twiddle at each of the three levels (72 instructions, 4 twiddle
// loads for 7) 1.51e-15 (754 us), the run-time kernels of transforms.cu 1.33e-15;
// FP32 here 4.29e-7, a twiddle at each level 4.52e-7, the run-time kernels 4.31e-7.
//
// Buffers are padded by one element every 128 bytes, so the first pass's
// stride-R writes spread over the banks.
#pragma once
#include <type_traits>
#include <utility>

#include "common.cuh"

namespace spectau {

template <int N>
struct FftPlan;   // R0, R1, R2 (1: two passes)
#define SP_FFT_PLAN(n, a, b, c)                       \
  template <>                                         \
  struct FftPlan<n> {                                 \
    static constexpr int R0 = a, R1 = b, R2 = c;      \
    static_assert(a * b * c == n, "radices");         \
  };
SP_FFT_PLAN(16, 4, 4, 1)
SP_FFT_PLAN(24, 6, 4, 1)
SP_FFT_PLAN(32, 8, 4, 1)
SP_FFT_PLAN(48, 3, 4, 4)
SP_FFT_PLAN(64, 4, 4, 4)
SP_FFT_PLAN(96, 6, 4, 4)
SP_FFT_PLAN(128, 8, 4, 4)
SP_FFT_PLAN(192, 6, 8, 4)
SP_FFT_PLAN(256, 8, 8, 4)
SP_FFT_PLAN(384, 6, 8, 8)
SP_FFT_PLAN(512, 8, 8, 8)
SP_FFT_PLAN(768, 12, 8, 8)
SP_FFT_PLAN(1024, 16, 8, 8)
SP_FFT_PLAN(1536, 12, 16, 8)
SP_FFT_PLAN(2048, 16, 16, 8)
SP_FFT_PLAN(3072, 12, 16, 16)
SP_FFT_PLAN(4096, 16, 16, 16)
#undef SP_FFT_PLAN

template <typename T>
__device__ __forceinline__ constexpr int fft_pad(int i) { return i + (sizeof(T) == 4 ? (i >> 4) : (i >> 3)); }
// elements of a padded buffer of N
template <typename T>
__host__ __device__ constexpr int fft_padded(int N) { return N + (sizeof(T) == 4 ? N / 16 : N / 8); }

// z times exp(SIGN i pi / 2)
template <typename T, int SIGN>
__device__ __forceinline__ C<T> rot90(C<T> z) { return SIGN < 0 ? mk<T>(z.y, -z.x) : mk<T>(-z.y, z.x); }

// E + w O, E - w O
template <typename T>
__device__ __forceinline__ void bfly(C<T> e, C<T> o, C<T> w, C<T>& p, C<T>& m) {
  p.x = fma(-w.y, o.y, fma(w.x, o.x, e.x));
  p.y = fma(w.y, o.x, fma(w.x, o.y, e.y));
  if constexpr (sizeof(T) == 8) {
    m.x = fma((T)2, e.x, -p.x);
    m.y = fma((T)2, e.y, -p.y);
  } else {
    m.x = fma(w.y, o.y, fma(-w.x, o.x, e.x));
    m.y = fma(-w.y, o.x, fma(-w.x, o.y, e.y));
  }
}

// DFT of length R (a power of two) of elements I, I + S, I + 2 S, ...: the two-point
// steps on the elements themselves by `leaf(i, j, p, m)`, which sets p, m to the
// sum and difference of elements i and j, the others with constant roots, the
// trivial ones as sums and differences.
template <typename T, int SIGN, int R, int S, int I, typename LEAF>
struct Dit {
  static __device__ __forceinline__ void run(C<T>* out, const LEAF& leaf) {
    C<T> e[R / 2], o[R / 2];
    Dit<T, SIGN, R / 2, 2 * S, I, LEAF>::run(e, leaf);
    Dit<T, SIGN, R / 2, 2 * S, I + S, LEAF>::run(o, leaf);
#pragma unroll
    for (int q = 0; q < R / 2; ++q) {
      if (q == 0) {
        out[0] = cadd<T>(e[0], o[0]);
        out[R / 2] = csub<T>(e[0], o[0]);
      } else if (4 * q == R) {
        const C<T> v = rot90<T, SIGN>(o[q]);
        out[q] = cadd<T>(e[q], v);
        out[q + R / 2] = csub<T>(e[q], v);
      } else {
        constexpr double c1 = 0.92387953251128675613, s1 = 0.38268343236508977173, h = 0.70710678118654752440;
        const int u = q * 16 / R;                // root exp(SIGN 2 pi i u / 16), u = 1, 2, 3, 5, 6, 7
        const double cr = u == 1 ? c1 : u == 2 ? h : u == 3 ? s1 : u == 5 ? -s1 : u == 6 ? -h : -c1;
        const double ci = u == 1 ? s1 : u == 2 ? h : u == 3 ? c1 : u == 5 ? c1 : u == 6 ? h : s1;
        bfly<T>(e[q], o[q], mk<T>((T)cr, (T)(SIGN < 0 ? -ci : ci)), out[q], out[q + R / 2]);
      }
    }
  }
};
template <typename T, int SIGN, int S, int I, typename LEAF>
struct Dit<T, SIGN, 2, S, I, LEAF> {
  static __device__ __forceinline__ void run(C<T>* out, const LEAF& leaf) { leaf(I, I + S, out[0], out[1]); }
};
template <typename T, int SIGN, int R>
__device__ __forceinline__ void dft_plain(const C<T>* a, C<T>* out) {
  if constexpr (R == 1) {
    out[0] = a[0];
  } else {
    auto leaf = [&](int i, int j, C<T>& p, C<T>& m) {
      p = cadd<T>(a[i], a[j]);
      m = csub<T>(a[i], a[j]);
    };
    Dit<T, SIGN, R, 1, 0, decltype(leaf)>::run(out, leaf);
  }
}
// The DFT of a[t] w^t; `at(t)` returns w^t.
template <typename T, int SIGN, int R, typename W>
__device__ __forceinline__ void dft_twiddled(const C<T>* a, C<T>* out, const W& at) {
  auto leaf = [&](int i, int j, C<T>& p, C<T>& m) {
    const C<T> e = i == 0 ? a[0] : cmul<T>(at(i), a[i]);
    if constexpr (sizeof(T) == 8) {
      bfly<T>(e, a[j], at(j), p, m);
    } else {
      const C<T> o = cmul<T>(at(j), a[j]);
      p = cadd<T>(e, o);
      m = csub<T>(e, o);
    }
  };
  Dit<T, SIGN, R, 1, 0, decltype(leaf)>::run(out, leaf);
}

// 3-point DFT: sums, differences and FMAs with -1/2 and sqrt(3)/2.  Z: an input
// known to be zero (-1: none).
template <typename T, int SIGN, int Z>
__device__ __forceinline__ void dft3(C<T> a0, C<T> a1, C<T> a2, C<T>& x0, C<T>& x1, C<T>& x2) {
  const T c = (SIGN < 0 ? (T)-1 : (T)1) * (T)0.86602540378443864676;
  const C<T> s = Z == 1 ? a2 : Z == 2 ? a1 : cadd<T>(a1, a2);
  const C<T> d = Z == 1 ? mk<T>(-a2.x, -a2.y) : Z == 2 ? a1 : csub<T>(a1, a2);
  const C<T> m = Z == 0 ? mk<T>((T)-0.5 * s.x, (T)-0.5 * s.y)
                        : mk<T>(fma((T)-0.5, s.x, a0.x), fma((T)-0.5, s.y, a0.y));
  x0 = Z == 0 ? s : cadd<T>(a0, s);
  x1 = mk<T>(fma(-c, d.y, m.x), fma(c, d.x, m.y));
  x2 = mk<T>(fma(c, d.y, m.x), fma(-c, d.x, m.y));
}

// f(integral_constant<int, 0>), ..., f(integral_constant<int, R - 1>)
template <typename F, int... Ts>
__device__ __forceinline__ void unroll_seq(F&& f, std::integer_sequence<int, Ts...>) {
  (f(std::integral_constant<int, Ts>()), ...);
}
template <int R, typename F>
__device__ __forceinline__ void unroll(F&& f) { unroll_seq(f, std::make_integer_sequence<int, R>()); }

// First-pass DFT of R0 = 2^a or 3 2^a elements.  The factor 3 by the prime
// factor map (coprime factors need no twiddles): with R = 3 H, input (H n1 + 3
// n2) mod R and output k = k1 mod 3, k2 mod H.
// PAD: the middle third of the inputs is zero (a spectrum padded by 3/2).
template <typename T, int SIGN, int R, bool PAD>
__device__ __forceinline__ void dft_first(const C<T>* a, C<T>* out) {
  if constexpr (R % 3 == 0) {
    constexpr int H = R / 3;
    C<T> b[3][H];
    unroll<H>([&](auto n) {
      constexpr int n2 = decltype(n)::value;
      constexpr int i0 = (3 * n2) % R, i1 = (H + 3 * n2) % R, i2 = (2 * H + 3 * n2) % R;
      // the three differ by R / 3, so exactly one lies in the middle third
      constexpr int Z = !PAD ? -1 : (i0 / H == 1 ? 0 : i1 / H == 1 ? 1 : 2);
      dft3<T, SIGN, Z>(a[i0], a[i1], a[i2], b[0][n2], b[1][n2], b[2][n2]);
    });
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) {
      C<T> o[H];
      dft_plain<T, SIGN, H>(b[k1], o);
#pragma unroll
      for (int k2 = 0; k2 < H; ++k2) {
        // the k in [0, R) with H k = k1 H (mod 3 H) after the maps: k = k1 (H
        // H^-1 mod 3) + k2 (3 3^-1 mod H)
        constexpr int hi = H % 3 == 1 ? 1 : 2;                        // H^-1 mod 3
        constexpr int ti = H == 1 ? 0 : H == 2 ? 1 : H == 4 ? 3 : 3;  // 3^-1 mod H (H = 1, 2, 4, 8)
        out[(H * hi * k1 + 3 * ti * k2) % R] = o[k2];
      }
    }
  } else {
    dft_plain<T, SIGN, R>(a, out);
  }
}

// First pass over nb sequences: `open(b, j)` gives a reader e of sequence b's
// elements j + t N / R0, e(integral_constant<int, t>).  PAD: elements [N/3, 2N/3)
// are zero and are not read.
template <int R, bool PAD>
constexpr bool fft_zero(int t) { return PAD && 3 * t >= R && 3 * t < 2 * R; }
template <typename T, int R, bool PAD, typename E>
__device__ __forceinline__ void fft_read(E&& e, C<T>* a) {
  unroll<R>([&](auto t) {
    if constexpr (fft_zero<R, PAD>(decltype(t)::value)) a[decltype(t)::value] = mk<T>(0, 0);
    else a[decltype(t)::value] = e(t);
  });
}
template <typename T, int N, int SIGN, int NT, bool PAD, typename OPEN, typename OUT>
__device__ __forceinline__ void fft_pass_first(int nb, OPEN&& open, OUT&& out) {
  constexpr int R = FftPlan<N>::R0, Q = N / R;
  for (int id = threadIdx.x; id < nb * Q; id += NT) {
    const int b = id / Q, j = id - b * Q;
    C<T> a[R], y[R];
    fft_read<T, R, PAD>(open(b, j), a);
    dft_first<T, SIGN, R, PAD>(a, y);
#pragma unroll
    for (int q = 0; q < R; ++q) out(b, j * R + q, y[q]);
  }
}

// element of a twiddle table by a 32-bit byte offset
template <typename T>
__device__ __forceinline__ C<T> fft_tw(const C<T>* tw, unsigned i) {
  return __ldg(reinterpret_cast<const C<T>*>(reinterpret_cast<const char*>(tw) + i * (unsigned)sizeof(C<T>)));
}

// A twiddled pass of radix R over sub-transforms of length Ns from padded
// buffers x (sequence stride NP): `out(b, i, v)` takes element i of sequence b.
template <typename T, int N, int SIGN, int NT, int R, int Ns, typename OUT>
__device__ __forceinline__ void fft_pass_tw(const C<T>* __restrict__ x, const C<T>* __restrict__ tw, int nb,
                                            OUT&& out) {
  constexpr int Q = N / R, NP = fft_padded<T>(N), STEP = N / (R * Ns);
  for (int id = threadIdx.x; id < nb * Q; id += NT) {
    const int b = id / Q, j = id - b * Q;
    const int k = j % Ns, g = j / Ns;
    const C<T>* xb = x + b * NP;
    C<T> a[R], y[R];
#pragma unroll
    for (int t = 0; t < R; ++t) a[t] = xb[fft_pad<T>(j + t * Q)];
    const unsigned w0 = k * STEP;
    dft_twiddled<T, SIGN, R>(a, y, [&](int t) {
      const C<T> w = fft_tw<T>(tw, t * w0);
      return SIGN > 0 ? mk<T>(w.x, -w.y) : w;
    });
    const int o = g * R * Ns + k;
#pragma unroll
    for (int q = 0; q < R; ++q) out(b, o + q * Ns, y[q]);
  }
}

// Transforms nb sequences: `open` as above, results to `fin(b, i, v)` in natural
// order.  A three-pass transform goes through buffer u, then v; a two-pass one
// through v only (fin may write where u is).  Ends after a barrier.
template <typename T, int N, int SIGN, int NT, bool PAD, typename OPEN, typename FIN>
__device__ __forceinline__ void fft_run(int nb, C<T>* u, C<T>* v, const C<T>* tw, OPEN&& open, FIN&& fin) {
  using P = FftPlan<N>;
  constexpr int NP = fft_padded<T>(N);
  C<T>* first = P::R2 > 1 ? u : v;
  fft_pass_first<T, N, SIGN, NT, PAD>(nb, open, [&](int b, int i, C<T> z) { first[b * NP + fft_pad<T>(i)] = z; });
  __syncthreads();
  if constexpr (P::R2 > 1) {
    fft_pass_tw<T, N, SIGN, NT, P::R1, P::R0>(u, tw, nb, [&](int b, int i, C<T> z) { v[b * NP + fft_pad<T>(i)] = z; });
    __syncthreads();
    fft_pass_tw<T, N, SIGN, NT, P::R2, P::R0 * P::R1>(v, tw, nb, fin);
  } else {
    fft_pass_tw<T, N, SIGN, NT, P::R1, P::R0>(v, tw, nb, fin);
  }
  __syncthreads();
}

// calls f(std::integral_constant<int, N>) for a length of the plans above
template <typename F>
cudaError_t fft_dispatch(int N, F&& f) {
  switch (N) {
#define SP_FFT_CASE(n) case n: return f(std::integral_constant<int, n>());
    SP_FFT_CASE(16) SP_FFT_CASE(24) SP_FFT_CASE(32) SP_FFT_CASE(48) SP_FFT_CASE(64) SP_FFT_CASE(96)
    SP_FFT_CASE(128) SP_FFT_CASE(192) SP_FFT_CASE(256) SP_FFT_CASE(384) SP_FFT_CASE(512) SP_FFT_CASE(768)
    SP_FFT_CASE(1024) SP_FFT_CASE(1536) SP_FFT_CASE(2048) SP_FFT_CASE(3072) SP_FFT_CASE(4096)
#undef SP_FFT_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace spectau
