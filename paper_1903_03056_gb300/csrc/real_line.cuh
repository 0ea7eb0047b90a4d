// Real line transforms in the registers of one thread.
//
// A line of N real values (N even) is one complex transform of N / 2 points plus a pass that
// joins (or splits) its even and odd samples.  The spectrum is kept in N / 2 complex values:
// entry 0 holds the two real modes, (X_0, X_{N/2}); entry k = 1..N/2-1 holds X_k; the rest is
// X_{N-k} = conj X_k.  Half the arithmetic and half the registers of a complex line.
#pragma once

#include "fft_line.cuh"
#include "simd2.cuh"

namespace dgfs {

template <typename T> __device__ __forceinline__ C<T> conj_(C<T> a) { return mk<T>(a.x, -a.y); }

// x * e^{2 pi i (A / B)}, A / B a compile-time fraction
template <typename T, int A, int B> __device__ __forceinline__ C<T> rot(C<T> x) { return twiddle<T, B, A, +1>(x); }

// inverse: Z_k = (X_k + conj X_{h-k}) + i w^k (X_k - conj X_{h-k}), w = e^{2 pi i / N}, h = N / 2,
// for the pair (K, h - K); X is replaced by Z
template <typename T, int N, int K>
__device__ __forceinline__ void c2r_join(C<T>* x) {
  constexpr int h = N / 2;
  if constexpr (2 * K < h) {
    const C<T> a = x[K], b = x[h - K];
    const C<T> s = mk<T>(a.x + b.x, a.y - b.y);
    const C<T> o = rot<T, 4 * K + N, 4 * N>(mk<T>(a.x - b.x, a.y + b.y));
    x[K] = add<T>(s, o);
    x[h - K] = mk<T>(s.x - o.x, o.y - s.y);
    c2r_join<T, N, K + 1>(x);
  } else if constexpr (2 * K == h) {
    x[K] = mk<T>(mulc(x[K].x, Const<T>(2)), mulc(x[K].y, Const<T>(-2)));
  }
}

// y[n] = sum_k X_k e^{2 pi i k n / N} (unnormalised, real): x holds X_1..X_{h-1} in entries 1..h-1
// and is destroyed; x0 = X_0, xh = X_{N/2}
template <typename T, int N>
__device__ __forceinline__ void c2r_line(C<T> (&x)[N / 2], T x0, T xh, T (&y)[N]) {
  x[0] = mk<T>(x0 + xh, x0 - xh);
  c2r_join<T, N, 1>(x);
  fft_line<T, N / 2, +1>(x);
#pragma unroll
  for (int n = 0; n < N / 2; ++n) {
    y[2 * n] = x[n].x;
    y[2 * n + 1] = x[n].y;
  }
}

// forward: X_k = (Z_k + conj Z_{h-k}) / 2 - i w^{-k} (Z_k - conj Z_{h-k}) / 2 for the pair (K, h - K)
template <typename T, int N, int K>
__device__ __forceinline__ void r2c_split(C<T>* x) {
  constexpr int h = N / 2;
  if constexpr (2 * K < h) {
    const C<T> a = x[K], b = conj_<T>(x[h - K]);
    const C<T> s = scale<T>(add<T>(a, b), T(0.5));
    const C<T> o = rot<T, 3 * N - 4 * K, 4 * N>(scale<T>(sub<T>(a, b), T(0.5)));
    x[K] = add<T>(s, o);
    x[h - K] = conj_<T>(sub<T>(s, o));
    r2c_split<T, N, K + 1>(x);
  } else if constexpr (2 * K == h) {
    x[K] = conj_<T>(x[K]);
  }
}

// X_k = sum_n y[n] e^{-2 pi i k n / N}, entry 0 = (X_0, X_{N/2})
template <typename T, int N>
__device__ __forceinline__ void r2c_line(const T (&y)[N], C<T> (&x)[N / 2]) {
#pragma unroll
  for (int n = 0; n < N / 2; ++n) x[n] = mk<T>(y[2 * n], y[2 * n + 1]);
  fft_line<T, N / 2, -1>(x);
  x[0] = mk<T>(x[0].x + x[0].y, x[0].x - x[0].y);
  r2c_split<T, N, 1>(x);
}

// Complex line of N values as two interleaved halves that run packed (FP32): the even and the odd
// samples are transforms of N / 2 points with the same twiddles, joined by
// X_k = E_k + w^k O_k, X_{k+h} = E_k - w^k O_k.  e[n] holds samples 2n (low halves) and 2n + 1.
template <int N, int DIR, int K>
__device__ __forceinline__ void eo_join(const C2 (&e)[N / 2], C<float> (&x)[N]) {
  constexpr int h = N / 2;
  if constexpr (K < h) {
    const float2 re = unpack2(e[K].x), im = unpack2(e[K].y);
    const float2 o = make_float2(re.y, im.y);
    if constexpr (K == 0) {
      x[0] = make_float2(re.x + o.x, im.x + o.y);
      x[h] = make_float2(re.x - o.x, im.x - o.y);
    } else if constexpr (4 * K == N) {
      x[K] = add_i<float, DIR>(make_float2(re.x, im.x), o);
      x[K + h] = add_i<float, -DIR>(make_float2(re.x, im.x), o);
    } else {
      constexpr float c = float(trig2pi(K, N, 0)), s = float(DIR * trig2pi(K, N, 1));
      x[K] = make_float2(fmaf(-s, o.y, fmaf(c, o.x, re.x)), fmaf(s, o.x, fmaf(c, o.y, im.x)));
      x[K + h] = make_float2(fmaf(s, o.y, fmaf(-c, o.x, re.x)), fmaf(-s, o.x, fmaf(-c, o.y, im.x)));
    }
    eo_join<N, DIR, K + 1>(e, x);
  }
}

// In-register transform of one complex line, packed in FP32 from 8 points on
template <typename T, int N, int DIR>
__device__ __forceinline__ void line_fft(C<T> (&x)[N]) {
  if constexpr (sizeof(T) == 4 && N >= 8) {
    C2 e[N / 2];
#pragma unroll
    for (int n = 0; n < N / 2; ++n) {
      e[n].x = pack2(x[2 * n].x, x[2 * n + 1].x);
      e[n].y = pack2(x[2 * n].y, x[2 * n + 1].y);
    }
    fft_stages<F2, N / 2, 1, DIR, RadixCode<T, N / 2>::value, 0>(e);
    eo_join<N, DIR, 0>(e, x);
  } else {
    fft_line<T, N, DIR>(x);
  }
}

}  // namespace dgfs
