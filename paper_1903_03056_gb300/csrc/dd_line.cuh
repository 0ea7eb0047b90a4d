// Line transforms that carry each value as an unevaluated sum of two (hi + lo), for the passes whose
// rounding every result keeps.
//
// B is float or F2 (two independent values).  A sum takes the exact rounding error of its leading parts
// along (Knuth's TwoSum, 8 operations); a product by a constant takes that of the leading product
// (one fused multiply-add) and the constant's own.  Nothing renormalises in between: lo stays a few
// units in the last place of hi over the stages of a line, so the result, hi + lo rounded once, is
// correct to about one rounding.
#pragma once

#include "real_line.cuh"

namespace dgfs {

template <typename B> struct DD {
  B hi, lo;
};
template <typename B> struct CDD {
  DD<B> x, y;
};
template <typename B> struct cplx_t<DD<B>> { using type = CDD<B>; };

// a constant as two floats
struct DDConst {
  float hi, lo;
  __host__ __device__ constexpr DDConst(double v) : hi(float(v)), lo(float(v - double(float(v)))) {}
  __host__ __device__ constexpr DDConst(float h, float l) : hi(h), lo(l) {}
  __host__ __device__ constexpr DDConst operator-() const { return DDConst(-hi, -lo); }
};
template <typename B> struct real_const<DD<B>> { using type = DDConst; };

// sums and products rounded on their own (never contracted into a multiply-add)
__device__ __forceinline__ float dd_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float dd_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float dd_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ F2 dd_add(F2 a, F2 b) { return a + b; }
__device__ __forceinline__ F2 dd_sub(F2 a, F2 b) { return a - b; }
__device__ __forceinline__ F2 dd_mul(F2 a, F2 b) { return a * b; }
__device__ __forceinline__ float dd_fma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ F2 dd_fma(F2 a, F2 b, F2 c) { return fma2(a, b, c); }
template <typename B> __device__ __forceinline__ B dd_const(float c);
template <> __device__ __forceinline__ float dd_const<float>(float c) { return c; }
template <> __device__ __forceinline__ F2 dd_const<F2>(float c) { return pack2(c, c); }

template <typename B> __device__ __forceinline__ DD<B> operator+(DD<B> a, DD<B> b) {
  const B s = dd_add(a.hi, b.hi), t = dd_sub(s, a.hi);
  const B e = dd_add(dd_sub(a.hi, dd_sub(s, t)), dd_sub(b.hi, t));
  return {s, dd_add(dd_add(a.lo, b.lo), e)};
}
template <typename B> __device__ __forceinline__ DD<B> operator-(DD<B> a, DD<B> b) {
  const B s = dd_sub(a.hi, b.hi), t = dd_sub(s, a.hi);
  const B e = dd_sub(dd_sub(a.hi, dd_sub(s, t)), dd_add(b.hi, t));
  return {s, dd_add(dd_sub(a.lo, b.lo), e)};
}
template <typename B> __device__ __forceinline__ DD<B> operator-(DD<B> a) { return {-a.hi, -a.lo}; }
template <typename B> __device__ __forceinline__ DD<B> mulc(DD<B> a, DDConst c) {
  const B ch = dd_const<B>(c.hi), cl = dd_const<B>(c.lo);
  const B p = dd_mul(a.hi, ch);
  return {p, dd_fma(a.hi, cl, dd_fma(a.lo, ch, dd_fma(a.hi, ch, -p)))};
}
template <typename B> __device__ __forceinline__ DD<B> fmac(DD<B> a, DDConst c, DD<B> b) { return mulc(a, c) + b; }

// DD of a value, and back (rounded once)
template <typename B> __device__ __forceinline__ DD<B> dd_of(B v) { return {v, dd_const<B>(0.0f)}; }
template <typename B> __device__ __forceinline__ CDD<B> dd_of(B x, B y) { return {dd_of(x), dd_of(y)}; }
template <typename B> __device__ __forceinline__ B dd_value(DD<B> a) { return dd_add(a.hi, a.lo); }

// line_fft with these sums, FP32: the even and odd samples packed, then joined
template <int N, int DIR, int K>
__device__ __forceinline__ void dd_join(const CDD<F2> (&e)[N / 2], float2 (&x)[N]) {
  constexpr int h = N / 2;
  if constexpr (K < h) {
    const float2 rh = unpack2(e[K].x.hi), rl = unpack2(e[K].x.lo), ih = unpack2(e[K].y.hi), il = unpack2(e[K].y.lo);
    const CDD<float> o = twiddle<DD<float>, N, K, DIR>(CDD<float>{{rh.y, rl.y}, {ih.y, il.y}});
    // (E + o, E - o) as one packed sum per component
    const DD<F2> ex = {pack2(rh.x, rh.x), pack2(rl.x, rl.x)}, ey = {pack2(ih.x, ih.x), pack2(il.x, il.x)};
    const DD<F2> ox = {pack2(o.x.hi, -o.x.hi), pack2(o.x.lo, -o.x.lo)}, oy = {pack2(o.y.hi, -o.y.hi), pack2(o.y.lo, -o.y.lo)};
    const float2 sx = unpack2(dd_value(ex + ox)), sy = unpack2(dd_value(ey + oy));
    x[K] = make_float2(sx.x, sy.x);
    x[K + h] = make_float2(sx.y, sy.y);
    dd_join<N, DIR, K + 1>(e, x);
  }
}
template <int N, int DIR>
__device__ __forceinline__ void dd_line_fft(float2 (&x)[N]) {
  CDD<F2> e[N / 2];
#pragma unroll
  for (int n = 0; n < N / 2; ++n) e[n] = dd_of(pack2(x[2 * n].x, x[2 * n + 1].x), pack2(x[2 * n].y, x[2 * n + 1].y));
  fft_stages<DD<F2>, N / 2, 1, DIR, RadixCode<float, N / 2>::value, 0>(e);
  dd_join<N, DIR, 0>(e, x);
}

}  // namespace dgfs
