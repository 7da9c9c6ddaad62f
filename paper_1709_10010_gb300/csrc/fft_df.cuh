// Complex operations and small DFTs of the double-float FFT passes.
//
// The generic code composes them from the accurate operators of df.cuh (20
// FP32 instructions an addition, 7 a product), every intermediate result
// renormalised.  Here a sum of products is formed at once: the leading products
// added with their exact errors (two-sum, FMA), the small terms summed in FP32,
// one renormalisation at the end, so fewer instructions and fewer roundings:
//
//   complex product        40 instructions, error 1.7e-15 (68, 1.9e-15)
//   sum                    11, 1.1e-15                    (20, 1.0e-15)
//   a + k b + l c          28                             (54)
//
// (rms error relative to the rms result, 4e5 random operands.)  Multiplications
// by +-1, +-i and 1/2 are sign changes and exact scalings.  The whole local part
// of H is no less accurate than with the composed operations: V psi of random
// bands and potentials against FP64, rms error relative to the result, 30: 8.0e-15
// (8.4e-15 composed), 48: 9.1e-15 (9.7e-15), 60: 1.09e-14 (1.17e-14), 90: 1.94e-14
// (1.94e-14), 144: 4.4e-14 (4.4e-14).  The plane pass of 128 bands on a 90^3 box:
// 6.54 -> 2.92 ms (with the coprime factorisation and blocks of 256 of
// fft_spec_impl.cuh), the z passes 0.83 -> 0.45 ms.
#pragma once
#include "df.cuh"
#include "fft_device.cuh"

namespace pwh {

// a + b: one FP32 rounding of the low parts' sum more than operator+ saves
__host__ __device__ __forceinline__ df df_sum(df a, df b) {
  float s, e;
  df_two_sum(a.hi, b.hi, s, e);
  e = df_add(e, df_add(a.lo, b.lo));
  df_fast_two_sum(s, e, s, e);
  return df(s, e);
}
// a b + c d
__host__ __device__ __forceinline__ df df_dot2(df a, df b, df c, df d) {
  const float p = df_mul(a.hi, b.hi), e = df_fma(a.hi, b.hi, -p);
  const float q = df_mul(c.hi, d.hi), g = df_fma(c.hi, d.hi, -q);
  float s, r;
  df_two_sum(p, q, s, r);
  float x = df_mul(a.hi, b.lo);
  x = df_fma(a.lo, b.hi, x);
  x = df_fma(c.hi, d.lo, x);
  x = df_fma(c.lo, d.hi, x);
  x = df_add(df_add(df_add(e, g), r), x);
  df_fast_two_sum(s, x, s, x);
  return df(s, x);
}
// z + a b + c d
__host__ __device__ __forceinline__ df df_dot3(df z, df a, df b, df c, df d) {
  const float p = df_mul(a.hi, b.hi), e = df_fma(a.hi, b.hi, -p);
  const float q = df_mul(c.hi, d.hi), g = df_fma(c.hi, d.hi, -q);
  float s, r, t, v;
  df_two_sum(p, q, s, r);
  df_two_sum(z.hi, s, t, v);
  float x = df_mul(a.hi, b.lo);
  x = df_fma(a.lo, b.hi, x);
  x = df_fma(c.hi, d.lo, x);
  x = df_fma(c.lo, d.hi, x);
  x = df_add(df_add(df_add(e, g), df_add(r, v)), df_add(x, z.lo));
  df_fast_two_sum(t, x, t, x);
  return df(t, x);
}

template <> __host__ __device__ __forceinline__ dfc add<df>(dfc a, dfc b) {
  return mk<df>(df_sum(a.x, b.x), df_sum(a.y, b.y));
}
template <> __host__ __device__ __forceinline__ dfc sub<df>(dfc a, dfc b) {
  return mk<df>(df_sum(a.x, -b.x), df_sum(a.y, -b.y));
}
template <> __host__ __device__ __forceinline__ dfc mul<df>(dfc a, dfc b) {
  return mk<df>(df_dot2(a.x, b.x, -a.y, b.y), df_dot2(a.x, b.y, a.y, b.x));
}

// z times +i or -i (sg = +-1)
__device__ __forceinline__ dfc df_rot(dfc z, bool plus) {
  return plus ? mk<df>(-z.y, z.x) : mk<df>(z.y, -z.x);
}

template <> __device__ __forceinline__ void dft<df, 3>(dfc* a, df sg) {
  const bool plus = sg.hi > 0.f;
  constexpr df s3(PWH_S3);
  const dfc t1 = add<df>(a[1], a[2]), d = sub<df>(a[1], a[2]);
  const dfc t2 = df_rot(mk<df>(d.x * s3, d.y * s3), plus);
  const dfc h = mk<df>(df(-0.5f * t1.x.hi, -0.5f * t1.x.lo), df(-0.5f * t1.y.hi, -0.5f * t1.y.lo));
  const dfc m = add<df>(a[0], h);
  a[0] = add<df>(a[0], t1);
  a[1] = add<df>(m, t2);
  a[2] = sub<df>(m, t2);
}
template <> __device__ __forceinline__ void dft<df, 4>(dfc* a, df sg) {
  const dfc s02 = add<df>(a[0], a[2]), d02 = sub<df>(a[0], a[2]);
  const dfc s13 = add<df>(a[1], a[3]), d13 = df_rot(sub<df>(a[1], a[3]), sg.hi > 0.f);
  a[0] = add<df>(s02, s13);
  a[2] = sub<df>(s02, s13);
  a[1] = add<df>(d02, d13);
  a[3] = sub<df>(d02, d13);
}
template <> __device__ __forceinline__ void dft<df, 5>(dfc* a, df sg) {
  const bool plus = sg.hi > 0.f;
  constexpr df ca(PWH_C5A), cb(PWH_C5B), sa(PWH_S5A), sb(PWH_S5B), nsa(-PWH_S5A);
  const dfc b1 = add<df>(a[1], a[4]), b2 = add<df>(a[2], a[3]);
  const dfc d1 = sub<df>(a[1], a[4]), d2 = sub<df>(a[2], a[3]);
  const dfc a0 = a[0];
  const dfc r1 = mk<df>(df_dot3(a0.x, b1.x, ca, b2.x, cb), df_dot3(a0.y, b1.y, ca, b2.y, cb));
  const dfc r2 = mk<df>(df_dot3(a0.x, b1.x, cb, b2.x, ca), df_dot3(a0.y, b1.y, cb, b2.y, ca));
  const dfc i1 = df_rot(mk<df>(df_dot2(d1.x, sa, d2.x, sb), df_dot2(d1.y, sa, d2.y, sb)), plus);
  const dfc i2 = df_rot(mk<df>(df_dot2(d1.x, sb, d2.x, nsa), df_dot2(d1.y, sb, d2.y, nsa)), plus);
  a[0] = add<df>(a0, add<df>(b1, b2));
  a[1] = add<df>(r1, i1);
  a[4] = sub<df>(r1, i1);
  a[2] = add<df>(r2, i2);
  a[3] = sub<df>(r2, i2);
}

// Double-float with the accurate operators only, for the compiled size whose
// transforms keep twiddles between their passes and would lose 7% of accuracy
// with the sums above (50 = 5 x 10; the coprime sizes have fewer products and
// gain accuracy).
struct dfa : df {
  using df::df;
  dfa() = default;
  __host__ __device__ constexpr dfa(df a) : df(a) {}
};
__host__ __device__ __forceinline__ dfa operator+(dfa a, dfa b) { return dfa((df)a + (df)b); }
__host__ __device__ __forceinline__ dfa operator-(dfa a) { return dfa(-(df)a); }
__host__ __device__ __forceinline__ dfa operator-(dfa a, dfa b) { return dfa((df)a - (df)b); }
__host__ __device__ __forceinline__ dfa operator*(dfa a, dfa b) { return dfa((df)a * (df)b); }
__host__ __device__ __forceinline__ dfa& operator*=(dfa& a, dfa b) { return a = a * b; }
struct dfac {
  dfa x, y;
};
template <> struct cplx<dfa> { using t = dfac; };

}  // namespace pwh
