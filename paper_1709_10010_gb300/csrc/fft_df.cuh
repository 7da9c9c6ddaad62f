// Complex operations and small DFTs of the double-float FFT passes.
//
// The generic code composes them from the operators of df.cuh (20 FP32
// instructions an addition, 7 a product), every intermediate result renormalised.
// Here a sum of products is formed at once: the leading products added with their
// exact errors (two-sum, FMA), the small terms summed in FP32, one renormalisation at
// the end, so fewer instructions and fewer roundings in a transform:
//
//   sum                    17 instructions, the composed result (20)
//   a b + c d              19, error 2.2e-15 (34, 1.8e-15)
//   z + a b + c d          26, error 2.3e-15 (54, 1.8e-15)
//
// (rms error relative to the rms result, 4e5 random operands; a sum's error is
// relative to the sum, also when it cancels, that of products relative to the
// products.)  Multiplications by +-1, +-i and 1/2 are sign changes and exact scalings.
//   A whole transform is more accurate than a composed one at every edge with coprime
// factors, which also saves the twiddles between the passes: rms error of a random
// one 30: -11%, 36: -11%, 40: -4%, 48: -8%, 60: -15%, 72: -7%, 80: -2%, 90: -7%, 120:
// -10%, 144: -2% (tests/test_df_transforms.py); V psi of random bands and potentials
// against FP64, 30: 7.5e-15 (8.4e-15 composed), 48: 8.7e-15 (9.7e-15), 90: 1.92e-14
// (1.94e-14), 144: 4.40e-14 (4.42e-14).  The FP64 local part of 64 bands, composed ->
// fused: 30 289 -> 100 us, 48 745 -> 507, 90 3.92 -> 2.56 ms, 120 10.4 -> 7.0, 144
// 23.6 -> 16.3.  (Sums that add the low parts in one rounding, 11 instructions,
// take 1.90 ms at 90 and 11.2 at 144, but lose the low parts under cancellation and
// raise the transform's error at 40, 72, 80 and 144.)
#pragma once
#include "df.cuh"
#include "fft_device.cuh"

namespace pwh {

// a + b.  Both the high and the low parts are added with their exact errors, so that
// the relative error stays below 2^-45 when the high parts cancel, as in operator+,
// whose second renormalisation is left out (3 of 20 instructions): |lo| is within
// 2^-24 |hi| + 2^-48 max(|a|, |b|).
__host__ __device__ __forceinline__ df df_sum(df a, df b) {
  float s, e, t, f;
  df_two_sum(a.hi, b.hi, s, e);
  df_two_sum(a.lo, b.lo, t, f);
  df_fast_two_sum(s, df_add(e, t), s, e);
  return df(s, df_add(e, f));
}
// a b + c d
__host__ __device__ __forceinline__ df df_dot2(df a, df b, df c, df d) {
  const float p = df_mul(a.hi, b.hi), e = df_fma(a.hi, b.hi, -p);
  const float q = df_mul(c.hi, d.hi), g = df_fma(c.hi, d.hi, -q);
  float s, r;
  df_two_sum(p, q, s, r);
  const float u = df_fma(a.lo, b.hi, df_fma(a.hi, b.lo, e));
  const float v = df_fma(c.lo, d.hi, df_fma(c.hi, d.lo, g));
  float x = df_add(df_add(u, v), r);
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
  const float u = df_fma(a.lo, b.hi, df_fma(a.hi, b.lo, e));
  const float w = df_fma(c.lo, d.hi, df_fma(c.hi, d.lo, g));
  float x = df_add(df_add(u, w), df_add(df_add(r, v), z.lo));
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
__host__ __device__ __forceinline__ dfc df_rot(dfc z, bool plus) {
  return plus ? mk<df>(-z.y, z.x) : mk<df>(z.y, -z.x);
}

template <> __host__ __device__ __forceinline__ void dft<df, 3>(dfc* a, df sg) {
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
template <> __host__ __device__ __forceinline__ void dft<df, 4>(dfc* a, df sg) {
  const dfc s02 = add<df>(a[0], a[2]), d02 = sub<df>(a[0], a[2]);
  const dfc s13 = add<df>(a[1], a[3]), d13 = df_rot(sub<df>(a[1], a[3]), sg.hi > 0.f);
  a[0] = add<df>(s02, s13);
  a[2] = sub<df>(s02, s13);
  a[1] = add<df>(d02, d13);
  a[3] = sub<df>(d02, d13);
}
template <> __host__ __device__ __forceinline__ void dft<df, 5>(dfc* a, df sg) {
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

// Double-float with the composed operators only, for the compiled edges without
// coprime factors (50 and 96).
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
