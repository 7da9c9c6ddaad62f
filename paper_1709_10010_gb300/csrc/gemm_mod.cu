// FP64-equivalent complex GEMM on the BF16 tensor cores by residues (Ozaki,
// Uchino and Imamura, "Ozaki Scheme II", 2025: an integer product through the
// Chinese remainder theorem): the operands are rounded to integers, the
// integer product is formed exactly modulo kMod pairwise coprime numbers of at
// most eight bits, and rebuilt from its residues.
//
//   C = alpha op(A) B + beta C.  Column j of B (and row i of op(A)) gets the
//   exponent e with 2-norm <= 2^e over the whole K and becomes the integers
//   X = round(x 2^(kT - e)), |X| <= 2^kT.  By Cauchy and Schwarz each real and
//   imaginary part of the integer product is below 2^(2 kT) < P / 2, P the
//   product of the moduli, so its residues determine it.  In A^H B, whose real
//   products keep real and imaginary parts apart, a column whose parts differ in norm
//   by more than 2^kPartGap gets an exponent for each, so that the smaller keeps its
//   bits; the real products then are rebuilt one by one.  The only errors are
//   the rounding to X (relative to |a| |b|: 2^-kT, 62 bits) and the final
//   FP64 rounding (the value within 2^-61, rounded once): no product of slices
//   is dropped, and the exponents follow the rows' norms, not their largest
//   elements.
//
// Work: 16 real BF16 products against the 36 of the integer-slice form (pairs
// of base-128 digits) that this replaced, and one byte a modulus of partial
// results instead of 36 FP32 partials per 4,096 of K.  Measured, a basis of
// 1088 columns over 161,235 plane waves: A^H B with 544 columns and A B onto 544
// columns together 28.2 ms, against 57.4 ms (12.6 and 15.4 ms; tensor pipe of the
// residue GEMMs 61-70% busy).
//
// Kernels: row and column norms; residues of the operands (BF16, K-major, one
// plane a modulus); k_mod_gemm, one persistent pair of CTAs per two SMs; the
// reconstruction.
#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "gemm.cuh"
#include "gemm_mod_geom.cuh"
#include "pair_ring.cuh"
#include "tc_ptx.cuh"

namespace pwh {

// ------------------------------------------------------------- the moduli ----
constexpr int kT = 62;  // operands are integers of 2-norm at most 2^kT
constexpr int kDigits = 6;
constexpr int kPartGap = 4;
struct ModTab {
  int p[kMod];
  // 2^16, 2^32 and 2^48 mod p, symmetric: the weights of X's 16-bit limbs
  float c1[kMod], c2[kMod], c3[kMod], inv[kMod];
  // (P/p)^-1 mod p over p as a 108-bit fraction, V / P = sum r_i K_i mod 1: its
  // 18-bit digits, leading first
  int k[kMod][kDigits];
  unsigned long long ph;  // P 2^-kPShift, rounded: in [2^63, 2^64)
};
constexpr int kPShift = 62;
constexpr ModTab make_mod_tab() {
  ModTab t{};
  const int p[kMod] = {256, 255, 253, 251, 247, 241, 239, 233,
                       229, 227, 223, 217, 211, 199, 197, 193};
  unsigned __int128 P = 1;  // 2^125.37
  for (int i = 0; i < kMod; ++i) {
    t.p[i] = p[i];
    P *= (unsigned)p[i];
    long long w = 1 << 16;
    auto sym = [&](long long v) {
      v %= p[i];
      return (float)(v > p[i] / 2 ? v - p[i] : v);
    };
    t.c1[i] = sym(w);
    t.c2[i] = sym((w % p[i]) * (w % p[i]));
    t.c3[i] = sym((w % p[i]) * (w % p[i]) % p[i] * (w % p[i]));
    t.inv[i] = 1.0f / (float)p[i];
    long long rest = 1;
    for (int j = 0; j < kMod; ++j)
      if (j != i) rest = rest * p[j] % p[i];
    long long iv = 1;
    while (rest * iv % p[i] != 1) ++iv;
    // iv 2^108 / p by long division
    long long rem = iv;
    for (int k = 0; k < kDigits; ++k) {
      rem <<= 18;
      t.k[i][k] = (int)(rem / p[i]);
      rem %= p[i];
    }
  }
  t.ph = (unsigned long long)((P + ((unsigned __int128)1 << (kPShift - 1))) >> kPShift);
  return t;
}
constexpr ModTab kTab = make_mod_tab();
static_assert(kTab.ph >> 63, "P 2^-kPShift has 64 bits");
__constant__ float c_mod_p[kMod] = {256, 255, 253, 251, 247, 241, 239, 233,
                                    229, 227, 223, 217, 211, 199, 197, 193};
constexpr float kMagic = 12582912.f;  // 1.5 2^23: adding it rounds to an integer
constexpr int kNonfinite = 0x7fffffff;  // exponent of a row with an infinity or NaN

// x mod p, symmetric and exact for integers |x| < 2^24 (|result| <= 0.51 p)
__device__ __forceinline__ float mod_sym(float x, float p, float inv) {
  const float q = fmaf(x, inv, kMagic) - kMagic;
  return fmaf(-p, q, x);
}

// ------------------------------------------------------------ row norms ----
// A partial sum of squares, sum x^2 = s 2^(2 (E - 1023)): E the largest biased
// exponent seen (that of the leading bit for a subnormal), s in FP32 from the
// 20 leading fraction bits (integer operations: conversions from FP64 issue on
// the narrow FP64 pipe).
struct NormAcc {
  int E = -100000;
  float s = 0.f;
  __device__ __forceinline__ void rescale(int En) {
    const int d = 2 * (E - En);  // <= 0
    s = d < -120 ? 0.f : s * __uint_as_float((unsigned)(127 + d) << 23);
    E = En;
  }
  __device__ __forceinline__ void add(double x) {
    const int h = __double2hiint(x) & 0x7fffffff;
    if (h < (1 << 20)) {  // zero or subnormal
      const unsigned l = (unsigned)__double2loint(x);
      const unsigned long long m = ((unsigned long long)h << 32) | l;
      if (m) {
        const int hb = 63 - __clzll((long long)m);  // x < 2^(hb + 1 - 1074)
        merge(hb + 1 - 51, 1.f);
      }
      return;
    }
    if ((h >> 20) > E) rescale(h >> 20);
    const int t = h - ((E - 127) << 20);  // exponent relative to E, FP32 bias
    const float f = t > 0 ? __uint_as_float((unsigned)t << 3) : 0.f;
    s = fmaf(f, f, s);
  }
  __device__ __forceinline__ void merge(int E2, float s2) {
    if (E2 > E) rescale(E2);
    const int d = 2 * (E2 - E);
    s += d < -120 ? 0.f : s2 * __uint_as_float((unsigned)(127 + d) << 23);
  }
};

// Real and imaginary parts c of column j of X (K x J, ld) split over gridDim.y
// blocks: partial (2 j + c) gridDim.y + y.
__global__ void __launch_bounds__(256) k_mod_colnorm(const double2* __restrict__ X, int64_t ld, int K,
                                                     int2* __restrict__ part) {
  __shared__ int2 red[2][8];
  const int j = blockIdx.x;
  const double2* x = X + (size_t)j * ld;
  NormAcc a[2];
  for (int k = blockIdx.y * 256 + threadIdx.x; k < K; k += gridDim.y * 256) {
    const double2 v = x[k];
    a[0].add(v.x);
    a[1].add(v.y);
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    for (int o = 16; o > 0; o >>= 1) {
      const int E2 = __shfl_down_sync(0xffffffffu, a[c].E, o);
      const float s2 = __shfl_down_sync(0xffffffffu, a[c].s, o);
      a[c].merge(E2, s2);
    }
    if ((threadIdx.x & 31) == 0) red[c][threadIdx.x >> 5] = make_int2(a[c].E, __float_as_int(a[c].s));
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    const int c = threadIdx.x;
    NormAcc t;
    for (int w = 0; w < 8; ++w) t.merge(red[c][w].x, __int_as_float(red[c][w].y));
    part[(2 * (size_t)j + c) * gridDim.y + blockIdx.y] = make_int2(t.E, __float_as_int(t.s));
  }
}
// Rows m of A (M x K, ld), columns split over gridDim.y blocks.
__global__ void __launch_bounds__(256) k_mod_rownorm(const double2* __restrict__ A, int64_t ld, int M,
                                                     int K, int2* __restrict__ part) {
  const int m = blockIdx.x * 256 + threadIdx.x;
  if (m >= M) return;
  NormAcc a;
  const int per = (K + gridDim.y - 1) / gridDim.y;
  const int k1 = min(K, (int)(blockIdx.y + 1) * per);
#pragma unroll 4
  for (int k = blockIdx.y * per; k < k1; ++k) {
    const double2 v = A[(size_t)k * ld + m];
    a.add(v.x);
    a.add(v.y);
  }
  part[(size_t)m * gridDim.y + blockIdx.y] = make_int2(a.E, __float_as_int(a.s));
}
// e with norm <= 2^e
__device__ __forceinline__ int mod_exp(const NormAcc& a) {
  if (a.E == 0x7ff) return kNonfinite;
  if (!(a.s > 0.f)) return 0;
  // s (1 + 1e-3) < 2^q covers the truncated fractions and the FP32 sum
  int q;
  frexpf(a.s * 1.001f, &q);
  return a.E - 1023 + ((q + 1) >> 1);
}
// Exponents from the partials of the rows of A (na of them; parts = 1: one each)
// and the columns of B (nb); parts = 2: two each, real and imaginary part, equal
// (the norm of both) unless `apart` and the parts are further apart than kPartGap.
__global__ void k_mod_exp(const int2* __restrict__ pa, int na, int Sa, int parts_a,
                          const int2* __restrict__ pb, int nb, int Sb, bool apart,
                          int* __restrict__ exa, int* __restrict__ exb) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= na + nb) return;
  const int S = i < na ? Sa : Sb, parts = i < na ? parts_a : 2;
  const int2* p = i < na ? pa + (size_t)i * S * parts : pb + (size_t)(i - na) * S * parts;
  int* ex = i < na ? exa + (size_t)i * parts : exb + 2 * (size_t)(i - na);
  NormAcc a;
  for (int k = 0; k < S; ++k) a.merge(p[k].x, __int_as_float(p[k].y));
  if (parts == 1) {
    ex[0] = mod_exp(a);
    return;
  }
  NormAcc b;
  for (int k = S; k < 2 * S; ++k) b.merge(p[k].x, __int_as_float(p[k].y));
  const int e0 = mod_exp(a), e1 = mod_exp(b);
  const bool two = apart && a.s > 0.f && b.s > 0.f && e0 != kNonfinite && e1 != kNonfinite &&
                   abs(e0 - e1) > kPartGap;
  a.merge(b.E, b.s);
  const int e = mod_exp(a);
  ex[0] = two ? e0 : e;
  ex[1] = two ? e1 : e;
}

// ---------------------------------------------------------------- residues ----
// X = round(x 2^(kT - e)) as four balanced 16-bit limbs, exact in FP32.
__device__ __forceinline__ void mod_limbs(double x, int e, float* l) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int eb = (int)((bits >> 52) & 0x7ff);
  const unsigned long long m = (bits & 0xfffffffffffffull) | (eb ? (1ull << 52) : 0ull);
  const int sh = (eb ? eb : 1) - 1075 + kT - e;  // X = m 2^sh
  long long X;
  if (e == kNonfinite) X = 0;
  else if (sh >= 0) X = (long long)(m << min(sh, 63));
  else if (sh > -64) X = (long long)((m + (1ull << (-sh - 1))) >> (-sh));
  else X = 0;
  if (bits >> 63) X = -X;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int d = (int)(short)(X & 0xffff);
    l[k] = __int_as_float(0x4B400000 + d) - kMagic;
    X = (X - d) >> 16;
  }
  l[3] = __int_as_float(0x4B400000 + (int)X) - kMagic;
}
// X mod p_i, symmetric, |.| <= 130: three limb products (|sum| < 1.1e7, exact)
template <int I> __device__ __forceinline__ float mod_res(const float* l) {
  constexpr float p = (float)kTab.p[I], inv = kTab.inv[I];
  constexpr float c1 = kTab.c1[I], c2 = kTab.c2[I], c3 = kTab.c3[I];
  return mod_sym(fmaf(l[3], c3, fmaf(l[2], c2, fmaf(l[1], c1, l[0]))), p, inv);
}
// four residues, first reduced to |.| <= p / 2, as signed bytes (128 and -128 of
// p = 256 are the same byte)
__device__ __forceinline__ unsigned pack_res(const float* x, float p) {
  const float top = 0.5f * (p - 1.f);
  unsigned b[4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
    b[u] = __float_as_uint((x[u] > top ? x[u] - p : x[u] < -top ? x[u] + p : x[u]) + kMagic);
  return __byte_perm(__byte_perm(b[0], b[1], 0x0040), __byte_perm(b[2], b[3], 0x0040), 0x5410);
}
// two small integers as BF16 (their FP32 patterns have 16 zero trailing bits)
__device__ __forceinline__ unsigned pack_bf16(float a, float b) {
  return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
}
template <int I, int E = kMod, class F> __device__ __forceinline__ void each_mod(F f) {
  if constexpr (I < E) {
    f(std::integral_constant<int, I>{});
    each_mod<I + 1, E>(f);
  }
}

// Rows 2j (real parts) and 2j+1 (imaginary parts), columns k, of the operand
// whose row pair j is column j of X (zero for K <= k < seg); plane i holds the
// residues mod p_i.  Four K positions a thread: 8-byte stores, 256 bytes a
// warp and row.  Bound by the FP32 pipes (6.5 operations a residue) and the
// 64 bytes written per 16 read.
__global__ void __launch_bounds__(256) k_mod_slice_cols(const double2* __restrict__ X, int64_t ld, int K,
                                                        int seg, const int* __restrict__ ex,
                                                        __nv_bfloat16* __restrict__ out,
                                                        int64_t plane) {
  const int j = blockIdx.y;
  const int k = 4 * (blockIdx.x * 256 + threadIdx.x);
  if (k >= seg) return;
  const double2* x = X + (size_t)j * ld;
  const int er = ex[2 * j], ei = ex[2 * j + 1];
  float lr[4][4], li[4][4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const double2 v = k + u < K ? x[k + u] : make_double2(0.0, 0.0);
    mod_limbs(v.x, er, lr[u]);
    mod_limbs(v.y, ei, li[u]);
  }
  char* o = (char*)(out + (size_t)(2 * j) * seg + k);
  each_mod<0>([&](auto I) {
    constexpr int i = decltype(I)::value;
    uint2 r, q;
    r.x = pack_bf16(mod_res<i>(lr[0]), mod_res<i>(lr[1]));
    r.y = pack_bf16(mod_res<i>(lr[2]), mod_res<i>(lr[3]));
    q.x = pack_bf16(mod_res<i>(li[0]), mod_res<i>(li[1]));
    q.y = pack_bf16(mod_res<i>(li[2]), mod_res<i>(li[3]));
    *(uint2*)(o + (size_t)i * plane * 2) = r;
    *(uint2*)(o + (size_t)i * plane * 2 + (size_t)seg * 2) = q;
  });
}

// Row m, columns 2k + c = (Re, Im) A[m][k] (zero for 2K <= 2k + c < seg): 32 x
// 32 tiles transposed through shared memory, two k a thread.
__global__ void __launch_bounds__(256) k_mod_slice_rows(const double2* __restrict__ A, int64_t ld, int M,
                                                        int K, int seg, const int* __restrict__ ex,
                                                        __nv_bfloat16* __restrict__ out,
                                                        int64_t plane) {
  __shared__ double2 tile[32][33];
  const int m0 = blockIdx.x * 32, k0 = blockIdx.y * 32;
  for (int t = threadIdx.x; t < 1024; t += 256) {
    const int mm = t & 31, kk = t >> 5;
    const int m = m0 + mm, k = k0 + kk;
    tile[kk][mm] = (m < M && k < K) ? A[(size_t)k * ld + m] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 512; t += 256) {
    const int kk = 2 * (t & 15), mm = t >> 4;
    const int m = m0 + mm, k = k0 + kk;
    if (m >= M || 2 * k >= seg) continue;
    const double2 v = tile[kk][mm], w = tile[kk + 1][mm];
    const int e = ex[m];
    float l[4][4];
    mod_limbs(v.x, e, l[0]);
    mod_limbs(v.y, e, l[1]);
    mod_limbs(w.x, e, l[2]);
    mod_limbs(w.y, e, l[3]);
    char* o = (char*)(out + (size_t)m * seg + 2 * k);
    each_mod<0>([&](auto I) {
      constexpr int i = decltype(I)::value;
      *(uint2*)(o + (size_t)i * plane * 2) =
          make_uint2(pack_bf16(mod_res<i>(l[0]), mod_res<i>(l[1])),
                     pack_bf16(mod_res<i>(l[2]), mod_res<i>(l[3])));
    });
  }
}

// B operand of op(A) = A, rows 2n and 2n+1 of B[k][n]:
//     B2[2n][2k] = Re, B2[2n][2k+1] = -Im, B2[2n+1][2k] = Im, B2[2n+1][2k+1] = Re
__global__ void __launch_bounds__(256) k_mod_slice_b2(const double2* __restrict__ B, int64_t ld, int K,
                                                      int seg, const int* __restrict__ ex,
                                                      __nv_bfloat16* __restrict__ out, int64_t plane) {
  const int n = blockIdx.y;
  const int k = blockIdx.x * 256 + threadIdx.x;
  if (2 * k >= seg) return;
  const double2 v = k < K ? B[(size_t)n * ld + k] : make_double2(0.0, 0.0);
  const int e = ex[2 * n];
  float lr[4], li[4];
  mod_limbs(v.x, e, lr);
  mod_limbs(v.y, e, li);
  char* o = (char*)(out + (size_t)(2 * n) * seg + 2 * k);
  each_mod<0>([&](auto I) {
    constexpr int i = decltype(I)::value;
    const float re = mod_res<i>(lr), im = mod_res<i>(li);
    *(unsigned*)(o + (size_t)i * plane * 2) = pack_bf16(re, -im);
    *(unsigned*)(o + (size_t)i * plane * 2 + (size_t)seg * 2) = pack_bf16(im, re);
  });
}

// --------------------------------------------------------------- the GEMM ----
// A pair of CTAs (cta_group::2, one cluster) forms a 256 x bn tile: each CTA
// loads its 128 rows of A and its half of the bn rows of B, two thirds of the
// shared-memory fill and reads of a 128 x 256 tile a CTA.  Roles per CTA: warps 0-7 the epilogue (warp w: TMEM lanes 32 (w
// mod 4).., column half w / 4), warp 8 the TMA producer, warp 9 of CTA 0 the
// MMA issuer.
//   A K range runs in chunks of kChunkKb stages (960 of K: 960 * 130^2 + 131 <
//   2^24, so the FP32 sums of a chunk are exact integers) into alternating
//   accumulators; the epilogue adds each chunk to its running residue (four
//   FP32 operations an element, 1.3k clocks of the chunk's 7.7k of MMA) in
//   registers, and stores one byte an element at the end.
constexpr int kPairThreads = 320;
constexpr int kPairStages = 6;
constexpr int kPairABytes = 128 * TC_BK * 2;
constexpr int kPairStageBytes = 2 * kPairABytes;  // A half and (at most) 128 rows of B
constexpr int kPairSmem = kPairStages * kPairStageBytes + 1024 + 256;
constexpr int kChunkKb = 15;

struct ModArgs {
  int Mr, Nr;        // rows of A and of B, per modulus plane
  int bn;            // tile width: a multiple of 32, at most 256
  int gm, gn, gz;    // tiles and K ranges
  int kb_total, kb_per;  // 64-wide K blocks, and a K range's share
  int accum;         // add to the residues of the earlier K segments
  int64_t Np;        // output pitch (bytes): gn bn
  unsigned char* out;  // [z][modulus][m][n]
  int* err;
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_to_cta0(uint32_t saddr) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(0));
  return r;
}
__device__ __forceinline__ void pair_sync() {
  asm volatile(
      "barrier.cluster.arrive.release.aligned;\n"
      "barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// TMA load into this CTA's shared memory that completes on an mbarrier of the
// pair (bar: shared::cluster address)
__device__ __forceinline__ void tma_load_pair(void* dst, const CUtensorMap* map, int x, int y,
                                              uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(su32(dst)),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void mma_bf16_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                              uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum)
      : "memory");
}
// arrive on this mbarrier in both CTAs once the MMAs issued so far are done
__device__ __forceinline__ void mma_commit_pair(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;" ::"r"(su32(bar)),
      "h"((uint16_t)3)
      : "memory");
}
// arrive on this CTA's mbarrier once the MMAs issued so far are done
__device__ __forceinline__ void mma_commit_pair_own(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   su32(bar))
               : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
    k_mod_gemm(const __grid_constant__ CUtensorMap tma_a, const __grid_constant__ CUtensorMap tma_b,
               ModArgs args) {
  extern __shared__ __align__(1024) uint8_t mod_smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)mod_smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + kPairStages * kPairStageBytes);  // CTA 0's is used
  uint64_t* empty = full + kPairStages;
  uint64_t* tfull = empty + kPairStages;  // [2]
  uint64_t* tempty = tfull + 2;           // [2], CTA 0's is used
  uint64_t* quiet = tempty + 2;           // CTA 0's: the MMAs after a time-out are done
  uint32_t* tmem_slot = (uint32_t*)(quiet + 1);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  volatile int* fills1 = abort_flag + 1;  // CTA 0's: slots that CTA 1 filled

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int pair = blockIdx.x >> 1, npair = gridDim.x >> 1;
  const int tiles = args.gm * args.gn, items = tiles * args.gz * kMod;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kPairStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 16);  // eight epilogue warps in each CTA
    }
    mbar_init(quiet, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  pair_sync();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // item -> modulus (slowest), K range, M tile, N tile (fastest): the pairs
  // work on one or two moduli at a time, whose operand planes they share in L2
  int issued = 0;  // producer: ring slots whose loads were started
  if (warp == 8 && lane == 0) {
    const int bytes = 2 * (kPairABytes + (args.bn / 2) * TC_BK * 2);  // both CTAs' loads
    for (int it = pair; it < items; it += npair) {
      const int mod = it / (tiles * args.gz), rz = it - mod * (tiles * args.gz);
      const int z = rz / tiles, rem = rz - z * tiles;
      const int ya = mod * args.Mr + (rem / args.gn) * 256 + (int)rank * 128;
      const int yb = mod * args.Nr + (rem % args.gn) * args.bn + (int)rank * (args.bn / 2);
      const int kb0 = z * args.kb_per, kb_end = min(args.kb_total, kb0 + args.kb_per);
      bool ok = true;
      for (int kb = kb0; kb < kb_end; ++kb) {
        const int s = issued % kPairStages;
        if (!mbar_wait(&empty[s], ((issued / kPairStages) & 1) ^ 1, abort_flag)) {
          *abort_flag = 1;
          ok = false;
          break;
        }
        uint8_t* sa = smem + s * kPairStageBytes;
        if (rank == 0) mbar_expect_tx(&full[s], bytes);
        const uint32_t bar = map_to_cta0(su32(&full[s]));
        tma_load_pair(sa, &tma_a, kb * TC_BK, ya, bar);
        tma_load_pair(sa + kPairABytes, &tma_b, kb * TC_BK, yb, bar);
        ++issued;
      }
      if (!ok) break;
    }
  } else if (warp == 9 && lane == 0 && rank == 0) {
    const uint32_t idesc = idesc_bf16(256, args.bn);
    int used = 0, lc = 0;  // ring slots consumed, chunks of this pair
    bool ok = true;
    for (int it = pair; it < items && ok; it += npair) {
      const int rz = it % (tiles * args.gz);
      const int kb0 = (rz / tiles) * args.kb_per, kb_end = min(args.kb_total, kb0 + args.kb_per);
      for (int kc = kb0; kc < kb_end && ok; kc += kChunkKb, ++lc) {
        const int buf = lc & 1;
        if (!mbar_wait(&tempty[buf], ((lc >> 1) & 1) ^ 1, abort_flag)) {
          *abort_flag = 1;
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t dst = tmem + (uint32_t)(buf * 256);
        const int ke = min(kb_end, kc + kChunkKb);
        for (int kb = kc; kb < ke; ++kb, ++used) {
          const int s = used % kPairStages;
          if (!mbar_wait(&full[s], (used / kPairStages) & 1, abort_flag)) {
            *abort_flag = 1;
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a0 = su32(smem + s * kPairStageBytes);
          const uint32_t b0 = a0 + kPairABytes;
#pragma unroll
          for (int k = 0; k < TC_BK / 16; ++k)
            mma_bf16_pair(dst, smem_desc(a0 + k * 32), smem_desc(b0 + k * 32), idesc,
                          (kb > kc || k > 0) ? 1u : 0u);
          mma_commit_pair(&empty[s]);
        }
        if (ok) mma_commit_pair(&tfull[buf]);
      }
    }
    if (!ok) {
      // no epilogue waits for the last MMAs: they read shared and write tensor memory
      mma_commit_pair_own(quiet);
      mbar_wait(quiet, 0, nullptr);
    }
  } else if (warp < 8) {
    const int sub = warp & 3, half = warp >> 2;
    // columns of this warp: the first 128 of the tile or the others
    const int hn = half ? args.bn - 128 : min(128, args.bn);
    const uint32_t tempty0 = map_to_cta0(su32(&tempty[0]));
    int lc = 0;
    bool ok = true;
    for (int it = pair; it < items && ok; it += npair) {
      const int mod = it / (tiles * args.gz), rz = it - mod * (tiles * args.gz);
      const int z = rz / tiles, rem = rz - z * tiles;
      const int m = (rem / args.gn) * 256 + (int)rank * 128 + sub * 32 + lane;
      const int n0 = (rem % args.gn) * args.bn + half * 128;
      const int kb0 = z * args.kb_per, kb_end = min(args.kb_total, kb0 + args.kb_per);
      const float p = c_mod_p[mod], inv = 1.f / p;
      // this thread's residues, one byte each, a row's columns side by side: 16-byte
      // accesses (a byte store a column, with the rows of a warp side by side, took
      // 45k clocks a tile, more than a short K's MMAs)
      unsigned char* o = args.out + (((size_t)z * kMod + mod) * args.Mr + m) * args.Np + n0;
      float acc[128];
#pragma unroll
      for (int j = 0; j < 128; ++j) acc[j] = 0.f;
      if (args.accum && m < args.Mr) {
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          if (c * 16 < hn) {
            const uint4 w = *(const uint4*)(o + c * 16);
            const unsigned v[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int u = 0; u < 16; ++u) acc[c * 16 + u] = (float)(signed char)(v[u / 4] >> (8 * (u % 4)));
          }
        }
      }
      for (int kc = kb0; kc < kb_end; kc += kChunkKb, ++lc) {
        const int buf = lc & 1;
        if (!mbar_wait(&tfull[buf], (lc >> 1) & 1, abort_flag)) {
          *abort_flag = 1;
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t src = tmem + ((uint32_t)(sub * 32) << 16) + (uint32_t)(buf * 256 + half * 128);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (c * 32 < hn) {
            float v[32];
            tmem_ld32(src + c * 32, v);
#pragma unroll
            for (int j = 0; j < 32; ++j) acc[c * 32 + j] = mod_sym(acc[c * 32 + j] + v[j], p, inv);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(tempty0 + (uint32_t)(buf * sizeof(uint64_t)));
      }
      if (!ok) break;
      if (m < args.Mr) {
        const float top = 0.5f * (p - 1.f);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          if (c * 16 < hn) {
            unsigned w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              unsigned b[4];
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                const float x = acc[c * 16 + q * 4 + u];
                b[u] = __float_as_uint((x > top ? x - p : x < -top ? x + p : x) + kMagic);
              }
              w[q] = __byte_perm(__byte_perm(b[0], b[1], 0x0040), __byte_perm(b[2], b[3], 0x0040),
                                 0x5410);
            }
            *(uint4*)(o + c * 16) = make_uint4(w[0], w[1], w[2], w[3]);
          }
        }
      }
    }
  }
  __syncwarp();
  // Shared memory goes away only after everything that comes in from outside the
  // thread has landed.  Each producer: the MMA issuer's releases of its last slots (none
  // come after a time-out, the flag then ends the wait).  CTA 0's: the copies of both
  // CTAs, whose counts differ after a time-out (pair_drain).
  if (warp == 8 && lane == 0) {
    for (int j = max(0, issued - kPairStages); j < issued; ++j)
      if (!mbar_wait(&empty[j % kPairStages], (j / kPairStages) & 1, abort_flag)) break;
    if (rank == 1)
      asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(map_to_cta0(su32((const void*)fills1))),
                   "r"(issued)
                   : "memory");
  }
  __syncwarp();
  pair_sync();
  if (warp == 8 && lane == 0 && rank == 0) {
    const PairDrain d = pair_drain(issued, *fills1, kPairStages);
    const int bytes = kPairABytes + (args.bn / 2) * TC_BK * 2;  // one CTA's loads
    for (int j = d.arm0; j < d.arm1; ++j) mbar_expect_tx(&full[j % kPairStages], bytes);
    for (int j = d.wait0; j < d.wait1; ++j)
      mbar_wait(&full[j % kPairStages], (j / kPairStages) & 1, nullptr);
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) atomicExch(args.err, (int)PWH_ERR_TIMEOUT);
  pair_sync();
  if (warp == 8) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512)
                 : "memory");
  }
}

// ---------------------------------------------------------- reconstruction ----
// V / P as a fraction (mod 1): the symmetric residues times the 18-bit digits of the
// constants, in 32-bit multiply-adds (16 residues of at most 256, the sum of two:
// below 2^31; 64-bit multiply-adds on 31-bit digits ran at a quarter of their rate),
// then carried into a 96-bit fraction.  Residues of several K ranges are added modulo
// p first, and those of two products added as they are: a product that is zero has
// residues that are all zero.  The fraction is off by at most 2^-95, which with P < 2^126
// and integers of at least half 2^kT is 2^-91 of |a| |b|: products of integers come out
// exact up to where |a| |b| passes 2^37 times the result (2^21 with five digits).
struct CrtDigits {
  int d[kDigits] = {0, 0, 0, 0, 0, 0};
  template <int I> __device__ __forceinline__ void add(int r) {
    constexpr int k0 = kTab.k[I][0], k1 = kTab.k[I][1], k2 = kTab.k[I][2], k3 = kTab.k[I][3],
                  k4 = kTab.k[I][4], k5 = kTab.k[I][5];
    d[0] += r * k0;
    d[1] += r * k1;
    d[2] += r * k2;
    d[3] += r * k3;
    d[4] += r * k4;
    d[5] += r * k5;
  }
};
struct CrtFrac {
  unsigned long long h;  // leading 64 bits
  unsigned l;            // 32 more
  unsigned exact;        // 1 when nothing was cut off below them
  __device__ __forceinline__ void set(const CrtDigits& c) {
    constexpr int M = (1 << 18) - 1;
    const int t4 = c.d[4] + (c.d[5] >> 18), t3 = c.d[3] + (t4 >> 18), t2 = c.d[2] + (t3 >> 18),
              t1 = c.d[1] + (t2 >> 18), t0 = c.d[0] + (t1 >> 18);
    const unsigned d1 = t1 & M, d2 = t2 & M, d3 = t3 & M, d4 = t4 & M, d5 = c.d[5] & M;
    const unsigned hi = ((unsigned)t0 << 14) | (d1 >> 4);
    const unsigned lo = (d1 << 28) | (d2 << 10) | (d3 >> 8);
    h = ((unsigned long long)hi << 32) | lo;
    l = (d3 << 24) | (d4 << 6) | (d5 >> 12);
    exact = (d5 & 0xfff) == 0 ? 1u : 0u;
  }
  // the signed value times 2^(ea + eb - 2 kT), rounded once: the truncations
  // below add up to less than 2^-61 of it
  __device__ __forceinline__ double value(int ea, int eb) const {
    const bool neg = (long long)h < 0;
    // the magnitude cut off, so that opposite values have the same bits
    const unsigned lx = neg ? ~l + exact : l;
    const unsigned long long hx = neg ? ~h + (l == 0 ? exact : 0u) : h;
    if (hx == 0 && lx == 0) return 0.0;
    int s;
    unsigned long long w;
    if (hx == 0) {
      s = 64 + __clz(lx);
      w = (unsigned long long)lx << (32 + __clz(lx));
    } else {
      s = __clzll((long long)hx);
      w = s ? (hx << s) | (((unsigned long long)lx << 32) >> (64 - s)) : hx;
    }
    // |V| = w 2^(-64 - s) P = (w ph 2^-64) 2^(kPShift - s), by integer operations
    // (conversions and products in FP64 issue on the narrow FP64 pipe)
    unsigned long long q = __umul64hi(w, kTab.ph);  // 2^62 .. 2^64
    if (!(q >> 63)) {
      q += q;
      ++s;
    }
    // to 53 bits; a double in [1, 2]
    const unsigned long long r = (q >> 11) + ((q >> 10) & 1);  // 2^52 .. 2^53
    double d = __longlong_as_double((long long)(r + (1022ull << 52)));
    const int sc = ea + eb - s + (kPShift + 63 - 2 * kT);
    const int ed = (int)((__double2hiint(d) >> 20) & 0x7ff);
    if (ed + sc >= 1 && ed + sc <= 2046)
      d = __hiloint2double(__double2hiint(d) + (sc << 20), __double2loint(d));
    else
      d = scalbn(d, sc);
    return neg ? -d : d;
  }
};

struct CrtOut {
  double2 alpha, beta;
  int mode;  // 0: alpha 1, beta 0; 1: alpha +-1, beta 1; 2: general
};
__device__ __forceinline__ void crt_store(const CrtOut& o, double re, double im, double2* c) {
  if (o.mode == 0) {
    *c = make_double2(re, im);
  } else if (o.mode == 1) {
    const double2 c0 = *c;
    *c = o.alpha.x > 0 ? make_double2(c0.x + re, c0.y + im) : make_double2(c0.x - re, c0.y - im);
  } else {
    double2 r = make_double2(o.alpha.x * re - o.alpha.y * im, o.alpha.x * im + o.alpha.y * re);
    if (o.beta.x != 0.0 || o.beta.y != 0.0) {
      const double2 c0 = *c;
      r.x += o.beta.x * c0.x - o.beta.y * c0.y;
      r.y += o.beta.x * c0.y + o.beta.y * c0.x;
    }
    *c = r;
  }
}

// Complex (m, n) from the residues res[z][modulus][m'][n'].  op(A) = A^H: from
// rows 2m, 2m+1 and columns 2n, 2n+1 (Re = C[2m][2n] + C[2m+1][2n+1], Im =
// C[2m][2n+1] - C[2m+1][2n], their residues added unless an operand's parts have
// two exponents); op(A) = A: (C[m][2n], C[m][2n+1]).  A block takes
// 32 m (a warp's lanes: coalesced C) by NB n, its residues through shared
// memory (16-byte loads, all in flight; pitch of an odd number of words), those of
// several K ranges (RANGES) added modulo p on the way.  Bound by its integer
// instructions (1,088^2 outputs of A^H B 34 us, 5,000,000 x 1 of A B, mostly padding of
// the 32 columns, 1.9 ms).
template <bool CONJ, bool RANGES>
__global__ void __launch_bounds__(256, 3)
    k_mod_crt(const unsigned char* __restrict__ res, int nz, int M, int N, int64_t Np,
              const int* __restrict__ exa, const int* __restrict__ exb,
              const double* __restrict__ rowscale, CrtOut o, double2* __restrict__ C, int64_t ldc) {
  constexpr int NB = CONJ ? 16 : 32, ROWS = CONJ ? 64 : 32;
  constexpr int RW = NB / 2, PW = RW + 1;  // words of a row, pitch
  constexpr int PAIRS = NB / 16;           // pairs of n a thread
  __shared__ unsigned sm[kMod * ROWS * PW];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int m = blockIdx.x * 32 + lane, n0 = blockIdx.y * NB;
  const int64_t rows = (CONJ ? 2 : 1) * (int64_t)M;
  {
    // 128 chunks of 16 bytes a modulus, eight moduli a thread
    const int c = threadIdx.x & 127, r = c / (RW / 4), q = c % (RW / 4), odd = threadIdx.x >> 7;
    const int64_t row = (int64_t)blockIdx.x * ROWS + r, col = 2 * (int64_t)n0 + 16 * q;
    const bool in = row < rows && col < Np;
    auto at = [&](int z, int mod) {
      return in ? __ldg((const uint4*)(res + (((size_t)z * kMod + mod) * rows + row) * Np + col))
                : make_uint4(0, 0, 0, 0);
    };
    auto put = [&](int mod, uint4 v) {
      unsigned* d = sm + (mod * ROWS + r) * PW + 4 * q;
      d[0] = v.x;
      d[1] = v.y;
      d[2] = v.z;
      d[3] = v.w;
    };
    if constexpr (!RANGES) {
      uint4 v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = at(0, 2 * i + odd);
#pragma unroll
      for (int i = 0; i < 8; ++i) put(2 * i + odd, v[i]);
    } else {
#pragma unroll 1
      for (int i = 0; i < 8; ++i) {
        const int mod = 2 * i + odd;
        const float p = c_mod_p[mod], inv = 1.f / p;
        int t[16] = {};
#pragma unroll 4
        for (int z = 0; z < nz; ++z) {
          const uint4 v = at(z, mod);
          const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int u = 0; u < 16; ++u) t[u] += (signed char)(w[u / 4] >> (8 * (u % 4)));
        }
        float x[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) x[u] = mod_sym((float)t[u], p, inv);
        put(mod, make_uint4(pack_res(x, p), pack_res(x + 4, p), pack_res(x + 8, p), pack_res(x + 12, p)));
      }
    }
  }
  __syncthreads();
  if (m >= M) return;
  const unsigned* mine = sm + (CONJ ? 2 : 1) * lane * PW + warp * PAIRS;
  CrtFrac re[2 * PAIRS], im[2 * PAIRS];
#pragma unroll
  for (int u = 0; u < 2 * PAIRS; ++u) {
    CrtDigits dr, di;
    const unsigned* p = mine + u / 2;
    each_mod<0>([&](auto I) {
      constexpr int i = decltype(I)::value;
      const unsigned x = p[i * ROWS * PW] >> (16 * (u & 1));
      const int a0 = (signed char)x, a1 = (signed char)(x >> 8);
      if constexpr (CONJ) {
        const unsigned y = p[i * ROWS * PW + PW] >> (16 * (u & 1));
        dr.template add<i>(a0 + (signed char)(y >> 8));
        di.template add<i>(a1 - (signed char)y);
      } else {
        dr.template add<i>(a0);
        di.template add<i>(a1);
      }
    });
    re[u].set(dr);
    im[u].set(di);
  }
  const int ea = exa[CONJ ? 2 * m : m], eai = CONJ ? exa[2 * m + 1] : ea;
  const double rs = rowscale ? rowscale[m] : 1.0;
#pragma unroll
  for (int u = 0; u < 2 * PAIRS; ++u) {
    const int n = n0 + 2 * PAIRS * warp + u;
    if (n >= N) break;
    const int eb = exb[2 * n], ebi = exb[2 * n + 1];
    double x, y;
    if (ea == kNonfinite || eb == kNonfinite) {
      x = y = __longlong_as_double(0x7ff8000000000000ll);
    } else if (CONJ && (ea != eai || eb != ebi)) {
      // Re Re + Im Im and Re Im - Im Re
      x = y = 0.0;
#pragma unroll 1
      for (int w = 0; w < 4; ++w) {
        const bool ima = w & 1, imb = w == 1 || w == 2;
        CrtDigits d;
        each_mod<0>([&](auto I) {
          constexpr int i = decltype(I)::value;
          d.template add<i>(
              (signed char)(mine[i * ROWS * PW + (ima ? PW : 0) + u / 2] >> (16 * (u & 1) + (imb ? 8 : 0))));
        });
        CrtFrac f;
        f.set(d);
        const double v = f.value(ima ? eai : ea, imb ? ebi : eb);
        if (w < 2) x += v;
        else y += w == 2 ? v : -v;
      }
    } else {
      x = re[u].value(ea, eb);
      y = im[u].value(ea, eb);
    }
    if (rowscale) {
      x *= rs;
      y *= rs;
    }
    crt_store(o, x, y, C + (size_t)n * ldc + m);
  }
}

// ------------------------------------------------------------------- host ----
// Number of CTA pairs resident at once.
static int mod_pairs() {
  static int pairs = 0;
  static std::once_flag once;
  std::call_once(once, [] {
    cudaFuncSetAttribute(k_mod_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmem);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * 76);
    cfg.blockDim = dim3(kPairThreads);
    cfg.dynamicSmemBytes = kPairSmem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&pairs, (void*)k_mod_gemm, &cfg) != cudaSuccess || pairs < 1)
      pairs = 76;
    cudaGetLastError();  // clear a refused query
  });
  return pairs;
}

void oz_reserve(System& s, bool conjA, int M, int N, int K) {
  if (M <= 0 || N <= 0 || K <= 0 || 8.0 * M * (double)N * K < kOzMinFlops) return;
  ensure(s.ws_oz, mod_bound(conjA, M, N, K));
}

static void oz_gemm_piece(System& s, bool conjA, int M, int N, int K, double2 alpha,
                          const double2* A, int64_t lda, const double2* B, int64_t ldb,
                          double2 beta, double2* C, int64_t ldc, cudaStream_t st,
                          const double* rowscale) {
  const ModGeom g = mod_geom(conjA, M, N, K, mod_pairs());
  ensure(s.ws_oz, g.total());
  char* base = s.ws_oz.p;
  __nv_bfloat16* pA = (__nv_bfloat16*)base;
  __nv_bfloat16* pB = (__nv_bfloat16*)(base + g.bytes_a);
  unsigned char* res = (unsigned char*)(base + g.bytes_a + g.bytes_b);
  int2* na = (int2*)(base + g.bytes_a + g.bytes_b + g.bytes_r);
  const int parts = conjA ? 2 : 1;  // exponents of a row of op(A)
  int2* nb = na + (size_t)M * g.Sa * parts;
  int* exa = (int*)((char*)na + g.bytes_n);
  int* exb = exa + (size_t)M * parts;
  // timed as its own family: the work is the real BF16 tensor-core GEMMs of
  // all moduli (2 Mr Nr Kr each)
  const double Kr = (double)g.seg * g.nseg;
  TimedScope ts(s, KF_GEMM_OZ, st, 2.0 * kMod * (double)g.Mr * g.Nr * Kr,
                4.0 * kMod * ((double)g.Mr + g.Nr) * Kr + 2.0 * g.gz * g.nseg * kMod * (double)g.Mr * g.Nr);
  if (conjA)
    k_mod_colnorm<<<dim3(M, g.Sa), 256, 0, st>>>(A, lda, K, na);
  else
    k_mod_rownorm<<<dim3((M + 255) / 256, g.Sa), 256, 0, st>>>(A, lda, M, K, na);
  PWH_LAUNCH_CHECK();
  k_mod_colnorm<<<dim3(N, g.Sb), 256, 0, st>>>(B, ldb, K, nb);
  PWH_LAUNCH_CHECK();
  k_mod_exp<<<(M + N + 255) / 256, 256, 0, st>>>(na, M, g.Sa, parts, nb, N, g.Sb, conjA, exa, exb);
  PWH_LAUNCH_CHECK();
  for (int sgi = 0; sgi < g.nseg; ++sgi) {
    const int k0 = sgi * g.kseg, kk = std::min(g.kseg, K - k0);
    const int64_t seg = round_up((int64_t)kk * (conjA ? 1 : 2), TC_BK);
    const int64_t pla = g.Mr * seg, plb = g.Nr * seg;
    if (conjA) {
      const unsigned gx = (unsigned)((seg + 1023) / 1024);
      k_mod_slice_cols<<<dim3(gx, M), 256, 0, st>>>(A + k0, lda, kk, (int)seg, exa, pA, pla);
      PWH_LAUNCH_CHECK();
      k_mod_slice_cols<<<dim3(gx, N), 256, 0, st>>>(B + k0, ldb, kk, (int)seg, exb, pB, plb);
      PWH_LAUNCH_CHECK();
    } else {
      k_mod_slice_rows<<<dim3((M + 31) / 32, (unsigned)((seg / 2 + 31) / 32)), 256, 0, st>>>(
          A + (int64_t)k0 * lda, lda, M, kk, (int)seg, exa, pA, pla);
      PWH_LAUNCH_CHECK();
      k_mod_slice_b2<<<dim3((unsigned)((seg / 2 + 255) / 256), N), 256, 0, st>>>(
          B + k0, ldb, kk, (int)seg, exb, pB, plb);
      PWH_LAUNCH_CHECK();
    }
    const CUtensorMap ma = make_map(pA, kMod * g.Mr, seg, seg, 128);
    const CUtensorMap mb = make_map(pB, kMod * g.Nr, seg, seg, g.bn / 2);
    ModArgs a{};
    a.Mr = (int)g.Mr;
    a.Nr = (int)g.Nr;
    a.bn = g.bn;
    a.gm = g.gm;
    a.gn = g.gn;
    a.gz = g.gz;
    a.kb_total = (int)(seg / TC_BK);
    a.kb_per = g.kb_per;
    a.accum = sgi > 0;
    a.Np = g.Np;
    a.out = res;
    a.err = device_error_word(s);
    const int64_t items = (int64_t)g.gm * g.gn * g.gz * kMod;
    const int pairs = (int)std::min<int64_t>(items, mod_pairs());
    k_mod_gemm<<<2 * pairs, kPairThreads, kPairSmem, st>>>(ma, mb, a);
    PWH_LAUNCH_CHECK();
  }
  CrtOut o;
  o.alpha = alpha;
  o.beta = beta;
  const bool pm1 = alpha.y == 0.0 && (alpha.x == 1.0 || alpha.x == -1.0);
  o.mode = pm1 && alpha.x == 1.0 && beta.x == 0.0 && beta.y == 0.0 ? 0
           : pm1 && beta.x == 1.0 && beta.y == 0.0                 ? 1
                                                                   : 2;
  const dim3 gc((M + 31) / 32, conjA ? (N + 15) / 16 : (N + 31) / 32);
  auto crt = [&](auto kernel) {
    kernel<<<gc, 256, 0, st>>>(res, g.gz, M, N, g.Np, exa, exb, rowscale, o, C, ldc);
  };
  if (conjA)
    g.gz > 1 ? crt(k_mod_crt<true, true>) : crt(k_mod_crt<true, false>);
  else
    g.gz > 1 ? crt(k_mod_crt<false, true>) : crt(k_mod_crt<false, false>);
  PWH_LAUNCH_CHECK();
}

void oz_gemm(System& s, bool conjA, int M, int N, int K, double2 alpha, const double2* A,
             int64_t lda, const double2* B, int64_t ldb, double2 beta, double2* C, int64_t ldc,
             cudaStream_t st, const double* rowscale) {
  if (M <= 0 || N <= 0) return;
  const ModSplit sp = mod_split(conjA, M, N, K);
  for (int64_t n0 = 0; n0 < N; n0 += sp.pn)
    for (int64_t m0 = 0; m0 < M; m0 += sp.pm)
      // rows m0.. of C: columns m0.. of A (A^H) or rows m0.. of A
      oz_gemm_piece(s, conjA, (int)std::min<int64_t>(sp.pm, M - m0), (int)std::min<int64_t>(sp.pn, N - n0), K, alpha,
                    A + (conjA ? m0 * lda : m0), lda, B + n0 * ldb, ldb, beta,
                    C + n0 * ldc + m0, ldc, st, rowscale ? rowscale + m0 : nullptr);
}

}  // namespace pwh
