// Learned preconditioner (not in the paper; the learned part of this library):
// a 4 -> 64 -> 64 -> 1 SiLU network s = MLP(f) corrects the Teter-Payne-Allan
// diagonal per (shell of equal |k+G|, band):  K = K_TPA(x) * exp(clip(s, -3, 3)).
//
//  * features/targets of (shell, band) rows from Ritz vectors X, their H X,
//    Ritz values and the converged bands X* (training data harvested from the
//    solver's own trajectories);
//  * forward, loss + backward (register-tiled products over row tiles), Adam;
//  * the per-iteration factors used by the eigensolver's preconditioner.
//
// Parameter vector (FP32): W1 (64x4 row-major), b1, W2 (64x64), b2, W3 (64), b3,
// then 8 floats of feature ranges (min f1..f4, max f1..f4) outside which the
// preconditioner falls back to plain TPA (s = 0).
#include <algorithm>
#include <mutex>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "gemm.cuh"

namespace pwh {

constexpr int MH = 64, MIN = 4;
constexpr int kMlpParams = MH * MIN + MH + MH * MH + MH + MH + 1;  // 4545
constexpr int kMlpBlob = kMlpParams + 8;

__device__ __forceinline__ float silu_f(float z) { return z / (1.f + __expf(-z)); }

// Load the parameters into shared memory (all threads).
__device__ void mlp_load(const float* __restrict__ p, float* sp) {
  for (int i = threadIdx.x; i < kMlpParams; i += blockDim.x) sp[i] = p[i];
  __syncthreads();
}

// Forward pass of one row.
__device__ float mlp_row(const float* sp, const float f[4]) {
  const float* W1 = sp;
  const float* b1 = W1 + MH * MIN;
  const float* W2 = b1 + MH;
  const float* b2 = W2 + MH * MH;
  const float* W3 = b2 + MH;
  const float b3 = W3[MH];
  float h1[MH];
#pragma unroll 8
  for (int i = 0; i < MH; ++i) {
    float z = b1[i] + W1[i * 4] * f[0] + W1[i * 4 + 1] * f[1] + W1[i * 4 + 2] * f[2] +
              W1[i * 4 + 3] * f[3];
    h1[i] = silu_f(z);
  }
  float s = b3;
  for (int i = 0; i < MH; ++i) {
    float z = b2[i];
#pragma unroll 16
    for (int j = 0; j < MH; ++j) z += W2[i * MH + j] * h1[j];
    s += W3[i] * silu_f(z);
  }
  return s;
}

__global__ void k_mlp_forward(const float* __restrict__ p, const float* __restrict__ F, int64_t rows,
                              float* __restrict__ s) {
  extern __shared__ float sp[];
  mlp_load(p, sp);
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < rows;
       r += (int64_t)gridDim.x * blockDim.x) {
    float f[4] = {F[4 * r], F[4 * r + 1], F[4 * r + 2], F[4 * r + 3]};
    s[r] = mlp_row(sp, f);
  }
}

// Loss sum w (s - y)^2 / wsum and its gradient, accumulated (atomically) into
// g (kMlpParams) and loss[0].
//
// Bound: the FP32 pipes.  The three 64 x 64 products of a row (forward, back
// through W2, gradient of W2) are 12,288 of its 13,250 multiply-adds, so each
// is a register-tiled matrix product over a tile of GR rows: activations and
// deltas lie transposed in shared memory ([unit][row], pitch GP: 16-byte
// loads, eight neighbouring units on distinct banks) and a thread owns an
// 8 x 4 (rows x units) tile of the first two products and a 4 x 4 tile of the
// W2 gradient, 24 and 32 multiply-adds per 16-byte load triple / pair.  Blocks
// are persistent (two per SM), so that every weight gradient stays in its
// thread's registers until the block's last tile and costs one atomic per
// block; z1 is recomputed in the backward pass (four multiply-adds) rather
// than kept.  A training step (this kernel, two memsets, Adam) of 32,768 rows:
// 85 us, against 356 us for a row per thread with scalar shared-memory weights.
constexpr int GR = 128;        // rows per tile
constexpr int GT = 256;        // threads per block
constexpr int GP = GR + 4;     // pitch of the transposed activations
constexpr int GLOADS = kMlpParams + 3;  // parameters, padded to 16 bytes
static_assert(GLOADS % 4 == 0 && (MH * MIN + MH) % 4 == 0, "16-byte loads of W2");

__device__ __forceinline__ float sigmoid_f(float z) { return 1.f / (1.f + __expf(-z)); }

__global__ void __launch_bounds__(GT, 2) k_mlp_grad(const float* __restrict__ p,
                                                    const float* __restrict__ F,
                                                    const float* __restrict__ y,
                                                    const float* __restrict__ w, int64_t rows,
                                                    float inv_wsum, float* __restrict__ g,
                                                    float* __restrict__ loss) {
  extern __shared__ __align__(16) float sm[];
  float* sp = sm;                  // parameters
  float* w2t = sp + GLOADS;        // W2 transposed: [j][i]
  float* h1t = w2t + MH * MH;      // h1, [j][row]
  float* d2t = h1t + MH * GP;      // dL/dz2, [i][row]
  float* sf = d2t + MH * GP;       // features, [row][4]
  float* ss = sf + GR * 4;         // partial outputs, [4][row]
  float* sds = ss + 4 * GR;        // dL/ds, [row]
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int i = t; i < kMlpParams; i += GT) sp[i] = p[i];
  __syncthreads();
  const float* W1 = sp;
  const float* b1 = W1 + MH * MIN;
  const float* W2 = b1 + MH;
  const float* b2 = W2 + MH * MH;
  const float* W3 = b2 + MH;
  const float b3 = W3[MH];
  for (int e = t; e < MH * MH; e += GT) w2t[(e % MH) * MH + e / MH] = W2[e];
  // tile of the first two products: rows r0..r0+3 and r0+64..r0+67, units c0..c0+3
  const int rg = (warp & 1) * 8 + (lane & 7), cg = (warp >> 1) * 4 + (lane >> 3);
  const int r0 = rg * 4, c0 = cg * 4;
  // tile of the W2 gradient: units gi + 16 q (rows of W2), gj + 16 q (columns)
  const int gi = (warp & 1) * 8 + (lane & 7), gj = (warp >> 1) * 4 + (lane >> 3);
  float g2[4][4] = {}, g1[4][4] = {}, gb1[4] = {}, gb2[4] = {}, g3[4] = {};
  float gb3 = 0.f, lsum = 0.f;
  const int64_t ntile = (rows + GR - 1) / GR;
  for (int64_t tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
    const int64_t base = tile * GR;
    __syncthreads();  // w2t written / the previous tile consumed
    for (int e = t; e < GR * 4; e += GT) sf[e] = base + e / 4 < rows ? F[base * 4 + e] : 0.f;
    __syncthreads();
    {  // first layer: a row and half of the units per thread
      const int r = t & (GR - 1), j0 = (t / GR) * (MH / 2);
      const float4 f = *(const float4*)(sf + 4 * r);
      const bool on = base + r < rows;
#pragma unroll 8
      for (int j = j0; j < j0 + MH / 2; ++j) {
        const float4 a = *(const float4*)(W1 + 4 * j);
        const float z = b1[j] + a.x * f.x + a.y * f.y + a.z * f.z + a.w * f.w;
        h1t[j * GP + r] = on ? z * sigmoid_f(z) : 0.f;
      }
    }
    __syncthreads();
    float acc[8][4];
    // z2 = b2 + W2 h1
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int r = 0; r < 8; ++r) acc[r][q] = b2[c0 + q];
#pragma unroll 2
    for (int j = 0; j < MH; ++j) {
      const float4 x0 = *(const float4*)(h1t + j * GP + r0);
      const float4 x1 = *(const float4*)(h1t + j * GP + r0 + 64);
      const float4 u = *(const float4*)(w2t + j * MH + c0);
      const float xr[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
      const float uc[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[r][q] = fmaf(xr[r], uc[q], acc[r][q]);
    }
    // s = b3 + W3 silu(z2): partial sums over the thread's units, then over
    // the warp's four unit groups and the block's four warp columns
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      float v = 0.f;
#pragma unroll
      for (int q = 0; q < 4; ++q) v += W3[c0 + q] * (acc[r][q] * sigmoid_f(acc[r][q]));
      v += __shfl_xor_sync(0xffffffffu, v, 8);
      v += __shfl_xor_sync(0xffffffffu, v, 16);
      if (lane < 8) ss[(warp >> 1) * GR + r0 + (r & 3) + 64 * (r >> 2)] = v;
    }
    __syncthreads();
    if (t < GR) {
      float ds = 0.f;
      if (base + t < rows) {
        const float s = b3 + ((ss[t] + ss[GR + t]) + (ss[2 * GR + t] + ss[3 * GR + t]));
        const float e = s - y[base + t], we = w[base + t] * e * inv_wsum;
        ds = 2.f * we;
        lsum += we * e;
      }
      sds[t] = ds;
      gb3 += ds;
    }
    __syncthreads();
    // dL/dz2 and the gradients of b2 and W3
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float4 d4 = *(const float4*)(sds + r0 + 64 * h);
      const float ds[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float o[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const float z = acc[4 * h + r][q], sg = sigmoid_f(z);
          // padding rows contribute nothing, whatever the parameters
          const bool on = base + r0 + 64 * h + r < rows;
          o[r] = on ? ds[r] * W3[c0 + q] * (sg * (1.f + z * (1.f - sg))) : 0.f;
          gb2[q] += o[r];
          g3[q] += on ? ds[r] * (z * sg) : 0.f;
        }
        *(float4*)(d2t + (c0 + q) * GP + r0 + 64 * h) = make_float4(o[0], o[1], o[2], o[3]);
      }
    }
    __syncthreads();
    // dL/dh1 = W2^T dL/dz2
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[r][q] = 0.f;
#pragma unroll 2
    for (int i = 0; i < MH; ++i) {
      const float4 x0 = *(const float4*)(d2t + i * GP + r0);
      const float4 x1 = *(const float4*)(d2t + i * GP + r0 + 64);
      const float4 u = *(const float4*)(W2 + i * MH + c0);
      const float xr[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
      const float uc[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
      for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[r][q] = fmaf(xr[r], uc[q], acc[r][q]);
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int row = r0 + (r & 3) + 64 * (r >> 2);
      const float4 f = *(const float4*)(sf + 4 * row);
      const bool on = base + row < rows;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 a = *(const float4*)(W1 + 4 * (c0 + q));
        const float z = b1[c0 + q] + a.x * f.x + a.y * f.y + a.z * f.z + a.w * f.w;
        const float sg = sigmoid_f(z);
        const float d = on ? acc[r][q] * (sg * (1.f + z * (1.f - sg))) : 0.f;
        gb1[q] += d;
        g1[q][0] += d * f.x;
        g1[q][1] += d * f.y;
        g1[q][2] += d * f.z;
        g1[q][3] += d * f.w;
      }
    }
    // gradient of W2: sum over the rows of dL/dz2[i] h1[j]
#pragma unroll 1
    for (int r = 0; r < GR; r += 4) {
      float4 a[4], b[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        a[q] = *(const float4*)(d2t + (gi + 16 * q) * GP + r);
        b[q] = *(const float4*)(h1t + (gj + 16 * q) * GP + r);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          g2[i][j] = fmaf(a[i].w, b[j].w,
                          fmaf(a[i].z, b[j].z, fmaf(a[i].y, b[j].y, fmaf(a[i].x, b[j].x, g2[i][j]))));
    }
  }
  float* gW1 = g;
  float* gB1 = gW1 + MH * MIN;
  float* gW2 = gB1 + MH;
  float* gB2 = gW2 + MH * MH;
  float* gW3 = gB2 + MH;
  float* gB3 = gW3 + MH;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) atomicAdd(&gW2[(gi + 16 * i) * MH + gj + 16 * j], g2[i][j]);
  // the other gradients: sums over the eight row groups of a warp, then atomics
  auto reduce = [&](float v, float* dst) {
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    if ((lane & 7) == 0) atomicAdd(dst, v);
  };
#pragma unroll
  for (int q = 0; q < 4; ++q) {
#pragma unroll
    for (int k = 0; k < MIN; ++k) reduce(g1[q][k], &gW1[(c0 + q) * MIN + k]);
    reduce(gb1[q], &gB1[c0 + q]);
    reduce(gb2[q], &gB2[c0 + q]);
    reduce(g3[q], &gW3[c0 + q]);
  }
  if (t < GR) {  // whole warps
    for (int o = 16; o > 0; o >>= 1) {
      gb3 += __shfl_xor_sync(0xffffffffu, gb3, o);
      lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    }
    if (lane == 0) {
      atomicAdd(gB3, gb3);
      atomicAdd(loss, lsum);
    }
  }
}

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// ---------------------------------------------------------- features / data --
__device__ __forceinline__ double tpa_k(double x) {
  const double q = 27.0 + x * (18.0 + x * (12.0 + 8.0 * x));
  return q / (q + 16.0 * x * x * x * x);
}

__device__ __forceinline__ void make_features(double Tg, double th, double rn, double E, double vbar,
                                              float f[4]) {
  const double x = Tg / E;
  f[0] = (float)log(x + 0.05);
  f[1] = (float)((th - vbar) / E);
  f[2] = (float)fmin(2.0, fmax(-12.0, log10(fmax(rn, 1e-300))));
  f[3] = (float)((Tg + vbar - th) / (Tg + E));
}

// per band: R = HX - X theta (internal order scratch), rn, eref = <x|T|x>/<x|x>;
// per (band, shell): num += Re conj(r) e, den += |r|^2 with e = corrections E.
__global__ void k_shell_stats(const double2* __restrict__ X, const double2* __restrict__ HX,
                              const double2* __restrict__ E, int64_t npw,
                              const double* __restrict__ theta, const int32_t* __restrict__ shell,
                              int nshell, double* __restrict__ num, double* __restrict__ den) {
  const int b = blockIdx.y;
  const double th = theta[b];
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < npw;
       i += (int64_t)gridDim.x * blockDim.x) {
    const size_t o = (size_t)b * npw + i;
    const double2 x = X[o], hx = HX[o], e = E[o];
    const double rx = hx.x - th * x.x, ry = hx.y - th * x.y;
    const int g = shell[i];
    atomicAdd(&num[(size_t)b * nshell + g], rx * e.x + ry * e.y);
    atomicAdd(&den[(size_t)b * nshell + g], rx * rx + ry * ry);
  }
}

__global__ void k_band_stats(const double2* __restrict__ X, const double2* __restrict__ HX,
                             int64_t npw, const double* __restrict__ theta,
                             const double* __restrict__ kin, double* __restrict__ rn,
                             double* __restrict__ eref) {
  const int b = blockIdx.x;
  const double th = theta[b];
  double s2 = 0, xt = 0, x2 = 0;
  for (int64_t i = threadIdx.x; i < npw; i += blockDim.x) {
    const size_t o = (size_t)b * npw + i;
    const double2 x = X[o], hx = HX[o];
    const double rx = hx.x - th * x.x, ry = hx.y - th * x.y;
    s2 += rx * rx + ry * ry;
    const double a = x.x * x.x + x.y * x.y;
    x2 += a;
    xt += kin[i] * a;
  }
  __shared__ double red[3][32];
  for (int o = 16; o > 0; o >>= 1) {
    s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    xt += __shfl_xor_sync(0xffffffffu, xt, o);
    x2 += __shfl_xor_sync(0xffffffffu, x2, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = s2;
    red[1][threadIdx.x >> 5] = xt;
    red[2][threadIdx.x >> 5] = x2;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0, c = 0, d = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      a += red[0][w];
      c += red[1][w];
      d += red[2][w];
    }
    rn[b] = sqrt(a);
    eref[b] = (d > 0 && c > 0) ? c / d : 1.0;
  }
}

// One block per band: features of every shell, target y and weight w.
__global__ void k_make_rows(const double* __restrict__ num, const double* __restrict__ den, int nshell,
                            const double* __restrict__ Tshell, const double* __restrict__ theta,
                            const double* __restrict__ rn, const double* __restrict__ eref,
                            double vbar, float* __restrict__ F, float* __restrict__ y,
                            float* __restrict__ w) {
  const int b = blockIdx.x;
  const double E = eref[b];
  __shared__ double red[2][32];
  double dsum = 0;
  for (int g = threadIdx.x; g < nshell; g += blockDim.x) dsum += den[(size_t)b * nshell + g];
  for (int o = 16; o > 0; o >>= 1) dsum += __shfl_xor_sync(0xffffffffu, dsum, o);
  if ((threadIdx.x & 31) == 0) red[0][threadIdx.x >> 5] = dsum;
  __syncthreads();
  double tot = 0;
  for (int q = 0; q < (int)(blockDim.x >> 5); ++q) tot += red[0][q];
  __syncthreads();
  // raw targets and weights, then the weighted mean
  double wy = 0, ws = 0;
  for (int g = threadIdx.x; g < nshell; g += blockDim.x) {
    const size_t o = (size_t)b * nshell + g;
    const double dn = den[o];
    const double d = dn > 0 ? -num[o] / dn : 0.0;
    const bool ok = d > 0 && dn > 0;
    const double yy = ok ? log(d) - log(tpa_k(Tshell[g] / E)) : 0.0;
    const double ww = ok ? dn / tot : 0.0;
    y[o] = (float)yy;
    w[o] = (float)ww;
    wy += ww * yy;
    ws += ww;
    float f[4];
    make_features(Tshell[g], theta[b], rn[b], E, vbar, f);
    for (int k = 0; k < 4; ++k) F[4 * o + k] = f[k];
  }
  for (int o = 16; o > 0; o >>= 1) {
    wy += __shfl_xor_sync(0xffffffffu, wy, o);
    ws += __shfl_xor_sync(0xffffffffu, ws, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = wy;
    red[1][threadIdx.x >> 5] = ws;
  }
  __syncthreads();
  double mwy = 0, mws = 0;
  for (int q = 0; q < (int)(blockDim.x >> 5); ++q) {
    mwy += red[0][q];
    mws += red[1][q];
  }
  const double mean = mws > 0 ? mwy / mws : 0.0;
  for (int g = threadIdx.x; g < nshell; g += blockDim.x) {
    const size_t o = (size_t)b * nshell + g;
    if (w[o] > 0) y[o] = (float)((double)y[o] - mean);
  }
}

// Preconditioner factors for the eigensolver: s[j * nshell + g] for the bands
// idx[j], clipped to [-3, 3], 0 (plain TPA) when a feature leaves the range
// the network was trained on.
__global__ void k_mlp_factors(const float* __restrict__ blob, const int* __restrict__ idx, int k,
                              const double* __restrict__ theta, const double* __restrict__ rn,
                              const double* __restrict__ eref, const double* __restrict__ Tshell,
                              int nshell, double vbar, float* __restrict__ s) {
  extern __shared__ float sp[];
  mlp_load(blob, sp);
  const float* lo = blob + kMlpParams;
  const float* hi = lo + 4;
  const int64_t rows = (int64_t)k * nshell;
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < rows;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int j = (int)(r / nshell), g = (int)(r % nshell);
    const int b = idx[j];
    float f[4];
    make_features(Tshell[g], theta[b], rn[b], eref[b], vbar, f);
    bool inside = true;
    for (int q = 0; q < 4; ++q) inside = inside && f[q] >= lo[q] && f[q] <= hi[q];
    float v = inside ? mlp_row(sp, f) : 0.f;
    s[r] = fminf(3.f, fmaxf(-3.f, v));
  }
}

static size_t grad_smem() {
  return (size_t)(GLOADS + MH * MH + 2 * MH * GP + GR * 4 + 4 * GR + GR) * sizeof(float);
}

void mlp_factors(System& s, const int* idx, int k, const double* theta, const double* rn,
                 const double* eref, float* out, cudaStream_t st) {
  const int64_t rows = (int64_t)k * s.nshell;
  const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(1024, (rows + 255) / 256));
  k_mlp_factors<<<blocks, 256, kMlpParams * sizeof(float), st>>>(s.d_mlp, idx, k, theta, rn, eref,
                                                                 s.d_Tshell, s.nshell, s.vbar, out);
  PWH_LAUNCH_CHECK();
}

}  // namespace pwh

using namespace pwh;

extern "C" {

pwh_status pwh_mlp_num_params(int32_t* n) {
  return guarded([&] {
    PWH_CHECK_ARG(n, "null argument");
    *n = kMlpBlob;
  });
}

pwh_status pwh_mlp_forward(pwh_system* sys, const float* params, const float* feats, int64_t rows,
                           float* s_out) {
  return guarded([&] {
    PWH_CHECK_ARG(sys && params && feats && s_out, "null argument");
    PWH_CHECK_ARG(rows >= 0, "rows < 0");
    if (rows == 0) return;
    const int blocks = (int)std::min<int64_t>(4096, (rows + 255) / 256);
    k_mlp_forward<<<blocks, 256, kMlpParams * sizeof(float), sys->s.stream>>>(params, feats, rows,
                                                                             s_out);
    PWH_LAUNCH_CHECK();
  });
}

pwh_status pwh_mlp_loss_grad(pwh_system* sys, const float* params, const float* feats,
                             const float* y, const float* w, int64_t rows, double wsum,
                             float* grad_out, float* loss_out) {
  return guarded([&] {
    PWH_CHECK_ARG(sys && params && feats && y && w && grad_out && loss_out, "null argument");
    PWH_CHECK_ARG(rows >= 1 && wsum > 0, "rows >= 1 and wsum > 0 required");
    System& s = sys->s;
    static std::once_flag attr_once;
    std::call_once(attr_once, [] {
      cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)grad_smem());
    });
    PWH_CUDA(cudaMemsetAsync(grad_out, 0, kMlpParams * sizeof(float), s.stream));
    PWH_CUDA(cudaMemsetAsync(loss_out, 0, sizeof(float), s.stream));
    // persistent: two blocks per SM
    const int blocks = (int)std::min<int64_t>(2 * 152, (rows + GR - 1) / GR);
    k_mlp_grad<<<blocks, GT, grad_smem(), s.stream>>>(params, feats, y, w, rows, (float)(1.0 / wsum),
                                                      grad_out, loss_out);
    PWH_LAUNCH_CHECK();
  });
}

pwh_status pwh_mlp_adam(pwh_system* sys, float* params, const float* grad, float* m, float* v,
                        int32_t step, float lr) {
  return guarded([&] {
    PWH_CHECK_ARG(sys && params && grad && m && v, "null argument");
    PWH_CHECK_ARG(step >= 1, "step counts from 1");
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - std::pow(b1, (float)step), c2 = 1.f - std::pow(b2, (float)step);
    k_adam<<<32, 256, 0, sys->s.stream>>>(params, grad, m, v, kMlpParams, lr, b1, b2, 1e-8f, c1, c2);
    PWH_LAUNCH_CHECK();
  });
}

pwh_status pwh_mlp_training_rows(pwh_system* sys, int32_t nb, const void* X, const void* HX,
                                 const double* theta, const void* Xstar, float* feats, float* y,
                                 float* w) {
  return guarded([&] {
    PWH_CHECK_ARG(sys && X && HX && theta && Xstar && feats && y && w, "null argument");
    System& s = sys->s;
    PWH_CHECK_ARG(nb >= 1, "nb < 1");
    if (!s.have_v) throw Error{PWH_ERR_STATE, "pwh_set_potential has not been called"};
    const int64_t npw = s.npw;
    cudaStream_t st = s.stream;
    // scratch: internal-order copies of X, HX, X*, corrections E, W (nb x nb), stats
    const size_t nv = (size_t)npw * nb;
    double2* buf = nullptr;
    PWH_CUDA(cudaMalloc((void**)&buf, (4 * nv + (size_t)nb * nb) * sizeof(double2) +
                                          (2 * (size_t)nb * s.nshell + 3 * (size_t)nb) * sizeof(double)));
    double2 *Xi = buf, *HXi = Xi + nv, *Si = HXi + nv, *Ei = Si + nv, *Wm = Ei + nv;
    double* num = (double*)(Wm + (size_t)nb * nb);
    double* den = num + (size_t)nb * s.nshell;
    double* th = den + (size_t)nb * s.nshell;
    double* rn = th + nb;
    double* eref = rn + nb;
    try {
      permute_public_to_internal(s, (const double2*)X, Xi, nb);
      permute_public_to_internal(s, (const double2*)HX, HXi, nb);
      permute_public_to_internal(s, (const double2*)Xstar, Si, nb);
      PWH_CUDA(cudaMemcpyAsync(th, theta, nb * sizeof(double), cudaMemcpyHostToDevice, st));
      // E = X* (X*^H X) - X
      const double2 one = make_double2(1, 0), zero = make_double2(0, 0);
      cgemm<double>(s, true, nb, nb, (int)npw, one, Si, npw, Xi, npw, zero, Wm, nb, st);
      PWH_CUDA(cudaMemcpyAsync(Ei, Xi, nv * sizeof(double2), cudaMemcpyDeviceToDevice, st));
      cgemm<double>(s, false, (int)npw, nb, nb, one, Si, npw, Wm, nb, make_double2(-1, 0), Ei, npw, st);
      PWH_CUDA(cudaMemsetAsync(num, 0, 2 * (size_t)nb * s.nshell * sizeof(double), st));
      dim3 g((unsigned)std::min<int64_t>(64, (npw + 255) / 256), nb);
      k_shell_stats<<<g, 256, 0, st>>>(Xi, HXi, Ei, npw, th, s.d_shell, s.nshell, num, den);
      PWH_LAUNCH_CHECK();
      k_band_stats<<<nb, 256, 0, st>>>(Xi, HXi, npw, th, s.d_kin, rn, eref);
      PWH_LAUNCH_CHECK();
      k_make_rows<<<nb, 256, 0, st>>>(num, den, s.nshell, s.d_Tshell, th, rn, eref, s.vbar, feats, y, w);
      PWH_LAUNCH_CHECK();
      PWH_CUDA(cudaStreamSynchronize(st));
    } catch (...) {
      cudaFree(buf);
      throw;
    }
    cudaFree(buf);
  });
}

pwh_status pwh_set_mlp(pwh_system* sys, const float* blob, int32_t n) {
  return guarded([&] {
    PWH_CHECK_ARG(sys && blob, "null argument");
    PWH_CHECK_ARG(n == kMlpBlob, "parameter blob has the wrong length");
    System& s = sys->s;
    if (!s.d_mlp) PWH_CUDA(cudaMalloc((void**)&s.d_mlp, kMlpBlob * sizeof(float)));
    PWH_CUDA(cudaMemcpyAsync(s.d_mlp, blob, kMlpBlob * sizeof(float), cudaMemcpyHostToDevice,
                             s.stream));
    PWH_CUDA(cudaStreamSynchronize(s.stream));
    s.have_mlp = true;
  });
}

pwh_status pwh_get_shells(const pwh_system* sys, int32_t* nshell, int32_t* shell_of_pw,
                          double* shell_kinetic) {
  return guarded([&] {
    PWH_CHECK_ARG(sys && nshell, "null argument");
    const System& s = sys->s;
    *nshell = s.nshell;
    if (shell_of_pw) std::copy(s.shell_pub.begin(), s.shell_pub.end(), shell_of_pw);
    if (shell_kinetic) std::copy(s.Tshell_h.begin(), s.Tshell_h.end(), shell_kinetic);
  });
}

}  // extern "C"
