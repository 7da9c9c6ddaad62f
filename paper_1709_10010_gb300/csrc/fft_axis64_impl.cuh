// Kernels of the FP64 axis transforms (fft_axis64.cuh).  A block holds 16 lines
// in shared memory (a 256-byte run of the fast axis when the lines are strided)
// and transforms them with fft_nat: NT = 16 max(N1, N2) threads, one small DFT
// each per pass.
#pragma once
#include "fft_axis64.cuh"
#include "fft_spec_impl.cuh"

namespace pwh {

constexpr int kAxLines = 16;
template <int N> constexpr int ax_threads() {
  constexpr int N1 = Fac<double, N>::N1, N2 = Fac<double, N>::N2;
  return (kAxLines * (N1 > N2 ? N1 : N2) + 31) / 32 * 32;
}
template <int N> constexpr size_t ax_smem() {
  return ((size_t)kAxLines * (N + 1) + N) * sizeof(double2);
}

template <int N, int OP>
__global__ void __launch_bounds__(ax_threads<N>()) k_ax_box(AxisArgs a, int n1, int n2, int n3, int tw_off,
                                                          const double2* __restrict__ tw_g) {
  constexpr int NT = ax_threads<N>(), LD = N + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* buf = (double2*)smem_raw;
  double2* tw = buf + kAxLines * LD;
  __shared__ int64_t base[kAxLines];
  double2* box = a.box + (int64_t)blockIdx.y * a.bstride;
  // element stride, and the strides of the slow and the fast other axis
  const int64_t s1 = (int64_t)n2 * n3, s2 = n3;
  const int64_t es = a.axis == 2 ? 1 : a.axis == 1 ? s2 : s1;
  const int64_t ss = a.axis == 0 ? s2 : s1, fs = a.axis == 2 ? s2 : 1;
  const int nfast = a.axis == 2 ? n2 : n3, nslow = a.axis == 0 ? n2 : n1;
  const int64_t l0 = (int64_t)blockIdx.x * kAxLines, nlines = (int64_t)nslow * nfast;
  const int nl = (int)min((int64_t)kAxLines, nlines - l0);
  for (int t = threadIdx.x; t < N; t += NT) tw[t] = tw_g[tw_off + t];
  if (threadIdx.x < nl) {
    const int64_t L = l0 + threadIdx.x;
    base[threadIdx.x] = (L / nfast) * ss + (L % nfast) * fs;
  }
  __syncthreads();
  // consecutive threads along the contiguous direction
  auto at = [&](int t, int& j, int& e) {
    if (a.axis == 2) {
      j = t / N;
      e = t - j * N;
    } else {
      e = t / kAxLines;
      j = t - e * kAxLines;
    }
  };
  const double2* U = OP == AX_PAIR ? a.U + (int64_t)blockIdx.y * a.bstride : nullptr;
  for (int t = threadIdx.x; t < kAxLines * N; t += NT) {
    int j, e;
    at(t, j, e);
    if (j >= nl) continue;
    const int64_t o = base[j] + e * es;
    if constexpr (OP == AX_PAIR) {
      const double2 u = U[o], p = a.P[o];
      buf[j * LD + e] = make_double2(u.x * p.x + u.y * p.y, u.x * p.y - u.y * p.x);
    } else {
      buf[j * LD + e] = box[o];
    }
  }
  __syncthreads();
  fft_nat<double, OP == AX_INV, N>(buf, nl, LD, tw);
  if constexpr (OP == AX_KERN) {
    for (int t = threadIdx.x; t < kAxLines * N; t += NT) {
      int j, e;
      at(t, j, e);
      if (j >= nl) continue;
      const double k = a.kern[base[j] + e * es];
      const double2 v = buf[j * LD + e];
      buf[j * LD + e] = make_double2(k * v.x, k * v.y);
    }
    __syncthreads();
    fft_nat<double, true, N>(buf, nl, LD, tw);
  }
  for (int t = threadIdx.x; t < kAxLines * N; t += NT) {
    int j, e;
    at(t, j, e);
    if (j < nl) box[base[j] + e * es] = buf[j * LD + e];
  }
}

// y transforms of 16 columns of a plane: blockIdx = (column group, z, band)
template <int N, bool INV>
__global__ void __launch_bounds__(ax_threads<N>()) k_ax_y(PlaneArgs a, int nsticks, int ncols,
                                                        const int32_t* __restrict__ stick_at, int tw_off,
                                                        const double2* __restrict__ tw_g) {
  constexpr int NT = ax_threads<N>(), LD = N + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* buf = (double2*)smem_raw;
  double2* tw = buf + kAxLines * LD;
  const int c0 = blockIdx.x * kAxLines, z = blockIdx.y, b = blockIdx.z;
  const int nc = min(kAxLines, ncols - c0);
  double2* plane = a.W + (size_t)b * a.wband + (size_t)z * nsticks;
  double2* cols = a.C + (((size_t)b * gridDim.y + z) * ncols + c0) * N;
  const int32_t* sa = stick_at + (size_t)c0 * N;
  for (int t = threadIdx.x; t < N; t += NT) tw[t] = tw_g[tw_off + t];
  for (int t = threadIdx.x; t < nc * N; t += NT) {
    const int j = t / N, e = t - j * N;
    double2 v;
    if (INV) {
      const int st = sa[t];
      v = st >= 0 ? plane[st] : make_double2(0.0, 0.0);
    } else {
      v = cols[t];
    }
    buf[j * LD + e] = v;
  }
  __syncthreads();
  fft_nat<double, INV, N>(buf, nc, LD, tw);
  for (int t = threadIdx.x; t < nc * N; t += NT) {
    const int j = t / N, e = t - j * N;
    const double2 v = buf[j * LD + e];
    if (INV) {
      cols[t] = v;
    } else {
      const int st = sa[t];
      if (st >= 0) plane[st] = v;
    }
  }
}

// x transforms of 16 rows y0.. of a plane: blockIdx = (row group, z, band or
// slice of bands)
template <int N, int OP>
__global__ void __launch_bounds__(ax_threads<N>()) k_ax_x(PlaneArgs a, int ncols, int n2,
                                                        const int16_t* __restrict__ xcol, int tw_off,
                                                        const double2* __restrict__ tw_g) {
  constexpr int NT = ax_threads<N>(), LD = N + 1;
  constexpr int PER = (kAxLines * N + NT - 1) / NT;  // elements a thread
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* buf = (double2*)smem_raw;
  double2* tw = buf + kAxLines * LD;
  const int y0 = blockIdx.x * kAxLines, z = blockIdx.y;
  const int nr = min(kAxLines, n2 - y0);
  const size_t grid0 = ((size_t)z * n2 + y0) * N;  // V and rho at (z, y0, x = 0)
  for (int t = threadIdx.x; t < N; t += NT) tw[t] = tw_g[tw_off + t];
  auto load = [&](int b) {
    const double2* cols = a.C + ((size_t)b * gridDim.y + z) * ncols * n2 + y0;
    for (int t = threadIdx.x; t < kAxLines * N; t += NT) {
      const int e = t / kAxLines, j = t - e * kAxLines;
      if (j >= nr) continue;
      const int c = xcol[e];
      buf[j * LD + e] = c >= 0 ? cols[(size_t)c * n2 + j] : make_double2(0.0, 0.0);
    }
    __syncthreads();
  };
  if constexpr (OP == PL_XV) {
    const int b = blockIdx.z;
    load(b);
    fft_nat<double, true, N>(buf, nr, LD, tw);
    for (int t = threadIdx.x; t < nr * N; t += NT) {
      const int j = t / N, e = t - j * N;
      const double v = a.V[grid0 + t];
      const double2 w = buf[j * LD + e];
      buf[j * LD + e] = make_double2(v * w.x, v * w.y);
    }
    __syncthreads();
    fft_nat<double, false, N>(buf, nr, LD, tw);
    double2* cols = a.C + ((size_t)b * gridDim.y + z) * ncols * n2 + y0;
    for (int t = threadIdx.x; t < kAxLines * N; t += NT) {
      const int e = t / kAxLines, j = t - e * kAxLines;
      if (j >= nr) continue;
      const int c = xcol[e];
      if (c >= 0) cols[(size_t)c * n2 + j] = buf[j * LD + e];
    }
  } else {
    // a slice of bands summed in registers, one atomic a point
    double acc[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) acc[i] = 0.0;
    const int b1 = min(a.bb, ((int)blockIdx.z + 1) * a.per_slice);
    for (int b = blockIdx.z * a.per_slice; b < b1; ++b) {
      __syncthreads();  // the previous band's values are consumed
      load(b);
      fft_nat<double, true, N>(buf, nr, LD, tw);
      const double f = a.occ[b];
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        const int t = threadIdx.x + i * NT;
        if (t < nr * N) {
          const int j = t / N, e = t - j * N;
          const double2 v = buf[j * LD + e];
          acc[i] += f * (v.x * v.x + v.y * v.y);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int t = threadIdx.x + i * NT;
      if (t < nr * N) atomicAdd(a.rho + grid0 + t, acc[i]);
    }
  }
}

template <int N> void ax_attributes() {
  static std::once_flag once;
  std::call_once(once, [] {
    const int b = (int)ax_smem<N>();
    auto set = [&](auto k) { cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, b); };
    set(k_ax_box<N, AX_FWD>);
    set(k_ax_box<N, AX_INV>);
    set(k_ax_box<N, AX_PAIR>);
    set(k_ax_box<N, AX_KERN>);
    set(k_ax_y<N, true>);
    set(k_ax_y<N, false>);
    set(k_ax_x<N, PL_XV>);
    set(k_ax_x<N, PL_XDENS>);
    cudaFuncSetAttribute(ks_zinv<double, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    cudaFuncSetAttribute(ks_zfwd<double, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  });
}

template <int N> void ax_box_launch(System& s, AxisOp op, const AxisArgs& a) {
  ax_attributes<N>();
  const int64_t nlines = (int64_t)s.n1 * s.n2 * s.n3 / N;
  const dim3 g((unsigned)((nlines + kAxLines - 1) / kAxLines), (unsigned)a.nbox);
  const int off = s.plan[a.axis].tw_off;
  auto run = [&](auto k) {
    k<<<g, ax_threads<N>(), ax_smem<N>(), s.stream>>>(a, s.n1, s.n2, s.n3, off, s.d_tw64);
  };
  switch (op) {
    case AX_FWD: run(k_ax_box<N, AX_FWD>); break;
    case AX_INV: run(k_ax_box<N, AX_INV>); break;
    case AX_PAIR: run(k_ax_box<N, AX_PAIR>); break;
    case AX_KERN: run(k_ax_box<N, AX_KERN>); break;
  }
  PWH_LAUNCH_CHECK();
}

template <int N> void ax_plane_launch(System& s, PlaneOp op, const PlaneArgs& a) {
  ax_attributes<N>();
  constexpr int NT = ax_threads<N>();
  if (op == PL_YINV || op == PL_YFWD) {
    const dim3 g((s.ncols + kAxLines - 1) / kAxLines, s.n3, a.bb);
    const int off = s.plan[1].tw_off;
    if (op == PL_YINV)
      k_ax_y<N, true><<<g, NT, ax_smem<N>(), s.stream>>>(a, s.nsticks, s.ncols, s.d_stick_at, off, s.d_tw64);
    else
      k_ax_y<N, false><<<g, NT, ax_smem<N>(), s.stream>>>(a, s.nsticks, s.ncols, s.d_stick_at, off, s.d_tw64);
  } else {
    const int slices = op == PL_XV ? a.bb : (a.bb + a.per_slice - 1) / a.per_slice;
    const dim3 g((s.n2 + kAxLines - 1) / kAxLines, s.n3, slices);
    const int off = s.plan[0].tw_off;
    if (op == PL_XV)
      k_ax_x<N, PL_XV><<<g, NT, ax_smem<N>(), s.stream>>>(a, s.ncols, s.n2, s.d_xcol, off, s.d_tw64);
    else
      k_ax_x<N, PL_XDENS><<<g, NT, ax_smem<N>(), s.stream>>>(a, s.ncols, s.n2, s.d_xcol, off, s.d_tw64);
  }
  PWH_LAUNCH_CHECK();
}

template <int N> void ax_z_launch(System& s, bool inverse, const PassArgs& a) {
  ax_attributes<N>();
  const dim3 gz((s.nsticks + a.spb - 1) / a.spb, a.bb);
  if (inverse)
    ks_zinv<double, N><<<gz, 256, a.zsmem, a.st>>>(a.psi, a.ldp, s.d_stick_off, s.d_stick_of, s.d_zpos,
                                                 s.nsticks, s.plan[2].tw_off, s.plan[2].perm_off, s.d_tw64,
                                                 s.d_perm, (double2*)a.W, a.wband, a.spb);
  else
    ks_zfwd<double, N><<<gz, 256, a.zsmem, a.st>>>((const double2*)a.W, a.wband, s.d_stick_off, s.d_stick_of,
                                                 s.d_zpos, s.nsticks, s.plan[2].tw_off, s.plan[2].perm_off,
                                                 s.d_tw64, s.d_perm, s.d_kin, a.psi, a.ldp, a.hpsi, a.ldh,
                                                 a.spb, a.vnl, a.ldv);
  PWH_LAUNCH_CHECK();
}

// One translation unit per list of sizes: false when n is not in it.
#define PWH_AXIS_UNIT(NAME, LIST)                                              \
  bool ax_has_##NAME(int n) {                                                  \
    switch (n) { LIST(PWH_AXIS_HAS) default: return false; }                   \
  }                                                                            \
  bool ax_box_##NAME(System& s, int n, AxisOp op, const AxisArgs& a) {         \
    switch (n) { LIST(PWH_AXIS_BOX) default: return false; }                   \
  }                                                                            \
  bool ax_plane_##NAME(System& s, int n, PlaneOp op, const PlaneArgs& a) {     \
    switch (n) { LIST(PWH_AXIS_PLANE) default: return false; }                 \
  }                                                                            \
  bool ax_z_##NAME(System& s, int n, bool inverse, const PassArgs& a) {        \
    switch (n) { LIST(PWH_AXIS_Z) default: return false; }                     \
  }
#define PWH_AXIS_HAS(n) case n: return true;
#define PWH_AXIS_BOX(n) case n: ax_box_launch<n>(s, op, a); return true;
#define PWH_AXIS_PLANE(n) case n: ax_plane_launch<n>(s, op, a); return true;
#define PWH_AXIS_Z(n) case n: ax_z_launch<n>(s, inverse, a); return true;

}  // namespace pwh
