// H|psi> = kinetic + local (FFT passes) + nonlocal sum_ij beta_i D_ij <beta_j|psi>
// (Eq. pauli_ks, S = 1), and the public entry points that apply it.
//
// Nonlocal step: becp = beta^H psi (the p_ij of Sec. "New parallelization
// levels"), becp' = D becp, hpsi += beta becp'.  FP64: complex GEMMs on the FP64
// pipe, with a diagonal D folded into the split-K reduction.  Mixed: the BF16
// tensor-core path of gemm_tc.cu.
#include <algorithm>

#include "common.cuh"
#include "gemm.cuh"

namespace pwh {

// dst[b][i] = src[b][idx[i]]: bands between the public and the internal order,
// both ways as gathers (idx = int_to_pub or pub_to_int).  Bound by L2: neighbouring
// threads take neighbouring elements of one band, whose 16-byte reads stay within
// the band (scattered 16-byte writes filled half a sector each: the way out took
// 1.40 ms for 512 bands of 161,235 plane waves and takes 0.46 as a gather).  One
// range over all bands, so that few short bands fill their blocks (30^3, 4 bands: H
// 24.8 us, with a row of blocks a band 26.9).  I: unsigned where that range has fewer
// than 2^31 elements; a 64-bit division is most of a thread's work (80^3, 8 bands: H
// 60.5 us with it, 57.6 without).
template <typename I>
__global__ void __launch_bounds__(256) k_permute(const double2* __restrict__ src, int64_t lds, I npw, I tot,
                                                 const int32_t* __restrict__ idx,
                                                 double2* __restrict__ dst, int64_t ldd) {
  for (I t = blockIdx.x * (I)256 + threadIdx.x; t < tot; t += gridDim.x * (I)256) {
    const I b = t / npw, i = t - b * npw;
    dst[(int64_t)b * ldd + i] = src[(int64_t)b * lds + idx[i]];
  }
}

static void permute(System& s, int nb, const double2* src, int64_t lds, const int32_t* idx, double2* dst,
                    int64_t ldd) {
  const int64_t tot = s.npw * (int64_t)nb;
  const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(152 * 16, (tot + 255) / 256));
  if (tot < ((int64_t)1 << 31))
    k_permute<unsigned><<<blocks, 256, 0, s.stream>>>(src, lds, (unsigned)s.npw, (unsigned)tot, idx, dst, ldd);
  else
    k_permute<int64_t><<<blocks, 256, 0, s.stream>>>(src, lds, s.npw, tot, idx, dst, ldd);
  PWH_LAUNCH_CHECK();
}

void permute_public_to_internal(System& s, const double2* src, double2* dst, int nb, int64_t lds) {
  permute(s, nb, src, lds > 0 ? lds : s.npw, s.d_int_to_pub, dst, s.npw);
}

void nonlocal_fp64(System& s, int nb, const double2* psi, int64_t ldp, double2* hpsi, int64_t ldh,
                   cudaStream_t st) {
  if (s.nproj == 0 || nb <= 0) return;
  const int P = s.nproj;
  ensure(s.ws_becp, (size_t)2 * P * nb * sizeof(double2));
  double2* becp = (double2*)s.ws_becp.p;
  double2* becp2 = becp + (size_t)P * nb;
  const double2 one = make_double2(1, 0), zero = make_double2(0, 0);
  if (s.d_diag) {
    cgemm<double>(s, true, P, nb, (int)s.npw, one, s.d_beta64, s.npw, psi, ldp, zero, becp, P, st,
                  s.d_ddiag);
  } else {
    cgemm<double>(s, true, P, nb, (int)s.npw, one, s.d_beta64, s.npw, psi, ldp, zero, becp2, P, st);
    cgemm<double>(s, false, P, nb, P, one, s.d_dfull, P, becp2, P, zero, becp, P, st);
  }
  cgemm<double>(s, false, (int)s.npw, nb, P, one, s.d_beta64, s.npw, becp, P, one, hpsi, ldh, st);
}

void ace_apply(System& s, int nb, const double2* psi, int64_t ldp, double2* hpsi, int64_t ldh,
               int precision);  // exx.cu

void apply_internal(System& s, int nb, const double2* psi, int64_t ldp, double2* hpsi, int64_t ldh,
                    int precision) {
  if (!s.have_v) throw Error{PWH_ERR_STATE, "pwh_set_potential has not been called"};
  if (nb <= 0) return;
  if (precision == PWH_FP64) {
    local_kinetic<double>(s, nb, psi, ldp, hpsi, ldh, s.stream);
    nonlocal_fp64(s, nb, psi, ldp, hpsi, ldh, s.stream);
    ace_apply(s, nb, psi, ldp, hpsi, ldh, precision);
  } else {
    // the nonlocal term first, into an FP32 buffer that the last FFT pass adds
    float2* vnl = nullptr;
    if (s.nproj > 0) {
      ensure(s.ws_vnl, (size_t)s.npw * nb * sizeof(float2));
      vnl = (float2*)s.ws_vnl.p;
      nonlocal_mixed(s, nb, psi, ldp, vnl, s.npw, s.stream, precision == PWH_MIXED_FAST ? 1 : 3);
    }
    local_kinetic<float>(s, nb, psi, ldp, hpsi, ldh, s.stream, vnl, s.npw);
    ace_apply(s, nb, psi, ldp, hpsi, ldh, precision);
  }
}

}  // namespace pwh

using namespace pwh;

extern "C" {

pwh_status pwh_apply_h_internal(pwh_system* sys, int32_t nb, const void* psi, int64_t ld_psi,
                                void* hpsi, int64_t ld_hpsi) {
  return guarded([&] {
    PWH_CHECK_ARG(sys, "null system");
    System& s = sys->s;
    PWH_CHECK_ARG(nb >= 0, "nb < 0");
    if (nb == 0) return;
    PWH_CHECK_ARG(psi && hpsi, "null band pointer");
    PWH_CHECK_ARG(ld_psi >= s.npw && ld_hpsi >= s.npw, "leading dimension < npw");
    apply_internal(s, nb, (const double2*)psi, ld_psi, (double2*)hpsi, ld_hpsi, s.precision);
  });
}

pwh_status pwh_apply_h(pwh_system* sys, int32_t nb, const void* psi, int64_t ld_psi, void* hpsi,
                       int64_t ld_hpsi) {
  return guarded([&] {
    PWH_CHECK_ARG(sys, "null system");
    System& s = sys->s;
    PWH_CHECK_ARG(nb >= 0, "nb < 0");
    if (nb == 0) return;
    PWH_CHECK_ARG(psi && hpsi, "null band pointer");
    PWH_CHECK_ARG(ld_psi >= s.npw && ld_hpsi >= s.npw, "leading dimension < npw");
    if (!s.have_v) throw Error{PWH_ERR_STATE, "pwh_set_potential has not been called"};
    const size_t n = (size_t)s.npw * nb;
    ensure(s.ws_psi, n * sizeof(double2));
    ensure(s.ws_hpsi, n * sizeof(double2));
    double2* pi = (double2*)s.ws_psi.p;
    double2* hi = (double2*)s.ws_hpsi.p;
    permute(s, nb, (const double2*)psi, ld_psi, s.d_int_to_pub, pi, s.npw);
    apply_internal(s, nb, pi, s.npw, hi, s.npw, s.precision);
    permute(s, nb, hi, s.npw, s.d_pub_to_int, (double2*)hpsi, ld_hpsi);
  });
}

pwh_status pwh_apply_h_host(pwh_system* sys, int32_t nb, const void* psi_host, void* hpsi_host) {
  return guarded([&] {
    PWH_CHECK_ARG(sys, "null system");
    System& s = sys->s;
    PWH_CHECK_ARG(nb >= 0, "nb < 0");
    if (nb == 0) return;
    PWH_CHECK_ARG(psi_host && hpsi_host, "null band pointer");
    const size_t n = (size_t)s.npw * nb;
    // ws_host holds the device copies of psi (first half) and hpsi (second half)
    ensure(s.ws_host, 2 * n * sizeof(double2));
    double2* dp = (double2*)s.ws_host.p;
    double2* dh = dp + n;
    PWH_CUDA(cudaMemcpyAsync(dp, psi_host, n * sizeof(double2), cudaMemcpyHostToDevice, s.stream));
    pwh_status st = pwh_apply_h(sys, nb, dp, s.npw, dh, s.npw);
    if (st != PWH_OK) throw Error{st, pwh_last_error()};
    PWH_CUDA(cudaMemcpyAsync(hpsi_host, dh, n * sizeof(double2), cudaMemcpyDeviceToHost, s.stream));
    PWH_CUDA(cudaStreamSynchronize(s.stream));
  });
}

}  // extern "C"
