// Double-float instances of the compile-time specialised FFT passes: the FP64
// local part of H on the FP32 pipes.
#include "fft_df.cuh"
#include "fft_spec_impl.cuh"

namespace pwh {
template <> bool spec_pass<df>(SpecPass pass, System& s, const PassArgs& a) {
  if (s.n1 != s.n2 || s.n2 != s.n3) return false;
  switch (s.n1) {
#define PWH_SPEC_CASE(n)                                                               \
  case n:                                                                              \
    spec_launch<DfPass<n>, n>(pass, s, a);                                             \
    return true;
    PWH_SPEC_SIZES(PWH_SPEC_CASE)
#undef PWH_SPEC_CASE
    default: return false;
  }
}
}  // namespace pwh
