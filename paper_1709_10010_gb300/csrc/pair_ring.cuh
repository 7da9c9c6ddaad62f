// The ring of a CTA pair at its end (gemm_mod.cu).  Both CTAs' copies into a slot
// complete on CTA 0's barrier, which CTA 0 arms for both as it fills the slot; CTA 1 may
// be ahead of it.
#pragma once

namespace pwh {

#ifdef __CUDACC__
#define PWH_HD __host__ __device__
#else
#define PWH_HD
#endif

// What CTA 0 does once both producers have stopped, after filling `own` slots here and
// `other` in CTA 1 (the two differ only after a time-out): the fills arm0.. < arm1, which
// only CTA 1 made, are armed for its copies alone; then the fills wait0.. < wait1 are
// waited for, each the last of its slot.
struct PairDrain {
  int arm0, arm1, wait0, wait1;
};
PWH_HD constexpr PairDrain pair_drain(int own, int other, int stages) {
  const int last = own > other ? own : other;
  return {own, other, last > stages ? last - stages : 0, last};
}

}  // namespace pwh
