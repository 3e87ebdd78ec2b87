// A converter group's place in the tensor-core router's ring of stages
// (router_tc.cu).  Plain C++, so that the host can run it too.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define XS_HD __host__ __device__ __forceinline__
#else
#define XS_HD inline
#endif

namespace xs {

// Group g of kGroups takes the K steps g, g + kGroups, ...; step i lies in
// stage i % stages, in its round i / stages (phase: the round's parity).  At least two stages.
template <int kGroups>
struct ConvRing {
  int stage, stages;
  uint32_t phase;

  XS_HD ConvRing(int group, int n_stages)
      : stage(group % n_stages), stages(n_stages), phase(static_cast<uint32_t>(group / n_stages) & 1u) {}

  XS_HD void next() {
    stage += kGroups;
    while (stage >= stages) {
      stage -= stages;
      phase ^= 1u;
    }
  }

  // True once the step's operands are in its stage; wait_empty and wait_full
  // (stage, parity) wait on the stage's barriers.  A parity wait cannot tell
  // round r from round r - 2: asked for round r while round r - 1 is still
  // loading, it passes at once.  The step of round r - 1 belongs to the other
  // group if `stages` is odd (3 and 5 are), and its load may land after loads
  // issued later, so nothing that this group has seen says that it is over.
  // The stage's release by the MMAs of round r - 1 does, and it cannot be a
  // round ahead, since round r's MMAs need this group.  The load of round r
  // is not issued before it either, so the extra wait costs no time.
  template <class Empty, class Full>
  XS_HD bool wait(Empty wait_empty, Full wait_full) const {
    return wait_empty(stage, phase ^ 1u) && wait_full(stage, phase);
  }
};

}  // namespace xs
