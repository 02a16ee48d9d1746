// stage_drain.h -- which stages of a ring a role still has to see released before its CTA
// leaves.  Plain C++: the rule is checked on the host.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define GBPIR_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define GBPIR_HOST_DEVICE inline
#endif

namespace gbpir {

// Of the stages group, group + groups, ... below `stages`, the first whose slot of the ring no
// later stage of any group takes: nobody waits for the release of that one or of the role's later
// ones in order to refill them.  `stages` if there is none.
GBPIR_HOST_DEVICE uint64_t first_undrained(uint64_t stages, uint32_t group, uint32_t groups, uint32_t ring) {
  if (stages <= group) return stages;
  const uint64_t from = stages > ring ? stages - ring : 0;
  return from <= group ? group : group + (from - group + groups - 1) / groups * groups;
}

}  // namespace gbpir
