// rules.h -- arithmetic of the searches that needs no GPU (plain C++ too).
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define SCUBA_HD __host__ __device__ __forceinline__
#else
#define SCUBA_HD inline
#endif

namespace scuba {

// Nanoseconds from `start` to `now`, two readings of the global timer by
// different SMs: a clock slightly behind the one that set the start reads as no
// time, not as 584 years.
SCUBA_HD uint64_t elapsed_ns(uint64_t start, uint64_t now) {
  return (int64_t)(now - start) < 0 ? 0 : now - start;
}

}  // namespace scuba
