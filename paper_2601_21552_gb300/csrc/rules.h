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

// Search steps between two flushes of a warp's 32-bit work counters into the
// caller's 64-bit ones: a power of two, at most 64, such that no counter can pass
// 32 bits in between. A step (one propagation to a fixpoint and what follows)
// visits every occurrence entry and every literal of a learned clause at most
// once, and undoes or reads the activity of every variable at most once.
SCUBA_HD uint32_t flush_steps(uint64_t entries, uint64_t learned_words, uint64_t variables) {
  const uint64_t most = entries + learned_words + variables;
  uint32_t steps = 64;
  while (steps > 1 && most > 0xffffffffull / steps) steps /= 2;
  return steps;
}

}  // namespace scuba
