// closure.cuh -- unit propagation of scuba_propagate_batch (included by solver.cu
// inside namespace scuba::dev). A closure's rounds are wide (whole input words
// are assumed at once, frontiers of hundreds of literals), unlike the searches'.
// One warp takes a batch of 32 frontier literals' entries as one list
// (close_rounds); where instances are few and large a block's warps share one:
// eight lanes take a literal's list, every lane claims what its entry implies by
// itself, and a round ends at a barrier (close_shared). The closure does not
// depend on the order of that.
// What a conflict leaves in the assignment does (the interface leaves those
// values open), so an instance that conflicts is done again by one warp
// (close_rounds): however many warps took it first, its values are those of one
// walk over the lists in their order. That order is the clauses' but for the
// entries of 32 neighbouring clauses, and the claims of one step take the order in
// which the SM serves a warp's shared-memory atomics; neither has been seen to
// differ between runs, and nothing promises it.

__device__ __forceinline__ void close_conflict(Warp& w, uint32_t a, uint32_t b, uint32_t c) {
  if (atomicCAS(&w.ws->conflict, 0u, 1u) == 0u) {
    w.ws->cl[0] = a;
    w.ws->cl[1] = b;
    w.ws->cl[2] = c;
  }
}

// Assign literal l true. Returns false on a clash with the opposite value.
__device__ __forceinline__ bool close_claim(Warp& w, uint32_t l) {
  uint32_t v = WIDX(w, l >> 1, w.V, 1);
  uint32_t sh = (v & 15u) * 2u;
  uint32_t mask = ((l & 1u) ? 2u : 1u) << sh;
  uint32_t old = atomicOr(&w.asg[v >> 4], mask);
  uint32_t ob = (old >> sh) & 3u;
  if (ob == 0u) {
    uint32_t pos = atomicAdd(&w.ws->tail, 1u);
    w.trail[WIDX(w, pos, w.V, 2)] = l;
    return true;
  }
  if (ob == (mask >> sh)) return true;
  if ((old & mask) == 0u) atomicAnd(&w.asg[v >> 4], ~mask);  // undo our bit
  return false;
}

__device__ void close_long(Warp& w, uint32_t local, uint32_t f) {
  const int64_t c = w.c0 + local;
  const int64_t b = w.cb[c], e = w.cb[c + 1];
  uint32_t open_lit = NONE;
  int n_open = 0;
  for (int64_t q = b; q < e; q++) {
    uint32_t x = code_of(__ldg(&w.lits[q]));
    uint32_t vx = lit_value(w.asg, x);
    if (vx == LV_T || vx == LV_X) return;
    if (vx == LV_U && x != open_lit) {
      n_open++;
      open_lit = x;
      if (n_open > 1) return;
    }
  }
  if (n_open == 0) {
    close_conflict(w, LONG_CLAUSE | local, NONE, NONE);
  } else if (!close_claim(w, open_lit)) {
    close_conflict(w, LONG_CLAUSE | local, NONE, NONE);
  }
}

// Visit one occurrence entry of the falsified literal f.
__device__ __forceinline__ void close_entry(Warp& w, uint32_t f, uint64_t e) {
  const uint32_t a0 = (uint32_t)e, b0 = (uint32_t)(e >> 32);
  if (a0 & LONG_CLAUSE) {
    close_long(w, a0 & ~LONG_CLAUSE, f);
    return;
  }
  const uint32_t a = WIDX(w, a0, 2u * w.V, 3);
  const uint32_t b = b0 == NONE ? NONE : WIDX(w, b0, 2u * w.V, 3);
  const uint32_t va = lit_value(w.asg, a);
  if (b == NONE) {  // binary (f | a)
    if (va == LV_T || va == LV_X) return;
    if (va == LV_F || !close_claim(w, a)) close_conflict(w, f, a, NONE);
    return;
  }
  const uint32_t vb = lit_value(w.asg, b);  // ternary (f | a | b)
  if (va == LV_T || vb == LV_T || va == LV_X || vb == LV_X) return;
  if (va == LV_F && vb == LV_F) {
    close_conflict(w, f, a, b);
  } else if (va == LV_F) {
    if (!close_claim(w, b)) close_conflict(w, f, a, b);
  } else if (vb == LV_F) {
    if (!close_claim(w, a)) close_conflict(w, f, a, b);
  }
}

// Unit propagation to a fixpoint by one warp. Returns true on conflict.
// Each round takes the trail literals assigned in the previous round (the
// frontier), 32 at a time, and spreads their occurrence entries over the lanes as
// one list. The values of a conflicting instance are what this order of visits
// leaves.
__device__ bool close_rounds(Warp& w) {
  for (;;) {
    __syncwarp();
    const uint32_t hi = *(volatile uint32_t*)&w.ws->tail;
    if (w.head >= hi) return false;
    const uint32_t lo = w.head;
    w.head = hi;
    for (uint32_t base = lo; base < hi; base += 32) {
      const uint32_t nlit = min(32u, hi - base);
      if (nlit == 1) {
        // one literal: every lane reads the same list bounds (broadcast)
        const uint32_t f = WIDX(w, w.trail[base] ^ 1u, 2u * w.V, 4);
        const uint32_t beg = __ldg(&w.occ[f]);
        const uint32_t cnt = __ldg(&w.occ[f + 1]) - beg;
        for (uint32_t e = w.lane; e < cnt; e += 32)
          close_entry(w, f, __ldg(&w.ent[WIDX(w, beg + e, w.ent_end, 5)]));
      } else {
        uint32_t f = 0, beg = 0, cnt = 0;
        if (w.lane < nlit) {
          f = WIDX(w, w.trail[base + w.lane] ^ 1u, 2u * w.V, 4);  // the literal that became false
          beg = __ldg(&w.occ[f]);
          cnt = __ldg(&w.occ[f + 1]) - beg;
        }
        uint32_t inc = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          uint32_t y = __shfl_up_sync(FULL, inc, d);
          if (w.lane >= d) inc += y;
        }
        const uint32_t excl = inc - cnt;
        const uint32_t total = __shfl_sync(FULL, inc, 31);
        if (total <= 32) {
          // owner of entry e = the lane whose segment starts at the last
          // segment start <= e: segment starts as a bit mask, ranks by popc
          const bool has = cnt > 0;
          const uint32_t starts = __reduce_or_sync(FULL, has ? (1u << excl) : 0u);
          const uint32_t nz = __ballot_sync(FULL, has);
          const uint32_t e = w.lane;
          int j = 0;
          if (e < total) {
            const int rank = __popc(starts & ((2u << e) - 1u)) - 1;
            j = __fns(nz, 0, rank + 1);
          }
          const uint32_t jbeg = __shfl_sync(FULL, beg, j);
          const uint32_t jex = __shfl_sync(FULL, excl, j);
          const uint32_t jf = __shfl_sync(FULL, f, j);
          if (e < total) close_entry(w, jf, __ldg(&w.ent[WIDX(w, jbeg + (e - jex), w.ent_end, 5)]));
        } else {
          for (uint32_t e0 = 0; e0 < total; e0 += 32) {
            const uint32_t e = e0 + w.lane;
            // owner = smallest lane j with inc_j > e
            int lo_j = 0, hi_j = 31;
#pragma unroll
            for (int s2 = 0; s2 < 5; s2++) {
              int mid = (lo_j + hi_j) >> 1;
              uint32_t v = __shfl_sync(FULL, inc, mid);
              if (v > e) hi_j = mid; else lo_j = mid + 1;
              if (lo_j > hi_j) lo_j = hi_j;
            }
            const int j = lo_j;
            const uint32_t jbeg = __shfl_sync(FULL, beg, j);
            const uint32_t jex = __shfl_sync(FULL, excl, j);
            const uint32_t jf = __shfl_sync(FULL, f, j);
            if (e < total) close_entry(w, jf, __ldg(&w.ent[WIDX(w, jbeg + (e - jex), w.ent_end, 5)]));
          }
        }
      }
      __syncwarp();
      if (*(volatile uint32_t*)&w.ws->conflict) return true;
    }
  }
}

// Unit propagation to a fixpoint by the whole block. Returns true on conflict.
// The next literal's list bounds are loaded before this one's entries are
// evaluated, and its first entries before those of this one's are used up.
__device__ __forceinline__ bool close_shared(Warp& w) {
  const uint32_t groups = blockDim.x >> 3, sub = threadIdx.x & 7u;
  uint32_t lo = 0;
  for (;;) {
    __syncthreads();
    const uint32_t hi = *(volatile uint32_t*)&w.ws->tail;
    const uint32_t bad = *(volatile uint32_t*)&w.ws->conflict;
    __syncthreads();  // everyone has read the tail before it moves again
    if (bad) return true;
    if (lo >= hi) return false;
    uint32_t p = lo + (threadIdx.x >> 3);
    uint32_t f = 0, beg = 0, end = 0;
    if (p < hi) {
      f = WIDX(w, w.trail[p] ^ 1u, 2u * w.V, 4);
      beg = __ldg(&w.occ[f]);
      end = __ldg(&w.occ[f + 1]);
    }
    while (p < hi) {
      uint32_t k = beg + sub;
      uint64_t e = 0;
      if (k < end) e = __ldg(&w.ent[WIDX(w, k, w.ent_end, 5)]);
      const uint32_t f0 = f, end0 = end;
      p += groups;
      if (p < hi) {
        f = WIDX(w, w.trail[p] ^ 1u, 2u * w.V, 4);
        beg = __ldg(&w.occ[f]);
        end = __ldg(&w.occ[f + 1]);
      }
      while (k < end0) {
        const uint64_t e0 = e;
        k += 8;
        if (k < end0) e = __ldg(&w.ent[WIDX(w, k, w.ent_end, 5)]);
        close_entry(w, f0, e0);
      }
    }
    lo = hi;
  }
}
