// prep.cuh -- from the caller's CSR to occurrence lists (included by solver.cu
// inside namespace scuba::dev).
//
// k_setup clears the call's control block and per-unit state and lays out the
// instances' occurrence offsets; k_prep then validates and normalises the
// clauses of every instance (duplicate literals removed, tautologies dropped,
// unit clauses collected) and writes its occurrence lists.
//
// One block takes one work item: an instance, or for an instance of more than
// `range` literal codes one range of them. Its warps own contiguous runs of the
// instance's clauses. Pass 1 counts, per warp and literal code of the range,
// the occurrences in shared memory; a scan over (literal, warp) turns the
// counts into list offsets and per-warp cursors; pass 2 reads the clauses again
// (from L2: an instance is a few 100 KB) and writes each entry where its warp's
// cursor stands. A list is therefore in the order of the clauses' groups of 32,
// the same in every run, and no count, cursor or normalised literal goes
// through global memory. The ranges of one large instance need nothing from
// each other: a block also counts the literals below its range, which is where
// its first list begins.

// Header checks, scratch layout and launch shape of one call's preparation.
struct Prep {
  int n;
  int64_t C, L;
  int64_t total_vars;  // model size promised by the caller
  int64_t occ_cap;     // allocated occurrence-offset entries
  int32_t vmax;
  uint32_t range;      // literal codes a work item covers (even)
  const int64_t* vb;
  Ctrl* ctrl;
  const int64_t* icb;
  const int64_t* cb;
  const int32_t* lits;
  const int32_t* nv;
  int64_t* occ_base;   // [n+1]
  uint32_t* occ_begin; // [occ_total]
  uint64_t* ent;       // [L]
  uint32_t* units;     // [C]
  uint32_t* nunits;    // [n]
  uint32_t* flags;     // [n]
  int2* items;         // {instance, range} of each work item; NULL: item i is instance i
  uint32_t item_cap;
};

// State a search starts from (n_units = 0: a propagation call, none of it).
struct SearchInit {
  int n_units;
  uint32_t* pending;
  uint32_t* done;
  unsigned long long* inst_dec;
  uint8_t* verdict;
  Job* ring;
  uint32_t ring_cap;
  unsigned long long* share_cur;   // clause-sharing cursors; NULL: no sharing
  unsigned long long* share_base;  // where this call's records begin
  uint32_t share_pools;
};

__device__ __forceinline__ int32_t clamp_nv(int32_t v, int32_t vmax) {
  return v < 0 ? 0 : (v > vmax ? vmax : v);
}

// Exclusive sum over the block's threads; total gets the block's sum.
template <class T>
__device__ __forceinline__ T block_exclusive(T v, T* part /* [32] shared */, T& total) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, nw = blockDim.x >> 5;
  T inc = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const T y = __shfl_up_sync(FULL, inc, d);
    if (lane >= d) inc += y;
  }
  __syncthreads();  // part may still be read from an earlier call
  if (lane == 31) part[wib] = inc;
  __syncthreads();
  T w = lane < nw ? part[lane] : T(0), winc = w;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const T y = __shfl_up_sync(FULL, winc, d);
    if (lane >= d) winc += y;
  }
  total = __shfl_sync(FULL, winc, 31);
  return __shfl_sync(FULL, winc - w, wib) + inc - v;
}

// Work items of an instance of V variables.
__device__ __forceinline__ uint32_t item_count(int32_t V, uint32_t range) {
  return max(1u, (2u * (uint32_t)V + range - 1u) / range);
}

// Block 0: the control block, then occ_base[i] = sum_{j<i} (2 nv[j] + 1) and
// the work items. The other blocks: the units' state, the verdicts (UNKNOWN
// until a unit is finished), the job ring and the sharing pools' bases.
__global__ void __launch_bounds__(1024) k_setup(Prep P, SearchInit I) {
  if (blockIdx.x > 0) {
    const int stride = (gridDim.x - 1) * blockDim.x;
    const int first = (blockIdx.x - 1) * blockDim.x + threadIdx.x;
    for (int i = first; i < I.n_units; i += stride) {
      I.pending[i] = 1u;
      I.done[i] = 0u;
      I.inst_dec[i] = 0ull;
      I.verdict[i] = SCUBA_UNKNOWN;
    }
    for (uint32_t i = first; i < I.ring_cap; i += stride) I.ring[i].seq = i;
    // records of earlier calls stay in the pools; this call's begin at the
    // cursors' present values, and no job reads below them
    if (I.share_cur)
      for (uint32_t i = first; i < I.share_pools; i += stride) I.share_base[i] = I.share_cur[i];
    return;
  }
  __shared__ long long part[32];
  __shared__ uint32_t ipart[32];
  constexpr int PER = 4;  // instances a thread takes per round
  const int n = P.n;
  if (threadIdx.x == 0) {
    Ctrl* c = P.ctrl;
    c->next_inst = 0;
    c->inst_left = (uint32_t)I.n_units;
    c->idle = 0;
    c->status = 0;
    c->q_head = 0;
    c->q_tail = 0;
    c->t0 = 0;
    c->jobs_split = 0;
    c->check_site = 0;
    c->check_index = 0;
    c->check_limit = 0;
    c->next_item = 0;
    c->n_items = (uint32_t)n;
  }
  long long carry = 0;
  uint32_t items = 0;
  for (int i0 = 0; i0 < n; i0 += PER * (int)blockDim.x) {
    const int b = i0 + PER * (int)threadIdx.x;
    int32_t v[PER];
    long long s = 0;
    uint32_t m = 0;
#pragma unroll
    for (int k = 0; k < PER; k++) v[k] = b + k < n ? clamp_nv(P.nv[b + k], P.vmax) : -1;
#pragma unroll
    for (int k = 0; k < PER; k++)
      if (v[k] >= 0) {
        s += 2 * (long long)v[k] + 1;
        m += item_count(v[k], P.range);
      }
    long long total;
    long long at = carry + block_exclusive(s, part, total);
    carry += total;
#pragma unroll
    for (int k = 0; k < PER; k++)
      if (v[k] >= 0) {
        P.occ_base[b + k] = at;
        at += 2 * (long long)v[k] + 1;
      }
    if (P.items) {
      uint32_t mtotal;
      uint32_t it = items + block_exclusive(m, ipart, mtotal);
      items += mtotal;
#pragma unroll
      for (int k = 0; k < PER; k++)
        if (v[k] >= 0)
          for (uint32_t r = 0, e = item_count(v[k], P.range); r < e; r++, it++)
            if (it < P.item_cap) P.items[it] = make_int2(b + k, (int)r);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    P.occ_base[n] = carry;
    if (P.items) P.ctrl->n_items = items;
    // more variables than the caller promised (the items then need not fit)
    if (carry > P.occ_cap || (P.items && items > P.item_cap))
      fail_batch(P.ctrl, SCUBA_ERR_MALFORMED);
  }
}

// One clause as a lane sees it: its literal range in the caller's CSR and, up
// to length 3, its literals.
struct RawClause {
  int64_t b, e;
  int32_t l[3];
};

__device__ __forceinline__ RawClause load_bounds(const Prep& P, int64_t c, int64_t c1) {
  RawClause R;
  R.b = R.e = 0;
  if (c < c1) {
    R.b = __ldg(P.cb + c);
    R.e = __ldg(P.cb + c + 1);
  }
  return R;
}

__device__ __forceinline__ void load_literals(const Prep& P, RawClause& R) {
  const int64_t len = R.b >= 0 && R.e <= P.L ? R.e - R.b : 0;
#pragma unroll
  for (int k = 0; k < 3; k++) R.l[k] = k < len ? __ldg(P.lits + R.b + k) : 0;
}

// The warp's clauses [s0, s1) in groups of 32, fn(group start, lane's clause):
// the literals of the next group and the bounds of the one after it are on
// their way while a group is handled.
template <class Fn>
__device__ __forceinline__ void each_group(const Prep& P, int64_t s0, int64_t s1, int lane,
                                           Fn&& fn) {
  RawClause R = load_bounds(P, s0 + lane, s1);
  RawClause N = load_bounds(P, s0 + 32 + lane, s1);
  load_literals(P, R);
  for (int64_t cs = s0; cs < s1; cs += 32) {
    load_literals(P, N);
    const RawClause M = load_bounds(P, cs + 64 + lane, s1);
    fn(cs, R);
    R = N;
    N = M;
  }
}

enum { CL_NONE, CL_SHORT, CL_UNIT, CL_LONG };

// Normalise a clause: CL_SHORT with its 2 or 3 distinct codes in u, CL_UNIT
// with u[0], CL_LONG (its codes are read from the CSR as they stand), CL_NONE
// (no clause, a tautology, or one that raised F_EMPTY / F_BAD in f).
__device__ __forceinline__ int classify(const Prep& P, const RawClause& R, bool valid, int V,
                                        uint32_t u[3], int& nk, uint32_t& f) {
  nk = 0;
  if (!valid) return CL_NONE;
  if (R.b < 0 || R.e < R.b || R.e > P.L) {
    f |= F_BAD;
    return CL_NONE;
  }
  const int64_t len = R.e - R.b;
  if (len == 0) {
    f |= F_EMPTY;
    return CL_NONE;
  }
  if (len > 3) return CL_LONG;
  bool bad = false, taut = false;
#pragma unroll
  for (int q = 0; q < 3; q++) {
    if (q >= len) break;
    const int32_t l = R.l[q];
    bad |= l == 0 || l > V || l < -V;
    const uint32_t x = code_of(l);
    bool dup = false;
#pragma unroll
    for (int r = 0; r < 2; r++)
      if (r < nk) {
        dup |= u[r] == x;
        taut |= u[r] == (x ^ 1u);
      }
    if (!dup) {
      if (nk == 0) u[0] = x;
      else if (nk == 1) u[1] = x;
      else u[2] = x;
      nk++;
    }
  }
  if (bad) {
    f |= F_BAD;
    nk = 0;
    return CL_NONE;
  }
  if (taut) {
    nk = 0;
    return CL_NONE;
  }
  if (nk == 1) {
    nk = 0;
    return CL_UNIT;
  }
  return CL_SHORT;
}

// WARPS = 8 for batches whose literals fit one item (several blocks per SM),
// 32 for larger ones (one block per SM; a large instance is cut into ranges).
// Per item the clauses are read twice; the passes are bound by the latency of
// their loads and shared-memory updates, which the loads issued ahead of their
// group and the other warps cover.
template <int WARPS>
__global__ void __launch_bounds__(32 * WARPS) k_prep(const __grid_constant__ Prep P) {
  extern __shared__ uint32_t smem[];
  __shared__ uint32_t part[32], s_units[WARPS], s_item, s_flags, s_wide, s_below;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const uint32_t below_me = (1u << lane) - 1u;
  if (batch_failed(P.ctrl)) return;
  const uint32_t n_items = P.ctrl->n_items;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) {
      s_item = atomicAdd(&P.ctrl->next_item, 1u);
      s_flags = s_wide = s_below = 0;
    }
    __syncthreads();
    const uint32_t it = s_item;
    if (it >= n_items) break;
    const int2 item = P.items ? P.items[it] : make_int2((int)it, 0);
    const int i = item.x;
    const bool first_range = item.y == 0;
    const int64_t c0 = P.icb[i], c1 = P.icb[i + 1];
    // the clause ranges must cover [0, C) in order, or nothing can be trusted
    if (c0 < 0 || c1 < c0 || c1 > P.C || (i == 0 && c0 != 0) || (i == P.n - 1 && c1 != P.C)) {
      if (threadIdx.x == 0) fail_batch(P.ctrl, SCUBA_ERR_MALFORMED);
      continue;
    }
    const int32_t nv = P.nv[i], V = clamp_nv(nv, P.vmax);
    const int64_t lbase = c0 < c1 ? P.cb[c0] : 0;
    const int64_t vb = P.vb[i];
    // occurrence offsets are 32-bit within an instance; the model must fit
    if (nv != V || (c0 < c1 && P.cb[c1] - lbase >= (1LL << 32)) || vb < 0 ||
        vb + (int64_t)V > P.total_vars) {
      if (first_range && threadIdx.x == 0) P.flags[i] = F_BAD;
      continue;
    }
    const uint32_t lo = (uint32_t)item.y * P.range;
    const uint32_t hi = min(lo + P.range, 2u * (uint32_t)V);
    const uint32_t nl = hi - lo, nl2 = (nl + 1u) >> 1;
    uint32_t* const begin = smem;                // [nl] first entry of each literal's list
    uint32_t* const packed = smem + P.range;     // [WARPS][nl2] two 16-bit counts, then cursors
    uint32_t* const my_packed = packed + (size_t)wib * nl2;
    for (uint32_t k = threadIdx.x; k < WARPS * nl2; k += 32 * WARPS) packed[k] = 0u;
    // this warp's clauses: whole groups of 32
    const int64_t seg = ((c1 - c0 + 32 * WARPS - 1) / (32 * WARPS)) * 32;
    const int64_t s0 = min(c1, c0 + wib * seg), s1 = min(c1, s0 + seg);
    __syncthreads();
    // ---- pass 1: counts ----
    uint32_t f = 0, below = 0, units = 0, wide = 0;
    auto count = [&](uint32_t x) {
      below += x < lo;
      if (x >= lo && x < hi) {
        const uint32_t sh = ((x - lo) & 1u) * 16u;
        const uint32_t old = atomicAdd(&my_packed[(x - lo) >> 1], 1u << sh);
        wide |= ((old >> sh) & 0xffffu) == 0xffffu;
      }
    };
    each_group(P, s0, s1, lane, [&](int64_t cs, const RawClause& R) {
      uint32_t u[3];
      int nk;
      const int kind = classify(P, R, cs + lane < s1, V, u, nk, f);
      if (kind == CL_SHORT) {
        count(u[0]);
        count(u[1]);
        if (nk == 3) count(u[2]);
      } else if (kind == CL_LONG) {
        bool bad = false;
        for (int64_t q = R.b; q < R.e; q++) {
          const int32_t l = __ldg(P.lits + q);
          if (l == 0 || l > V || l < -V) bad = true;
          else count(code_of(l));
        }
        if (bad) f |= F_BAD;
      }
      units += __popc(__ballot_sync(FULL, kind == CL_UNIT));
    });
    f = __reduce_or_sync(FULL, f);
    wide = __reduce_or_sync(FULL, wide);
    below = __reduce_add_sync(FULL, below);
    if (lane == 0) {
      if (f) atomicOr(&s_flags, f);
      if (wide) s_wide = 1;
      if (below) atomicAdd(&s_below, below);
      s_units[wib] = units;
    }
    __syncthreads();
    f = s_flags;
    if (first_range && threadIdx.x == 0) P.flags[i] = f;
    if (f & F_BAD) continue;
    // ---- scan: list begins, and each warp's cursor within each list ----
    uint32_t* const occ = P.occ_begin + P.occ_base[i];
    uint32_t run = s_below;
    for (uint32_t k0 = 0; k0 < nl2; k0 += 32 * WARPS) {
      const uint32_t k = k0 + threadIdx.x;
      uint32_t a = 0, b = 0;  // occurrences of codes lo + 2k, lo + 2k + 1
      if (k < nl2) {
#pragma unroll 8
        for (int w = 0; w < WARPS; w++) {
          const uint32_t c = packed[(size_t)w * nl2 + k];
          packed[(size_t)w * nl2 + k] = (a & 0xffffu) | (b << 16);
          a += c & 0xffffu;
          b += c >> 16;
        }
        if (a > 0xffffu || b > 0xffffu) s_wide = 1;
      }
      uint32_t total;
      const uint32_t at = run + block_exclusive(a + b, part, total);
      run += total;
      if (k < nl2) {
        begin[2 * k] = at;
        occ[lo + 2 * k] = at;
        if (2 * k + 1 < nl) {
          begin[2 * k + 1] = at + a;
          occ[lo + 2 * k + 1] = at + a;
        }
      }
    }
    __syncthreads();
    if (s_wide) {
      // more than 65,535 occurrences of a literal: 32-bit counts for the whole
      // block, and one warp fills the lists
      for (uint32_t k = threadIdx.x; k < nl; k += 32 * WARPS) begin[k] = 0u;
      __syncthreads();
      for (int64_t c = c0 + threadIdx.x; c < c1; c += 32 * WARPS) {
        RawClause Q = load_bounds(P, c, c1);
        load_literals(P, Q);
        uint32_t u[3], g = 0;
        int nk;
        const int kind = classify(P, Q, true, V, u, nk, g);
        const int64_t len = kind == CL_LONG ? Q.e - Q.b : nk;
        for (int64_t q = 0; q < len; q++) {
          const uint32_t x = kind == CL_LONG ? code_of(__ldg(P.lits + Q.b + q))
                                             : (q == 0 ? u[0] : q == 1 ? u[1] : u[2]);
          if (x >= lo && x < hi) atomicAdd(&begin[x - lo], 1u);
        }
      }
      __syncthreads();
      run = s_below;
      for (uint32_t k0 = 0; k0 < nl; k0 += 32 * WARPS) {
        const uint32_t k = k0 + threadIdx.x;
        const uint32_t a = k < nl ? begin[k] : 0u;
        uint32_t total;
        const uint32_t at = run + block_exclusive(a, part, total);
        run += total;
        if (k < nl) {
          begin[k] = at;
          occ[lo + k] = at;
        }
      }
      __syncthreads();
    }
    const bool one_warp = s_wide != 0;
    if (hi == 2u * (uint32_t)V && threadIdx.x == 0) occ[hi] = run;
    uint32_t nunit = 0;
    if (first_range) {
      uint32_t all = 0;
      for (int w = 0; w < WARPS; w++) {
        if (w < wib) nunit += s_units[w];
        all += s_units[w];
      }
      if (threadIdx.x == 0) P.nunits[i] = all;
    }
    if (one_warp && wib != 0) continue;
    // ---- pass 2: entries and unit literals ----
    uint16_t* const cur = reinterpret_cast<uint16_t*>(my_packed);
    uint64_t* const ent = P.ent + lbase;
    const int64_t e1 = one_warp ? c1 : s1;
    each_group(P, s0, e1, lane, [&](int64_t cs, const RawClause& R) {
      uint32_t u[3], g = 0;
      int nk;
      const int kind = classify(P, R, cs + lane < e1, V, u, nk, g);
      if (first_range) {
        const uint32_t ub = __ballot_sync(FULL, kind == CL_UNIT);
        if (kind == CL_UNIT) P.units[c0 + nunit + __popc(ub & below_me)] = u[0];
        nunit += __popc(ub);
      }
      // literal k of every clause of the group at once
      auto place = [&](bool has, uint32_t x, uint64_t entry) {
        has = has && x >= lo && x < hi;
        if (!__any_sync(FULL, has)) return;
        const uint32_t grp = __match_any_sync(FULL, has ? x : (0x80000000u | (uint32_t)lane));
        const int leader = __ffs(grp) - 1;
        uint32_t at = 0;
        if (has && lane == leader) {
          if (one_warp) {
            at = begin[x - lo];
            begin[x - lo] = at + __popc(grp);
          } else {
            const uint32_t used = cur[x - lo];
            at = begin[x - lo] + used;
            cur[x - lo] = (uint16_t)(used + __popc(grp));
          }
        }
        at = __shfl_sync(FULL, at, leader);
        if (has) ent[at + __popc(grp & below_me)] = entry;
        __syncwarp();
      };
      const bool sh = kind == CL_SHORT;
      const uint32_t third = nk == 3 ? u[2] : NONE;
      place(sh, u[0], (uint64_t)u[1] | ((uint64_t)third << 32));
      place(sh, u[1], (uint64_t)u[0] | ((uint64_t)third << 32));
      place(sh && nk == 3, u[2], (uint64_t)u[0] | ((uint64_t)u[1] << 32));
      if (__any_sync(FULL, kind == CL_LONG)) {
        const uint32_t len = kind == CL_LONG ? (uint32_t)(R.e - R.b) : 0u;
        const uint32_t rounds = __reduce_max_sync(FULL, len);
        const uint64_t entry = (uint64_t)(LONG_CLAUSE | (uint32_t)(cs + lane - c0));
        for (uint32_t k = 0; k < rounds; k++) {
          const bool has = k < len;
          place(has, has ? code_of(__ldg(P.lits + R.b + k)) : 0u, entry);
        }
      }
    });
  }
}
