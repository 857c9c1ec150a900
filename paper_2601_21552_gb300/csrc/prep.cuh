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
// cursor stands. A list is therefore in the order of the clauses' groups of 32
// (within a group: first literals, then second, then third, each in the order
// in which the SM serves a warp's shared-memory atomics), and no count, cursor
// or normalised literal goes through global memory. The ranges of one large
// instance need nothing from each other: a block also counts the literals below
// its range, which is where its first list begins.

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
  uint32_t* flags;     // [n] F_EMPTY, F_BAD
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

// The clauses of one instance: literal slots [base, end) of the CSR.
struct Slots {
  int64_t base, end;
};

// One clause as a lane sees it: its first literal slot (from the instance's),
// its length (0 past the last clause too) and, up to length 3, its literals.
struct RawClause {
  uint32_t at, len;
  bool bad;
  int32_t l[3];
};

__device__ __forceinline__ RawClause load_bounds(const Prep& P, const Slots& S, int64_t c,
                                                 int64_t c1) {
  RawClause R;
  R.at = R.len = 0;
  R.bad = false;
  if (c < c1) {
    const int64_t b = __ldg(P.cb + c), e = __ldg(P.cb + c + 1);
    R.bad = b < S.base || e < b || e > S.end;
    if (!R.bad) {
      R.at = (uint32_t)(b - S.base);
      R.len = (uint32_t)(e - b);
    }
  }
  return R;
}

__device__ __forceinline__ void load_literals(const int32_t* lits, RawClause& R) {
#pragma unroll
  for (int k = 0; k < 3; k++) R.l[k] = k < R.len ? __ldg(lits + R.at + k) : 0;
}

// The warp's clauses [s0, s1) in groups of 32, fn(group start, lane's clause):
// the literals of the next two groups and the bounds of the one after them are
// on their way while a group is handled. lits: the instance's first literal.
template <class Fn>
__device__ __forceinline__ void each_group(const Prep& P, const Slots& S, const int32_t* lits,
                                           int64_t s0, int64_t s1, int lane, Fn&& fn) {
  RawClause R = load_bounds(P, S, s0 + lane, s1);
  RawClause N = load_bounds(P, S, s0 + 32 + lane, s1);
  RawClause M = load_bounds(P, S, s0 + 64 + lane, s1);
  load_literals(lits, R);
  load_literals(lits, N);
  for (int64_t cs = s0; cs < s1; cs += 32) {
    load_literals(lits, M);
    const RawClause Q = load_bounds(P, S, cs + 96 + lane, s1);
    fn(cs, R);
    R = N;
    N = M;
    M = Q;
  }
}

enum { CL_NONE, CL_SHORT, CL_UNIT, CL_LONG };

// Normalise a clause: CL_SHORT with its 2 or 3 distinct codes in u, CL_UNIT
// with u[0], CL_LONG (its codes are read from the CSR as they stand), CL_NONE
// (no clause, an empty one, or a tautology).
__device__ __forceinline__ int classify(const RawClause& R, uint32_t u[3], int& nk) {
  const uint32_t x0 = code_of(R.l[0]), x1 = code_of(R.l[1]), x2 = code_of(R.l[2]);
  const bool h1 = R.len > 1, h2 = R.len > 2;
  const bool d1 = h1 && x1 == x0;               // a literal said before
  const bool d2 = h2 && (x2 == x0 || x2 == x1);
  const bool taut = (h1 && x1 == (x0 ^ 1u)) || (h2 && (x2 == (x0 ^ 1u) || x2 == (x1 ^ 1u)));
  nk = (int)h1 - (int)d1 + (int)h2 - (int)d2 + 1;
  u[0] = x0;
  u[1] = h1 && !d1 ? x1 : x2;
  u[2] = x2;
  if (R.len > 3) return CL_LONG;
  return R.len == 0 || taut ? CL_NONE : nk == 1 ? CL_UNIT : CL_SHORT;
}

// A literal of 0, or of a variable the instance does not have.
__device__ __forceinline__ bool bad_literal(int32_t l, int V) { return l == 0 || l > V || l < -V; }

// WARPS = 8 for batches whose literals fit one item (several blocks per SM),
// 32 for larger ones (one block per SM; a large instance is cut into ranges).
// Per item the clauses are read twice; the passes are bound by instruction
// issue and by the latency of their loads and shared-memory updates, which the
// loads issued ahead of their group and the other warps cover. (Ranks within a
// group by __match_any_sync, about 380 cycles when all lanes differ, cost more
// than the rest of pass 2.) 4,096 partition queries of 16 bits, 460 MB of CSR: 537 us
// at 52 % of the issue slots, 1.2 GB of DRAM traffic; counting, scanning and filling
// through global memory took four kernels and 1,319 us.
template <int WARPS>
__global__ void __launch_bounds__(32 * WARPS) k_prep(const __grid_constant__ Prep P) {
  extern __shared__ uint32_t smem[];
  __shared__ uint32_t part[32], s_units[WARPS], s_item, s_flags, s_below;
  // a warp's own count ran over 16 bits (pass 1) / a list's did (scan): two words,
  // since the scan sets its one while slower threads still read the other
  __shared__ uint32_t s_wide, s_long;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const uint32_t below_me = (1u << lane) - 1u;
  const uint32_t n_items = P.ctrl->n_items;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) {
      // another block may set the status at any time (a malformed range below):
      // one thread reads it for the block, which leaves as a whole
      s_item = batch_failed(P.ctrl) ? n_items : atomicAdd(&P.ctrl->next_item, 1u);
      s_flags = s_wide = s_long = s_below = 0;
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
    Slots slots{0, 0};
    if (c0 < c1) slots = Slots{P.cb[c0], P.cb[c1]};
    const int64_t vb = P.vb[i];
    // occurrence offsets are 32-bit within an instance; the model must fit
    if (nv != V || slots.base < 0 || slots.end < slots.base || slots.end > P.L ||
        slots.end - slots.base >= (1LL << 32) || vb < 0 || vb + (int64_t)V > P.total_vars) {
      if (first_range && threadIdx.x == 0) P.flags[i] = F_BAD;
      continue;
    }
    const int32_t* const lits = P.lits + slots.base;
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
      const uint32_t r = x - lo;
      if (r < nl) {
        const uint32_t sh = (r & 1u) * 16u;
        const uint32_t old = atomicAdd(&my_packed[r >> 1], 1u << sh);
        wide |= ((old >> sh) & 0xffffu) == 0xffffu;
      }
    };
    each_group(P, slots, lits, s0, s1, lane, [&](int64_t cs, const RawClause& R) {
      uint32_t u[3];
      int nk;
      const int kind = classify(R, u, nk);
      bool bad = R.bad;
#pragma unroll
      for (int k = 0; k < 3; k++) bad |= k < R.len && R.len <= 3 && bad_literal(R.l[k], V);
      if (bad) {
        f |= F_BAD;
      } else if (kind == CL_SHORT) {
        count(u[0]);
        count(u[1]);
        if (nk == 3) count(u[2]);
      } else if (kind == CL_LONG) {
        for (uint32_t q = 0; q < R.len; q++) {
          const int32_t l = __ldg(lits + R.at + q);
          if (bad_literal(l, V)) f |= F_BAD;
          else count(code_of(l));
        }
      } else if (kind == CL_NONE && R.len == 0 && cs + lane < s1) {
        f |= F_EMPTY;
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
    // ---- scan: where the lists begin, and each warp's cursor within each list ----
    uint32_t* const occ = P.occ_begin + P.occ_base[i];
    auto head = [&](uint32_t r, uint32_t at) {  // literal lo + r's list begins at `at`
      begin[r] = at;
      occ[lo + r] = at;
    };
    uint32_t run = s_below;
    const bool recount = s_wide != 0;  // a 16-bit count ran over: the counts are void
    for (uint32_t k0 = 0; k0 < nl2 && !recount; k0 += 32 * WARPS) {
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
        if (a > 0xffffu || b > 0xffffu) s_long = 1;
      }
      uint32_t total;
      const uint32_t at = run + block_exclusive(a + b, part, total);
      run += total;
      if (k < nl2) {  // nl is even
        head(2 * k, at);
        head(2 * k + 1, at + a);
      }
    }
    __syncthreads();
    const bool one_warp = recount || s_long != 0;
    if (one_warp) {
      // more than 65,535 occurrences of a literal: 32-bit counts for the whole
      // block, and one warp fills the lists
      uint32_t* const cnt32 = packed;  // [nl]: WARPS * nl2 words or more
      for (uint32_t k = threadIdx.x; k < nl; k += 32 * WARPS) cnt32[k] = 0u;
      __syncthreads();
      for (int64_t c = c0 + threadIdx.x; c < c1; c += 32 * WARPS) {
        RawClause Q = load_bounds(P, slots, c, c1);
        load_literals(lits, Q);
        uint32_t u[3];
        int nk;
        const int kind = classify(Q, u, nk);
        const uint32_t len = kind == CL_LONG ? Q.len : kind == CL_SHORT ? (uint32_t)nk : 0u;
        for (uint32_t q = 0; q < len; q++) {
          const uint32_t x = kind == CL_LONG ? code_of(__ldg(lits + Q.at + q))
                                             : (q == 0 ? u[0] : q == 1 ? u[1] : u[2]);
          if (x - lo < nl) atomicAdd(&cnt32[x - lo], 1u);
        }
      }
      __syncthreads();
      run = s_below;
      for (uint32_t k0 = 0; k0 < nl; k0 += 32 * WARPS) {
        const uint32_t k = k0 + threadIdx.x;
        const uint32_t a = k < nl ? cnt32[k] : 0u;
        uint32_t total;
        const uint32_t at = run + block_exclusive(a, part, total);
        run += total;
        if (k < nl) {
          head(k, at);
          cnt32[k] = 0u;  // from here on the list's cursor
        }
      }
      __syncthreads();
    }
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
    uint64_t* const ent = P.ent + slots.base;
    const int64_t e1 = one_warp ? c1 : s1;
    each_group(P, slots, lits, s0, e1, lane, [&](int64_t cs, const RawClause& R) {
      uint32_t u[3];
      int nk;
      const int kind = classify(R, u, nk);
      if (first_range) {
        const uint32_t ub = __ballot_sync(FULL, kind == CL_UNIT);
        if (kind == CL_UNIT) P.units[c0 + nunit + __popc(ub & below_me)] = u[0];
        nunit += __popc(ub);
      }
      // literal x of the lane's clause: its entry {a, b} at the list's next place
      auto place = [&](bool has, uint32_t x, uint32_t a, uint32_t b) {
        const uint32_t r = x - lo;
        if (!has || r >= nl) return;
        uint32_t p;
        if (one_warp) {
          p = atomicAdd(&packed[r], 1u);
        } else {
          const uint32_t sh = (r & 1u) * 16u;
          p = (atomicAdd(&my_packed[r >> 1], 1u << sh) >> sh) & 0xffffu;
        }
        ent[begin[r] + p] = (uint64_t)a | ((uint64_t)b << 32);
      };
      const bool sh = kind == CL_SHORT;
      const uint32_t third = nk == 3 ? u[2] : NONE;
      place(sh, u[0], u[1], third);
      place(sh, u[1], u[0], third);
      place(sh && nk == 3, u[2], u[0], u[1]);
      if (__any_sync(FULL, kind == CL_LONG)) {
        const uint32_t len = kind == CL_LONG ? R.len : 0u;
        const uint32_t rounds = __reduce_max_sync(FULL, len);
        for (uint32_t k = 0; k < rounds; k++)
          place(k < len, k < len ? code_of(__ldg(lits + R.at + k)) : 0u,
                LONG_CLAUSE | (uint32_t)(cs + lane - c0), 0u);
      }
    });
  }
}
