// cdcl.cuh -- conflict-driven clause learning mode of the persistent search
// (included by solver.cu after the DPLL search; same prep layout, shared
// assignment, BCP frontier rounds and worker loop).
//
// The paper's solver (Sec. V-B, OR-Tools' SAT solver) learns clauses
// internally and says no more about it; this mode puts the textbook
// first-UIP scheme on top of the GPU propagation of the DPLL mode:
//
//  * The assignment takes two bit sets over literal codes in shared memory: the
//    true literals, and the settled ones, true literals whose own propagation
//    has begun (a literal assigned during a BCP round is "fresh" until then).
//    Every assigned variable keeps its reason (the occurrence entry or
//    clause reference that implied it) and its decision level.
//  * Propagation rounds are frontier-parallel, so two lanes can assign
//    variables of the same round in either trail order. An implication may
//    therefore only rely on false literals assigned BEFORE the current round;
//    a clause whose unit-ness depends on a literal falsified during the round
//    is left for the next round, where that literal's own occurrence list
//    brings it back. Every reason then precedes its literal on the trail, and
//    the trail is a topological order of the implication graph. Conflicts
//    need no such rule: a falsified clause is a conflict whenever found.
//  * Learned clauses live in a per-warp arena with two watched literals per
//    clause. Each literal's watch list is an array in a per-warp pool (grown
//    by doubling); an entry is {clause, blocker}, the blocker being a literal
//    of the clause (the other watch when the entry was made) whose truth
//    settles the clause without reading it. After the static occurrence
//    entries of each frontier batch, the watchers of every literal in the
//    batch are spread over the 32 lanes like the static entries, and the
//    clauses whose blocker is not true are visited by eight lanes each. A
//    clause can sit on two lists of one pass only when both its watches are
//    false; its second visit then waits until the first has moved its watch.
//    Moved watches are appended to their new lists all at once (the warp
//    copies a list when it grows) and a list closes up while it is read.
//  * Conflict analysis resolves the falsified clause with the reasons of
//    current-level literals, newest first on the trail, until one
//    current-level literal (the first UIP) is left; the lanes take the
//    literals of each clause, and the next literal to resolve is the newest
//    of the waiting ones, each kept in a lane's registers (a warp-wide
//    backward scan of the trail if more than 32 wait). Every variable met is
//    bumped. (Dropping the literals that the rest of the clause implies, a lane
//    per literal, saved 2 % of the conflicts on partition queries and 7 % on
//    random 3-SAT, and cost as much as it saved or more.)
//  * Hard instances are shared cube-and-conquer style through the DPLL mode's
//    job ring: a busy warp that sees idle warps gives away the negation of
//    its first free decision, together with the assumptions above it, as a
//    cube, and keeps that decision as one more assumption itself (backjumps
//    and restarts never undo assumptions). An instance is UNSAT once every
//    cube is; a cube starts from its donor's activities and its short,
//    low-LBD learned clauses. A unit of scuba_solve_units (an instance under
//    the caller's assumptions) starts the same way, as a job with a prefix.
//  * The search backjumps to the second-highest level of the learned clause
//    and asserts its UIP literal there; decisions take the saved phase (the
//    variable's last value, false at first); restarts follow the Luby
//    sequence times `restart_unit` conflicts. The first restart after 2000
//    conflicts (then 2300, 2600, ... more) also halves the learned clauses,
//    keeping the newer half and every clause of LBD <= 3 (the number of
//    distinct decision levels in it at learning time, after Glucose). When
//    the arena or the watch pool runs out the same reduction happens at once;
//    if even that does not fit, every learned clause is dropped (all of them
//    are implied by the formula, so any of this is sound).
//
// Clause arena layout (32-bit words, 16-byte aligned clauses): [len, 0, LBD,
// 0, lit0 .. lit_{len-1}, padding to a multiple of 4]; lit0 and lit1 are the
// watched literals.

constexpr uint32_t LEARNT_REF = 0xC0000000u;  // clause reference: learned clause at offset
constexpr uint32_t CD_HDR = 4;
// Shared memory of a clause-learning warp beyond its assignment: its profile, the
// literals and reasons of the CD_RING newest trail positions (a power of two), the
// first LSM literals of the clause under
// construction and, where they fit (Solve::cd_smem), per variable its
// activity (CD_SMEM_ACT), its trail position and level packed into 32 bits and
// its mark (both CD_SMEM_POS; at most 65,535 variables). The analysis walks from
// variable to variable, so what it reads of each has to be near: with these in
// global memory a resolution step took about 2,700 cycles. Where the activities
// do not fit, a bound per group of them does (CD_SMEM_GMAX, see pick_grouped).
enum { CD_SMEM_POS = 1, CD_SMEM_ACT = 2, CD_SMEM_GMAX = 4 };
constexpr uint32_t CD_RING = 64, LSM = 64;
constexpr size_t CD_FIXED = 8 * 8 + CD_RING * 12 + LSM * 4 + 16 + 32 * 12;

__host__ __device__ __forceinline__ size_t cd_area_bytes(int what, int32_t vmax) {
  const size_t v16 = ((size_t)vmax + 15) & ~(size_t)15;
  return CD_FIXED + (what & CD_SMEM_ACT ? 4 * v16 : 0) + (what & CD_SMEM_POS ? 5 * v16 : 0) +
         (what & CD_SMEM_GMAX ? (4 * (((size_t)vmax + 127) / 128) + 15) & ~(size_t)15 : 0);
}
// A warp's area is never taken smaller than this: the largest instance that fits
// an SM is part of the interface.
constexpr size_t CD_AREA_MIN = 1792;
static_assert(CD_FIXED <= CD_AREA_MIN, "largest instance");
__device__ __forceinline__ float* cd_area_act(unsigned char* area) {
  return reinterpret_cast<float*>(area + CD_FIXED);
}
// (an area has either the activities or the groups' bounds)
__device__ __forceinline__ uint32_t* cd_area_gmax(unsigned char* area) {
  return reinterpret_cast<uint32_t*>(area + CD_FIXED);
}

// A variable's mark: bit 0 the saved phase, bits 1-7 the number (1..127, mod
// 127) of the last analysis that met it, so that nothing is cleared after one.
constexpr uint32_t MK_PHASE = 1, MK_EPOCHS = 127;
constexpr uint32_t GMAX_LOOK = 0xffffffffu;  // a group's bound that is not known
constexpr uint32_t DEEP_CUBE = 20;  // cube levels from which two-level clauses are shared

// Profile counters (only when the caller passed a profile array): lane 0
// adds the clock cycles of each phase to its warp's profile.
enum { PF_BCP = 0, PF_LEARNED = 1, PF_ANALYZE = 2, PF_DECIDE = 3, PF_DB = 4, PF_NDB = 5,
       PF_NLEARNT = 6 };

__device__ __forceinline__ long long pf_now(const Solve& S) {
  return S.prof ? clock64() : 0;
}

__device__ __forceinline__ void pf_add(const Solve& S, Warp& w, int k, long long t0) {
  if (S.prof && w.lane == 0) w.cyc[k] += (unsigned long long)(clock64() - t0);
}

__device__ __forceinline__ bool is_learnt_ref(uint32_t a) {
  return a != NONE && (a & LEARNT_REF) == LEARNT_REF;
}

struct WList {       // one literal's learned watch list in the pool
  uint32_t off, len, cap, pad;
};

// Per assigned variable, one 16-byte record written by one store: the reason
// (the occurrence entry {a, b} that implied it, or a clause reference in the
// low word, ~0 for decisions and assumptions), its trail position and level.
struct VarInfo {
  uint32_t reason_lo, reason_hi, pos, level;
};

struct CdWarp {
  VarInfo* var;       // [V] reason, trail position, decision level
  uint8_t* mark;      // [V] saved phase and last analysis (MK_PHASE, MK_EPOCHS)
  WList* wl;          // [2V] learned watch list per literal code
  uint64_t* pool;     // [pool_cap] watch entries {clause, blocker}
  uint32_t* arena;    // [arena_words]
  uint32_t* cl_off;   // [arena_words / 8] arena offset of each learned clause, oldest first
  uint32_t* learnt;   // [V] clause under construction
  uint32_t* pl;       // [V] trail position | level << 16 in shared memory, or NULL
  unsigned char* area; // the warp's shared-memory area:
  // reason of the literal in the ring's same slot; ring[p mod CD_RING] = trail[p]
  // as in WarpShared; learnt[0 .. LSM)
  __device__ __forceinline__ uint2* why() const { return reinterpret_cast<uint2*>(area + 64); }
  __device__ __forceinline__ uint32_t* ring() const {
    return reinterpret_cast<uint32_t*>(area + 64 + 8 * CD_RING);
  }
  __device__ __forceinline__ uint32_t* lsm() const {
    return reinterpret_cast<uint32_t*>(area + 64 + 12 * CD_RING);
  }
  __device__ __forceinline__ uint4* next() const {  // the literal to resolve next, its reason
    return reinterpret_cast<uint4*>(area + 64 + 12 * CD_RING + 4 * LSM);
  }
  __device__ __forceinline__ uint2* visit() const {  // [32] clauses to visit {clause, false watch}
    return reinterpret_cast<uint2*>(area + 64 + 12 * CD_RING + 4 * LSM + 16);
  }
  __device__ __forceinline__ uint32_t* outcome() const {  // [32] what became of their entries
    return reinterpret_cast<uint32_t*>(area + 64 + 12 * CD_RING + 4 * LSM + 16 + 32 * 8);
  }
  uint32_t arena_words, pool_cap;
  uint32_t top;       // first free arena word
  uint32_t ncl;       // learned clauses in the arena
  uint32_t pool_top;  // first free pool entry
  uint32_t full;      // the pool ran out during propagation: drop the learned clauses
  uint32_t epoch;     // number of the last analysis (marks)
};

// Literal k of the clause under construction.
__device__ __forceinline__ uint32_t learnt_at(const CdWarp& cd, uint32_t k) {
  return k < LSM ? cd.lsm()[k] : cd.learnt[k];
}
__device__ __forceinline__ void set_learnt(CdWarp& cd, uint32_t k, uint32_t l) {
  if (k < LSM) cd.lsm()[k] = l;
  else cd.learnt[k] = l;
}
// Decision level of an assigned variable.
__device__ __forceinline__ uint32_t level_of(const CdWarp& cd, uint32_t v) {
  return cd.pl ? cd.pl[v] >> 16 : cd.var[v].level;
}

// Value (LV_U, LV_T, LV_F) of literal l.
__device__ __forceinline__ uint32_t lit_value_cd(const uint32_t* asg, uint32_t l) {
  const uint32_t x = asg[2 * (l >> 5)];
  if ((x >> (l & 31u)) & 1u) return LV_T;
  return (x >> ((l & 31u) ^ 1u)) & 1u ? LV_F : LV_U;
}

// The two words {true, settled} that hold literal l and its negation.
__device__ __forceinline__ uint2 lit_words(const uint32_t* asg, uint32_t l) {
  return *reinterpret_cast<const uint2*>(asg + 2 * (l >> 5));
}
__device__ __forceinline__ bool has_bit(uint32_t x, uint32_t l) { return (x >> (l & 31u)) & 1u; }

// Make literal l of every lane with want set true at the current level, with
// its reason (all lanes). Returns true in a lane whose literal's negation was
// claimed by another lane of this call.
__device__ __forceinline__ bool claim_cd(Warp& w, CdWarp& cd, bool want, uint32_t l,
                                         uint32_t why_lo, uint32_t why_hi) {
  bool won;
  const bool clash = claim_bits<2>(w, want, l, won);
  const uint32_t pos = push_trail<CD_RING>(w, cd.ring(), won, l);
  if (won) {
    const uint32_t v = l >> 1;
    cd.why()[pos & (CD_RING - 1u)] = make_uint2(why_lo, why_hi);
    if (cd.pl) cd.pl[v] = pos | (w.nd << 16);
    *reinterpret_cast<uint4*>(&cd.var[v]) = make_uint4(why_lo, why_hi, pos, w.nd);
  }
  return clash;
}

// Assign l, unassigned, for a decision, an assumption, a learned or an imported
// clause (all lanes, uniform).
__device__ __forceinline__ void assign_one_cd(Warp& w, CdWarp& cd, uint32_t l, uint32_t why_lo,
                                              uint32_t why_hi) {
  claim_cd(w, cd, w.lane == 0, l, why_lo, why_hi);
  __syncwarp();
}

// A long clause of the caller's CSR: unit or false, or nothing if it is true,
// has two open literals, or its last open literal rests on a fresh one (that
// literal's own list brings it back next round).
__device__ __noinline__ Found eval_long_cd(const uint32_t* asg, const int32_t* lits, int64_t b,
                                           int64_t e, uint32_t local) {
  uint32_t open_lit = NONE;
  bool fresh_false = false;
  for (int64_t q = b; q < e; q++) {
    const uint32_t x = code_of(__ldg(&lits[q]));
    const uint2 ws = lit_words(asg, x);
    if (has_bit(ws.x, x)) return Found{false, false, NONE, 0, 0, 0};
    if (!has_bit(ws.x, x ^ 1u)) {
      if (open_lit != NONE && x != open_lit) return Found{false, false, NONE, 0, 0, 0};
      open_lit = x;
    } else {
      fresh_false |= !has_bit(ws.y, x ^ 1u);
    }
  }
  return Found{open_lit != NONE && !fresh_false, open_lit == NONE, open_lit, LONG_CLAUSE | local,
               NONE, NONE};
}

// One occurrence entry of the falsified (settled) literal f: (f | a) with b ==
// NONE, (f | a | b), or a long clause; without branches but for those. A
// literal is implied only by settled false literals. For a wanted literal c0
// and c1 are its reason, for a conflict c0..c2 the clause.
__device__ __forceinline__ Found eval_entry_cd(const Warp& w, uint32_t f, uint64_t e) {
  const uint32_t a0 = (uint32_t)e, b0 = (uint32_t)(e >> 32);
  if (a0 & LONG_CLAUSE) {
    const uint32_t local = a0 & ~LONG_CLAUSE;
    const int64_t c = w.c0 + local;
    return eval_long_cd(w.asg, w.lits, w.cb[c], w.cb[c + 1], local);
  }
  const bool tern = b0 != NONE;
  const uint32_t a = WIDX(w, a0, 2u * w.V, 13), b = tern ? WIDX(w, b0, 2u * w.V, 13) : a;
  const uint2 xa = lit_words(w.asg, a), xb = lit_words(w.asg, b);
  const bool ta = has_bit(xa.x, a), fa = has_bit(xa.x, a ^ 1u), sa = has_bit(xa.y, a ^ 1u);
  const bool tb = tern && has_bit(xb.x, b), fb = !tern || has_bit(xb.x, b ^ 1u);
  const bool sb = !tern || has_bit(xb.y, b ^ 1u);
  const bool ua = !ta && !fa && sb, ub = !tb && !fb && sa;
  const bool confl = fa && fb;
  return Found{ua || ub, confl, ua ? a : b, f, confl ? a : ua ? b0 : a, confl ? b0 : NONE};
}

// A literal's watch list with room for more entries: copied to the pool's top
// with twice the capacity. Returns the new top, or NONE if the pool is full.
__device__ __noinline__ uint32_t grow_list(WList* wl, uint64_t* pool, uint32_t pool_top,
                                           uint32_t pool_cap, uint32_t g, int lane) {
  WList L = wl[g];
  const uint32_t ncap = L.cap ? 2u * L.cap : 8u;
  if ((uint64_t)pool_top + ncap > pool_cap) return NONE;
  for (uint32_t k = lane; k < L.len; k += 32) pool[pool_top + k] = pool[L.off + k];
  __syncwarp();
  if (lane == 0) wl[g] = WList{pool_top, L.len, ncap, 0u};
  __syncwarp();
  return pool_top + ncap;
}

// Append entry e to literal g's watch list in every lane with mover set (all
// lanes): lists with room take theirs at once, the others grow one by one.
// Sets cd.full and a conflict (which ends the propagation) if the pool is full.
template <bool DISTINCT>
__device__ __forceinline__ void append_watches(Warp& w, CdWarp& cd, bool mover, uint32_t g,
                                               uint64_t e) {
  uint32_t todo = __ballot_sync(FULL, mover);
  while (todo) {
    uint4 L = make_uint4(0, 0, 0, 0);  // {offset, length, capacity}
    if (mover) L = *reinterpret_cast<const uint4*>(&cd.wl[g]);
    uint32_t grp = 1u << w.lane;
    if (!DISTINCT && (todo & (todo - 1u))) {
      if (__popc(todo) <= 3) {
        for (uint32_t left = todo; left;) {
          const uint32_t g0 = __shfl_sync(FULL, g, __ffs(left) - 1);
          const uint32_t same = __ballot_sync(FULL, mover && g == g0);
          if (mover && g == g0) grp = same;
          left &= ~same;
        }
      } else {
        grp = __match_any_sync(FULL, mover ? g : ~(uint32_t)w.lane);
      }
    }
    const uint32_t rank = __popc(grp & ((1u << w.lane) - 1u)), size = __popc(grp);
    const bool fits = mover && L.y + size <= L.z;
    if (fits) {
      cd.pool[L.x + L.y + rank] = e;
      if (rank == 0) cd.wl[g].len = L.y + size;
      mover = false;
    }
    __syncwarp();
    todo = __ballot_sync(FULL, mover);
    if (todo) {
      const uint32_t gj = __shfl_sync(FULL, g, __ffs(todo) - 1);
      const uint32_t top = grow_list(cd.wl, cd.pool, cd.pool_top, cd.pool_cap, gj, w.lane);
      if (top == NONE) {
        cd.full = 1;
        w.confl = 1;
        return;
      }
      cd.pool_top = top;
    }
  }
}

// Outcome of a visited clause for its entry in the list: the new blocker, or
constexpr uint32_t OUT_SAME = 0xffffffffu, OUT_MOVED = 0xfffffffeu;

// Visit the `total` clauses in cd.visit(): eight lanes take a clause, four
// clauses at a time, a lane each literal, so that a search for a new watch is
// one trip to memory per eight literals whatever the lanes' clauses are (one
// lane per clause took about 1,900 cycles on random 3-SAT, each four literals
// of the longest clause one after another). A clause whose other watch is
// true gets it as its blocker; else the watch moves to the first literal from
// position 2 on that is not false, or if there is none the first that was
// falsified during this round (its own list brings the clause back next
// round); else the clause implies its other watch or is a conflict. dups: a
// clause may be there twice (both its watches false): the second is visited
// after the first has moved its watch. Stops at a conflict.
__device__ __forceinline__ void visit_clauses(Warp& w, CdWarp& cd, uint32_t total, bool dups) {
  const uint32_t sub = (uint32_t)w.lane & 7u, group = (uint32_t)w.lane >> 3;
  const uint32_t shift = (uint32_t)w.lane & 24u;  // this group's bits in a ballot
  for (uint32_t r0 = 0; r0 < total && !w.confl; r0 += 4) {
    uint32_t todo = (1u << min(4u, total - r0)) - 1u;  // groups whose clause is not done
    while (todo && !w.confl) {
      const uint32_t r = r0 + group;
      bool go = (todo >> group) & 1u;
      uint2 v = make_uint2(0, 0);
      if (go) v = cd.visit()[r];
      if (dups)
        for (uint32_t q = 0; q < 3; q++)
          if (go && q < group && ((todo >> q) & 1u) && cd.visit()[r0 + q].x == v.x) go = false;
      uint32_t* const L = cd.arena + v.x + CD_HDR;
      uint32_t lit = 0, len = 0;
      if (go) {
        lit = L[sub];  // past the clause's end too: not used then
        len = L[-(int)CD_HDR];
      }
      const bool in = sub < len;
      if (!in) lit = 0;
      uint2 ws = lit_words(w.asg, lit);
      const uint32_t m_true = __ballot_sync(FULL, in && has_bit(ws.x, lit));
      const uint32_t m_open = __ballot_sync(FULL, in && !has_bit(ws.x, lit ^ 1u));
      const uint32_t m_fresh =
          __ballot_sync(FULL, in && has_bit(ws.x, lit ^ 1u) && !has_bit(ws.y, lit ^ 1u));
      const uint32_t m_f = __ballot_sync(FULL, in && sub < 2 && lit == v.y);
      const uint32_t which = (m_f >> shift) & 1u ? 0u : 1u, op = which ^ 1u;
      const uint32_t other = __shfl_sync(FULL, lit, shift + op);
      const bool o_true = (m_true >> (shift + op)) & 1u, o_open = (m_open >> (shift + op)) & 1u;
      uint32_t cand = (m_open >> shift) & 0xfcu, fresh = (m_fresh >> shift) & 0xfcu;
      // position and literal of the new watch (fresh_*: the fallback)
      uint32_t at = __ffs(cand) - 1u, fresh_at = __ffs(fresh) - 1u;
      uint32_t g = __shfl_sync(FULL, lit, shift + (at & 7u));
      uint32_t fresh_g = __shfl_sync(FULL, lit, shift + (fresh_at & 7u));
      for (uint32_t q = 8; __any_sync(FULL, go && !o_true && at == NONE && q < len); q += 8) {
        const bool more = go && !o_true && at == NONE && q + sub < len;
        lit = more ? L[q + sub] : 0u;
        ws = lit_words(w.asg, lit);
        const bool isf = has_bit(ws.x, lit ^ 1u);
        cand = (__ballot_sync(FULL, more && !isf) >> shift) & 0xffu;
        fresh = (__ballot_sync(FULL, more && isf && !has_bit(ws.y, lit ^ 1u)) >> shift) & 0xffu;
        const uint32_t a = __ffs(cand) - 1u, b = __ffs(fresh) - 1u;
        const uint32_t la = __shfl_sync(FULL, lit, shift + (a & 7u));
        const uint32_t lb = __shfl_sync(FULL, lit, shift + (b & 7u));
        if (cand) {
          at = q + a;
          g = la;
        }
        if (fresh && fresh_at == NONE) {
          fresh_at = q + b;
          fresh_g = lb;
        }
      }
      if (at == NONE) {
        at = fresh_at;
        g = fresh_g;
      }
      // the group's first lane acts
      const bool act = go && sub == 0, moves = act && !o_true && at != NONE;
      const bool want = act && !o_true && at == NONE && o_open;
      bool confl = act && !o_true && at == NONE && !o_open;
      if (moves) {
        L[at] = v.y;
        L[which] = g;
      }
      if (act && (o_true || moves)) cd.outcome()[r] = moves ? OUT_MOVED : other;
      const uint32_t done = __ballot_sync(FULL, act);
      for (uint32_t q = 0; q < 4; q++)
        if ((done >> (8 * q)) & 1u) todo &= ~(1u << q);
      if (__any_sync(FULL, want || confl)) {
        confl |= claim_cd(w, cd, want, other, LEARNT_REF | v.x, 0u);
        note_conflict(w, confl, LEARNT_REF | v.x, NONE, NONE);
      }
      __syncwarp();
      if (__any_sync(FULL, moves) && !cd.full)
        append_watches<false>(w, cd, moves, g, (uint64_t)v.x | ((uint64_t)other << 32));
    }
  }
}

// Learned clauses watching the literals falsified in this batch: lane j <
// nlit holds falsified literal f and its watch list pool[beg, beg + cnt). Every
// list is read to its end, also after a conflict, since it closes up as its
// entries leave.
__device__ __forceinline__ void learned_batch(Warp& w, CdWarp& cd, const LaneMap& m,
                                              uint32_t nlit, uint32_t f, uint32_t beg,
                                              uint32_t cnt) {
  if (!__any_sync(FULL, cnt != 0)) return;
  const long long t0 = pf_now(*w.S);
  if (counts_list(m)) WADD(w, visits, cnt);
  const uint32_t below = (1u << w.lane) - 1u, mates = 0xffu << ((uint32_t)w.lane & 24u);
  for (uint32_t s = 0; s < nlit; s += 4) {
    uint32_t jb = beg, jf = f, jc = cnt;
    if (!m.few) {
      const uint32_t j = s + m.group;
      jb = __shfl_sync(FULL, beg, j);
      jf = __shfl_sync(FULL, f, j);
      jc = __shfl_sync(FULL, cnt, j);
      if (j >= nlit) jc = 0;
    }
    uint32_t kept = 0;
    bool more = __any_sync(FULL, m.sub < jc);
    for (uint32_t k = m.sub; more; k += 8) {
      const bool in = k < jc;
      uint64_t entry = 0;
      bool pending = false;
      if (in) {
        entry = cd.pool[WIDX(w, jb + k, cd.pool_cap, 16)];
        const uint32_t blocker = WIDX(w, (uint32_t)(entry >> 32), 2u * w.V, 18);
        pending = !has_bit(w.asg[2 * (blocker >> 5)], blocker);
      }
      more = __any_sync(FULL, k + 8 < jc);
      const uint32_t c = WIDX(w, (uint32_t)entry, cd.top, 17);
      const uint32_t pm = w.confl ? 0u : __ballot_sync(FULL, pending);
      bool stay = in;
      uint64_t now = entry;  // the entry that stays in this list
      if (pm) {
        const uint32_t rank = __popc(pm & below);
        if (pending) {
          cd.visit()[rank] = make_uint2(c, jf);
          cd.outcome()[rank] = OUT_SAME;
        }
        __syncwarp();
        visit_clauses(w, cd, __popc(pm), nlit > 1);
        __syncwarp();
        if (pending) {
          const uint32_t o = cd.outcome()[rank];
          stay = o != OUT_MOVED;
          if (stay && o != OUT_SAME) now = (uint64_t)c | ((uint64_t)o << 32);
        }
      }
      // close the list up behind the entries that left
      const uint32_t stays = __ballot_sync(FULL, stay);
      const uint32_t to = kept + __popc(stays & mates & below);
      if (stay && (to != k || now != entry)) cd.pool[jb + to] = now;
      kept += __popc(stays & mates);
      __syncwarp();
    }
    if (m.sub == 0 && kept != jc) cd.wl[jf].len = kept;
  }
  __syncwarp();
  pf_add(*w.S, w, PF_LEARNED, t0);
}

// Unit propagation to a fixpoint (true on conflict: w.confl, ws->cl), in the
// frontier rounds of the DPLL search. Per batch of up to 32 frontier literals
// the lanes read their literal, mark it settled, and load both its
// occurrence-list bounds and its learned watch list before the static entries
// and then the learned watchers are evaluated.
__device__ __forceinline__ bool bcp_cd(Warp& w, CdWarp& cd) {
  while (w.head < w.tail) {
    const uint32_t lo = w.head, hi = w.tail;
    w.head = hi;
    WCOUNT(w, props, hi - lo);
    for (uint32_t base = lo; base < hi; base += 32) {
      const uint32_t nlit = min(32u, hi - base);
      const LaneMap m = lane_map<true>(w.lane, nlit);
      uint32_t f = 0, beg = 0, cnt = 0, lbeg = 0, lcnt = 0;
      if (m.mine < nlit) {
        const uint32_t t = WIDX(w, frontier_lit<CD_RING>(w, cd.ring(), base + m.mine), 2u * w.V, 14);
        f = t ^ 1u;
        beg = __ldg(&w.occ[f]);
        cnt = __ldg(&w.occ[f + 1]) - beg;
        if (cd.top) {
          const uint2 L = *reinterpret_cast<const uint2*>(&cd.wl[f]);  // {offset, length}
          lbeg = L.x;
          lcnt = L.y;
        }
        if (!m.few || m.sub == 0) atomicOr(&w.asg[2 * (t >> 5) + 1], 1u << (t & 31u));  // settled
      }
      __syncwarp();
      spread_lists(m, nlit, f, beg, cnt, [&](uint32_t jf, uint32_t at, bool in) {
        Found r{false, false, 0, 0, 0, 0};
        if (in) r = eval_entry_cd(w, jf, __ldg(&w.ent[WIDX(w, at, w.ent_end, 15)]));
        if (__any_sync(FULL, r.want || r.confl)) {
          const bool clash = claim_cd(w, cd, r.want, r.lit, r.c0, r.c1);
          // a clash: the clause's wanted literal is false after all
          note_conflict(w, r.confl || clash, r.c0, r.c1,
                        clash && !(r.c0 & LONG_CLAUSE) ? r.lit : r.c2);
          __syncwarp();
        }
        return w.confl != 0;
      });
      if (counts_list(m)) WADD(w, visits, cnt);
      if (w.confl) return true;
      if (cd.top) {
        learned_batch(w, cd, m, nlit, f, lbeg, lcnt);
        if (w.confl) return true;
      }
    }
  }
  return false;
}

// First-UIP analysis of the recorded conflict (all lanes). Leaves the learned
// clause in cd.learnt[0 .. n): the asserting literal first, then a literal of
// the backjump level; returns n, the backjump level in blev and the clause's
// LBD (distinct decision levels, counted per group of 32 literals) in lbd.
// Returns 0 if a consistency check fails.
//
// A resolution step is a chain of dependent latencies on one warp, so it stays
// near: marks, positions and levels in shared memory, recent reasons in the
// ring's slots, and each current-level literal not yet resolved waits, with
// its reason, in the registers of the lane that met it. The lanes that hold
// none take the next clause's literals; the newest waiting literal is found
// with one warp-wide maximum of trail positions, and marks carry the
// analysis' number instead of being cleared on the way. If all 32 lanes hold a
// literal, the rest of this analysis scans the trail for seen marks instead.
__device__ __forceinline__ uint32_t analyze_cd(Warp& w, CdWarp& cd, uint32_t& blev,
                                               uint32_t& lbd) {
  const uint32_t lvl = w.nd, below = (1u << w.lane) - 1u;
  uint32_t n = 1, path = 0, p = NONE;
  uint32_t r0 = w.ws->cl[0], r1 = w.ws->cl[1], r2 = w.ws->cl[2];
  uint32_t idx = w.tail;  // the trail below this position is not resolved yet
  if (++cd.epoch > MK_EPOCHS) {  // every number used: start over on clean marks
    for (uint32_t v = w.lane; v < w.V; v += 32) cd.mark[v] &= (uint8_t)MK_PHASE;
    cd.epoch = 1;
    __syncwarp();
  }
  const uint32_t seen = cd.epoch << 1;
  uint32_t key = 0, mylit = 0, my0 = 0, my1 = 0;  // waiting literal (key: position + 1; 0: none)
  bool overflow = false;
  bool big = false;
  for (;;) {
    // the literals of the clause: static entry (up to three codes), a long
    // clause of the caller's CSR, or a learned clause
    const uint32_t* src = nullptr;
    const int32_t* csr = nullptr;
    uint32_t cnt = 3;
    if (is_learnt_ref(r0)) {
      const uint32_t off = r0 & ~LEARNT_REF;
      cnt = cd.arena[off];
      src = cd.arena + off + CD_HDR;
    } else if (r0 & LONG_CLAUSE) {
      const int64_t cl = w.c0 + (r0 & ~LONG_CLAUSE);
      const int64_t b = w.cb[cl];
      csr = w.lits + b;
      cnt = (uint32_t)(w.cb[cl + 1] - b);
    }
    for (uint32_t k0 = 0; k0 < cnt;) {
      uint32_t idle = __ballot_sync(FULL, key == 0);
      if (idle == 0) overflow = true;
      if (overflow) idle = FULL;
      const uint32_t k = k0 + __popc(idle & below);
      k0 += __popc(idle);
      uint32_t q = NONE;
      if (k < cnt && ((idle >> w.lane) & 1u))
        q = src ? src[k] : csr ? code_of(csr[k]) : (k == 0 ? r0 : k == 1 ? r1 : r2);
      const uint32_t v = q == NONE ? NONE >> 1 : WIDX(w, q >> 1, w.V, 21);
      bool take = false;
      uint32_t mk = 0, pos = 0, lev = 0;
      uint2 why = make_uint2(0, 0);
      float a = 0.0f;
      if (q != NONE && (p == NONE || v != (p >> 1))) {
        mk = cd.mark[v];  // independent loads
        a = w.act[v];
        if (cd.pl) {
          const uint32_t x = cd.pl[v];
          pos = x & 0xffffu;
          lev = x >> 16;
        } else {
          const uint4 rec = *reinterpret_cast<const uint4*>(&cd.var[v]);
          why = make_uint2(rec.x, rec.y);
          pos = rec.z;
          lev = rec.w;
        }
        take = (mk & ~MK_PHASE) != seen && lev > 0;
      }
      if (csr) {  // one lane per variable: a long clause may repeat a literal
        const uint32_t grp = __match_any_sync(FULL, take ? v : NONE);
        if (take && __ffs(grp) - 1 != w.lane) take = false;
      }
      const bool cur = take && lev >= lvl;
      const uint32_t lowm = __ballot_sync(FULL, take && !cur);
      path += __popc(__ballot_sync(FULL, cur));
      if (take) {
        cd.mark[v] = (uint8_t)((mk & MK_PHASE) | seen);
        a += w.inc;
        w.act[v] = a;
        big |= a > 1e20f;
        if (!cur) {
          set_learnt(cd, WIDX(w, n + __popc(lowm & below), w.V, 20), q);
        } else if (!overflow) {
          key = pos + 1u;
          mylit = q ^ 1u;
          if (cd.pl) {
            // the slot of a literal's position holds its reason as long as the
            // ring still names that literal there
            why = cd.why()[pos & (CD_RING - 1u)];
            if (w.tail - pos > CD_RING || cd.ring()[pos & (CD_RING - 1u)] != mylit)
              why = *reinterpret_cast<const uint2*>(&cd.var[v].reason_lo);
          }
          my0 = why.x;
          my1 = why.y;
        }
      }
      n += __popc(lowm);
      __syncwarp();
    }
    // a conflict without a current-level literal, or a scan that runs off the
    // trail, means the search state is inconsistent: give up (n = 0)
    if (path == 0) return 0;
    if (!overflow) {
      // the newest waiting literal (trail positions are distinct)
      const uint32_t top = __reduce_max_sync(FULL, key);
      if (top == 0) return 0;
      if (key == top) {  // through shared memory: finding the lane takes longer
        *cd.next() = make_uint4(mylit, my0, my1, 0u);
        key = 0;
      }
      __syncwarp();
      const uint4 c = *cd.next();
      p = c.x;
      r0 = c.y;
      r1 = c.z;
      idx = top - 1u;
    } else {
      for (;;) {  // the newest seen literal on the trail
        if (idx == 0) return 0;
        const uint32_t pos = idx - 1u - w.lane;
        bool sn = false;
        if (w.lane < idx) sn = (cd.mark[w.trail[pos] >> 1] & ~MK_PHASE) == seen;
        const uint32_t m = __ballot_sync(FULL, sn);
        if (m) {
          idx -= __ffs(m);
          break;
        }
        idx = idx > 32u ? idx - 32u : 0u;
      }
      p = w.trail[idx];
      const uint2 rw = *reinterpret_cast<const uint2*>(&cd.var[p >> 1].reason_lo);
      r0 = rw.x;
      r1 = rw.y;
    }
    if (--path == 0) break;
    r2 = NONE;
  }
  if (w.lane == 0) set_learnt(cd, 0, p ^ 1u);
  // backjump level: the highest level among learnt[1..n), moved to position 1
  uint32_t best_l = 0, best_k = 1, levels = 1;  // learnt[0] is alone at level lvl
  for (uint32_t k0 = 1; k0 < n; k0 += 32) {
    const uint32_t k = k0 + w.lane;
    uint32_t lv = NONE;
    if (k < n) {
      lv = level_of(cd, learnt_at(cd, k) >> 1);
      if (lv > best_l) {
        best_l = lv;
        best_k = k;
      }
    }
    const uint32_t grp = __match_any_sync(FULL, lv);
    levels += __popc(__ballot_sync(FULL, k < n && __ffs(grp) - 1 == w.lane));
  }
  lbd = levels;
  for (int d = 16; d > 0; d >>= 1) {
    const uint32_t ol = __shfl_xor_sync(FULL, best_l, d);
    const uint32_t ok = __shfl_xor_sync(FULL, best_k, d);
    if (ol > best_l || (ol == best_l && ok < best_k)) {
      best_l = ol;
      best_k = ok;
    }
  }
  __syncwarp();
  if (w.lane == 0 && n > 2 && best_k != 1) {
    const uint32_t t = learnt_at(cd, 1);
    set_learnt(cd, 1, learnt_at(cd, best_k));
    set_learnt(cd, best_k, t);
  }
  big = __any_sync(FULL, big);
  if (big) {
    for (uint32_t v = w.lane; v < w.V; v += 32) w.act[v] *= 1e-20f;
    w.inc *= 1e-20f;
    if (w.S->cd_smem & CD_SMEM_GMAX)
      for (uint32_t g = w.lane; 128u * g < w.V; g += 32) cd_area_gmax(cd.area)[g] = GMAX_LOOK;
  }
  __syncwarp();
  blev = best_l;
  return n;
}

// Undo every assignment above level lev, saving phases.
__device__ void backjump_cd(Warp& w, CdWarp& cd, uint32_t lev) {
  if (w.nd <= lev) return;
  const uint32_t pos = w.dstack[lev];
  const uint32_t tail = w.tail;
  WCOUNT(w, undone, tail - pos);
  for (uint32_t t = pos + w.lane; t < tail; t += 32) {
    const uint32_t l = w.trail[t], v = l >> 1;
    const uint32_t keep = ~(3u << (l & 30u));
    atomicAnd(&w.asg[2 * (l >> 5)], keep);
    atomicAnd(&w.asg[2 * (l >> 5) + 1], keep);
    cd.mark[v] = (l & 1u) ? 0 : (uint8_t)MK_PHASE;
    if (w.S->cd_smem & CD_SMEM_GMAX)
      atomicMax(&cd_area_gmax(cd.area)[v >> 7], __float_as_uint(w.act[v]) + 1u);
  }
  __syncwarp();
  w.nd = lev;
  w.head = w.tail = pos;
}

// Arena words a learned clause of n literals takes.
__device__ __forceinline__ uint32_t clause_words(uint32_t n) {
  return CD_HDR + ((n + 3u) & ~3u);
}

// Store learnt[0..n) (n >= 2) at the arena top and watch its first two
// literals. The caller checked the arena has room; the pool may run out
// (cd.full).
__device__ __forceinline__ uint32_t add_learnt(Warp& w, CdWarp& cd, uint32_t n, uint32_t lbd) {
  const uint32_t c = cd.top;
  for (uint32_t k = w.lane; k < ((n + 3u) & ~3u); k += 32)
    cd.arena[c + CD_HDR + k] = k < n ? learnt_at(cd, k) : NONE;
  if (w.lane == 0) {
    cd.arena[c] = n;
    cd.arena[c + 1] = 0u;
    cd.arena[c + 2] = lbd;
    cd.arena[c + 3] = 0u;
  }
  if (w.lane == 0) {
    cd.cl_off[cd.ncl] = c;
    if (w.S->prof) w.cyc[PF_NLEARNT]++;
  }
  __syncwarp();
  cd.top = c + clause_words(n);
  cd.ncl++;
  const uint32_t l0 = cd.lsm()[0], l1 = cd.lsm()[1];
  append_watches<true>(w, cd, w.lane < 2, w.lane == 0 ? l0 : l1,
                 (uint64_t)c | ((uint64_t)(w.lane == 0 ? l1 : l0) << 32));
  return c;
}

// Room every watch list gets before its first entry (a list grows one at a time,
// the warp copying it): four entries, a sector, where that takes little of the pool.
__device__ __forceinline__ uint32_t list_room(const Warp& w, const CdWarp& cd) {
  return (uint64_t)w.V * 32u <= cd.pool_cap ? 4u : 0u;
}

__device__ __noinline__ void clear_learnts(Warp& w, CdWarp& cd) {
  const uint32_t room = list_room(w, cd);
  for (uint32_t k = w.lane; k < 2u * w.V; k += 32) cd.wl[k] = WList{room * k, 0u, room, 0u};
  cd.top = 0;
  cd.ncl = 0;
  cd.pool_top = room * 2u * w.V;
  cd.full = 0;
  __syncwarp();
}

__device__ bool rebuild_watches(Warp& w, CdWarp& cd);

// Learned-clause database maintenance at the bottom level (no reason above it
// refers to a learned clause). With drop_half, keep the newer half of the
// clauses and every clause whose LBD is at most 3 (the "glue" clauses that
// tie few decision levels together); otherwise keep them all.
// Kept clauses move down the arena in order; then every watch list is built
// afresh from the clauses' first two literals (count, scan, fill), which
// also compacts the pool. Returns false when the lists would take more than
// half of the pool.
__device__ bool reduce_db(Warp& w, CdWarp& cd, bool drop_half) {
  const uint32_t n = cd.ncl;
  uint32_t run_words = 0, run_cl = 0;
  for (uint32_t k0 = 0; k0 < n; k0 += 32) {
    const uint32_t k = k0 + w.lane;
    uint32_t off = 0, words = 0;
    bool keep = false;
    if (k < n) {
      off = cd.cl_off[k];
      const uint32_t len = cd.arena[off];
      keep = !drop_half || k >= n / 2 || cd.arena[off + 2] <= 3u;
      if (keep) words = clause_words(len);
    }
    uint32_t inc = words;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(FULL, inc, d);
      if (w.lane >= d) inc += y;
    }
    const uint32_t dst = run_words + inc - words;
    const uint32_t km = __ballot_sync(FULL, keep);
    __syncwarp();
    // move the kept clauses down one at a time, in order (dst <= src)
    for (uint32_t m = km; m; m &= m - 1u) {
      const int j = __ffs(m) - 1;
      const uint32_t src = __shfl_sync(FULL, off, j), to = __shfl_sync(FULL, dst, j);
      const uint32_t wd = __shfl_sync(FULL, words, j);
      if (src != to)
        for (uint32_t q0 = 0; q0 < wd; q0 += 32) {
          const uint32_t q = q0 + w.lane;
          const uint32_t x = q < wd ? cd.arena[src + q] : 0u;
          __syncwarp();
          if (q < wd) cd.arena[to + q] = x;
          __syncwarp();
        }
    }
    if (keep) cd.cl_off[run_cl + __popc(km & ((1u << w.lane) - 1u))] = dst;
    run_words += __shfl_sync(FULL, inc, 31);
    run_cl += __popc(km);
    __syncwarp();
  }
  cd.top = run_words;
  cd.ncl = run_cl;
  return rebuild_watches(w, cd);
}

// Every watch list built afresh from the learned clauses' first two literals
// (count, exclusive scan of capacities, fill); this also compacts the pool.
// Returns false when the lists would take more than half of the pool.
__device__ bool rebuild_watches(Warp& w, CdWarp& cd) {
  const uint32_t run_cl = cd.ncl;
  const uint32_t nl = 2u * w.V;
  for (uint32_t k = w.lane; k < nl; k += 32) cd.wl[k] = WList{0u, 0u, 0u, 0u};
  __syncwarp();
  for (uint32_t k = w.lane; k < run_cl; k += 32) {
    const uint32_t c = cd.cl_off[k];
    atomicAdd(&cd.wl[cd.arena[c + CD_HDR]].len, 1u);
    atomicAdd(&cd.wl[cd.arena[c + CD_HDR + 1]].len, 1u);
  }
  __syncwarp();
  const uint32_t room = list_room(w, cd);
  uint32_t base = 0;
  for (uint32_t k0 = 0; k0 < nl; k0 += 32) {
    const uint32_t k = k0 + w.lane;
    const uint32_t len = k < nl ? cd.wl[k].len : 0u;
    const uint32_t cap = k < nl ? len + (len ? max(4u, len / 2u) : room) : 0u;
    uint32_t inc = cap;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(FULL, inc, d);
      if (w.lane >= d) inc += y;
    }
    if (k < nl) cd.wl[k] = WList{base + inc - cap, 0u, cap, 0u};
    base += __shfl_sync(FULL, inc, 31);
  }
  __syncwarp();
  cd.pool_top = 0;
  cd.full = 0;
  if (base > cd.pool_cap / 2) return false;  // leave room for the lists to grow
  for (uint32_t k = w.lane; k < run_cl; k += 32) {
    const uint32_t c = cd.cl_off[k];
    const uint32_t l0 = cd.arena[c + CD_HDR], l1 = cd.arena[c + CD_HDR + 1];
    const uint32_t p0 = atomicAdd(&cd.wl[l0].len, 1u);
    cd.pool[cd.wl[l0].off + p0] = (uint64_t)c | ((uint64_t)l1 << 32);
    const uint32_t p1 = atomicAdd(&cd.wl[l1].len, 1u);
    cd.pool[cd.wl[l1].off + p1] = (uint64_t)c | ((uint64_t)l0 << 32);
  }
  cd.pool_top = base;
  __syncwarp();
  return true;
}

// Bring the database back within its limits at the bottom level: compact
// (drop_half false) or halve it, and if the lists still do not fit, drop it.
// Afterwards the bottom levels are propagated again from the first trail
// entry, over the rebuilt watch lists too.
__device__ __noinline__ void maintain_db(Warp& w, CdWarp& cd, bool drop_half) {
  const long long t0 = pf_now(*w.S);
  if (w.S->prof && w.lane == 0) w.cyc[PF_NDB]++;
  backjump_cd(w, cd, w.nd_fixed);
  if (!reduce_db(w, cd, drop_half) && (drop_half || !reduce_db(w, cd, true)))
    clear_learnts(w, cd);
  w.confl = 0;
  // the head moves back: the ring has to hold the last positions below the tail
  // again (undone claims may have overwritten them)
  for (uint32_t k = w.lane; k < min(w.tail, CD_RING); k += 32) {
    const uint32_t p = w.tail - 1u - k;
    cd.ring()[p & (CD_RING - 1u)] = w.trail[p];
  }
  __syncwarp();
  w.head = 0;
  pf_add(*w.S, w, PF_DB, t0);
}

// luby(i), i >= 1: 1 1 2 1 1 2 4 1 1 2 1 1 2 4 8 ...: luby(2^k - 1) = 2^(k-1);
// otherwise the sequence repeats itself, luby(i) = luby(i - 2^(k-1) + 1) for
// 2^(k-1) <= i < 2^k - 1 (Luby, Sinclair and Zuckerman).
__device__ uint32_t luby_cd(uint32_t i) {
  for (;;) {
    uint32_t k = 1;
    while (k < 31 && (1u << k) - 1u < i) k++;
    if (i == (1u << k) - 1u || k == 31) return 1u << (k - 1);
    i -= (1u << (k - 1)) - 1u;
  }
}

// Learned clauses handed to a cube with its assumptions (all lanes): the
// newest clauses of at most 12 literals and LBD at most 4, as many as fit
// dst[JOB_CLS_WORDS] = [count, words used, offsets[JOB_CLS_MAX], records
// {len, lbd, literals}]. Every learned clause is implied by the formula, so
// the cube may use them whatever its assumptions.
__device__ __noinline__ void export_clauses(Warp& w, CdWarp& cd, uint32_t* dst) {
  constexpr uint32_t base = 2 + JOB_CLS_MAX;
  uint32_t m = 0, used = base;
  for (int64_t k0 = (int64_t)cd.ncl - 1; k0 >= 0 && m < JOB_CLS_MAX; k0 -= 32) {
    const int64_t k = k0 - w.lane;
    uint32_t off = 0, len = 0, lbd = 0, words = 0;
    if (k >= 0) {
      off = cd.cl_off[k];
      len = cd.arena[off];
      lbd = cd.arena[off + 2];
      if (len <= 12u && lbd <= 4u) words = len + 2u;
    }
    uint32_t inc = words;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(FULL, inc, d);
      if (w.lane >= d) inc += y;
    }
    const bool ok = words > 0 && used + inc <= JOB_CLS_WORDS;
    const uint32_t okm = __ballot_sync(FULL, ok);
    const uint32_t rank = __popc(okm & ((1u << w.lane) - 1u));
    if (ok && m + rank < JOB_CLS_MAX) {
      const uint32_t at = used + inc - words;
      dst[2 + m + rank] = at;
      dst[at] = len;
      dst[at + 1] = lbd;
      for (uint32_t q = 0; q < len; q++) dst[at + 2 + q] = cd.arena[off + CD_HDR + q];
    }
    const uint32_t taken = min((uint32_t)__popc(okm), JOB_CLS_MAX - m);
    // the prefix sums grow with the lane, so the clauses that fit are a prefix
    const int last = taken ? __fns(okm, 0, taken) : -1;
    if (taken) used += __shfl_sync(FULL, inc, last);
    m += taken;
    if (__popc(okm) < __popc(__ballot_sync(FULL, words > 0))) break;  // buffer full
  }
  if (w.lane == 0) {
    dst[0] = m;
    dst[1] = used;
  }
  __syncwarp();
}

// The clauses a donor attached to this cube (see export_clauses) into the
// empty database, then its watch lists. Returns false (the database is left
// empty) if they do not fit.
__device__ __noinline__ bool import_clauses(Warp& w, CdWarp& cd, const uint32_t* src) {
  const uint32_t m = min(src[0], JOB_CLS_MAX);
  uint32_t top = 0;
  for (uint32_t k0 = 0; k0 < m; k0 += 32) {
    const uint32_t k = k0 + w.lane;
    uint32_t at = 0, len = 0, words = 0;
    if (k < m) {
      at = src[2 + k];
      if (at >= 2 + JOB_CLS_MAX && at + 2 < JOB_CLS_WORDS) {
        len = src[at];
        if (at + 2 + len <= JOB_CLS_WORDS && len >= 2u && len <= 12u) words = clause_words(len);
      }
    }
    uint32_t inc = words;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(FULL, inc, d);
      if (w.lane >= d) inc += y;
    }
    const uint32_t c = top + inc - words;
    const uint32_t okm = __ballot_sync(FULL, words > 0);
    if (!__all_sync(FULL, !words || c + words <= cd.arena_words)) {  // no room
      clear_learnts(w, cd);
      return false;
    }
    if (words) {
      cd.arena[c] = len;
      cd.arena[c + 1] = 0u;
      cd.arena[c + 2] = src[at + 1];
      cd.arena[c + 3] = 0u;
      for (uint32_t q = 0; q < words - CD_HDR; q++)
        cd.arena[c + CD_HDR + q] = q < len ? src[at + 2 + q] : NONE;
      cd.cl_off[cd.ncl + __popc(okm & ((1u << w.lane) - 1u))] = c;
    }
    top += __shfl_sync(FULL, inc, 31);
    cd.ncl += __popc(okm);
    __syncwarp();
  }
  cd.top = top;
  if (!rebuild_watches(w, cd)) {
    clear_learnts(w, cd);
    return false;
  }
  return true;
}

// pick_max where the activities are in global memory: for every 128 variables
// shared memory holds a bound on the activities of the unassigned ones (0: none
// left, else the bits of the bound plus 1). Assigning and bumping (an analysis
// bumps assigned variables only) leave a bound valid; backjump_cd raises it for
// what it unassigns, and looking at a group makes it exact. So a decision looks
// at the few groups whose bound reaches the best variable found, not at 40 KB
// of activities of an instance of 10,000 variables: on 128 large queries 20,000
// cycles a decision became 3,200, 28 % of all cycles 6 %, and 65 ms 58.
__device__ __forceinline__ uint32_t pick_grouped(const Warp& w, uint32_t* gmax) {
  uint32_t best = 0, best_v = NONE;
  for (;;) {
    // the group of the highest bound, the lowest one of equals
    uint32_t top = 0, g = NONE;
    for (uint32_t k = w.lane; 128u * k < w.V; k += 32) {
      const uint32_t x = gmax[k];
      if (x > top) {
        top = x;
        g = k;
      }
    }
    const uint32_t high = __reduce_max_sync(FULL, top);
    if (high == 0u || high < best) return best_v;
    g = __reduce_min_sync(FULL, top == high ? g : NONE);
    if (high == best && g >= (best_v >> 7)) return best_v;
    const uint32_t v = 128u * g + 4u * w.lane;
    uint32_t un = 0;
    if (v < w.V) {
      const uint32_t word = w.asg[2 * (v >> 4)];
      un = (~(word | (word >> 1)) >> (2u * (v & 15u))) & 0x55u;
      if (w.V - v < 4u) un &= (1u << (2u * (w.V - v))) - 1u;
    }
    uint32_t key = 0, kv = NONE;
    if (un) {
      const float4 a = *reinterpret_cast<const float4*>(w.act + v);
      const float x[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
      for (int q = 0; q < 4; q++)
        if (((un >> (2 * q)) & 1u) && __float_as_uint(x[q]) + 1u > key) {
          key = __float_as_uint(x[q]) + 1u;
          kv = v + q;
        }
    }
    const uint32_t most = __reduce_max_sync(FULL, key);
    kv = __reduce_min_sync(FULL, key == most ? kv : NONE);
    if (w.lane == 0) gmax[g] = most;
    __syncwarp();
    if (most > best || (most == best && kv < best_v)) {
      best = most;
      best_v = kv;
    }
  }
}

__device__ uint32_t pick_cd(Warp& w, unsigned char* area) {
  if (!(w.S->cd_smem & CD_SMEM_GMAX)) return pick_max<2>(w);
  const uint32_t v = pick_grouped(w, cd_area_gmax(area));
#ifdef SCUBA_CHECKED
  (void)WIDX(w, v == pick_max<2>(w) ? 0u : 1u, 1u, 27);
#endif
  return v;
}

// ---- clauses shared between the jobs of one instance ----------------------
//
// Every learned clause is implied by the formula alone (assumption literals
// enter it as decisions, level-0 literals are dropped only when false at
// level 0), so any job of the same instance may use it, whatever its own
// assumptions. Jobs that run beside others of their instance publish their
// short, low-LBD learned clauses to a per-instance pool and read the others'
// at each restart. A pool is a ring of fixed-size records in global memory:
// a writer reserves record r with one atomicAdd on the pool's cursor, writes
// the body, then the header r + 1 with a release store. A reader takes record r only
// if its header reads r + 1 before the body and the cursor shows, after the
// body, that no writer can have reserved the record's slot again (cursor <=
// r + cap). Records that fail either check are skipped, never guessed.

// Publish learnt[0..n) (1 <= n <= SHARE_MAXLEN) with its LBD (all lanes).
__device__ void share_publish(const Solve& S, Warp& w, CdWarp& cd, uint32_t n, uint32_t lbd,
                              int64_t slot) {
  const uint32_t p = (uint32_t)w.inst & S.share_mask;
  unsigned long long r = 0;
  if (w.lane == 0) r = atomicAdd(&S.share_cur[p], 1ull);
  r = __shfl_sync(FULL, r, 0);
  uint32_t* rec =
      S.share + ((size_t)p * S.share_cap + (uint32_t)(r & (S.share_cap - 1u))) * SHARE_REC;
  if (w.lane >= 1 && w.lane < (int)SHARE_REC) {
    uint32_t x;
    if (w.lane == 1) x = (uint32_t)w.inst;
    else if (w.lane == 2) x = n | (min(lbd, 255u) << 8);
    else if (w.lane == 3) x = (uint32_t)slot;
    else x = (uint32_t)(w.lane - 4) < n ? cd.lsm()[w.lane - 4] : NONE;
    *(volatile uint32_t*)&rec[w.lane] = x;
  }
  __syncwarp();
  if (w.lane == 0) store_release(&rec[0], (uint32_t)(r + 1ull));
  __syncwarp();
}

// Read the pool's records published since *rd by other jobs of this
// instance, at most 256 per call, into the learned-clause database (all
// lanes, at the bottom level after a restart). Each clause is watched on two
// literals that are not false if it has them, else on its one such literal
// and the false literal of highest level; a clause with one open literal
// left implies it, one with none refutes the job. Returns false in that
// case (the job's assumptions contradict the formula), true otherwise.
__device__ __noinline__ bool share_import(const Solve& S, Warp& w, CdWarp& cd, int64_t slot,
                             unsigned long long& rd) {
  const uint32_t p = (uint32_t)w.inst & S.share_mask;
  const unsigned long long cap = S.share_cap;
  unsigned long long cur = 0;
  if (w.lane == 0) cur = *(volatile unsigned long long*)&S.share_cur[p];
  cur = __shfl_sync(FULL, cur, 0);
  unsigned long long from = rd;
  if (cur > cap / 2 && from < cur - cap / 2) from = cur - cap / 2;  // skip what may be overwritten
  const unsigned long long to = min(cur, from + 256ull);
  bool ok_all = true;
  for (unsigned long long base = from; base < to && ok_all; base += 32) {
    const unsigned long long r = base + (unsigned long long)w.lane;
    bool ok = r < to;
    uint32_t n = 0, lbd = 0, lit[SHARE_MAXLEN];
    const uint32_t* rec = S.share + ((size_t)p * S.share_cap + (uint32_t)(r & (cap - 1u))) * SHARE_REC;
    if (ok) ok = *(const volatile uint32_t*)&rec[0] == (uint32_t)(r + 1ull);
    if (ok) {
      __threadfence();
      const uint32_t ins = *(const volatile uint32_t*)&rec[1];
      const uint32_t nl = *(const volatile uint32_t*)&rec[2];
      const uint32_t prod = *(const volatile uint32_t*)&rec[3];
      n = nl & 255u;
      lbd = nl >> 8;
      ok = ins == (uint32_t)w.inst && prod != (uint32_t)slot && n >= 1 && n <= SHARE_MAXLEN;
#pragma unroll
      for (uint32_t k = 0; k < SHARE_MAXLEN; k++) {
        lit[k] = *(const volatile uint32_t*)&rec[4 + k];
        if (k < n && lit[k] >= 2u * w.V) ok = false;
      }
      __threadfence();
      const unsigned long long now = *(volatile unsigned long long*)&S.share_cur[p];
      if (now > r + cap) ok = false;  // the slot may hold a newer record by now
    }
    for (uint32_t todo = __ballot_sync(FULL, ok); todo && ok_all; todo &= todo - 1u) {
      const int j = __ffs(todo) - 1;
      const uint32_t nj = __shfl_sync(FULL, n, j), lbdj = __shfl_sync(FULL, lbd, j);
      uint32_t my = NONE;
#pragma unroll
      for (uint32_t k = 0; k < SHARE_MAXLEN; k++) {
        const uint32_t x = __shfl_sync(FULL, lit[k], j);
        if ((uint32_t)w.lane == k) my = x;
      }
      const bool have = (uint32_t)w.lane < nj;
      const uint32_t val = have ? lit_value_cd(w.asg, my) : LV_F;
      const uint32_t lvl = have && val == LV_F ? level_of(cd, my >> 1) : 0u;
      const uint32_t nf = __ballot_sync(FULL, have && val != LV_F);
      if (nf == 0u) {  // every literal false: the job's assumptions are refuted
        ok_all = false;
        break;
      }
      const int w0 = __ffs(nf) - 1;
      int w1 = -1;
      if (__popc(nf) >= 2) {
        w1 = __fns(nf, 0, 2);
      } else if (nj >= 2) {  // the false literal of the highest level (lowest lane on ties)
        const bool cand = have && w.lane != w0;
        uint32_t best = cand ? lvl : 0u;
        for (int d = 16; d > 0; d >>= 1) best = max(best, __shfl_xor_sync(FULL, best, d));
        w1 = __ffs(__ballot_sync(FULL, cand && lvl == best)) - 1;
      }
      const bool unit = __popc(nf) == 1 && __shfl_sync(FULL, val, w0) == LV_U;
      const uint32_t first = __shfl_sync(FULL, my, w0);
      if (nj == 1) {  // a unit clause: its literal holds in every model
        if (unit) assign_one_cd(w, cd, first, NONE, NONE);
        continue;
      }
      if ((uint64_t)cd.top + clause_words(nj) > cd.arena_words || cd.full) break;
      // the two watches first, then the rest in record order
      const uint32_t rest = __ballot_sync(FULL, have) & ~(1u << w0) & ~(1u << w1);
      if (have) {
        uint32_t at;
        if (w.lane == w0) at = 0;
        else if (w.lane == w1) at = 1;
        else at = 2u + __popc(rest & ((1u << w.lane) - 1u));
        cd.lsm()[at] = my;
      }
      __syncwarp();
      const uint32_t c = add_learnt(w, cd, nj, lbdj);
      if (unit) assign_one_cd(w, cd, first, LEARNT_REF | c, 0u);
    }
  }
  rd = to;
  __syncwarp();
  return ok_all;
}

// One job: an instance, or a cube of it (the job's literals as assumptions,
// from the subtree-sharing ring), start to verdict. Returns SAT, UNSAT (for a
// cube: no model extends it) or UNKNOWN.
__device__ int run_cdcl(const Solve& S, Warp& w, int64_t slot, int unit, int inst,
                        const TakenJob* job, unsigned char* area, int& abort_code) {
  CdWarp cd;
  cd.area = area;
  cd.epoch = 0;
  cd.var = reinterpret_cast<VarInfo*>(S.cd_var) + slot * S.vmax;
  cd.pl = nullptr;
  cd.mark = S.cd_mark + slot * S.vmax;
  if (S.cd_smem & CD_SMEM_POS) {
    const size_t v16 = ((size_t)S.vmax + 15) & ~(size_t)15;
    unsigned char* at = area + cd_area_bytes(S.cd_smem & ~CD_SMEM_POS, S.vmax);
    cd.pl = reinterpret_cast<uint32_t*>(at);
    cd.mark = at + 4 * v16;
  }
  cd.wl = S.cd_wl + slot * 2 * S.vmax;
  cd.pool = S.cd_pool + slot * S.cd_pool_cap;
  cd.arena = S.cd_arena + slot * S.cd_arena_words;
  cd.learnt = S.cd_learnt + slot * S.vmax;
  cd.cl_off = S.cd_clidx + slot * (S.cd_arena_words / 8);
  cd.arena_words = (uint32_t)S.cd_arena_words;
  cd.ncl = 0;
  cd.pool_cap = (uint32_t)S.cd_pool_cap;
  cd.top = 0;
  cd.pool_top = 0;
  cd.full = 0;
  w.inst = inst;
  w.V = (uint32_t)S.nv[inst];
  w.c0 = S.icb[inst];
  w.occ = S.occ_begin + S.occ_base[inst];
  const int64_t lbase = S.icb[inst] < S.icb[inst + 1] ? S.cb[S.icb[inst]] : 0;
  w.ent = S.ent + lbase;
  warp_checks(w, S.ctrl);
  w.head = 0;
  w.nd = 0;
  w.nd_fixed = 0;
  w.inc = job ? job->inc : 1.0f;  // a cube starts from its donor's activities
  const uint32_t nwords = 2u * ((w.V + 15u) >> 4);
  for (uint32_t k = w.lane; k < nwords; k += 32) w.asg[k] = 0u;
  for (uint32_t v = w.lane; v < w.V; v += 32) {
    if (!job) w.act[v] = 0.0f;
    cd.mark[v] = 0;
  }
  if (S.cd_smem & CD_SMEM_GMAX)
    for (uint32_t g = w.lane; 128u * g < w.V; g += 32) cd_area_gmax(area)[g] = GMAX_LOOK;
  w.tail = 0;
  w.confl = 0;
  // Calls of the rarely used parts work on copies of w and cd, so that the
  // search itself can keep them in registers. (All of them come back, also the
  // pointers, which do not change: a compiler that knows that computes them from
  // the launch's arguments each time, which measured 4 % slower.)
  auto apart = [&](auto&& fn) {
    Warp w2 = w;
    CdWarp cd2 = cd;
    fn(w2, cd2);
    w = w2;
    cd = cd2;
  };
  apart([&](Warp& a, CdWarp& b) {
    clear_learnts(a, b);
    if (job && job->cls) import_clauses(a, b, job->cls);  // the donor's clauses
  });
  __syncwarp();
  if (S.flags[inst] & F_EMPTY) return SCUBA_UNSAT;
  const uint32_t nu = S.nunits[inst];
  const uint32_t* un = S.units + w.c0;
  for (uint32_t k0 = 0; k0 < nu; k0 += 32) {
    const uint32_t l = k0 + w.lane < nu ? un[k0 + w.lane] : NONE;
    const bool clash = claim_cd(w, cd, l != NONE, l, NONE, NONE);
    __syncwarp();
    // a unit clause against an earlier one's value, or another lane's
    const bool bad = l != NONE && lit_value_cd(w.asg, l) != LV_T;
    if (__any_sync(FULL, clash || bad)) return SCUBA_UNSAT;
  }
  // the cube's literals become decisions of levels 1, 2, ..., one after each
  // propagation of the main loop
  int next_asm = 0;
  const int n_asm = job ? job->len : 0;

  // fixed levels that are the unit's own assumptions, not cube literals
  const uint32_t asm_levels =
      S.unit_asm_begin ? (uint32_t)min(S.unit_asm_begin[unit + 1] - S.unit_asm_begin[unit],
                                       (int64_t)MAX_PREFIX)
                       : 0u;
  uint32_t conflicts = 0, since_restart = 0, restart_no = 1;
  auto steps = [&] {  // counted down: a register less than a mask
    return flush_steps(__ldg(&w.occ[2u * w.V]), (uint64_t)S.cd_arena_words, w.V);
  };
  uint32_t until_flush = steps();
  uint32_t next_reduce = 2000u, reductions = 0;  // periodic database reduction
  uint32_t restart_at = (uint32_t)S.restart_unit * luby_cd(1);
  // clause sharing with the other jobs of this instance: on for a cube and
  // once this job has given one away or sees others running
  bool shared = S.share_lbd > 0 && job != nullptr;
  unsigned long long share_rd =
      S.share_lbd > 0 ? S.share_base[(uint32_t)inst & S.share_mask] : 0ull;
  for (;;) {
    if (--until_flush == 0u) {
      until_flush = steps();
      flush_counters(S, w, unit);
      int stop = 0;
      if (w.lane == 0) {
        if (S.abort_flag && *S.abort_flag) stop = 1;
        else if (search_ns(S) > S.time_ns) stop = 2;
        else if (*(volatile uint32_t*)&S.done[unit] & 1u) stop = 3;
#ifdef SCUBA_CHECKED
        else if (batch_failed(S.ctrl)) stop = 4;  // a bounds check failed: stop
#endif
      }
      stop = __shfl_sync(FULL, stop, 0);
      if (stop == 4) { abort_code = SCUBA_ERR_INTERNAL; return SCUBA_UNKNOWN; }
      if (stop == 1) { abort_code = SCUBA_ERR_ABORTED; return SCUBA_UNKNOWN; }
      if (stop == 2) { abort_code = SCUBA_ERR_TIMEOUT; return SCUBA_UNKNOWN; }
      if (stop == 3) return SCUBA_UNSAT;  // the instance is SAT already; this cube is moot
    }
    long long t0 = pf_now(S);
    const bool confl = bcp_cd(w, cd);
    pf_add(S, w, PF_BCP, t0);
    if (cd.full) {  // the watch pool ran out: compact it (or halve the clauses)
      apart([](Warp& a, CdWarp& b) { maintain_db(a, b, false); });
      continue;
    }
    if (confl) {
      if (next_asm < n_asm) return SCUBA_UNSAT;  // the assumptions alone
      WCOUNT(w, conflicts, 1);
      if (w.nd <= w.nd_fixed) return SCUBA_UNSAT;
      conflicts++;
      since_restart++;
      t0 = pf_now(S);
      uint32_t blev, lbd;
      const uint32_t n = analyze_cd(w, cd, blev, lbd);
      if (n == 0) {
        abort_code = SCUBA_ERR_INTERNAL;
        return SCUBA_UNKNOWN;
      }
      // Cubes many levels deep share clauses of two levels whatever the bound: such a
      // tree is growing out of hand, and they keep it from it. With a bound of one
      // level throughout, 16 to 24 solves of 512 partition queries of 16 bits took a
      // mean of 116-288 ms (slowest 2,179), so 76 (175); 128 of them 259-316 and 79, 512
      // of 18 bits 266-395 and 93, 256 of 20 bits 240-1,196 (11,241) and 146 (471). With
      // two levels throughout 50, 61, 74 and 155, but 4,096 of 16 bits 92 (86 and 87
      // so), 256 bounds queries of 16 bits 56 (33 and 33), units 6.9 (6.1). From 14
      // levels 55, 68, 109, 144 and 87, 39; from 28 62, 80, 103, 254 and 88, 33.
      if (shared && n <= SHARE_MAXLEN &&
          (n == 1 || lbd <= S.share_lbd || (lbd <= 2u && w.nd_fixed >= asm_levels + DEEP_CUBE)))
        share_publish(S, w, cd, n, lbd, slot);
      // Activities fade quickly while the search learns clauses that join few
      // levels (a conflict of one part of the formula: stay there), slowly
      // otherwise. Against 0.95 throughout: 4,096 partition queries 95.0 -> 90.5
      // ms, units 6.45 -> 6.0, 12 bounds queries 2.22 -> 2.15, large queries 54 -> 50,
      // random 3-SAT, whose clauses join many levels, 45.0 -> 45.4. (0.90 throughout
      // 88.6 and 51 ms on partition queries and 3-SAT; 5 levels in place of 4
      // 92.5 and 47.5.)
      w.inc *= lbd <= 4u ? (1.0f / 0.86f) : (1.0f / 0.97f);
      w.confl = 0;
      const uint32_t target = max(blev, w.nd_fixed);
      if (n >= 2 && (uint64_t)cd.top + clause_words(n) > cd.arena_words) {
        apart([&](Warp& a, CdWarp& b) {
          maintain_db(a, b, true);  // arena full: restart with half the clauses
          if ((uint64_t)b.top + clause_words(n) > b.arena_words) clear_learnts(a, b);
        });
        since_restart = 0;
      } else {
        backjump_cd(w, cd, target);
      }
      uint32_t why = NONE;
      const uint32_t uip = cd.lsm()[0];
      if (n >= 2) {
        uint32_t c = add_learnt(w, cd, n, lbd);
        if (cd.full)  // the pool ran out: compact it, the new clause included
          apart([&](Warp& a, CdWarp& b) {
            maintain_db(a, b, false);
            // the newest clause survives a compaction or a halving; after a
            // full drop it is added again to the empty database
            c = b.ncl > 0 ? b.cl_off[b.ncl - 1] : add_learnt(a, b, n, lbd);
          });
        why = LEARNT_REF | c;
      }
      // the clause is unit once every literal but the first is false
      if (n == 1 || blev <= w.nd) assign_one_cd(w, cd, uip, why, n == 1 ? NONE : 0u);
      pf_add(S, w, PF_ANALYZE, t0);
      if (S.budget > 0) {  // conflicts of the instance, all of its cubes together
        unsigned long long tot = 0;
        if (w.lane == 0) tot = atomicAdd(&S.inst_dec[unit], 1ull) + 1ull;
        tot = __shfl_sync(FULL, tot, 0);
        if ((int64_t)tot >= S.budget) return SCUBA_UNKNOWN;
      }
      continue;
    }
    if (next_asm < n_asm) {
      const uint32_t l = job->lit[next_asm++];
      const uint32_t val = lit_value_cd(w.asg, l);
      if (val == LV_F) return SCUBA_UNSAT;
      if (val == LV_U) {
        if (w.lane == 0) w.dstack[WIDX(w, w.nd, (uint32_t)S.vmax, 19)] = w.tail;
        w.nd++;
        w.nd_fixed = w.nd;
        assign_one_cd(w, cd, l, NONE, NONE);
      }
      continue;
    }
    if (since_restart >= restart_at) {
      since_restart = 0;
      restart_no++;
      restart_at = (uint32_t)S.restart_unit * luby_cd(restart_no);
      if (conflicts >= next_reduce) {  // a restart that also halves the database
        reductions++;
        next_reduce = conflicts + 2000u + 300u * reductions;
        apart([](Warp& a, CdWarp& b) { maintain_db(a, b, true); });
      } else {
        backjump_cd(w, cd, w.nd_fixed);
      }
      if (S.share_lbd > 0 && !shared) {
        uint32_t others = 0;
        if (w.lane == 0) others = (*(volatile uint32_t*)&S.pending[unit] & PEND_JOBS) > 1u;
        shared = __shfl_sync(FULL, others, 0) != 0u;
      }
      if (shared) {
        bool ok = true;
        apart([&](Warp& a, CdWarp& b) { ok = share_import(S, a, b, slot, share_rd); });
        if (!ok) return SCUBA_UNSAT;
      }
      continue;
    }
    WCOUNT(w, act_reads, w.V - w.tail);
    t0 = pf_now(S);
    const uint32_t v = pick_cd(w, area);
    pf_add(S, w, PF_DECIDE, t0);
    if (v == NONE) {
      // the first cube of the instance to reach a model writes it
      uint32_t won = 0;
      if (w.lane == 0) won = !(atomicOr(&S.done[unit], 8u) & 8u);
      won = __shfl_sync(FULL, won, 0);
      if (won && S.model)
        for (uint32_t x = w.lane; x < w.V; x += 32) {
          S.model[(S.unit_vb ? S.unit_vb[unit] : S.vb[inst]) + x] =
              lit_value_cd(w.asg, 2u * x) == LV_T ? 1 : 0;
        }
      __syncwarp();
      return SCUBA_SAT;
    }
    // cube-and-conquer: hand the other side of the first free decision to an
    // idle warp and keep this side as an assumption, up to split_depth cube
    // levels below the instance. A cube relearns almost from scratch, so a
    // job should share only once it has shown itself hard: sharing after 2 to 4
    // decisions whenever warps are idle took 48 ms for 12 bounds queries that need
    // 2.1 (16 decisions). split_min and split_interval hold while more than 7/8 of
    // the warps are idle, where a few hard instances decide the time and the
    // tree has to reach the idle warps quickly; both double with the busy share from
    // there on, up to 128 and 16 decisions, when most warps are busy and sharing
    // gains least. (16 and 4 so, against 32 and 16 throughout: 12
    // and 256 bounds queries 4.2 -> 2.8 and 6.6 -> 5.0 ms, units 10.0 -> 7.9, random
    // 3-SAT 51.5 -> 47.6, 4,096 partition queries 100 -> 97; three seeds.)
    if (S.split && w.decisions >= (uint32_t)S.split_min &&
        w.decisions % (uint32_t)S.split_interval == 0 && w.nd > w.nd_fixed &&
        w.nd_fixed + 1 <= (uint32_t)MAX_PREFIX &&
        w.nd_fixed < asm_levels + (uint32_t)S.split_depth) {
      uint32_t idle = 0;
      if (w.lane == 0) idle = *(volatile uint32_t*)&S.ctrl->idle;
      idle = __shfl_sync(FULL, idle, 0);
      const uint32_t warps = gridDim.x * (blockDim.x >> 5), busy = warps - min(idle, warps);
      const uint32_t times = busy > warps / 2 ? 8 : busy > warps / 4 ? 4 : busy > warps / 8 ? 2 : 1;
      // (a setting beyond the limits is taken as it is)
      const uint32_t gate = max((uint32_t)S.split_min, min((uint32_t)S.split_min * times, 128u));
      const uint32_t interval =
          max((uint32_t)S.split_interval, min((uint32_t)S.split_interval * times, 16u));
      if (idle > 0 && w.decisions >= gate && w.decisions % interval == 0) {
        const uint32_t k = w.nd_fixed;
        if (w.lane == 0) atomicAdd(&S.pending[unit], 1u);
        __syncwarp();
        if (ring_push(S, w, unit, k + 1, w.trail, w.dstack, k, [&](uint32_t cell) {
              apart([&](Warp& a, CdWarp& b) {
                export_clauses(a, b, S.job_cls + (size_t)cell * JOB_CLS_WORDS);
              });
            })) {
          w.nd_fixed = k + 1;
          shared = S.share_lbd > 0;
          if (w.lane == 0) {
            atomicAdd(&S.ctrl->jobs_split, 1u);
            if (S.prof) {
              atomicAdd(&S.prof[0], 1ull);
              atomicAdd(&S.prof[2], (unsigned long long)(k + 1));
              atomicAdd(&S.prof[3], (unsigned long long)(w.nd - k));
            }
          }
        } else if (w.lane == 0) {
          atomicSub(&S.pending[unit], 1u);
          if (S.prof) atomicAdd(&S.prof[4], 1ull);
        }
        __syncwarp();
      }
    }
    w.decisions++;
    WCOUNT(w, decisions, 1);
    const uint32_t lit = 2u * v + ((cd.mark[v] & MK_PHASE) ? 0u : 1u);
    if (w.lane == 0) w.dstack[WIDX(w, w.nd, (uint32_t)S.vmax, 19)] = w.tail;
    w.nd++;
    assign_one_cd(w, cd, lit, NONE, NONE);
  }
}
