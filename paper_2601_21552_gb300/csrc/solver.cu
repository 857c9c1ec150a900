// solver.cu -- GPU DPLL over batches of CNFs (the satisfiability step of
// Sec. V-B, step 10, applied to one query per static memory instruction).
//
// Layout in HBM (per batch, built by the prep kernels from the caller's CSR):
//   occ_begin[..]  u32  per instance 2V+1 offsets: occurrence list of each
//                       literal code 2(v-1)+neg (clauses that contain it)
//   ent[L]         u64  occurrence entries, clause group by clause group within a list:
//                       binary (x|y) in x's list = {y, NONE}; ternary
//                       (x|y|z) in x's list = {y, z}; longer clauses =
//                       {LONG_CLAUSE|local clause index, 0}
//   units[C]       u32  unit-clause literal codes, compacted per instance
// Per worker slot (one warp): trail[Vmax], dstack[Vmax], act[Vmax] in global
// memory; the assignment (2 bits per variable) in shared memory.
//
// Search per instance (complete DPLL): unit propagation to a fixpoint over
// occurrence lists, frontier-parallel across the 32 lanes; on conflict bump
// the activity of the falsified clause's variables and backtrack
// chronologically to the deepest decision not yet flipped; otherwise decide
// the unassigned variable of highest activity (ties: lowest id), value false
// first. A busy warp hands the untried branch of its shallowest open decision
// to an idle warp (subtree splitting) so that hard instances spread over the
// whole GPU.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/scuba.h"
#include "learn.cuh"
#include "rules.h"
#include "scuba_internal.h"

namespace scuba {
namespace dev {

constexpr uint32_t FULL = 0xffffffffu;
constexpr uint32_t NONE = 0xffffffffu;
constexpr uint32_t LONG_CLAUSE = 0x80000000u;
constexpr uint32_t FLIP = 0x80000000u;
constexpr uint32_t F_EMPTY = 1u, F_BAD = 2u;
// A unit's word of open jobs: their number, a job found a model, a job gave up.
constexpr uint32_t PEND_JOBS = 0x3fffffffu, PEND_SAT = 0x40000000u, PEND_GAVE_UP = 0x80000000u;
constexpr int MAX_PREFIX = 248;   // literals in a split job's prefix
// Learned clauses a clause-learning donor attaches to a cube: [count, words
// used, offset of each clause (JOB_CLS_MAX), records {len, lbd, literals}].
constexpr uint32_t JOB_CLS_MAX = 256, JOB_CLS_WORDS = 4096;
// Clause-learning records shared between the jobs of one instance: {seq,
// instance, len | lbd << 8, producer slot, up to SHARE_MAXLEN literals}.
constexpr uint32_t SHARE_REC = 16, SHARE_MAXLEN = 12;

__device__ __forceinline__ uint32_t code_of(int32_t l) {
  int32_t v = l > 0 ? l : -l;
  return 2u * (uint32_t)(v - 1) + (l < 0 ? 1u : 0u);
}

__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// --------------------------------------------------------------------------
// Prep
// --------------------------------------------------------------------------

struct Ctrl {
  uint32_t next_inst;   // fresh-instance counter
  uint32_t inst_left;   // instances not finished yet
  uint32_t idle;        // warps waiting for work
  int32_t status;       // first error (scuba status code)
  uint32_t q_head, q_tail;
  uint64_t t0;          // globaltimer when the search began (0: not yet)
  uint32_t jobs_split;  // statistics
  uint32_t next_item, n_items;  // preparation work items
  int32_t check_site;   // checked build: site of the first failed bounds check (0: none)
  uint64_t check_index; // ... the index it saw
  uint64_t check_limit; // ... and the bound it broke
};

__device__ void fail_batch(Ctrl* c, int32_t st) { atomicCAS(&c->status, 0, st); }

// Bounds checks of the checked build (-DSCUBA_CHECKED; compute-sanitizer is
// not available everywhere). SCUBA_IDX(ctrl, i, limit, site) is i when
// i < limit; otherwise the first failure records its site, index and bound,
// the call's status becomes SCUBA_ERR_INTERNAL and the access goes to index 0
// instead, so it stays inside its buffer (the call's results are void from
// then on). Without SCUBA_CHECKED the macro is the index itself.
#ifdef SCUBA_CHECKED
__device__ __noinline__ uint64_t check_fail(Ctrl* c, uint64_t i, uint64_t lim, int site) {
  if (atomicCAS(&c->check_site, 0, site) == 0) {
    c->check_index = i;
    c->check_limit = lim;
  }
  fail_batch(c, -8 /* SCUBA_ERR_INTERNAL */);
  return 0;
}
// The index expression is evaluated exactly once (it may be an atomicAdd).
template <class T>
__device__ __forceinline__ T checked_idx(Ctrl* c, T i, uint64_t lim, int site) {
  return (uint64_t)i < lim ? i : (T)check_fail(c, (uint64_t)i, lim, site);
}
#define SCUBA_IDX(ctrl, i, lim, site) \
  ::scuba::dev::checked_idx((ctrl), (i), (uint64_t)(lim), (site))
#else
#define SCUBA_IDX(ctrl, i, lim, site) (i)
#endif

__device__ __forceinline__ bool batch_failed(Ctrl* c) {
  return *(volatile int32_t*)&c->status != 0;
}

// --------------------------------------------------------------------------
// Solve
// --------------------------------------------------------------------------

struct Job {            // a DPLL subtree: the instance plus assumed literals
  int32_t inst;
  int32_t len;
  uint32_t lit[MAX_PREFIX];
  uint32_t seq;         // ring-buffer sequence number (Vyukov MPMC queue)
  float inc;            // donor's activity increment; its activities are in job_act
};

#include "prep.cuh"

// Decision-trace buffers (training data for the branching network).
struct TraceDev {
  unsigned long long* cursor;  // [2]: nodes, rows reserved
  int64_t max_nodes, max_rows;
  int32_t* node_inst;
  int32_t* node_depth;
  int64_t* node_row;
  int32_t* node_nrows;
  int32_t* node_closed;
  __nv_bfloat16* x;            // [max_rows][NFEAT]
  float* target;               // [max_rows]
  int32_t* var;                // [max_rows]
};

// MODE_CDCL1: clause learning where an SM holds one block only (large instances),
// which may then have 8 warps and 255 registers a thread. MODE_CDCL8: two blocks of
// 8 warps (128 registers) for batches that keep every warp busy.
enum { MODE_PLAIN = 0, MODE_TRACE = 1, MODE_LEARNED = 2, MODE_CDCL = 3, MODE_CDCL1 = 4,
       MODE_CDCL8 = 5 };
constexpr bool is_cdcl(int mode) { return mode >= MODE_CDCL; }

// Activities of a slot: whole groups of 16, what one 2-bit assignment word covers.
__host__ __device__ __forceinline__ int64_t act_stride(int32_t vmax) {
  return ((int64_t)vmax + 15) & ~(int64_t)15;
}

struct WList;  // a learned watch list (clause-learning mode)

struct Solve {
  int n;
  int32_t vmax;
  uint32_t assign_words;   // per-warp shared words (2 bits per variable)
  const int64_t* icb;
  const int64_t* cb;
  const int32_t* lits;
  const int32_t* nv;
  const int64_t* vb;
  const int64_t* occ_base;
  const uint32_t* occ_begin;
  const uint64_t* ent;
  const uint32_t* units;
  const uint32_t* nunits;
  const uint32_t* flags;
  const int32_t* order;
  // units: instance + assumption literals (solve_units); without a unit table
  // every instance is one unit with no assumptions
  int n_units;
  const int32_t* unit_inst;        // [n_units] or NULL (unit u is instance u)
  const int64_t* unit_asm_begin;   // [n_units+1] or NULL
  const int32_t* unit_asm;         // DIMACS assumption literals
  const int64_t* unit_vb;          // [n_units] model offset of each unit, or NULL
  uint8_t* verdict;
  uint8_t* model;
  int64_t* stats;
  // per instance bookkeeping
  uint32_t* pending;       // open jobs of a unit (PEND_JOBS), and what its finished ones found
  uint32_t* done;          // 1 once a model was found, 8 once a job writes it
  unsigned long long* inst_dec;  // decisions so far (budget)
  // per slot
  uint32_t* trail;
  uint32_t* dstack;
  float* act;
  // job ring
  Job* ring;
  float* job_act;          // [ring_cap x vmax] donor activity snapshot per cell
  uint32_t* prefix;        // [slots x MAX_PREFIX] the running job's assumptions
  uint32_t ring_cap;       // power of two
  int32_t split_min;       // decisions a job makes before it may donate
  int32_t split_depth;     // CDCL: cube levels below the instance a donor may reach
  Ctrl* ctrl;
  int64_t budget;
  uint64_t time_ns;
  const volatile int32_t* abort_flag;
  int split;
  int split_interval;
  int trail_smem;          // 1: each warp's trail lives in shared memory
  int64_t* finish_ns;      // optional [n]: completion time of each instance
  unsigned long long* prof;  // optional [8]: search counters
  // learned branching and trace recording
  const learn::MlpWeights* mlp;
  int learned_depth;           // MLP decides at decision depth < learned_depth
  const int32_t* inst_num_inputs;  // optional [n]: input bits (numbered first)
  int trace_depth;             // record decisions at depth < trace_depth
  TraceDev tr;
  uint32_t* lvlcnt;            // [slots][MAX_TRACE_DEPTH][vmax] conflict counts
  int64_t* lvl_node;           // [slots][MAX_TRACE_DEPTH] node of each open level
  // conflict-driven clause learning (per slot)
  uint4* cd_var;               // [slots][vmax] reason, trail position, level (16 B)
  uint8_t* cd_mark;            // [slots][vmax]
  int cd_smem;                 // per-variable state kept in shared memory (CD_SMEM_*)
  uint32_t cd_smem_warp;       // bytes of shared memory per warp beyond the assignment
  WList* cd_wl;                // [slots][2 vmax] learned watch lists
  uint64_t* cd_pool;           // [slots][cd_pool_cap] watch entries
  uint32_t* cd_learnt;         // [slots][vmax]
  uint32_t* cd_arena;          // [slots][cd_arena_words]
  uint32_t* cd_clidx;          // [slots][cd_arena_words / 8] clause offsets
  int64_t cd_arena_words, cd_pool_cap;
  uint32_t* job_cls;           // [ring_cap][JOB_CLS_WORDS] clauses shared with a cube
  uint32_t* cls_copy;          // [slots][JOB_CLS_WORDS] a taken cube's clauses
  int restart_unit;            // conflicts per Luby unit
  // clauses shared between the jobs (cubes, units) of one instance: pool
  // (inst & share_mask) is a ring of share_cap records of SHARE_REC words
  uint32_t* share;             // [pools][share_cap][SHARE_REC]
  unsigned long long* share_cur;  // [pools] records reserved so far
  const unsigned long long* share_base;  // [pools] ... before this call
  uint32_t share_mask;         // pools - 1 (a power of two)
  uint32_t share_cap;          // records per pool (a power of two)
  uint32_t share_lbd;          // publish learned clauses of LBD <= this; 0: off
};

// Recent trail literals a warp keeps in shared memory (a power of two; the
// clause-learning search keeps more, with their reasons: cdcl.cuh).
constexpr uint32_t RING = 16;

struct alignas(16) WarpShared {
  uint32_t tail, conflict;  // closures only: the searches keep theirs in registers
  uint32_t cl[3];
  uint32_t pad[3];
  // ring[p mod RING] = trail[p] for the positions p in [head, tail) that are
  // at most RING below the tail: a propagation round reads its literals here
  // instead of waiting for the global trail (DPLL)
  uint32_t ring[RING];
  // work counters, kept out of registers: added to without waiting (WADD), moved
  // to the caller's 64-bit ones every 64 steps of the search, oftener where 64
  // could pass 32 bits (flush_counters, flush_steps)
  uint32_t decisions, conflicts, props, visits, act_reads, undone;
  uint32_t pad2[6];
};
// The largest instance that fits an SM's shared memory beside this struct is part
// of the interface.
static_assert(sizeof(WarpShared) == 144, "per-warp shared memory");

enum : uint32_t { LV_U = 0, LV_T = 1, LV_F = 2, LV_X = 3 };

__device__ __forceinline__ uint32_t lit_value(const uint32_t* asg, uint32_t l) {
  uint32_t v = l >> 1;
  uint32_t bits = (asg[v >> 4] >> ((v & 15u) * 2u)) & 3u;
  if (bits == 0u || bits == 3u) return bits == 0u ? LV_U : LV_X;
  // bits 1 = variable true, 2 = variable false
  bool lit_true = (bits == 1u) ^ ((l & 1u) != 0u);
  return lit_true ? LV_T : LV_F;
}

struct Warp {
  const Solve* S;
  uint32_t* asg;
  WarpShared* ws;
  uint32_t* trail;
  uint32_t* dstack;
  float* act;
  unsigned long long* cyc; // clause learning: profile (cycles of lane 0 per phase; counts)
  int lane;
  int inst;
  uint32_t V;
  const uint32_t* occ;
  const uint64_t* ent;
  const int64_t* cb;       // the caller's clause_begin (long clauses)
  const int32_t* lits;     // the caller's literals (long clauses)
  int64_t c0;
  uint32_t head;
  uint32_t tail;           // trail length (the same in all lanes)
  uint32_t confl;          // a clause of the last bcp() is false (ws->cl)
  uint32_t nd;
  uint32_t nd_fixed;       // decisions below this index are assumptions
  float inc;
  uint32_t decisions;      // decisions of the current job
  uint32_t* lvlcnt;        // trace: per-level conflict counts of this slot
  int64_t* lvl_node;       // trace: node of each open level
  __nv_bfloat16* xtile;    // learned: 32 x NFEAT feature tile in shared memory
#ifdef SCUBA_CHECKED
  Ctrl* ck;                // where a failed bounds check is recorded
  uint32_t ent_end;        // occurrence entries of the instance (occ[2V])
#endif
};

// A checked index into a buffer of the current warp's instance.
#define WIDX(w, i, lim, site) SCUBA_IDX((w).ck, (i), (lim), (site))

// Checked build: the instance's bounds for WIDX (a no-op otherwise).
__device__ __forceinline__ void warp_checks(Warp& w, Ctrl* c) {
#ifdef SCUBA_CHECKED
  w.ck = c;
  w.ent_end = __ldg(&w.occ[2u * w.V]);
#else
  (void)w;
  (void)c;
#endif
}

// Add to a work counter, by the lanes that have something to add / by lane 0;
// nothing waits for the sum.
#define WADD(w, field, amount) atomicAdd(&(w).ws->field, (uint32_t)(amount))
#define WCOUNT(w, field, amount)               \
  do {                                         \
    if ((w).lane == 0) WADD(w, field, amount); \
  } while (0)

// The work counters into unit's statistics (all lanes).
__device__ __forceinline__ void flush_counters(const Solve& S, Warp& w, int unit) {
  __syncwarp();
  if (w.lane < SCUBA_NSTATS) {
    uint32_t* c = &w.ws->decisions + w.lane;
    if (S.stats)
      atomicAdd((unsigned long long*)&S.stats[SCUBA_NSTATS * (int64_t)unit + w.lane],
                (unsigned long long)*c);
    *c = 0;
  }
  __syncwarp();
}

#include "closure.cuh"

// Trail literal p of the current frontier, from a ring of SIZE.
template <uint32_t SIZE>
__device__ __forceinline__ uint32_t frontier_lit(const Warp& w, const uint32_t* ring, uint32_t p) {
  return w.tail - p <= SIZE ? ring[p & (SIZE - 1u)] : w.trail[p];
}

// Append the literals of the lanes with won set to the trail (all lanes): in
// lane order, so no counter in memory is involved. A ring of fewer slots than
// lanes takes the newest positions only: two lanes must not write one slot.
// Returns the lane's position.
template <uint32_t SIZE>
__device__ __forceinline__ uint32_t push_trail(Warp& w, uint32_t* ring, bool won, uint32_t l) {
  const uint32_t m = __ballot_sync(FULL, won);
  const uint32_t pos = w.tail + __popc(m & ((1u << w.lane) - 1u));
  w.tail += __popc(m);
  if (won) {
    w.trail[WIDX(w, pos, w.V, 2)] = l;
    if (SIZE >= 32u || w.tail - pos <= SIZE) ring[pos & (SIZE - 1u)] = l;
  }
  return pos;
}

// Make literal l of every lane with want set true (all lanes). The assignment is
// a bit set over literal codes, STRIDE words apart: bit l set = l is true. Of
// the lanes that claim one variable the first wins; returns true in a lane
// whose literal's negation was claimed by another lane of this call (seeing
// both bits, a lane agrees with the winner or the undo of the lane that saw
// one covers it); won is set where the lane's literal is new.
template <int STRIDE>
__device__ __forceinline__ bool claim_bits(Warp& w, bool want, uint32_t l, bool& won) {
  bool clash = false;
  won = false;
  if (want) {
    const uint32_t at = WIDX(w, l, 2u * w.V, 1);
    uint32_t* word = &w.asg[STRIDE * (at >> 5)];
    const uint32_t old = atomicOr(word, 1u << (at & 31u));
    const uint32_t t = (old >> (at & 31u)) & 1u, f = (old >> ((at & 31u) ^ 1u)) & 1u;
    won = !(t | f);
    clash = f && !t;
    if (clash) atomicAnd(word, ~(1u << (at & 31u)));
  }
  return clash;
}

// Assign l, unassigned, for a decision or an assumption (all lanes, uniform).
__device__ __forceinline__ void assign_one(Warp& w, uint32_t l) {
  bool won;
  claim_bits<1>(w, w.lane == 0, l, won);
  push_trail<RING>(w, w.ws->ring, won, l);
  __syncwarp();
}

// What one visited clause asks for: a literal to make true, or a conflict with
// the clause's falsified literals (or its reference) in c0..c2.
struct Found {
  bool want, confl;
  uint32_t lit, c0, c1, c2;
};

__device__ __noinline__ Found eval_long(const uint32_t* asg, const int32_t* lits, int64_t b,
                                        int64_t e, uint32_t local) {
  uint32_t open_lit = NONE;
  for (int64_t q = b; q < e; q++) {
    const uint32_t x = code_of(__ldg(&lits[q]));
    const uint32_t vx = lit_value(asg, x);
    if (vx == LV_T || (vx == LV_U && open_lit != NONE && x != open_lit))
      return Found{false, false, NONE, 0, 0, 0};
    if (vx == LV_U) open_lit = x;
  }
  return Found{open_lit != NONE, open_lit == NONE, open_lit, LONG_CLAUSE | local, NONE, NONE};
}

// One occurrence entry of the falsified literal f, without branches but for
// long clauses: bit a of the assignment says a is true, bit a ^ 1 that it is
// false; a binary entry's missing literal counts as false.
__device__ __forceinline__ Found eval_entry(const Warp& w, uint32_t f, uint64_t e) {
  const uint32_t a0 = (uint32_t)e, b0 = (uint32_t)(e >> 32);
  if (a0 & LONG_CLAUSE) {
    const uint32_t local = a0 & ~LONG_CLAUSE;
    const int64_t c = w.c0 + local;
    return eval_long(w.asg, w.lits, w.cb[c], w.cb[c + 1], local);
  }
  const bool tern = b0 != NONE;
  const uint32_t a = WIDX(w, a0, 2u * w.V, 3), b = tern ? WIDX(w, b0, 2u * w.V, 3) : a;
  const uint32_t xa = w.asg[a >> 5], xb = w.asg[b >> 5];
  const bool ta = (xa >> (a & 31u)) & 1u, fa = (xa >> ((a & 31u) ^ 1u)) & 1u;
  const bool tb = tern && ((xb >> (b & 31u)) & 1u);
  const bool fb = !tern || ((xb >> ((b & 31u) ^ 1u)) & 1u);
  const bool ua = !ta && !fa && fb, ub = !tb && !fb && fa;
  return Found{ua || ub, fa && fb, ua ? a : b, f, a, b0};
}

// How the lanes share a batch of nlit frontier literals: 8 lanes each, four at a
// time; in the DPLL search (NARROW false) a single literal has the whole warp and
// two have 16 lanes each. (DPLL on 256 bounds queries: 9.0 ms so, 10.0 with 8
// lanes always; clause learning on random 3-SAT 55.5 and 53.0, elsewhere equal.)
// Most lists hold 3 to 8 entries and most rounds 1 to 4 literals, so a round is
// usually one pass -- no scan over the list lengths, no search for the owner
// of an entry. With up to four literals (few) every lane reads its own
// literal and list bounds; with more, lane j reads those of literal j and
// each pass fetches its four with shuffles.
struct LaneMap {
  uint32_t lg;     // log2 of lanes per literal
  uint32_t sub;    // this lane's place among its literal's lanes
  uint32_t group;  // which of the pass's literals is this lane's
  uint32_t mine;   // the literal of the batch whose bounds this lane reads
  bool few;
};

template <bool NARROW>
__device__ __forceinline__ LaneMap lane_map(uint32_t lane, uint32_t nlit) {
  LaneMap m;
  m.lg = NARROW || nlit > 2 ? 3u : nlit == 1 ? 5u : 4u;
  m.sub = lane & ((1u << m.lg) - 1u);
  m.group = lane >> m.lg;
  m.few = nlit <= 4;
  m.mine = m.few ? m.group : lane;
  return m;
}

// The lane holds literal m.mine's falsified code f and list [beg, beg + cnt) (cnt 0
// past the last literal); visit(f, index, in) runs for every index of every
// list (all lanes, in = the lane has one) until it returns true.
template <class Visit>
__device__ __forceinline__ bool spread_lists(const LaneMap& m, uint32_t nlit, uint32_t f,
                                             uint32_t beg, uint32_t cnt, Visit&& visit) {
  for (uint32_t s = 0; s < nlit; s += 32u >> m.lg) {
    uint32_t jb = beg, jf = f, jc = cnt;
    if (!m.few) {
      const uint32_t j = s + m.group;
      jb = __shfl_sync(FULL, beg, j);
      jf = __shfl_sync(FULL, f, j);
      jc = __shfl_sync(FULL, cnt, j);
      if (j >= nlit) jc = 0;
    }
    bool more;
    uint32_t k = m.sub;
    do {
      const bool in = k < jc;
      const uint32_t at = jb + k;
      k += 1u << m.lg;
      more = __any_sync(FULL, k < jc);  // asked before it is needed
      if (visit(jf, at, in)) return true;
    } while (more);
  }
  return false;
}

// Whether this lane counts its list among the batch's.
__device__ __forceinline__ bool counts_list(const LaneMap& m) { return !m.few || m.sub == 0; }

// Remember the conflict of the first lane that has one (all lanes).
__device__ __forceinline__ void note_conflict(Warp& w, bool confl, uint32_t c0, uint32_t c1,
                                              uint32_t c2) {
  const uint32_t m = __ballot_sync(FULL, confl);
  if (!m) return;
  if (w.lane == __ffs(m) - 1) {
    w.ws->cl[0] = c0;
    w.ws->cl[1] = c1;
    w.ws->cl[2] = c2;
  }
  w.confl = 1;
  __syncwarp();
}

// Unit propagation to a fixpoint. Returns true on conflict (w.confl, ws->cl).
// Each round takes the trail literals assigned in the previous round (the
// frontier) and spreads their occurrence entries over the 32 lanes. A round is
// one chain of dependent latencies -- literal, list bounds, entry, assignment
// words, claim -- so the lanes evaluate without branching and claim together:
// one shared-memory atomic per claimed literal, positions from a ballot.
__device__ __forceinline__ bool bcp(Warp& w) {
  while (w.head < w.tail) {
    const uint32_t lo = w.head, hi = w.tail;
    w.head = hi;
    WCOUNT(w, props, hi - lo);
    for (uint32_t base = lo; base < hi; base += 32) {
      const uint32_t nlit = min(32u, hi - base);
      const LaneMap m = lane_map<false>(w.lane, nlit);
      uint32_t f = 0, beg = 0, cnt = 0;
      if (m.mine < nlit) {
        f = WIDX(w, frontier_lit<RING>(w, w.ws->ring, base + m.mine) ^ 1u, 2u * w.V, 4);  // became false
        beg = __ldg(&w.occ[f]);
        cnt = __ldg(&w.occ[f + 1]) - beg;
      }
      spread_lists(m, nlit, f, beg, cnt, [&](uint32_t jf, uint32_t at, bool in) {
        Found r{false, false, 0, 0, 0, 0};
        if (in) r = eval_entry(w, jf, __ldg(&w.ent[WIDX(w, at, w.ent_end, 5)]));
        if (__any_sync(FULL, r.want || r.confl)) {
          bool won;
          const bool clash = claim_bits<1>(w, r.want, r.lit, won);
          push_trail<RING>(w, w.ws->ring, won, r.lit);
          note_conflict(w, r.confl || clash, r.c0, r.c1, r.c2);
          __syncwarp();
        }
        return w.confl != 0;
      });
      if (counts_list(m)) WADD(w, visits, cnt);
      if (w.confl) return true;
    }
  }
  return false;
}

template <int MODE>
__device__ void bump(Warp& w) {
  // activity += inc for the variables of the falsified clause
  const uint32_t a = w.ws->cl[0], b = w.ws->cl[1], c = w.ws->cl[2];
  if (MODE == MODE_TRACE) {
    // every open traced level counts the falsified clause's variables
    const uint32_t levels = min(w.nd, (uint32_t)w.S->trace_depth);
    if ((uint32_t)w.lane < levels) {
      uint32_t* cnt = w.lvlcnt + (size_t)w.lane * w.S->vmax;
      if (a & LONG_CLAUSE) {
        const int64_t cl = w.c0 + (a & ~LONG_CLAUSE);
        for (int64_t q = w.cb[cl]; q < w.cb[cl + 1]; q++) cnt[code_of(w.lits[q]) >> 1]++;
      } else {
        if (a != NONE) cnt[a >> 1]++;
        if (b != NONE) cnt[b >> 1]++;
        if (c != NONE) cnt[c >> 1]++;
      }
    }
    __syncwarp();
  }
  bool big = false;
  if (a & LONG_CLAUSE) {
    if (w.lane == 0) {
      const int64_t cl = w.c0 + (a & ~LONG_CLAUSE);
      for (int64_t q = w.cb[cl]; q < w.cb[cl + 1]; q++) {
        uint32_t v = code_of(w.lits[q]) >> 1;
        w.act[v] += w.inc;
        big |= w.act[v] > 1e20f;
      }
    }
  } else {  // at most three literals of distinct variables: a lane each
    const uint32_t x = w.lane == 0 ? a : w.lane == 1 ? b : w.lane == 2 ? c : NONE;
    if (x != NONE) {
      const float v = w.act[x >> 1] + w.inc;
      w.act[x >> 1] = v;
      big = v > 1e20f;
    }
  }
  w.inc *= (1.0f / 0.95f);
  big = __any_sync(FULL, big) || w.inc > 1e20f;
  __syncwarp();
  if (big) {
    for (uint32_t v = w.lane; v < w.V; v += 32) w.act[v] *= 1e-20f;
    w.inc *= 1e-20f;
    __syncwarp();
  }
}

// ---- features of the residual formula (learned branching, traces) -------
//
// For variable v (0-based) and each polarity: how many clauses containing the
// literal are not yet satisfied with 2 / 3 open literals, its static
// occurrence count, plus activity, input-bit flags and search progress.
template <class Out>
__device__ void var_features(const Warp& w, uint32_t v, uint32_t ninputs, Out&& put) {
  uint32_t c2[2] = {0, 0}, c3[2] = {0, 0}, occn[2];
#pragma unroll
  for (int pol = 0; pol < 2; pol++) {
    const uint32_t lit = 2u * v + (uint32_t)pol;
    const uint32_t beg = __ldg(&w.occ[lit]), end = __ldg(&w.occ[lit + 1]);
    occn[pol] = end - beg;
    for (uint32_t e = beg; e < end; e++) {
      const uint64_t en = __ldg(&w.ent[e]);
      const uint32_t a = (uint32_t)en, b = (uint32_t)(en >> 32);
      if (a & LONG_CLAUSE) continue;
      const uint32_t va = lit_value(w.asg, a);
      if (va == LV_T || va == LV_X) continue;
      uint32_t open = 1 + (va == LV_U);
      if (b != NONE) {
        const uint32_t vb = lit_value(w.asg, b);
        if (vb == LV_T || vb == LV_X) continue;
        open += (vb == LV_U);
      }
      if (open == 2) c2[pol]++;
      else if (open == 3) c3[pol]++;
    }
  }
  const float tail = (float)w.tail;
  put(0, c2[0] * 0.25f);
  put(1, c3[0] * 0.25f);
  put(2, c2[1] * 0.25f);
  put(3, c3[1] * 0.25f);
  put(4, occn[0] * 0.125f);
  put(5, occn[1] * 0.125f);
  put(6, fminf(w.act[v] / w.inc, 16.0f) * 0.0625f);
  put(7, v < ninputs ? 1.0f : 0.0f);
  put(8, v < ninputs ? (float)v / (float)ninputs : 0.0f);
  put(9, (float)w.nd * (1.0f / 32.0f));
  put(10, w.V ? tail / (float)w.V : 0.0f);
  put(11, (c2[0] + c2[1]) * 0.125f);
  put(12, (c3[0] + c3[1]) * 0.125f);
  put(13, log2f(1.0f + occn[0] + occn[1]) * (1.0f / 6.0f));
  put(14, ((float)(c2[0] + c3[0]) - (float)(c2[1] + c3[1])) * 0.125f);
  put(15, 1.0f);
}

__device__ __forceinline__ bool var_unassigned(const uint32_t* asg, uint32_t v) {
  return ((asg[v >> 4] >> ((v & 15u) * 2u)) & 3u) == 0u;
}

// Trace: open a node for the decision about to be made at level `depth`.
__device__ void trace_open(Warp& w, uint32_t depth) {
  const Solve& S = *w.S;
  const TraceDev& T = S.tr;
  uint32_t nun = 0;
  for (uint32_t base = 0; base < w.V; base += 32) {
    const uint32_t v = base + w.lane;
    nun += __popc(__ballot_sync(FULL, v < w.V && var_unassigned(w.asg, v)));
  }
  long long node = -1, row0 = 0;
  if (w.lane == 0) {
    node = (long long)atomicAdd(&T.cursor[0], 1ull);
    row0 = (long long)atomicAdd(&T.cursor[1], (unsigned long long)nun);
    if (node >= T.max_nodes || row0 + nun > T.max_rows) node = -1;
  }
  node = __shfl_sync(FULL, node, 0);
  row0 = __shfl_sync(FULL, row0, 0);
  if (w.lane == 0) w.lvl_node[depth] = node;
  if (node < 0) return;
  if (w.lane == 0) {
    T.node_inst[node] = w.inst;
    T.node_depth[node] = (int32_t)depth;
    T.node_row[node] = row0;
    T.node_nrows[node] = (int32_t)nun;
    T.node_closed[node] = 0;
  }
  const uint32_t ni = S.inst_num_inputs ? (uint32_t)S.inst_num_inputs[w.inst] : 0u;
  long long r = row0;
  for (uint32_t base = 0; base < w.V; base += 32) {
    const uint32_t v = base + w.lane;
    const bool un = v < w.V && var_unassigned(w.asg, v);
    const uint32_t m = __ballot_sync(FULL, un);
    if (un) {
      const long long row = r + __popc(m & ((1u << w.lane) - 1u));
      __nv_bfloat16* xr = T.x + row * learn::NFEAT;
      var_features(w, v, ni, [&](int k, float x) { xr[k] = __float2bfloat16(x); });
      T.var[row] = (int32_t)v;
      T.target[row] = 0.0f;
    }
    r += __popc(m);
  }
  __syncwarp();
}

// Trace: the subtree of level l is finished; write its conflict counts.
__device__ void trace_close(Warp& w, uint32_t l) {
  const TraceDev& T = w.S->tr;
  const long long node = w.lvl_node[l];
  uint32_t* cnt = w.lvlcnt + (size_t)l * w.S->vmax;
  if (node >= 0) {
    const long long row0 = T.node_row[node];
    const int32_t nr = T.node_nrows[node];
    for (int k = w.lane; k < nr; k += 32) T.target[row0 + k] = (float)cnt[T.var[row0 + k]];
    __syncwarp();
    if (w.lane == 0) T.node_closed[node] = 1;
  }
  for (uint32_t v = w.lane; v < w.V; v += 32) cnt[v] = 0u;
  __syncwarp();
  if (w.lane == 0) w.lvl_node[l] = -1;
  __syncwarp();
}

// Learned decision: the unassigned variable with the highest MLP score
// (ties: higher activity, then lower id). NONE if all are assigned.
__device__ uint32_t pick_learned(Warp& w) {
  const Solve& S = *w.S;
  const uint32_t ni = S.inst_num_inputs ? (uint32_t)S.inst_num_inputs[w.inst] : 0u;
  float best_s = -INFINITY, best_a = -1.0f;
  uint32_t best_v = NONE;
  for (uint32_t base = 0; base < w.V; base += 32) {
    const uint32_t v = base + w.lane;
    const bool un = v < w.V && var_unassigned(w.asg, v);
    if (!__any_sync(FULL, un)) continue;
    __nv_bfloat16* xr = w.xtile + w.lane * learn::NFEAT;
    if (un) {
      var_features(w, v, ni, [&](int k, float x) { xr[k] = __float2bfloat16(x); });
    } else {
#pragma unroll
      for (int k = 0; k < 16; k++) xr[k] = __float2bfloat16(0.0f);
    }
    __syncwarp();
    float a_lo, a_hi, b_lo, b_hi;
    learn::mlp_tile_scores(S.mlp, w.xtile, w.lane, a_lo, a_hi);
    learn::mlp_tile_scores(S.mlp, w.xtile + 16 * learn::NFEAT, w.lane, b_lo, b_hi);
    // lane 4g holds rows g, g+8 (first tile) and 16+g, 24+g (second tile)
    const int src = 4 * (w.lane & 7);
    const float r0 = __shfl_sync(FULL, a_lo, src), r1 = __shfl_sync(FULL, a_hi, src);
    const float r2 = __shfl_sync(FULL, b_lo, src), r3 = __shfl_sync(FULL, b_hi, src);
    const float sc = w.lane < 8 ? r0 : (w.lane < 16 ? r1 : (w.lane < 24 ? r2 : r3));
    if (un) {
      const float a = w.act[v];
      if (sc > best_s || (sc == best_s && (a > best_a || (a == best_a && v < best_v)))) {
        best_s = sc;
        best_a = a;
        best_v = v;
      }
    }
    __syncwarp();
  }
  for (int d = 16; d > 0; d >>= 1) {
    const float os = __shfl_xor_sync(FULL, best_s, d), oa = __shfl_xor_sync(FULL, best_a, d);
    const uint32_t ov = __shfl_xor_sync(FULL, best_v, d);
    if (os > best_s || (os == best_s && (oa > best_a || (oa == best_a && ov < best_v)))) {
      best_s = os;
      best_a = oa;
      best_v = ov;
    }
  }
  return best_v;
}

// Chronological backtrack after a conflict. Returns false when no decision
// above the assumptions is left to flip (the subtree is refuted).
template <int MODE>
__device__ bool backtrack(Warp& w) {
  // the deepest decision not yet flipped, 32 at a time
  uint32_t nd = w.nd, pos = 0;
  for (;; nd -= 32) {
    if (nd <= w.nd_fixed) return false;
    const uint32_t at = nd - 1u - (uint32_t)w.lane;
    const bool in = (uint32_t)w.lane < nd - w.nd_fixed;
    const uint32_t d = in ? w.dstack[at] : FLIP;
    const uint32_t open = __ballot_sync(FULL, !(d & FLIP));
    if (open) {
      const int j = __ffs(open) - 1;
      nd -= (uint32_t)j;
      pos = __shfl_sync(FULL, d, j);
      break;
    }
    if (nd - w.nd_fixed <= 32) return false;
  }
  if (MODE == MODE_TRACE) {
    // levels nd .. w.nd-1 are popped: their subtrees are complete
    const uint32_t hi_l = min(w.nd, (uint32_t)w.S->trace_depth);
    for (uint32_t l = nd; l < hi_l; l++) trace_close(w, l);
  }
  const uint32_t tail = w.tail;
  const uint32_t d = w.trail[pos];
  WCOUNT(w, undone, tail - pos);
  for (uint32_t t = pos + w.lane; t < tail; t += 32) {
    uint32_t v = w.trail[t] >> 1;
    atomicAnd(&w.asg[v >> 4], ~(3u << ((v & 15u) * 2u)));
  }
  __syncwarp();
  if (w.lane == 0) w.dstack[nd - 1] = pos | FLIP;
  w.nd = nd;
  w.head = w.tail = pos;
  w.confl = 0;
  assign_one(w, d ^ 1u);
  return true;
}

// The best (activity, then lowest id) of the lanes' candidates.
__device__ __forceinline__ uint32_t best_of_warp(float a, uint32_t v) {
  // activities are not negative, so their bits order as the numbers do; a
  // lane without a candidate has a = -1
  const uint32_t key = v == NONE ? 0u : __float_as_uint(a) + 1u;
  const uint32_t top = __reduce_max_sync(FULL, key);
  return __reduce_min_sync(FULL, key == top ? v : NONE);
}

// Highest-activity unassigned variable (ties: lowest id); NONE if all are
// assigned. STRIDE: words between the assignment words of 16 variables (2 with
// clause learning). The activities of four neighbouring variables are one load
// (a slot's activities begin on a 64-byte boundary), all those of a lane's
// assignment word are on their way together, and a word without an unassigned
// variable loads nothing.
template <int STRIDE>
__device__ __forceinline__ uint32_t pick_max(const Warp& w) {
  float best_a = -1.0f;
  uint32_t best_v = NONE;
  const uint32_t nwords = (w.V + 15u) >> 4;
  for (uint32_t k = w.lane; k < nwords; k += 32) {
    const uint32_t word = w.asg[STRIDE * k];
    uint32_t un = ~(word | (word >> 1)) & 0x55555555u;  // 00 pairs
    const uint32_t lim = w.V - 16u * k;
    if (lim < 16u) un &= (1u << (2u * lim)) - 1u;
    if (!un) continue;
    const float4* a4 = reinterpret_cast<const float4*>(w.act + 16 * k);
    float4 a[4];
#pragma unroll
    for (uint32_t q = 0; q < 4; q++) a[q] = a4[q];
#pragma unroll
    for (uint32_t q = 0; q < 16; q++) {
      const float x = q % 4 == 0 ? a[q / 4].x : q % 4 == 1 ? a[q / 4].y : q % 4 == 2 ? a[q / 4].z
                                                                                  : a[q / 4].w;
      if (((un >> (2 * q)) & 1u) && x > best_a) {  // ids ascend: ties keep the lower one
        best_a = x;
        best_v = 16 * k + q;
      }
    }
  }
  return best_of_warp(best_a, best_v);
}

__device__ uint32_t pick(Warp& w) { return pick_max<1>(w); }

// When the search began. Warps of one launch start at different times, so the
// first of them sets it (start_clock) and every read goes to memory.
__device__ __forceinline__ void start_clock(Ctrl* c) {
  atomicCAS(reinterpret_cast<unsigned long long*>(&c->t0), 0ull,
            (unsigned long long)globaltimer());
}

__device__ __forceinline__ uint64_t search_ns(const Solve& S) {
  return elapsed_ns(*(volatile uint64_t*)&S.ctrl->t0, globaltimer());
}

__device__ __forceinline__ void set_status(const Solve& S, int32_t st) {
  atomicCAS(&S.ctrl->status, 0, st);
}

// Publish x to other SMs after every write that this thread has made or seen
// (the warp's, after a __syncwarp). A release store waits for those writes and
// nothing more; a __threadfence would also empty this SM's L1, which the
// other 15 or more searching warps of the SM live in.
__device__ __forceinline__ void store_release(uint32_t* p, uint32_t x) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(x) : "memory");
}

// ---- job ring (bounded MPMC queue, Vyukov) --------------------------------

// extra(cell) runs (all lanes) after the cell is filled and before it is
// published: the clause-learning search attaches learned clauses there.
template <class Extra>
__device__ bool ring_push(const Solve& S, const Warp& w, int inst, uint32_t plen,
                          const uint32_t* prefix_src_trail, const uint32_t* dpos,
                          uint32_t flip_index, Extra&& extra) {
  // called by all lanes; lane 0 reserves
  Ctrl* C = S.ctrl;
  uint32_t slot = NONE;
  if (w.lane == 0) {
    for (int it = 0; it < 64; it++) {
      uint32_t pos = *(volatile uint32_t*)&C->q_tail;
      Job* cell = &S.ring[pos & (S.ring_cap - 1)];
      uint32_t seq = *(volatile uint32_t*)&cell->seq;
      int32_t dif = (int32_t)(seq - pos);
      if (dif == 0) {
        if (atomicCAS(&C->q_tail, pos, pos + 1) == pos) { slot = pos; break; }
      } else if (dif < 0) {
        break;  // full
      }
    }
  }
  slot = __shfl_sync(FULL, slot, 0);
  if (slot == NONE) return false;
  Job* cell = &S.ring[slot & (S.ring_cap - 1)];
  // prefix = decision literals 0..flip_index-1 as assigned now, then the
  // negation of decision flip_index
  for (uint32_t k = w.lane; k < plen; k += 32) {
    uint32_t lit = prefix_src_trail[dpos[k] & ~FLIP];
    if (k == flip_index) lit ^= 1u;
    cell->lit[k] = lit;
  }
  // the thief continues with the donor's activity ordering
  float* snap = S.job_act + (size_t)(slot & (S.ring_cap - 1)) * S.vmax;
  for (uint32_t v = w.lane; v < w.V; v += 32) snap[v] = w.act[v];
  if (w.lane == 0) {
    cell->inst = inst;
    cell->len = (int32_t)plen;
    cell->inc = w.inc;
  }
  extra(slot & (S.ring_cap - 1));
  __syncwarp();
  if (w.lane == 0) store_release(&cell->seq, slot + 1);
  __syncwarp();
  return true;
}

__device__ bool ring_push(const Solve& S, const Warp& w, int inst, uint32_t plen,
                          const uint32_t* prefix_src_trail, const uint32_t* dpos,
                          uint32_t flip_index) {
  return ring_push(S, w, inst, plen, prefix_src_trail, dpos, flip_index, [](uint32_t) {});
}

// Try to take a job; returns slot or NONE. Only a warp that takes one fences: a
// fence empties the SM's L1, and idle warps come by every 2 us (fencing on each
// visit left the busy warps of a mostly idle GPU without an L1).
__device__ uint32_t ring_pop(const Solve& S, int lane) {
  Ctrl* C = S.ctrl;
  uint32_t slot = NONE;
  if (lane == 0) {
    for (int it = 0; it < 64; it++) {
      uint32_t pos = *(volatile uint32_t*)&C->q_head;
      Job* cell = &S.ring[pos & (S.ring_cap - 1)];
      uint32_t seq = *(volatile uint32_t*)&cell->seq;
      int32_t dif = (int32_t)(seq - (pos + 1));
      if (dif == 0) {
        if (atomicCAS(&C->q_head, pos, pos + 1) == pos) {
          slot = pos;
          __threadfence();  // acquire: the cell's contents after its sequence number
          break;
        }
      } else if (dif < 0) {
        break;  // empty
      }
    }
  }
  slot = __shfl_sync(FULL, slot, 0);
  __syncwarp();
  return slot;
}

__device__ void ring_release(const Solve& S, uint32_t slot, int lane) {
  __syncwarp();
  if (lane == 0) store_release(&S.ring[slot & (S.ring_cap - 1)].seq, slot + S.ring_cap);
  __syncwarp();
}

// A unit's job finished with result r (SCUBA_SAT / SCUBA_UNSAT /
// SCUBA_UNKNOWN). The last open job of a unit (an instance, or an instance
// under assumptions) writes its verdict. What a job found goes into the word that
// counts the open jobs: atomics of one thread on one word take effect in order,
// so the last job sees what every other one found before it left (on two words
// nothing but a fence would order them).
__device__ void finish_job(const Solve& S, Warp& w, int unit, int r) {
  flush_counters(S, w, unit);
  if (w.lane == 0) {
    if (r == SCUBA_SAT) {
      S.verdict[unit] = SCUBA_SAT;
      atomicOr(&S.done[unit], 1u);  // the unit's other jobs may stop
      atomicOr(&S.pending[unit], PEND_SAT);
    } else if (r == SCUBA_UNKNOWN) {
      atomicOr(&S.pending[unit], PEND_GAVE_UP);
    }
    const uint32_t p = atomicSub(&S.pending[unit], 1u);
    if ((p & PEND_JOBS) == 1u) {  // the last one
      if (!(p & PEND_SAT)) S.verdict[unit] = p & PEND_GAVE_UP ? SCUBA_UNKNOWN : SCUBA_UNSAT;
      atomicSub(&S.ctrl->inst_left, 1u);
      if (S.finish_ns) S.finish_ns[unit] = (int64_t)search_ns(S);
    }
    if (S.prof) {
      atomicAdd(&S.prof[1], 1ull);  // jobs run
      for (int k = 0; w.cyc && k < 8; k++)
        if (w.cyc[k]) atomicAdd(&S.prof[8 + k], w.cyc[k]);
    }
  }
  __syncwarp();
}

// Solve one subtree (inst + assumptions). Returns SAT / UNSAT / UNKNOWN.
// A taken job (a shared subtree) in slot-private memory: the ring cell is
// released as soon as it has been copied.
struct TakenJob {
  const uint32_t* lit;  // assumptions, in order
  int32_t len;
  float inc;            // activities were copied into the warp's act[] already
  const uint32_t* cls;  // clause learning: the donor's clauses (slot copy), or NULL
};

template <int MODE>
__device__ int run_job_body(const Solve& S, Warp& w, int unit, int inst, const TakenJob* job,
                            int& abort_code);

// A unit's assumption literals as the job of a fresh search (all lanes):
// converted into the slot's prefix buffer, activities zeroed. Returns true
// if a literal is out of range or there are more than MAX_PREFIX of them.
__device__ __noinline__ bool unit_job(const Solve& S, int unit, int inst, int64_t slot, int lane,
                                      float* act, TakenJob* out) {
  const int64_t ab = S.unit_asm_begin[unit], ae = S.unit_asm_begin[unit + 1];
  const int32_t V = min(S.nv[inst], S.vmax);
  bool bad = ae - ab > MAX_PREFIX;
  uint32_t* pre = S.prefix + slot * MAX_PREFIX;
  for (int64_t q = ab + lane; !bad && q < ae; q += 32) {
    const int32_t l = S.unit_asm[q];
    if (l == 0 || l > V || l < -V) bad = true;
    else pre[q - ab] = code_of(l);
  }
  bad = __any_sync(FULL, bad);
  for (int v = lane; v < V; v += 32) act[v] = 0.0f;  // fresh activities
  out->lit = pre;
  out->len = (int32_t)(ae - ab < MAX_PREFIX ? ae - ab : MAX_PREFIX);
  out->inc = 1.0f;
  out->cls = nullptr;
  __syncwarp();
  return bad;
}

// Runs one job; in trace mode every level still open at the end is closed.
template <int MODE>
__device__ int run_job(const Solve& S, Warp& w, int unit, int inst, const TakenJob* job,
                       int& abort_code) {
  const int r = run_job_body<MODE>(S, w, unit, inst, job, abort_code);
  if (MODE == MODE_TRACE) {
    const uint32_t hi_l = min(w.nd, (uint32_t)S.trace_depth);
    for (uint32_t l = 0; l < hi_l; l++) trace_close(w, l);
  }
  return r;
}

template <int MODE>
__device__ int run_job_body(const Solve& S, Warp& w, int unit, int inst, const TakenJob* job,
                            int& abort_code) {
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
  w.inc = 1.0f;
  const uint32_t nwords = (w.V + 15u) >> 4;
  for (uint32_t k = w.lane; k < nwords; k += 32) w.asg[k] = 0u;
  if (job) {
    w.inc = job->inc;
  } else {
    for (uint32_t v = w.lane; v < w.V; v += 32) w.act[v] = 0.0f;
  }
  w.tail = 0;
  w.confl = 0;
  __syncwarp();
  if (S.flags[inst] & F_EMPTY) return SCUBA_UNSAT;
  // level 0: unit clauses; the job's assumptions follow as fixed decisions, one
  // after each propagation of the main loop
  const uint32_t nu = S.nunits[inst];
  const uint32_t* un = S.units + w.c0;
  for (uint32_t k0 = 0; k0 < nu; k0 += 32) {
    const uint32_t l = k0 + w.lane < nu ? un[k0 + w.lane] : NONE;
    bool won;
    const bool clash = claim_bits<1>(w, l != NONE, l, won);
    push_trail<RING>(w, w.ws->ring, won, l);
    __syncwarp();
    // a unit clause against an earlier one's value, or another lane's
    const bool bad = l != NONE && !won && lit_value(w.asg, l) != LV_T;
    if (__any_sync(FULL, clash || bad)) return SCUBA_UNSAT;
  }
  int next_asm = 0;
  const int n_asm = job ? job->len : 0;
  uint32_t iter = 0;
  const uint32_t flush_mask = flush_steps(__ldg(&w.occ[2u * w.V]), 0, w.V) - 1u;
  for (;;) {
    if ((++iter & flush_mask) == 0u) {
      flush_counters(S, w, unit);
      int stop = 0;
      if (w.lane == 0) {
        if (S.abort_flag && *S.abort_flag) stop = 1;
        else if (search_ns(S) > S.time_ns) stop = 2;
        else if (*(volatile uint32_t*)&S.done[unit] & 1u) stop = 3;  // solved elsewhere
#ifdef SCUBA_CHECKED
        else if (batch_failed(S.ctrl)) stop = 4;  // a bounds check failed: stop
#endif
      }
      stop = __shfl_sync(FULL, stop, 0);
      if (stop == 4) { abort_code = SCUBA_ERR_INTERNAL; return SCUBA_UNKNOWN; }
      if (stop == 1) { abort_code = SCUBA_ERR_ABORTED; return SCUBA_UNKNOWN; }
      if (stop == 2) { abort_code = SCUBA_ERR_TIMEOUT; return SCUBA_UNKNOWN; }
      if (stop == 3) return SCUBA_UNSAT;  // the instance is SAT already; this subtree is moot
    }
    if (bcp(w)) {
      if (next_asm < n_asm) return SCUBA_UNSAT;  // the assumptions alone
      WCOUNT(w, conflicts, 1);
      bump<MODE>(w);
      if (!backtrack<MODE>(w)) return SCUBA_UNSAT;
      continue;
    }
    if (next_asm < n_asm) {
      const uint32_t l = job->lit[next_asm++];
      const uint32_t val = lit_value(w.asg, l);
      if (val == LV_F) return SCUBA_UNSAT;
      if (val == LV_U) {
        if (w.lane == 0) w.dstack[WIDX(w, w.nd, (uint32_t)w.S->vmax, 6)] = w.tail | FLIP;
        w.nd++;
        w.nd_fixed = w.nd;
        assign_one(w, l);
      }
      continue;
    }
    WCOUNT(w, act_reads, w.V - w.tail);
    uint32_t v;
    if (MODE == MODE_LEARNED && w.nd < (uint32_t)S.learned_depth) v = pick_learned(w);
    else v = pick(w);
    if (MODE == MODE_TRACE && v != NONE && w.nd < (uint32_t)S.trace_depth) trace_open(w, w.nd);
    if (v == NONE) {
      // the first subtree of the instance to reach a model writes it
      uint32_t won = 0;
      if (w.lane == 0) won = !(atomicOr(&S.done[unit], 8u) & 8u);
      won = __shfl_sync(FULL, won, 0);
      if (won && S.model)
        for (uint32_t x = w.lane; x < w.V; x += 32) {
          uint32_t bits = (w.asg[x >> 4] >> ((x & 15u) * 2u)) & 3u;
          S.model[(S.unit_vb ? S.unit_vb[unit] : S.vb[inst]) + x] = bits == 1u ? 1 : 0;
        }
      __syncwarp();
      return SCUBA_SAT;
    }
    // budget: decisions of the instance across all of its subtrees
    if (S.budget > 0 && (w.decisions & 255) == 0) {
      unsigned long long tot = 0;
      if (w.lane == 0) tot = atomicAdd(&S.inst_dec[unit], 256ull);
      tot = __shfl_sync(FULL, tot, 0);
      if ((int64_t)tot >= S.budget) return SCUBA_UNKNOWN;
    }
    // share the untried branch of the shallowest open decision
    if (S.split && w.decisions >= S.split_min && (w.decisions % S.split_interval) == 0 &&
        w.nd > w.nd_fixed) {
      uint32_t idle = 0;
      if (w.lane == 0) idle = *(volatile uint32_t*)&S.ctrl->idle;
      idle = __shfl_sync(FULL, idle, 0);
      if (idle > 0) {
        uint32_t k = w.nd_fixed;
        if (w.lane == 0)
          while (k < w.nd && (w.dstack[k] & FLIP)) k++;
        k = __shfl_sync(FULL, k, 0);
        if (k < w.nd && k + 1 <= (uint32_t)MAX_PREFIX) {
          if (w.lane == 0) atomicAdd(&S.pending[unit], 1u);
          __syncwarp();
          if (ring_push(S, w, unit, k + 1, w.trail, w.dstack, k)) {
            if (w.lane == 0) {
              w.dstack[k] |= FLIP;
              atomicAdd(&S.ctrl->jobs_split, 1u);
              if (S.prof) {
                atomicAdd(&S.prof[0], 1ull);                       // jobs shared
                atomicAdd(&S.prof[2], (unsigned long long)(k + 1)); // prefix literals
                atomicAdd(&S.prof[3], (unsigned long long)(w.nd - k)); // depth left
              }
            }
          } else if (w.lane == 0) {
            atomicSub(&S.pending[unit], 1u);
            if (S.prof) atomicAdd(&S.prof[4], 1ull);  // ring full
          }
          __syncwarp();
        }
      }
    }
    w.decisions++;
    WCOUNT(w, decisions, 1);
    if (w.lane == 0) w.dstack[WIDX(w, w.nd, (uint32_t)w.S->vmax, 6)] = w.tail;
    w.nd++;
    assign_one(w, 2u * v + 1u);  // false first
  }
}

#include "cdcl.cuh"

// Blocks of 8 warps that stay resident on an SM, which sets the registers a
// thread gets. Plain search: 3 (80 registers, against 5 blocks of 48 that spilled
// 116 bytes). More warps do not pay: a subtree given away repeats part of its
// donor's work, so idle warps multiply the decisions. With 64 decisions before
// the first share, 4,096 partition queries of 16 bits take a median of 0.74 s on 3
// blocks, 0.87 on 2 (means over 32 solves 0.98 and 1.23: one solve in five meets an
// unlucky split on either), and took 1.59 on 5 (512 of 10 bits 15.4 ms on 3, 12.6 on
// 2 and 24.5 on 5), and
// 8,192 random 3-SAT of 250 variables with a budget, where no warp is idle, 85 ms
// on 3 against 92 on 2.
// The learned variant takes up to 3 as well (80 registers, no spills; 2 blocks of 6
// warps for small batches, see scuba_solve_units), trace recording, which shares
// nothing, 5. Clause learning takes 2 blocks of 6 warps, three warps for
// each quarter of the SM, which leaves a thread 168 registers (162 used, no spills); 16
// warps (128 registers, 206 bytes spilled) are the better choice only where the
// search keeps every warp at work of its own for long: 511 random 3-SAT instances
// of 150 variables take 45.0 ms against 41.7, 256 of them 27.5 against 27.0, but 511
// of 100 variables 8.0 against 9.0, 24 to 2,048 bounds queries of 8 bits 8 to 13 % less,
// partition queries of 10 bits 6 to 11 % less.
#ifndef SCUBA_PLAIN_MINBLOCKS
#define SCUBA_PLAIN_MINBLOCKS 3
#endif
#ifndef SCUBA_LEARNED_MINBLOCKS
#define SCUBA_LEARNED_MINBLOCKS 3
#endif
#ifndef SCUBA_CDCL_MINBLOCKS
#define SCUBA_CDCL_MINBLOCKS 2
#endif
constexpr int CDCL_WARPS = 6;
template <int MODE>
__global__ void __launch_bounds__(MODE == MODE_CDCL ? 32 * CDCL_WARPS : 256,
                                  MODE == MODE_LEARNED ? SCUBA_LEARNED_MINBLOCKS
                                  : MODE == MODE_CDCL || MODE == MODE_CDCL8 ? SCUBA_CDCL_MINBLOCKS
                                  : MODE == MODE_PLAIN ? SCUBA_PLAIN_MINBLOCKS
                                  : MODE == MODE_CDCL1 ? 1
                                                       : 5)
    k_solve(const __grid_constant__ Solve S) {
  extern __shared__ uint32_t smem[];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const int wpb = blockDim.x >> 5;
  const int64_t slot = (int64_t)blockIdx.x * wpb + wib;
  WarpShared* wsh = reinterpret_cast<WarpShared*>(smem);
  Warp w;
  w.S = &S;
  w.ws = &wsh[wib];
  w.asg = smem + (sizeof(WarpShared) / 4) * wpb + (size_t)S.assign_words * wib;
  w.trail = S.trail_smem
                ? smem + (sizeof(WarpShared) / 4) * wpb + (size_t)S.assign_words * wpb +
                      (size_t)S.vmax * wib
                : S.trail + slot * S.vmax;
  w.dstack = S.dstack + slot * S.vmax;
  w.act = S.act + slot * act_stride(S.vmax);
  w.cb = S.cb;
  w.lits = S.lits;
  w.lane = lane;
  w.lvlcnt = nullptr;
  w.lvl_node = nullptr;
  w.xtile = nullptr;
  w.cyc = nullptr;
  if (MODE == MODE_TRACE) {
    w.lvlcnt = S.lvlcnt + (size_t)slot * learn::MAX_TRACE_DEPTH * S.vmax;
    w.lvl_node = S.lvl_node + (size_t)slot * learn::MAX_TRACE_DEPTH;
  }
  if (MODE == MODE_LEARNED) {
    // feature tile after the per-warp assignment (and trail) areas
    unsigned char* tiles = reinterpret_cast<unsigned char*>(
        smem + (sizeof(WarpShared) / 4) * wpb + (size_t)S.assign_words * wpb +
        (S.trail_smem ? (size_t)S.vmax * wpb : 0));
    w.xtile = reinterpret_cast<__nv_bfloat16*>(tiles) + (size_t)wib * 32 * learn::NFEAT;
  }
  unsigned char* area = nullptr;
  if (is_cdcl(MODE)) {
    // the warp's own area after the per-warp assignment (and trail) areas,
    // 16-byte aligned
    const size_t off = ((sizeof(WarpShared) / 4) * wpb + (size_t)S.assign_words * wpb +
                        (S.trail_smem ? (size_t)S.vmax * wpb : 0)) * 4;
    area = reinterpret_cast<unsigned char*>(smem) + ((off + 15) & ~(size_t)15) +
           (size_t)wib * S.cd_smem_warp;
    w.cyc = reinterpret_cast<unsigned long long*>(area);
    if (S.cd_smem & CD_SMEM_ACT) w.act = cd_area_act(area);
  }
  // the warp's lanes agree (other warps set the status while this one starts)
  if (__any_sync(FULL, batch_failed(S.ctrl))) return;
  if (lane == 0) start_clock(S.ctrl);
  bool counted_idle = false;
  for (;;) {
    // 1) a shared subtree, 2) a fresh unit (an instance, possibly under
    // assumptions), 3) wait for shared work
    int inst = -1, unit = -1;
    bool bad_unit = false;
    uint32_t slot_j = ring_pop(S, lane);
    TakenJob taken;
    const TakenJob* job = nullptr;
    if (slot_j != NONE) {
      // copy the cell out (prefix, activity snapshot) and release it at once
      const Job* cell = &S.ring[slot_j & (S.ring_cap - 1)];
      unit = cell->inst;
      inst = S.unit_inst ? S.unit_inst[unit] : unit;
      const int32_t len = cell->len;
      uint32_t* pre = S.prefix + slot * MAX_PREFIX;
      for (int k = lane; k < len; k += 32) pre[k] = cell->lit[k];
      const float* snap = S.job_act + (size_t)(slot_j & (S.ring_cap - 1)) * S.vmax;
      const int32_t V = min(S.nv[inst], S.vmax);
      for (int v = lane; v < V; v += 32) w.act[v] = snap[v];
      taken.lit = pre;
      taken.len = len;
      taken.inc = cell->inc;
      taken.cls = nullptr;
      if (is_cdcl(MODE)) {  // the donor's learned clauses, copied out too
        const uint32_t* src = S.job_cls + (size_t)(slot_j & (S.ring_cap - 1)) * JOB_CLS_WORDS;
        uint32_t* dst = S.cls_copy + slot * JOB_CLS_WORDS;
        const uint32_t words = min(src[1], JOB_CLS_WORDS);
        for (uint32_t k = lane; k < words; k += 32) dst[k] = src[k];
        taken.cls = dst;
      }
      __syncwarp();
      ring_release(S, slot_j, lane);
      job = &taken;
    } else {
      // look before taking a number: idle warps come by every 2 us, and an
      // atomic from each of them would hold up the working warps' (and wrap)
      uint32_t k = 0;
      if (lane == 0) {
        k = *(volatile uint32_t*)&S.ctrl->next_inst;
        if (k < (uint32_t)S.n_units) k = atomicAdd(&S.ctrl->next_inst, 1u);
      }
      k = __shfl_sync(FULL, k, 0);
      if (k < (uint32_t)S.n_units) {
        unit = S.order ? S.order[k] : (int)k;
        inst = S.unit_inst ? S.unit_inst[unit] : unit;
        if (inst < 0 || inst >= S.n) {
          bad_unit = true;
          inst = 0;
        } else if (S.unit_asm_begin &&
                   S.unit_asm_begin[unit + 1] > S.unit_asm_begin[unit]) {
          bad_unit = unit_job(S, unit, inst, slot, lane, w.act, &taken);
          job = &taken;
        }
      } else {
        if (!counted_idle) {
          if (lane == 0) atomicAdd(&S.ctrl->idle, 1u);
          counted_idle = true;
        }
        int stop = 0;
        if (lane == 0) {
          if (*(volatile uint32_t*)&S.ctrl->inst_left == 0u) stop = 1;
          else if (*(volatile int32_t*)&S.ctrl->status != 0) stop = 1;
          else if (S.abort_flag && *S.abort_flag) { stop = 1; set_status(S, SCUBA_ERR_ABORTED); }
          else if (search_ns(S) > S.time_ns) { stop = 1; set_status(S, SCUBA_ERR_TIMEOUT); }
          else {
            if (S.prof) atomicAdd(&S.prof[5], 1ull);  // idle polls
            __nanosleep(2000);
          }
        }
        stop = __shfl_sync(FULL, stop, 0);
        if (stop) break;
        continue;
      }
    }
    if (counted_idle) {
      if (lane == 0) atomicSub(&S.ctrl->idle, 1u);
      counted_idle = false;
    }
    int abort_code = 0;
    int r;
    w.decisions = 0;
    if (lane == 0) {
      w.ws->decisions = w.ws->conflicts = w.ws->props = 0;
      w.ws->visits = w.ws->act_reads = w.ws->undone = 0;
      for (int k = 0; w.cyc && k < 8; k++) w.cyc[k] = 0;
    }
    __syncwarp();
    uint32_t moot = 0;
    if (lane == 0) moot = *(volatile uint32_t*)&S.done[unit] & 1u;
    moot = __shfl_sync(FULL, moot, 0);
    if (bad_unit) {  // an instance index or assumption literal out of range
      r = SCUBA_UNKNOWN;
      if (lane == 0) set_status(S, SCUBA_ERR_MALFORMED);
    } else if (S.flags[inst] & F_BAD) {
      r = SCUBA_UNKNOWN;
      if (lane == 0) set_status(S, SCUBA_ERR_MALFORMED);
    } else if (S.nv[inst] > S.vmax) {
      r = SCUBA_UNKNOWN;
      if (lane == 0) set_status(S, SCUBA_ERR_TOO_LARGE);
    } else if (moot) {
      r = SCUBA_UNSAT;  // moot: another subtree already found a model
    } else if constexpr (is_cdcl(MODE)) {
      r = run_cdcl(S, w, slot, unit, inst, job, area, abort_code);
    } else {
      r = run_job<MODE>(S, w, unit, inst, job, abort_code);
    }
    finish_job(S, w, unit, r);
    if (abort_code) {
      if (lane == 0) set_status(S, abort_code);
      break;
    }
  }
  if (counted_idle && lane == 0) atomicSub(&S.ctrl->idle, 1u);
}

// Unit-propagation closure of each instance under its unit clauses and the
// caller's assumption literals, one block per instance. values[vb[i] + v] = 0
// open, 1 true, 2 false; conflict[i] = 1 when propagation falsifies a clause
// (values are then unspecified).
struct PropArgs {
  int n;
  int32_t vmax;
  uint32_t assign_words;
  const int64_t* icb;
  const int64_t* cb;
  const int32_t* lits;
  const int32_t* nv;
  const int64_t* vb;
  const int64_t* occ_base;
  const uint32_t* occ_begin;
  const uint64_t* ent;
  const uint32_t* units;
  const uint32_t* nunits;
  const uint32_t* flags;
  const int64_t* asm_begin;   // [n+1]
  const int32_t* asm_lits;    // DIMACS
  uint32_t* trail;            // [blocks][vmax], or NULL: in shared memory
  uint8_t* values;
  uint8_t* conflict;
  Ctrl* ctrl;
};

__global__ void __launch_bounds__(512) k_propagate(const __grid_constant__ PropArgs A) {
  extern __shared__ uint32_t smem[];
  const int lane = threadIdx.x & 31;
  Warp w;
  w.S = nullptr;  // the propagate kernel has no search state
  w.cb = A.cb;
  w.lits = A.lits;
  w.ws = reinterpret_cast<WarpShared*>(smem);
  w.asg = smem + sizeof(WarpShared) / 4;
  w.lane = lane;
  w.trail = A.trail ? A.trail + (int64_t)blockIdx.x * A.vmax : w.asg + A.assign_words;
  // the block's threads agree (a failed bounds check of the checked build sets
  // the status while other blocks start)
  if (__syncthreads_or(batch_failed(A.ctrl))) return;
  for (int i = blockIdx.x; i < A.n; i += gridDim.x) {
    if (A.flags[i] & F_BAD) continue;
    w.V = (uint32_t)A.nv[i];
    w.c0 = A.icb[i];
    w.occ = A.occ_begin + A.occ_base[i];
    const int64_t lbase = A.icb[i] < A.icb[i + 1] ? A.cb[A.icb[i]] : 0;
    w.ent = A.ent + lbase;
    warp_checks(w, A.ctrl);
    const bool empty = (A.flags[i] & F_EMPTY) != 0;
    // the assignment cleared, the unit clauses and assumptions claimed by threads
    // first, first + step, ...
    auto clear = [&](uint32_t first, uint32_t step) {
      for (uint32_t k = first; k < (w.V + 15u) >> 4; k += step) w.asg[k] = 0u;
      if (first == 0) w.ws->tail = w.ws->conflict = 0;
    };
    auto start = [&](uint32_t first, uint32_t step) {
      for (uint32_t k = first; k < A.nunits[i] && !empty; k += step)
        if (!close_claim(w, A.units[w.c0 + k])) close_conflict(w, 0, NONE, NONE);
      for (int64_t k = A.asm_begin[i] + first; k < A.asm_begin[i + 1]; k += step) {
        const int32_t l = A.asm_lits[k];
        if (l == 0 || l > (int32_t)w.V || l < -(int32_t)w.V) continue;
        if (!close_claim(w, code_of(l))) close_conflict(w, 0, NONE, NONE);
      }
    };
    __syncthreads();  // the previous instance's values have been read
    clear(threadIdx.x, blockDim.x);
    __syncthreads();
    start(threadIdx.x, blockDim.x);
    __syncthreads();
    bool confl = empty || *(volatile uint32_t*)&w.ws->conflict != 0;
    const bool alone = blockDim.x == 32;
    w.head = 0;
    if (!confl) confl = alone ? close_rounds(w) : close_shared(w);
    __syncthreads();
    if (confl && !alone) {  // again, in the fixed order
      if (threadIdx.x < 32) {
        clear(lane, 32);
        __syncwarp();
        start(lane, 32);
        __syncwarp();
        if (!empty && w.ws->conflict == 0) close_rounds(w);
      }
      __syncthreads();
    }
    if (threadIdx.x == 0) A.conflict[i] = confl ? 1 : 0;
    for (uint32_t x = threadIdx.x; x < w.V; x += blockDim.x) {
      const uint32_t bits = (w.asg[x >> 4] >> ((x & 15u) * 2u)) & 3u;
      A.values[A.vb[i] + x] = (uint8_t)(bits == 3u ? 0u : bits);
    }
  }
}

}  // namespace dev

// --------------------------------------------------------------------------
// Host side: scratch, launch
// --------------------------------------------------------------------------

namespace {

struct Buf {
  void* p = nullptr;
  size_t cap = 0;
};

struct Scratch {
  Buf occ_base, occ_begin, ent, units, nunits, flags, items;
  Buf pending, done, inst_dec, trail, dstack, act, ring, job_act, prefix, ctrl;
  Buf lvlcnt, lvl_node;
  Buf cd_var, cd_mark, cd_wl, cd_pool, cd_learnt, cd_arena, cd_clidx;
  Buf share, share_cur, share_base;
  Buf job_cls, cls_copy;
  Buf h_icb, h_cb, h_lits, h_nv, h_vb, h_verdict, h_model, h_stats;  // for the host entry
  int sms = 0;
  int32_t last_status = 0;
  int smem_set[6] = {0, 0, 0, 0, 0, 0};  // dynamic shared memory granted per search mode
  int smem_prop = 0;
};

std::map<int, Scratch>& scratch_map() {
  static std::map<int, Scratch> m;
  return m;
}

int ensure(Buf& b, size_t bytes) {
  if (bytes == 0) bytes = 16;
  if (b.cap >= bytes) return 0;
  if (b.p) cudaFree(b.p);
  b.p = nullptr;
  b.cap = 0;
  size_t want = bytes + bytes / 4;
  if (cudaMalloc(&b.p, want) != cudaSuccess) {
    cudaGetLastError();
    if (cudaMalloc(&b.p, bytes) != cudaSuccess) {
      cudaGetLastError();
      return -1;
    }
    want = bytes;
  }
  b.cap = want;
  return 0;
}

template <class T>
T* P(Buf& b) { return reinterpret_cast<T*>(b.p); }

int cuda_fail(const char* what, cudaError_t e) {
  set_error(std::string(what) + ": " + cudaGetErrorString(e));
  return SCUBA_ERR_CUDA;
}

// Launch shape of the preparation kernel: a batch whose literals fit 72 KB of
// counters of 8 warps (1,843 variables) takes one block of 256 threads per
// instance, three or more of them on an SM; larger instances take blocks of
// 1,024 threads, one per SM, each a range of up to 3,264 literals.
constexpr size_t kPrepSmem8 = 72 * 1024, kPrepSmem32 = 3264 * 68;

struct PrepShape {
  int warps;
  uint32_t range;
  size_t smem;
  int64_t items;  // upper bound of the work items
  bool table;     // more than one item per instance is possible
};

PrepShape prep_shape(int64_t n, int64_t total_vars, int vmax) {
  PrepShape s;
  const uint32_t lits = 2u * (uint32_t)vmax;
  s.warps = (size_t)lits * 20 <= kPrepSmem8 ? 8 : 32;
  s.range = s.warps == 8 ? lits : std::min(lits, 3264u);
  s.smem = (size_t)s.range * 4 * (1 + s.warps / 2);
  s.table = lits > s.range;
  s.items = n + (s.table ? 2 * total_vars / s.range : 0);
  return s;
}

// The batch's arrays and sizes; the caller fills in the scratch.
dev::Prep prep_args(const scuba_cnf_batch* b, int vmax, const PrepShape& shape) {
  dev::Prep pr;
  pr.n = b->num_instances;
  pr.C = b->total_clauses;
  pr.L = b->total_lits;
  pr.total_vars = b->total_vars;
  pr.occ_cap = 2LL * b->total_vars + b->num_instances;
  pr.vmax = vmax;
  pr.range = shape.range;
  pr.vb = b->inst_var_begin;
  pr.icb = b->inst_clause_begin;
  pr.cb = b->clause_begin;
  pr.lits = b->lits;
  pr.nv = b->inst_num_vars;
  pr.items = nullptr;
  pr.item_cap = (uint32_t)std::min<int64_t>(shape.items, 0xffffffffll);
  return pr;
}

// Set-up and preparation of one call on `st`: two launches.
cudaError_t launch_prep(const dev::Prep& pr, const dev::SearchInit& init, const PrepShape& shape,
                        int sms, cudaStream_t st) {
  const int64_t words = std::max<int64_t>(
      {(int64_t)init.n_units, (int64_t)init.ring_cap, init.share_cur ? (int64_t)init.share_pools : 0});
  const int others = (int)std::min<int64_t>((words + 1023) / 1024, 2 * (int64_t)sms);
  dev::k_setup<<<1 + others, 1024, 0, st>>>(pr, init);
  auto kern = shape.warps == 8 ? dev::k_prep<8> : dev::k_prep<32>;
  // always the same value, so that calls of different batches agree on it
  const cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(shape.warps == 8 ? kPrepSmem8 : kPrepSmem32));
  if (e != cudaSuccess) return e;
  const int64_t per_sm =
      shape.warps == 8
          ? std::max<int64_t>(1, std::min<int64_t>(8, 226 * 1024 / ((int64_t)shape.smem + 2048)))
          : 1;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(shape.items, sms * per_sm));
  kern<<<grid, 32 * shape.warps, shape.smem, st>>>(pr);
  return cudaSuccess;
}

}  // namespace

}  // namespace scuba

using namespace scuba;

extern "C" int scuba_abi_sizes(int64_t* out) {
  if (!out) return SCUBA_ERR_ARG;
  out[0] = (int64_t)sizeof(scuba_cnf_batch);
  out[1] = (int64_t)sizeof(scuba_options);
  return SCUBA_OK;
}

extern "C" int scuba_options_init(scuba_options* o) {
  if (!o) return SCUBA_ERR_ARG;
  std::memset(o, 0, sizeof(*o));
  o->heuristic = SCUBA_HEUR_ACTIVITY;
  o->learned_depth = 0;
  o->decision_budget = 0;
  o->time_budget_ms = 0;
  o->split = 1;
  o->split_interval = 0;
  return SCUBA_OK;
}

// Units for scuba_solve_units: unit u is instance inst[u] under the
// assumption literals asm_lits[asm_begin[u] .. asm_begin[u+1]).
struct UnitArgs {
  int32_t n;
  const int32_t* inst;
  const int64_t* asm_begin;
  const int32_t* asm_lits;
  const int64_t* model_begin;
};

// clause-sharing pools of the clause-learning search: instance i uses pool
// i & (kSharePools - 1), a ring of kShareCap records of 64 bytes (128 MiB)
constexpr uint32_t kSharePools = 1024, kShareCap = 2048;

static int solve_impl(const scuba_cnf_batch* b, uint8_t* verdict, uint8_t* model,
                      cudaStream_t st, const scuba_options* opt, const UnitArgs* ua = nullptr) {
  if (!b || b->num_instances < 0 || b->total_clauses < 0 || b->total_lits < 0 ||
      b->max_vars < 0 || b->total_vars < 0) {
    set_error("scuba_solve_batch: bad arguments");
    return SCUBA_ERR_ARG;
  }
  scuba_options defaults;
  scuba_options_init(&defaults);
  if (!opt) opt = &defaults;
  const int n = b->num_instances;
  const int n_units = ua ? ua->n : n;
  if (n_units == 0) return SCUBA_OK;
  if (n == 0 || n_units < 0 || (ua && (!ua->inst || (ua->asm_begin && !ua->asm_lits)))) {
    set_error("scuba_solve_units: units need instances, a unit table and assumption literals");
    return SCUBA_ERR_ARG;
  }
  if (!verdict) {
    set_error("scuba_solve_batch: NULL verdict array");
    return SCUBA_ERR_ARG;
  }
  if (!b->inst_clause_begin || !b->clause_begin || !b->inst_num_vars || !b->inst_var_begin ||
      (b->total_lits > 0 && !b->lits)) {
    set_error("scuba_solve_batch: NULL batch array");
    return SCUBA_ERR_ARG;
  }
  if (opt->heuristic != SCUBA_HEUR_ACTIVITY && opt->heuristic != SCUBA_HEUR_LEARNED) {
    set_error("scuba_solve_batch: unknown heuristic");
    return SCUBA_ERR_ARG;
  }
  if (opt->search != SCUBA_SEARCH_DPLL && opt->search != SCUBA_SEARCH_CDCL) {
    set_error("scuba_solve_batch: unknown search algorithm");
    return SCUBA_ERR_ARG;
  }
  if (opt->search == SCUBA_SEARCH_CDCL &&
      (opt->trace || opt->heuristic != SCUBA_HEUR_ACTIVITY || opt->restart_unit < 0 ||
       opt->learnt_words < 0 || opt->learnt_words >= (1LL << 30))) {
    set_error("scuba_solve_batch: CDCL takes activity branching, no trace, restart_unit >= 0 "
              "and 0 <= learnt_words < 2^30");
    return SCUBA_ERR_ARG;
  }
  if (b->max_vars >= (1 << 29)) {
    set_error("scuba_solve_batch: instance too large (max_vars >= 2^29)");
    return SCUBA_ERR_TOO_LARGE;
  }
  int mode = dev::MODE_PLAIN;
  if (opt->trace) {
    const scuba_trace* T = opt->trace;
    if (T->depth < 1 || T->depth > learn::MAX_TRACE_DEPTH || T->max_nodes < 0 ||
        T->max_rows < 0 || !T->counts || !T->node_inst || !T->node_depth || !T->node_row ||
        !T->node_nrows || !T->node_closed || !T->x || !T->target || !T->var) {
      set_error("scuba_solve_batch: bad trace buffers (depth 1..8, all arrays set)");
      return SCUBA_ERR_ARG;
    }
    if (ua) {
      set_error("scuba_solve_units: trace recording takes whole instances");
      return SCUBA_ERR_ARG;
    }
    mode = dev::MODE_TRACE;
  } else if (opt->heuristic == SCUBA_HEUR_LEARNED) {
    if (!opt->mlp_weights || opt->learned_depth < 0) {
      set_error("scuba_solve_batch: learned branching needs mlp_weights and learned_depth >= 0");
      return SCUBA_ERR_ARG;
    }
    mode = dev::MODE_LEARNED;
  } else if (opt->search == SCUBA_SEARCH_CDCL) {
    mode = dev::MODE_CDCL;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail("cudaGetDevice", e);
  Scratch& S = scratch_map()[dev];
  if (!S.sms) {
    e = cudaDeviceGetAttribute(&S.sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return cuda_fail("cudaDeviceGetAttribute", e);
  }
  const int64_t C = b->total_clauses, L = b->total_lits;
  const int vmax = std::max(1, (int)b->max_vars);
  // occurrence offsets: sum over instances of (2V+1)
  const int64_t occ_total = 2LL * b->total_vars + n;

  // shape: warps per block x blocks per SM (shared memory bounds the warps)
  // Learned branching: two blocks of 6 warps unless the batch has a unit for every
  // warp of three blocks of 8. 512 partition queries of 10 bits take 24.2 ms so and
  // 26.3 on three blocks, 2,048 bounds queries of 8 bits 16.1 and 17.7. A batch that
  // large may hold long searches, which want the warps (4,096 partition queries of
  // 16 bits: 1,041 and 755 ms, with an untrained network 4.1 and 2.8 s; bounds
  // queries of 16 bits: 1,741 and 1,217 ms), or short ones, which do not (partition
  // queries of 10 bits: 28-33 and 43-49 ms); the former cost more to get wrong.
  const bool many = n_units >= 24 * S.sms;
  int wpb = opt->warps_per_block > 0 ? opt->warps_per_block
            : mode == dev::MODE_LEARNED && !many ? 6
                                                 : 8;
  int bps = opt->blocks_per_sm > 0 ? opt->blocks_per_sm
            : mode == dev::MODE_LEARNED && !many ? 2
                                                 : 5;
  wpb = std::min(wpb, 8);
  // 2 bits per variable; the clause-learning search keeps 4 (true, settled)
  const uint32_t assign_words = mode == dev::MODE_CDCL ? 2u * (uint32_t)((vmax + 15) / 16)
                                                       : (uint32_t)((vmax + 15) / 16);
  const size_t smem_cap = 227 * 1024, sm_cap = 228 * 1024;
  const size_t per_warp_g = sizeof(dev::WarpShared) + (size_t)assign_words * 4;
  const size_t per_warp_s = per_warp_g + (size_t)vmax * 4;
  // The trail in global memory unless the caller asks otherwise: a small
  // shared-memory carve-out leaves a larger L1 for the read-only occurrence lists,
  // which measured faster.
  const int trail_smem = opt->trail_placement == 1 ? 1 : 0;
  size_t per_warp = trail_smem ? per_warp_s : per_warp_g;
  if (mode == dev::MODE_LEARNED) per_warp += 32 * learn::NFEAT * sizeof(__nv_bfloat16);
  int cd_smem = 0;
  bool wide = false;  // clause learning: two blocks of 8 warps
  uint32_t cd_smem_warp = 0;
  if (mode == dev::MODE_CDCL) {
    // per-variable state in shared memory: 9 or 5 bytes a variable, or bounds of
    // the activities only, the first that fits `blocks` blocks of `warps` on an SM
    auto place = [&](int warps, int blocks) {
      for (int what : {dev::CD_SMEM_POS | dev::CD_SMEM_ACT, dev::CD_SMEM_POS | dev::CD_SMEM_GMAX,
                       (int)dev::CD_SMEM_GMAX, 0}) {
        if (vmax >= 65536 && (what & dev::CD_SMEM_POS)) continue;
        cd_smem = what;
        cd_smem_warp = (uint32_t)dev::cd_area_bytes(what, vmax);
        if (!what) cd_smem_warp = std::max(cd_smem_warp, (uint32_t)dev::CD_AREA_MIN);
        const size_t block = (per_warp + cd_smem_warp) * warps + 16;
        if (blocks == 2 ? (block + 1024) * 2 <= sm_cap : block <= smem_cap) return true;
      }
      return false;
    };
    // Two blocks on an SM if blocks of CDCL_WARPS (or of what the caller asks for)
    // fit so, else one of up to 8 warps. A batch with more units than one block
    // an SM has warps takes what lets two of them fit, others as much state as one
    // allows. (4,000 random 3-SAT and 32-bit bounds queries, 4,905 variables at most:
    // 2,047 ms on one block with positions and marks in shared memory, 1,542 on two
    // with the activities' bounds only; 2,048 partition queries of 20 bits 270 and
    // 249; but 64 of them 88 and 94, 16 bounds queries of 32 bits 22.6 and 23.1.)
    // A budget says that units are not expected to finish; with more of them than
    // two blocks of CDCL_WARPS have warps every warp stays busy, and two blocks of 8
    // do more in spite of their spills: 2,000 random 3-SAT instances of 200 to 400
    // variables 600 -> 419 ms, 9,000 2,726 -> 2,243. (Without a budget the last
    // instances decide, and partition and bounds queries take 3 to 13 % longer.)
    wide = bps > 1 && wpb == 8 && opt->decision_budget > 0 &&
           n_units > 2 * dev::CDCL_WARPS * S.sms && place(8, 2);
    const int w2 = wide ? 8 : std::min(wpb, dev::CDCL_WARPS);
    bool two = wide || (bps > 1 && n_units > 8 * S.sms && place(w2, 2));
    if (!two) {
      place(8, 1);
      two = bps > 1 && ((per_warp + cd_smem_warp) * w2 + 16 + 1024) * 2 <= sm_cap;
    }
    per_warp += cd_smem_warp;
    if (two) wpb = w2;
    else bps = 1;
  }
  size_t smem = per_warp * wpb + (mode == dev::MODE_CDCL ? 16 : 0);  // ring alignment
  while (wpb > 1 && smem > smem_cap) {
    wpb--;
    smem = per_warp * wpb + (mode == dev::MODE_CDCL ? 16 : 0);
  }
  if (smem > smem_cap) {
    set_error("scuba_solve_batch: instance too large for the shared-memory assignment");
    return SCUBA_ERR_TOO_LARGE;
  }
  while (bps > 1 && (smem + 1024) * bps > sm_cap) bps--;
  if (mode == dev::MODE_PLAIN) bps = std::min(bps, SCUBA_PLAIN_MINBLOCKS);
  if (mode == dev::MODE_LEARNED) bps = std::min(bps, SCUBA_LEARNED_MINBLOCKS);
  if (mode == dev::MODE_CDCL) bps = std::min(bps, SCUBA_CDCL_MINBLOCKS);
  const bool one_block = mode == dev::MODE_CDCL && bps == 1;
  const int64_t slots = (int64_t)S.sms * bps * wpb;
  const uint32_t ring_cap = 2048;

  const PrepShape shape = prep_shape(n, b->total_vars, vmax);
  if (ensure(S.occ_base, 8 * (size_t)(n + 1)) ||
      ensure(S.items, shape.table ? 8 * (size_t)shape.items : 0) ||
      ensure(S.occ_begin, 4 * (size_t)occ_total) ||
      ensure(S.ent, 8 * (size_t)L) || ensure(S.units, 4 * (size_t)std::max<int64_t>(C, 1)) ||
      ensure(S.nunits, 4 * (size_t)n) || ensure(S.flags, 4 * (size_t)n) ||
      ensure(S.pending, 4 * (size_t)n_units) || ensure(S.done, 4 * (size_t)n_units) ||
      ensure(S.inst_dec, 8 * (size_t)n_units) || ensure(S.trail, 4 * (size_t)slots * vmax) ||
      ensure(S.dstack, 4 * (size_t)slots * vmax) || ensure(S.act, 4 * (size_t)(slots * dev::act_stride(vmax))) ||
      ensure(S.ring, sizeof(dev::Job) * (size_t)ring_cap) ||
      ensure(S.job_act, 4 * (size_t)ring_cap * vmax) ||
      ensure(S.prefix, 4 * (size_t)slots * dev::MAX_PREFIX) || ensure(S.ctrl, sizeof(dev::Ctrl))) {
    set_error("scuba_solve_batch: out of device memory for scratch");
    return SCUBA_ERR_NOMEM;
  }
  if (mode == dev::MODE_TRACE &&
      (ensure(S.lvlcnt, 4 * (size_t)slots * learn::MAX_TRACE_DEPTH * vmax) ||
       ensure(S.lvl_node, 8 * (size_t)slots * learn::MAX_TRACE_DEPTH))) {
    set_error("scuba_solve_batch: out of device memory for trace scratch");
    return SCUBA_ERR_NOMEM;
  }
  int64_t arena_words = 0;
  if (mode == dev::MODE_CDCL) {
    arena_words = (opt->learnt_words > 0 ? opt->learnt_words : (1LL << 18)) & ~3LL;
    if (arena_words < std::max<int64_t>((int64_t)vmax + 2 * dev::CD_HDR, 64)) {
      set_error("scuba_solve_batch: learnt_words must be at least max(max_vars + 8, 64)");
      return SCUBA_ERR_ARG;
    }
    const size_t share_bytes = 4 * (size_t)kSharePools * kShareCap * dev::SHARE_REC;
    const bool share_ready = S.share.p && S.share_cur.p && S.share_base.p;
    if (ensure(S.cd_var, 16 * (size_t)slots * vmax) ||
        ensure(S.cd_mark, (size_t)slots * vmax) ||
        ensure(S.cd_wl, 32 * (size_t)slots * vmax) ||
        ensure(S.cd_pool, 8 * (size_t)slots * arena_words) ||
        ensure(S.cd_learnt, 4 * (size_t)slots * vmax) ||
        // a clause's reader takes eight literals at a time, past its end too
        ensure(S.cd_arena, 4 * (size_t)slots * arena_words + 64) ||
        ensure(S.cd_clidx, 4 * (size_t)slots * (arena_words / 8)) ||
        ensure(S.job_cls, 4 * (size_t)ring_cap * dev::JOB_CLS_WORDS) ||
        ensure(S.cls_copy, 4 * (size_t)slots * dev::JOB_CLS_WORDS) ||
        ensure(S.share, share_bytes) || ensure(S.share_cur, 8 * (size_t)kSharePools) ||
        ensure(S.share_base, 8 * (size_t)kSharePools)) {
      set_error("scuba_solve_batch: out of device memory for clause-learning scratch");
      return SCUBA_ERR_NOMEM;
    }
    if (!share_ready) {  // fresh pools: no record, cursors at zero
      cudaMemsetAsync(S.share.p, 0, share_bytes, st);
      cudaMemsetAsync(S.share_cur.p, 0, 8 * (size_t)kSharePools, st);
    }
  }
  dev::Prep pr = prep_args(b, vmax, shape);
  pr.occ_base = P<int64_t>(S.occ_base);
  pr.occ_begin = P<uint32_t>(S.occ_begin);
  pr.ent = P<uint64_t>(S.ent);
  pr.units = P<uint32_t>(S.units);
  pr.nunits = P<uint32_t>(S.nunits);
  pr.flags = P<uint32_t>(S.flags);
  if (shape.table) pr.items = P<int2>(S.items);
  pr.ctrl = P<dev::Ctrl>(S.ctrl);

  dev::Solve sv;
  sv.n = n;
  sv.vmax = vmax;
  sv.assign_words = assign_words;
  sv.icb = b->inst_clause_begin;
  sv.cb = b->clause_begin;
  sv.lits = b->lits;
  sv.nv = b->inst_num_vars;
  sv.vb = b->inst_var_begin;
  sv.occ_base = pr.occ_base;
  sv.occ_begin = pr.occ_begin;
  sv.ent = pr.ent;
  sv.units = pr.units;
  sv.nunits = pr.nunits;
  sv.flags = pr.flags;
  sv.order = opt->order;
  sv.n_units = n_units;
  sv.unit_inst = ua ? ua->inst : nullptr;
  sv.unit_asm_begin = ua ? ua->asm_begin : nullptr;
  sv.unit_asm = ua ? ua->asm_lits : nullptr;
  sv.unit_vb = ua ? ua->model_begin : nullptr;
  sv.verdict = verdict;
  sv.model = model;
  sv.stats = opt->stats;
  sv.pending = P<uint32_t>(S.pending);
  sv.done = P<uint32_t>(S.done);
  sv.inst_dec = P<unsigned long long>(S.inst_dec);
  sv.trail = P<uint32_t>(S.trail);
  sv.dstack = P<uint32_t>(S.dstack);
  sv.act = P<float>(S.act);
  sv.ring = P<dev::Job>(S.ring);
  sv.ring_cap = ring_cap;
  sv.job_act = P<float>(S.job_act);
  sv.prefix = P<uint32_t>(S.prefix);
  sv.split_min = opt->split_min > 0 ? opt->split_min : 256;
  sv.split_depth = opt->split_depth > 0 ? opt->split_depth : dev::MAX_PREFIX;
  sv.ctrl = P<dev::Ctrl>(S.ctrl);
  sv.budget = opt->decision_budget;
  int64_t tb = opt->time_budget_ms > 0 ? opt->time_budget_ms : 600000;
  sv.time_ns = (uint64_t)tb * 1000000ull;
  sv.abort_flag = opt->abort_flag;
  sv.split = opt->split ? 1 : 0;
  sv.split_interval = opt->split_interval > 0 ? opt->split_interval : 16;
  sv.trail_smem = trail_smem;
  sv.finish_ns = opt->finish_ns;
  sv.prof = reinterpret_cast<unsigned long long*>(opt->profile);
  sv.mlp = static_cast<const learn::MlpWeights*>(opt->mlp_weights);
  sv.learned_depth = opt->learned_depth;
  sv.inst_num_inputs = opt->inst_num_inputs;
  sv.trace_depth = 0;
  sv.lvlcnt = nullptr;
  sv.lvl_node = nullptr;
  sv.cd_var = P<uint4>(S.cd_var);
  sv.cd_mark = P<uint8_t>(S.cd_mark);
  sv.cd_smem = cd_smem;
  sv.cd_smem_warp = cd_smem_warp;
  sv.cd_wl = P<dev::WList>(S.cd_wl);
  sv.cd_pool = P<uint64_t>(S.cd_pool);
  sv.cd_pool_cap = arena_words;
  sv.cd_learnt = P<uint32_t>(S.cd_learnt);
  sv.cd_arena = P<uint32_t>(S.cd_arena);
  sv.cd_clidx = P<uint32_t>(S.cd_clidx);
  sv.job_cls = P<uint32_t>(S.job_cls);
  sv.cls_copy = P<uint32_t>(S.cls_copy);
  sv.cd_arena_words = arena_words;
  sv.restart_unit = opt->restart_unit > 0 ? opt->restart_unit : 100;
  sv.share = nullptr;
  sv.share_cur = nullptr;
  sv.share_base = nullptr;
  sv.share_mask = 0;
  sv.share_cap = 0;
  sv.share_lbd = 0;
  if (mode == dev::MODE_CDCL && opt->share_lbd >= 0) {
    // the pools keep earlier calls' records; this call's jobs read from where
    // the cursors stood when it began (share_base)
    sv.share = P<uint32_t>(S.share);
    sv.share_cur = P<unsigned long long>(S.share_cur);
    sv.share_base = P<unsigned long long>(S.share_base);
    sv.share_mask = kSharePools - 1;
    sv.share_cap = kShareCap;
    sv.share_lbd = opt->share_lbd > 0 ? (uint32_t)opt->share_lbd : 2u;
  }
  std::memset(&sv.tr, 0, sizeof(sv.tr));
  if (mode == dev::MODE_TRACE) {
    const scuba_trace* T = opt->trace;
    sv.trace_depth = T->depth;
    sv.split = 0;  // a traced subtree must be explored by one warp
    sv.tr.cursor = reinterpret_cast<unsigned long long*>(T->counts);
    sv.tr.max_nodes = T->max_nodes;
    sv.tr.max_rows = T->max_rows;
    sv.tr.node_inst = T->node_inst;
    sv.tr.node_depth = T->node_depth;
    sv.tr.node_row = T->node_row;
    sv.tr.node_nrows = T->node_nrows;
    sv.tr.node_closed = T->node_closed;
    sv.tr.x = reinterpret_cast<__nv_bfloat16*>(T->x);
    sv.tr.target = T->target;
    sv.tr.var = T->var;
    sv.lvlcnt = P<uint32_t>(S.lvlcnt);
    sv.lvl_node = P<int64_t>(S.lvl_node);
    cudaMemsetAsync(sv.lvlcnt, 0, 4 * (size_t)slots * learn::MAX_TRACE_DEPTH * vmax, st);
    cudaMemsetAsync(sv.lvl_node, 0xff, 8 * (size_t)slots * learn::MAX_TRACE_DEPTH, st);
  }

  NvtxRange prep_range("scuba prep + search launch");
  const dev::SearchInit init{n_units, sv.pending, sv.done, sv.inst_dec, verdict, sv.ring, ring_cap,
                             sv.share_cur, P<unsigned long long>(S.share_base), kSharePools};
  e = launch_prep(pr, init, shape, S.sms, st);
  if (e != cudaSuccess) return cuda_fail("preparation launch", e);
  auto kern = mode == dev::MODE_TRACE     ? dev::k_solve<dev::MODE_TRACE>
              : mode == dev::MODE_LEARNED ? dev::k_solve<dev::MODE_LEARNED>
              : one_block                 ? dev::k_solve<dev::MODE_CDCL1>
              : wide                      ? dev::k_solve<dev::MODE_CDCL8>
              : mode == dev::MODE_CDCL    ? dev::k_solve<dev::MODE_CDCL>
                                          : dev::k_solve<dev::MODE_PLAIN>;
  // raise the dynamic shared-memory limit only when it grows, so that a
  // repeated call (for example while a CUDA graph is being captured) issues
  // no attribute change
  int& granted = S.smem_set[one_block ? (int)dev::MODE_CDCL1 : wide ? (int)dev::MODE_CDCL8 : mode];
  if ((int)smem > granted) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail("cudaFuncSetAttribute", e);
    granted = (int)smem;
  }
  if (opt->search_event_begin) cudaEventRecord((cudaEvent_t)opt->search_event_begin, st);
  kern<<<S.sms * bps, 32 * wpb, smem, st>>>(sv);
  if (opt->search_event_end) cudaEventRecord((cudaEvent_t)opt->search_event_end, st);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail("kernel launch", e);
  return SCUBA_OK;
}

extern "C" int scuba_solve_batch_ex(const scuba_cnf_batch* b, uint8_t* verdict, uint8_t* model,
                                    void* stream, const scuba_options* opt) {
  return solve_impl(b, verdict, model, (cudaStream_t)stream, opt);
}

extern "C" int scuba_solve_units(const scuba_cnf_batch* b, int32_t n_units,
                                 const int32_t* unit_inst, const int64_t* asm_begin,
                                 const int32_t* asm_lits, const int64_t* unit_model_begin,
                                 uint8_t* verdict, uint8_t* model, void* stream,
                                 const scuba_options* opt) {
  if (n_units < 0 || (n_units > 0 && (!unit_inst || !verdict)) || (model && !unit_model_begin)) {
    set_error("scuba_solve_units: bad arguments");
    return SCUBA_ERR_ARG;
  }
  UnitArgs ua{n_units, unit_inst, asm_begin, asm_lits, unit_model_begin};
  return solve_impl(b, verdict, model, (cudaStream_t)stream, opt, &ua);
}

extern "C" int scuba_solve_batch(const scuba_cnf_batch* b, uint8_t* verdict, uint8_t* model,
                                 void* stream) {
  return solve_impl(b, verdict, model, (cudaStream_t)stream, nullptr);
}

extern "C" int scuba_sync_status(void* stream) {
  cudaError_t e = cudaStreamSynchronize((cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_fail("cudaStreamSynchronize", e);
  int dev = 0;
  cudaGetDevice(&dev);
  auto it = scratch_map().find(dev);
  if (it == scratch_map().end() || !it->second.ctrl.p) return SCUBA_OK;
  dev::Ctrl c;
  e = cudaMemcpy(&c, it->second.ctrl.p, sizeof(c), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail("cudaMemcpy", e);
  if (c.status != 0) {
    std::string msg = "device status " + std::to_string(c.status);
    if (c.check_site != 0)
      msg += " (bounds check " + std::to_string(c.check_site) + " failed: index " +
             std::to_string(c.check_index) + ", limit " + std::to_string(c.check_limit) + ")";
    set_error(msg);
  }
  return c.status;
}

extern "C" int scuba_solve_batch_host(const scuba_cnf_batch* hb, uint8_t* verdict,
                                      uint8_t* model, void* stream, const scuba_options* opt) {
  if (!hb || !verdict || hb->num_instances < 0) return SCUBA_ERR_ARG;
  const int n = hb->num_instances;
  if (n == 0) return SCUBA_OK;
  int dev = 0;
  cudaGetDevice(&dev);
  Scratch& S = scratch_map()[dev];
  cudaStream_t st = (cudaStream_t)stream;
  const int64_t C = hb->total_clauses, L = hb->total_lits;
  const int64_t nvars = hb->inst_var_begin[n];
  if (ensure(S.h_icb, 8 * (size_t)(n + 1)) || ensure(S.h_cb, 8 * (size_t)(C + 1)) ||
      ensure(S.h_lits, 4 * (size_t)L) || ensure(S.h_nv, 4 * (size_t)n) ||
      ensure(S.h_vb, 8 * (size_t)(n + 1)) || ensure(S.h_verdict, (size_t)n) ||
      ensure(S.h_model, (size_t)std::max<int64_t>(nvars, 1)) ||
      ensure(S.h_stats, 8 * SCUBA_NSTATS * (size_t)n))
    return SCUBA_ERR_NOMEM;
  cudaError_t e;
  NvtxRange range("scuba host-buffer solve (upload, solve, download)");
  e = cudaMemcpyAsync(S.h_icb.p, hb->inst_clause_begin, 8 * (size_t)(n + 1), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(S.h_cb.p, hb->clause_begin, 8 * (size_t)(C + 1), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess && L > 0) e = cudaMemcpyAsync(S.h_lits.p, hb->lits, 4 * (size_t)L, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(S.h_nv.p, hb->inst_num_vars, 4 * (size_t)n, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(S.h_vb.p, hb->inst_var_begin, 8 * (size_t)(n + 1), cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return cuda_fail("cudaMemcpyAsync H2D", e);
  scuba_cnf_batch db = *hb;
  db.inst_clause_begin = P<int64_t>(S.h_icb);
  db.clause_begin = P<int64_t>(S.h_cb);
  db.lits = P<int32_t>(S.h_lits);
  db.inst_num_vars = P<int32_t>(S.h_nv);
  db.inst_var_begin = P<int64_t>(S.h_vb);
  scuba_options o;
  if (opt) o = *opt; else scuba_options_init(&o);
  int64_t* host_stats = o.stats;
  if (host_stats) {
    cudaMemsetAsync(S.h_stats.p, 0, 8 * SCUBA_NSTATS * (size_t)n, st);
    o.stats = P<int64_t>(S.h_stats);
  }
  int r = solve_impl(&db, P<uint8_t>(S.h_verdict), model ? P<uint8_t>(S.h_model) : nullptr, st, &o);
  if (r != SCUBA_OK) return r;
  e = cudaMemcpyAsync(verdict, S.h_verdict.p, (size_t)n, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess && model && nvars > 0)
    e = cudaMemcpyAsync(model, S.h_model.p, (size_t)nvars, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess && host_stats)
    e = cudaMemcpyAsync(host_stats, S.h_stats.p, 8 * SCUBA_NSTATS * (size_t)n, cudaMemcpyDeviceToHost, st);
  if (e != cudaSuccess) return cuda_fail("cudaMemcpyAsync D2H", e);
  return scuba_sync_status(stream);
}

extern "C" void scuba_release(void) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return;
  auto it = scratch_map().find(dev);
  if (it == scratch_map().end()) return;
  Scratch& S = it->second;
  Buf* all[] = {&S.occ_base, &S.items, &S.occ_begin, &S.ent, &S.units, &S.nunits,
                &S.flags, &S.pending, &S.done, &S.inst_dec, &S.trail, &S.dstack, &S.act,
                &S.ring, &S.job_act, &S.prefix, &S.ctrl, &S.lvlcnt, &S.lvl_node,
                &S.cd_var, &S.cd_mark, &S.cd_wl, &S.cd_pool,
                &S.cd_learnt, &S.cd_arena, &S.cd_clidx, &S.job_cls, &S.cls_copy,
                &S.share, &S.share_cur, &S.share_base, &S.h_icb,
                &S.h_cb, &S.h_lits,
                &S.h_nv, &S.h_vb,
                &S.h_verdict, &S.h_model, &S.h_stats};
  for (Buf* x : all) {
    if (x->p) cudaFree(x->p);
    x->p = nullptr;
    x->cap = 0;
  }
  scratch_map().erase(it);
}

// --------------------------------------------------------------------------
// Allocation-free variant
//
// Some callers cannot call cudaMalloc: code that runs inside another
// framework's memory pool or allocator hooks, inside a plugin whose host
// forbids device allocation, or on a path where a synchronous allocation would
// stall other streams. For them scuba_solve_batch_noalloc runs the same
// preparation and search kernels with every scratch buffer carved out of one
// file-scope device array of fixed size. Every GPU that loads this library
// holds that array until the process exits.
// --------------------------------------------------------------------------

namespace scuba {
namespace {
constexpr size_t kNoAllocScratchBytes = 64ull << 20;  // 64 MiB
constexpr int kNoAllocWarpsPerBlock = 4;
constexpr uint32_t kNoAllocRingCap = 256;
constexpr int kMaxDevices = 256;
void* g_noalloc_scratch_addr[kMaxDevices];  // device address of the array, per device
std::mutex g_noalloc_mu;  // guards the per-device set-up and the shared attribute cache
}  // namespace
}  // namespace scuba

static __device__ __align__(256) unsigned char g_noalloc_scratch[scuba::kNoAllocScratchBytes];

extern "C" int scuba_solve_batch_noalloc(const scuba_cnf_batch* b, uint8_t* verdict,
                                         uint8_t* model, void* stream,
                                         const scuba_options* opt) {
  using namespace scuba;
  if (!b || b->num_instances < 0 || b->total_clauses < 0 || b->total_lits < 0 ||
      b->max_vars < 0 || b->total_vars < 0) {
    set_error("scuba_solve_batch_noalloc: bad arguments");
    return SCUBA_ERR_ARG;
  }
  scuba_options defaults;
  scuba_options_init(&defaults);
  if (!opt) opt = &defaults;
  const int n = b->num_instances;
  if (n == 0) return SCUBA_OK;
  if (!verdict || !b->inst_clause_begin || !b->clause_begin || !b->inst_num_vars ||
      !b->inst_var_begin || (b->total_lits > 0 && !b->lits)) {
    set_error("scuba_solve_batch_noalloc: NULL array");
    return SCUBA_ERR_ARG;
  }
  if (opt->heuristic != SCUBA_HEUR_ACTIVITY || opt->search != SCUBA_SEARCH_DPLL) {
    set_error("scuba_solve_batch_noalloc: only DPLL with activity branching is supported");
    return SCUBA_ERR_ARG;
  }
  if (b->max_vars >= (1 << 29) || b->total_lits >= (1LL << 32)) {
    set_error("scuba_solve_batch_noalloc: instance too large");
    return SCUBA_ERR_TOO_LARGE;
  }
  cudaStream_t st = (cudaStream_t)stream;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail("cudaGetDevice", e);
  if (dev < 0 || dev >= kMaxDevices) {
    set_error("scuba_solve_batch_noalloc: device ordinal out of range");
    return SCUBA_ERR_ARG;
  }
  // set-up, once per device, with that device current: the host-side name of
  // the array is not a device address, so ask the runtime for it
  {
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_scratch_addr[dev]) {
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e != cudaSuccess) return cuda_fail("cudaGetSymbolAddress", e);
      g_noalloc_scratch_addr[dev] = p;
    }
  }
  int sms = 0;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return cuda_fail("cudaDeviceGetAttribute", e);

  const int64_t C = b->total_clauses, L = b->total_lits;
  const int vmax = std::max(1, (int)b->max_vars);
  const int64_t occ_total = 2LL * b->total_vars + n;
  const int wpb = kNoAllocWarpsPerBlock;
  const uint32_t assign_words = (uint32_t)((vmax + 15) / 16);
  const size_t smem = (sizeof(dev::WarpShared) + (size_t)assign_words * 4) * wpb;
  if (smem > 227 * 1024) {
    set_error("scuba_solve_batch_noalloc: instance too large for the shared-memory assignment");
    return SCUBA_ERR_TOO_LARGE;
  }
  const int64_t slots = (int64_t)sms * wpb;  // one block per SM
  const uint32_t ring_cap = kNoAllocRingCap;

  // carve every buffer out of the static array, 256-byte aligned
  size_t off = 0;
  auto carve = [&](size_t bytes) {
    size_t at = off;
    off += (std::max<size_t>(bytes, 16) + 255) & ~(size_t)255;
    return at;
  };
  // 4 L + 4 occ_total bytes are set aside and not used (but for the padding of
  // the activities): the limit on what a batch may need is part of the interface,
  // which states it
  carve(4 * (size_t)L);
  carve(4 * (size_t)occ_total);
  const size_t act_bytes = 4 * (size_t)(slots * dev::act_stride(vmax));
  const size_t act_pad = ((act_bytes + 255) & ~(size_t)255) -
                         ((4 * (size_t)slots * vmax + 255) & ~(size_t)255);
  off -= std::min(off, act_pad);
  const size_t o_occ_base = carve(8 * (size_t)(n + 1)), o_occ_begin = carve(4 * (size_t)occ_total),
               o_ent = carve(8 * (size_t)L), o_units = carve(4 * (size_t)std::max<int64_t>(C, 1)),
               o_nunits = carve(4 * (size_t)n), o_flags = carve(4 * (size_t)n),
               o_pending = carve(4 * (size_t)n), o_done = carve(4 * (size_t)n),
               o_inst_dec = carve(8 * (size_t)n), o_trail = carve(4 * (size_t)slots * vmax),
               o_dstack = carve(4 * (size_t)slots * vmax), o_act = carve(act_bytes),
               o_ring = carve(sizeof(dev::Job) * (size_t)ring_cap),
               o_job_act = carve(4 * (size_t)ring_cap * vmax),
               o_prefix = carve(4 * (size_t)slots * dev::MAX_PREFIX),
               o_ctrl = carve(sizeof(dev::Ctrl));
  if (off > kNoAllocScratchBytes) {
    set_error("scuba_solve_batch_noalloc: batch needs " + std::to_string(off) +
              " bytes of scratch, more than the fixed " +
              std::to_string(kNoAllocScratchBytes) + " bytes");
    return SCUBA_ERR_TOO_LARGE;
  }
  unsigned char* base = static_cast<unsigned char*>(g_noalloc_scratch_addr[dev]);
  auto at = [&](size_t o) { return static_cast<void*>(base + o); };

  const PrepShape shape = prep_shape(n, b->total_vars, vmax);
  dev::Prep pr = prep_args(b, vmax, shape);
  pr.occ_base = static_cast<int64_t*>(at(o_occ_base));
  pr.occ_begin = static_cast<uint32_t*>(at(o_occ_begin));
  pr.ent = static_cast<uint64_t*>(at(o_ent));
  pr.units = static_cast<uint32_t*>(at(o_units));
  pr.nunits = static_cast<uint32_t*>(at(o_nunits));
  pr.flags = static_cast<uint32_t*>(at(o_flags));
  pr.ctrl = static_cast<dev::Ctrl*>(at(o_ctrl));
  if (shape.table) {
    // in the search's trail, decision and activity arrays, not in use yet: 12 *
    // slots * vmax bytes with vmax > 1,843, while a batch within the limit has
    // fewer than 64 MiB / 40 instances (12.8 MiB of items; the arrays hold 12.8
    // MiB from 152 SMs on, so only a smaller GPU could meet this error)
    pr.items = static_cast<int2*>(at(o_trail));
    if (8 * (size_t)shape.items > o_ring - o_trail) {
      set_error("scuba_solve_batch_noalloc: too many instances beside a large one");
      return SCUBA_ERR_TOO_LARGE;
    }
  }

  dev::Solve sv;
  std::memset(&sv, 0, sizeof(sv));
  sv.n = n;
  sv.vmax = vmax;
  sv.assign_words = assign_words;
  sv.icb = b->inst_clause_begin;
  sv.cb = b->clause_begin;
  sv.lits = b->lits;
  sv.nv = b->inst_num_vars;
  sv.vb = b->inst_var_begin;
  sv.occ_base = pr.occ_base;
  sv.occ_begin = pr.occ_begin;
  sv.ent = pr.ent;
  sv.units = pr.units;
  sv.nunits = pr.nunits;
  sv.flags = pr.flags;
  sv.n_units = n;
  sv.order = opt->order;
  sv.verdict = verdict;
  sv.model = model;
  sv.stats = opt->stats;
  sv.pending = static_cast<uint32_t*>(at(o_pending));
  sv.done = static_cast<uint32_t*>(at(o_done));
  sv.inst_dec = static_cast<unsigned long long*>(at(o_inst_dec));
  sv.trail = static_cast<uint32_t*>(at(o_trail));
  sv.dstack = static_cast<uint32_t*>(at(o_dstack));
  sv.act = static_cast<float*>(at(o_act));
  sv.ring = static_cast<dev::Job*>(at(o_ring));
  sv.ring_cap = ring_cap;
  sv.job_act = static_cast<float*>(at(o_job_act));
  sv.prefix = static_cast<uint32_t*>(at(o_prefix));
  sv.split_min = opt->split_min > 0 ? opt->split_min : 256;
  sv.split_depth = opt->split_depth > 0 ? opt->split_depth : dev::MAX_PREFIX;
  sv.ctrl = pr.ctrl;
  sv.budget = opt->decision_budget;
  int64_t tb = opt->time_budget_ms > 0 ? opt->time_budget_ms : 600000;
  sv.time_ns = (uint64_t)tb * 1000000ull;
  sv.abort_flag = opt->abort_flag;
  sv.split = opt->split ? 1 : 0;
  sv.split_interval = opt->split_interval > 0 ? opt->split_interval : 16;
  sv.trail_smem = 0;
  sv.finish_ns = nullptr;
  sv.prof = nullptr;

  // the array keeps the previous call's contents: set-up writes everything that
  // must have a value before the search, the rest is written before it is read
  const dev::SearchInit init{n, sv.pending, sv.done, sv.inst_dec, verdict, sv.ring, ring_cap,
                             nullptr, nullptr, 0};
  e = launch_prep(pr, init, shape, sms, st);
  if (e != cudaSuccess) return cuda_fail("preparation launch", e);
  // the kernel attribute is shared with the regular entry points: only ever
  // raise it, through the same per-device cache, so that a later regular
  // call that needs more shared memory still finds its own grant in place
  {
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    int& granted = scratch_map()[dev].smem_set[dev::MODE_PLAIN];
    if ((int)smem > granted) {
      e = cudaFuncSetAttribute(dev::k_solve<dev::MODE_PLAIN>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return cuda_fail("cudaFuncSetAttribute", e);
      granted = (int)smem;
    }
  }
  dev::k_solve<dev::MODE_PLAIN><<<sms, 32 * wpb, smem, st>>>(sv);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail("kernel launch", e);
  // report the device-side status of this call (the control block lives in
  // the static array, so the normal status query cannot see it)
  e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail("cudaStreamSynchronize", e);
  int32_t status = 0;
  e = cudaMemcpy(&status, reinterpret_cast<unsigned char*>(pr.ctrl) + offsetof(dev::Ctrl, status),
                 sizeof(status), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail("cudaMemcpy", e);
  if (status != 0) set_error("scuba_solve_batch_noalloc: device status " + std::to_string(status));
  return status;
}

extern "C" int scuba_propagate_batch(const scuba_cnf_batch* b, const int64_t* asm_begin,
                                     const int32_t* asm_lits, uint8_t* values,
                                     uint8_t* conflict, void* stream) {
  using namespace scuba;
  if (!b || b->num_instances < 0 || b->max_vars < 0 || b->total_vars < 0 ||
      b->total_clauses < 0 || b->total_lits < 0) {
    set_error("scuba_propagate_batch: bad arguments");
    return SCUBA_ERR_ARG;
  }
  const int n = b->num_instances;
  if (n == 0) return SCUBA_OK;
  if (!asm_begin || !values || !conflict || !b->inst_clause_begin || !b->clause_begin ||
      !b->inst_num_vars || !b->inst_var_begin || (b->total_lits > 0 && !b->lits)) {
    set_error("scuba_propagate_batch: NULL array");
    return SCUBA_ERR_ARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail("cudaGetDevice", e);
  Scratch& S = scratch_map()[dev];
  if (!S.sms) {
    e = cudaDeviceGetAttribute(&S.sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return cuda_fail("cudaDeviceGetAttribute", e);
  }
  const int64_t C = b->total_clauses, L = b->total_lits;
  const int vmax = std::max(1, (int)b->max_vars);
  const int64_t occ_total = 2LL * b->total_vars + n;
  const uint32_t assign_words = (uint32_t)((vmax + 15) / 16);
  if ((sizeof(dev::WarpShared) + (size_t)assign_words * 4) * 8 > 227 * 1024)
    return SCUBA_ERR_TOO_LARGE;
  // warps per instance: as many as keep about 48 on an SM, one per 512 variables
  // at most (a round has to have work for them), 16 at most. (33 instances of up to
  // 46,000 variables: 1.30, 0.89, 0.62, 0.47, 0.40 ms for 1, 2, 4, 8, 16 warps,
  // preparation included; one warp in close_rounds 1.31 ms. 4,096 instances of
  // 1,800 variables: one warp in close_rounds 0.99 ms, two to eight sharing an
  // instance 1.32 to 1.51 ms.)
  int wpb = 1;
  while (wpb < 16 && 2LL * wpb * n <= 48LL * S.sms && 1024 * wpb <= vmax) wpb *= 2;
  // a shared instance's trail in shared memory where it fits; not for one warp
  // each, whose lists then lose the L1 (1.26 against 0.99 ms)
  const bool trail_smem = wpb > 1 && (size_t)vmax * 4 <= (size_t)wpb * 12 * 1024;
  const size_t smem = sizeof(dev::WarpShared) + (size_t)assign_words * 4 +
                      (trail_smem ? (size_t)vmax * 4 : 0);
  const int per_sm = (int)std::max<size_t>(1, std::min<size_t>(64 / wpb > 32 ? 32 : 64 / wpb,
                                                               227 * 1024 / (smem + 1024)));
  const int blocks = std::min(n, S.sms * per_sm);
  const PrepShape shape = prep_shape(n, b->total_vars, vmax);
  if (ensure(S.occ_base, 8 * (size_t)(n + 1)) ||
      ensure(S.items, shape.table ? 8 * (size_t)shape.items : 0) ||
      ensure(S.occ_begin, 4 * (size_t)occ_total) ||
      ensure(S.ent, 8 * (size_t)L) || ensure(S.units, 4 * (size_t)std::max<int64_t>(C, 1)) ||
      ensure(S.nunits, 4 * (size_t)n) || ensure(S.flags, 4 * (size_t)n) ||
      ensure(S.trail, trail_smem ? 0 : 4 * (size_t)blocks * vmax) ||
      ensure(S.ctrl, sizeof(dev::Ctrl)))
    return SCUBA_ERR_NOMEM;
  dev::Prep pr = prep_args(b, vmax, shape);
  pr.occ_base = P<int64_t>(S.occ_base);
  pr.occ_begin = P<uint32_t>(S.occ_begin);
  pr.ent = P<uint64_t>(S.ent);
  pr.units = P<uint32_t>(S.units);
  pr.nunits = P<uint32_t>(S.nunits);
  pr.flags = P<uint32_t>(S.flags);
  if (shape.table) pr.items = P<int2>(S.items);
  pr.ctrl = P<dev::Ctrl>(S.ctrl);
  const dev::SearchInit no_search{};
  e = launch_prep(pr, no_search, shape, S.sms, st);
  if (e != cudaSuccess) return cuda_fail("preparation launch", e);
  dev::PropArgs A;
  A.n = n;
  A.vmax = vmax;
  A.assign_words = assign_words;
  A.icb = b->inst_clause_begin;
  A.cb = b->clause_begin;
  A.lits = b->lits;
  A.nv = b->inst_num_vars;
  A.vb = b->inst_var_begin;
  A.occ_base = pr.occ_base;
  A.occ_begin = pr.occ_begin;
  A.ent = pr.ent;
  A.units = pr.units;
  A.nunits = pr.nunits;
  A.flags = pr.flags;
  A.asm_begin = asm_begin;
  A.asm_lits = asm_lits;
  A.trail = trail_smem ? nullptr : P<uint32_t>(S.trail);
  A.values = values;
  A.conflict = conflict;
  A.ctrl = pr.ctrl;
  if ((int)smem > S.smem_prop) {
    e = cudaFuncSetAttribute(dev::k_propagate, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem);
    if (e != cudaSuccess) return cuda_fail("cudaFuncSetAttribute", e);
    S.smem_prop = (int)smem;
  }
  dev::k_propagate<<<blocks, 32 * wpb, smem, st>>>(A);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail("kernel launch", e);
  return SCUBA_OK;
}
