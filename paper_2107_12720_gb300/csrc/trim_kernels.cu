// trim_kernels.cu -- the persistent round-synchronous trimming kernel.
//
// One cooperative launch runs every round of the trimming of Guo & Sekerinski
// (arXiv 2107.12720): round 0 removes the vertices without out-edges, round r
// the vertices whose successors were all removed in rounds < r (Definition 2).
// Each round runs one of three kernels, chosen per round:
//
//   AC-4 push   (Section 5, Algorithm 6): each removed vertex w decrements the
//               out-degree counter of every predecessor through G^T; the atomic
//               decrement that returns 1 removes the predecessor (it is unique,
//               so no CAS on the status is needed).
//   AC-6 support (Section 6, Algorithms 7/8, Definition 3): every live vertex
//               keeps one support (edge_index) and sits in that support's
//               supporting set S; when a support is removed, the members of its
//               S re-scan forward for the next live successor. Rounds replace the
//               paper's spin locks: a set is only read after the round in which
//               its owner was removed, and no vertex joins the S of a vertex
//               removed in an earlier round.
//   AC-3 pull   (Section 4, Algorithm 4 with the edge_index jump of Section 8):
//               a sweep over a compacted list of the vertices still live.
//
// All three read "u removed before round r" as level[u] < r, so mixing them
// round by round yields the same levels.
//
// Rounds end at a grid-wide barrier (a monotone arrival counter, bounded spin).
// No CTA hands anything to another between rounds: every CTA advances its own
// copy of the schedule state (Sched, in shared memory) from the same global
// inputs, so the copies agree. Appends to the dead log, the AC-4 work list and
// the AC-3 live list go to per-warp shared-memory slices and reach global
// memory with one atomic per counter per CTA per round.
//
// A scheduled run may span several launches (segments): at the start of a
// round every CTA can decide from the same state to stop (the kernel lacks the
// variant the scheduler chose); CTA 0 then saves the schedule state in the
// control block, and the next launch resumes from it at the same round. A
// scheduler that commits to its choice stays in the same kernel: the rounds
// of a committed stretch skip the scheduler and its features (and in the AC-4
// + schedulers flavour may run as local rounds).
#include "trim_internal.cuh"

// This file is compiled once per kernel flavour: TRIM_MODES is a bit set of the
// variants the kernel can run (1 AC-4, 2 AC-6, 4 AC-3) plus 8 for the
// per-round schedulers (features, heuristic, MLP, scripted lists), or 17 for
// in+out trimming. A fixed variant gets a kernel with only its own path,
// hence fewer registers.
#ifndef TRIM_MODES
#define TRIM_MODES 15
#endif
#define TRIM_CAT2(a, b) a##b
#define TRIM_CAT(a, b) TRIM_CAT2(a, b)
#ifdef TRIM_KERNEL_SUFFIX
#define TRIM_KERNEL TRIM_CAT(trim_persistent_kernel_m, TRIM_KERNEL_SUFFIX)
#else
#define TRIM_KERNEL TRIM_CAT(trim_persistent_kernel_m, TRIM_MODES)
#endif

using namespace trimk;

namespace {

constexpr int MODES = TRIM_MODES;
// In the all-variant flavour each round function keeps its own register
// allocation, so the heavier AC-6 code cannot push the AC-4 loop into spills.
#if TRIM_MODES == 15
#define ROUND_FN __noinline__
#else
#define ROUND_FN __forceinline__
#endif
constexpr int M_AC4 = 1, M_AC6 = 2, M_AC3 = 4, M_SCHED = 8;
// in+out trimming: AC-4 pushes on both G^T (out-degree counters) and G
// (in-degree counters); its own flavour, with no other variant
constexpr int M_INOUT = 16;
// implicit graph (Section 2.1, on-the-fly): successors computed, no CSR; with
// AC-6 (34) or AC-3 (36) only
constexpr int M_IMPLICIT = 32;
constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int MAX_WARPS = 16;   // blockDim.x <= 512
constexpr int WBUF = 64;        // per-warp staging of supporting-set members

// Work counters (TRIM_FLAG_STATS). Each round function keeps its own in registers and
// adds a warp's to the CTA's 64-bit totals (stats_flush) before they can pass 2^32: at its
// end where an edge or a vertex counts once, after every round where each round counts
// them again (AC-3).
struct Counters {
  unsigned edges = 0, pushed = 0, cand = 0, swept = 0;
};

// Per-warp append slices. Each warp buffers what it removes (and, in AC-3
// rounds, what survives) in its own slice of shared memory; no shared atomics
// and no CTA-wide synchronisation inside the variant loops. A full slice is
// flushed by its warp alone; at the end of a round one CTA-wide flush moves
// all slices with one global atomic per counter.
constexpr uint32_t LW = 256;  // entries per warp slice (per buffer)
struct WarpSlice {
  uint32_t nlog, nw4, nedge, nlive;   // entries in the slices; edges of the w4 entries
  uint32_t ncount;                    // removals counted in the log but not written to it
  uint32_t log_base, w4_base, edge_base, live_base;  // global bases at the CTA flush
  uint32_t sum_in, sum_out;  // feature sums (distinct removed vertices: at most m < 2^32)
  uint32_t hist[3];
  uint32_t max_din;          // largest in-degree among this warp's work-list entries
};

// Local AC-4 rounds (the AC-4-only flavour, and the AC-4 + schedulers flavour
// inside committed stretches): while the pending work is small,
// each CTA keeps the vertices it removes in a shared-memory queue together with
// their predecessors (their G^T rows, loaded when they are removed) and
// decrements those predecessors' counters itself in the next round. A round then
// needs neither the dead log nor the work list in global memory, nor space
// reservations, nor a read of the control block: it ends at a barrier that
// carries the round's totals (see local_barrier). A removal that does not fit
// the queue goes to the global lists, and the run returns to ordinary rounds.
//
// In+out trimming (flavour 17) runs local rounds too: its queue holds, per
// removed vertex, the one row that still matters (see inout_round), and per
// queued neighbour which of its two counters the push decrements.
// So does AC-6 (flavours 2 and 34, the ones that run nothing else), with the dead log
// as the queue of all CTAs (see its local_stretch). And so does AC-3 (flavours 4 and 36), with a live list per CTA.
#if TRIM_MODES == 1 || TRIM_MODES == 9
#define TRIM_LOCAL 1
#define TRIM_ASYNC 1
#elif TRIM_MODES == 17 || TRIM_MODES == 2 || TRIM_MODES == 34 || TRIM_MODES == 4 || TRIM_MODES == 36
#define TRIM_LOCAL 1
#define TRIM_ASYNC 0
#else
#define TRIM_LOCAL 0
#define TRIM_ASYNC 0
#endif
#define TRIM_AC6_ONLY (TRIM_MODES == 2 || TRIM_MODES == 34)
#define TRIM_AC3_ONLY (TRIM_MODES == 4 || TRIM_MODES == 36)
#if TRIM_LOCAL
constexpr uint32_t LQ_EDGES = 1024;   // predecessors queued per CTA per round
constexpr uint32_t LQ_ENTRIES = 256;  // removed vertices queued per CTA per round
constexpr uint32_t LQ_FLOOR = 512;     // least bound of a stretch's queues
constexpr uint32_t LQ_SKEW = 4;        // ... and the bound as a multiple of the mean load
constexpr uint32_t LQ_LATE_MIN = 1u << 14;  // from here on offsets are loaded for removals only
constexpr uint32_t LQ_DMAX = 64;      // larger in-degrees always go to the global work list
#endif
#if TRIM_ASYNC
// asynchronous AC-4 tail (see async_tail)
constexpr uint32_t ASYNC_MIN_ROUND = 128;  // rounds before the tail may take over
constexpr uint32_t ASYNC_RETRY = 64;       // local stretches end for it at multiples of this
constexpr uint32_t AQ_LOCAL_DMAX = 1024; // larger in-degrees always go to the global pieces
constexpr uint32_t AQ_PIECE = 32;        // in-edges per piece of a CTA's ring (one batch)
constexpr uint32_t ASYNC_LOOK = 128;     // rows handed on by a CTA before the first look at the tail's worth
constexpr uint32_t ASYNC_PATIENCE = 16;  // ... and turns of its control warp with a crowded ring
constexpr uint32_t ASYNC_CLOSE = 192;  // ... and rebalances in a row at most four levels apart that end it
constexpr uint32_t ASYNC_WAIT = 128;     // rounds before a tail that was not may start again
#endif

// Per-CTA shared state.
struct Cta {
  Sched S;
  WarpSlice ws[MAX_WARPS];
  unsigned epoch;     // grid barriers passed by this kernel
  unsigned bar_base;  // barrier counter when this kernel started
  unsigned resume;    // this launch continues a run a segment handed over
  unsigned skip;      // continuation launch of a run that needs none: return at once
  unsigned mode;      // trim_variant_t of the run
  unsigned err;
  unsigned w4_wide;   // initial pass: the work-list slices take all four buffers
  unsigned lq_scratch;  // initial pass with a dead mask: deferred heavy rows
  unsigned long long kstat[4];  // TRIM_FLAG_STATS totals of this CTA (see stats_flush)
  uint32_t wbuf[(TRIM_MODES & 2) && !TRIM_AC6_ONLY ? MAX_WARPS : 1][WBUF];  // (AC-6 in schedules)
#if TRIM_LOCAL
#if TRIM_AC3_ONLY
  uint32_t live_n[2];  // local AC-3 rounds: the CTA's live list, by local-round parity
#elif !TRIM_AC6_ONLY
  // local queues, double-buffered by local-round parity: buffer b is filled in
  // the round whose lround parity is b and read in the next one
  uint32_t lq_ids[2][LQ_EDGES];       // predecessors to decrement
  uint32_t lq_row[2][LQ_ENTRIES];     // the queued vertices' G^T rows ...
  uint32_t lq_din[2][LQ_ENTRIES];     // ... and in-degrees
#endif
  unsigned long long lq_cnt[2];       // reserved: entries (low 32) | predecessors (high 32)
  uint32_t lq_vend[2];                // end of the reservations that fit (entries)
  uint32_t lq_k;                      // this round's removals kept local
  uint32_t lq_ovf;                    // 1: a removal of this round went to the global lists
  uint32_t lq_pushed;                 // predecessors decremented from the queue this round
  uint32_t lq_next;                   // how the stretch goes on after the local barrier
#if TRIM_MODES & 16
  uint8_t lq_dir[2][LQ_EDGES];        // 1: the neighbour is a successor (its in-degree counter)
#endif
#endif
#if TRIM_ASYNC
  // asynchronous tail (see async_tail). The ring of row pieces in dynamic
  // shared memory: pieces taken out and put in so far. The idle workers (a bit
  // each), their wake-up barriers and the rows in their mailboxes. What the CTA does next (read by every worker
  // before each batch); the share of the last rebalance still to claim (global
  // entries, rows and pieces); removals and top level not yet published;
  // entries and rows written out by a rebalance; whether the CTA holds a
  // token, asks for a rebalance; rebalances passed; first piece of the global
  // list not yet shared out; batches so far (shows progress); bases of
  // the entries and rows it writes out; its channels' last tags
  uint32_t r_head, r_tail;
  uint32_t a_idle;
  unsigned long long w_bar[MAX_WARPS];
  uint32_t w_rows[MAX_WARPS];
  uint32_t a_next;
  uint32_t sh_elo, sh_ehi, sh_rlo, sh_rhi, sh_plo, sh_phi;
  uint32_t a_removed, a_maxlev;
  uint32_t a_ne, a_nr;
  uint32_t a_token;
  uint32_t a_want;
  uint32_t a_gen;
  uint32_t a_plo;
  uint32_t a_prog;
  uint32_t a_ebase, a_rbase;
  // is the tail worth it (see async_rebalance): the level above which vertices are parked
  // (NIL: none yet); rows handed on since the last rebalance, how many at least bring the
  // next, and the batches before it;
  // the run's removals before the tail; totals of removals and rows and the top level at the
  // last rebalance, and how many of them came soon after each other; turns of the control
  // warp with a crowded ring that bring the next one
  uint32_t a_cap;
  uint32_t a_hand, a_look;
  uint32_t a_base;
  uint32_t a_seen_removed, a_seen_hand;
  uint32_t a_seen_top, a_close;
  uint32_t a_prog0;
  uint32_t a_patience;
  uint32_t ch_sent[32], ch_taken[32];
#endif
};

// This CTA's state, and its copy of the launch's parameters, for the functions that
// are not inlined: they read both from shared memory at known addresses instead of
// through generic pointers (to the state and to the kernel's parameters), and the
// parameters, whose address no longer leaves the kernel, stay in the constant
// bank for the inlined code. Kernel us before and after: AC-3 of 100,000 vertices (23
// rounds) 163.3 and 159.4, in+out of 5,000,011 (1,001 rounds) 7,863 and 7,602, AC-4 of
// 2^24 (2,868 levels) 6,700 and 6,555, 4,096 packed graphs 2,056 and 2,041.
__shared__ Cta cta_state;
__shared__ Dev cta_dev;
// What the two CTAs of an SM take of its 256 KB decides how much is left as L1: with 512
// threads (64 KB of append slices each) and some 200 bytes of scratch they stay within a
// carve-out of 164 KB. Past it the next size is 196 KB, and rounds that push millions of
// edges have a third less L1: in+out of R-MAT 2^23, round 1 in us, 211 with 20 KB of state
// per CTA and 167 with 9 KB.
#if TRIM_LOCAL
static_assert(sizeof(Cta) + sizeof(Dev) + 256 + 1024 + 65536 <= (164 << 10) / 2,
              "the CTA's state pushes the shared memory past the 164 KB carve-out");
#endif

// Are scheduler features gathered in round S.round? The learned scheduler (and
// a round log of a scheduled run) reads them after every round in which it is
// consulted, i.e. every round outside a committed stretch.
__device__ __forceinline__ bool feats_on(const Dev& D, const Sched& S) {
  return (MODES & M_SCHED) && (D.flags & F_NEED_FEATURES) &&
         !(S.cstop != 0u && S.round < S.cstop);
}

// dynamic shared memory: per warp w, 4 slices of LW words at w * 4 * LW:
// dead-log entries | work-list rows | work-list edge offsets (warp-local) | live-list entries
extern __shared__ __align__(16) uint32_t dyn_smem[];  // (AC-6 stages 16-byte records there)
__device__ __forceinline__ uint32_t* slice(unsigned warp, int which) {
  return dyn_smem + (warp * 4u + (unsigned)which) * LW;
}

__device__ __forceinline__ unsigned long long ld_relaxed64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void fence_acq_rel() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ void red_relaxed_add(unsigned* p, unsigned v) {
  asm volatile("red.relaxed.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// A read of data that no other push needs soon: it leaves the L2 first.
__device__ __forceinline__ uint32_t ld_stream(const uint32_t* p) {
  unsigned long long policy;
  uint32_t v;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  asm volatile("ld.global.nc.L2::cache_hint.u32 %0, [%1], %2;"
               : "=r"(v)
               : "l"(p), "l"(policy));
  return v;
}

// ------------------------------------------------------------------ rows

#if TRIM_MODES & 32
// The implicit planted graph of trim_create_implicit (include/trim.h gives the
// definition): SplitMix64 (Steele, Lea & Flood) as a counter-based generator,
// key(v) = mix(seed ^ mix(salt + v + GAMMA)), word(v, i) = mix(key + (i+1) GAMMA),
// and Lemire's multiply-shift for a uniform integer below k.
constexpr uint64_t IG_GAMMA = 0x9E3779B97F4A7C15ull;
__device__ __forceinline__ uint64_t ig_mix(uint64_t z) {
  z ^= z >> 30;
  z *= 0xBF58476D1CE4E5B9ull;
  z ^= z >> 27;
  z *= 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__device__ __forceinline__ uint64_t ig_word(const Dev& D, uint32_t v, uint64_t i) {
  const uint64_t key = ig_mix(D.ig.seed ^ ig_mix(D.ig.salt + v + IG_GAMMA));
  return ig_mix(key + (i + 1ull) * IG_GAMMA);
}
__device__ __forceinline__ uint32_t ig_below(uint64_t w, uint64_t k) {
  return (uint32_t)__umul64hi(w, k);
}
// number of successors of v
__device__ uint32_t ig_degree(const Dev& D, uint32_t v) {
  const trim_implicit_graph_t& g = D.ig;
  const uint64_t w0 = ig_word(D, v, 0);
  const uint32_t nCR = g.nC + g.nR;
  if (v < g.nC) return g.c_kmin + ig_below(w0, (uint64_t)g.c_kmax - g.c_kmin + 1u);
  if (v < nCR) return g.r_kmin + ig_below(w0, (uint64_t)g.r_kmax - g.r_kmin + 1u);
  const uint32_t rank = v - nCR;
  const uint32_t k = g.t_kmin + ig_below(w0, (uint64_t)g.t_kmax - g.t_kmin + 1u);
  if (g.n_chains == 0u) return rank < g.t_sinks ? 0u : k;
  return rank < g.n_chains ? 0u : 1u + k;
}
// successor j of v (j below its degree)
__device__ uint32_t ig_successor(const Dev& D, uint32_t v, uint32_t j) {
  const trim_implicit_graph_t& g = D.ig;
  const uint64_t w = ig_word(D, v, 1ull + j);
  const uint32_t nCR = g.nC + g.nR;
  if (v < g.nC) return ig_below(w, g.nC);
  if (v < nCR) return ig_below(w, j == 0u ? g.nC : nCR);
  const uint32_t rank = v - nCR;
  if (g.n_chains == 0u) return nCR + ig_below(w, rank);
  if (j == 0u) return v - g.n_chains;
  return nCR + ig_below(w, (uint64_t)(rank / g.n_chains) * g.n_chains);
}
#endif

// Row access of the scans: out-CSR loads, or computed successors on an
// implicit graph (where s is unused).
__device__ __forceinline__ void row_bounds(const Dev& D, uint32_t v, uint32_t& s, uint32_t& d) {
#if TRIM_MODES & 32
  s = 0u;
  d = ig_degree(D, v);
#else
  s = __ldg(&D.off[v]);
  d = __ldg(&D.off[v + 1]) - s;
#endif
}
__device__ __forceinline__ uint32_t row_target(const Dev& D, uint32_t v, uint32_t s, uint32_t j) {
#if TRIM_MODES & 32
  (void)s;
  return ig_successor(D, v, j);
#else
  (void)v;
  return __ldg(&D.tgt[s + j]);
#endif
}

// ------------------------------------------------------------------ appends

// Warp-collective: writes the chunk-owner index of the work-list entries the
// lanes hold: every chunk start 32c inside an entry's edge range [es, ee) is
// owned by that entry (pos). An entry with at most two chunk starts marks them
// itself; a longer one (a hub) is marked by the whole warp, so one lane never
// serialises thousands of stores.
__device__ __forceinline__ void mark_chunks(const Dev& D, bool has, uint32_t pos, uint32_t es,
                                            uint32_t ee) {
  const uint32_t c0 = (es + 31u) >> 5, c1 = (ee + 31u) >> 5;  // chunk starts in [es, ee)
  const bool big = has && c1 > c0 + 2u;
  if (has && !big) {
    if (c0 < c1) D.chunk_first[c0] = pos;
    if (c0 + 1u < c1) D.chunk_first[c0 + 1u] = pos;
  }
  unsigned bm = __ballot_sync(FULL, big);
  while (bm) {
    const int j = __ffs(bm) - 1;
    bm &= bm - 1u;
    const uint32_t p = __shfl_sync(FULL, pos, j), a = __shfl_sync(FULL, c0, j),
                   z = __shfl_sync(FULL, c1, j);
    for (uint32_t c = a + lane_id(); c < z; c += 32u) D.chunk_first[c] = p;
  }
}

// AC-4 work-list slices of a warp: G^T row starts and in-edge offsets. The
// initial pass writes no dead log and no live list, so there they span two
// buffers each (rows over buffers 0-1, offsets over 2-3): fewer warp flushes.
__device__ __forceinline__ uint32_t* w4_rows(const Cta& B, unsigned warp) {
  return slice(warp, B.w4_wide ? 0 : 1);
}
__device__ __forceinline__ uint32_t w4_cap(const Cta& B) { return B.w4_wide ? 2u * LW : LW; }

// One push from a removed vertex to its neighbour u: the predecessor's
// live-successor counter. In+out trimming keeps both counters of a vertex in one
// word (in-degree << 32 | out-degree); dir 1 pushes to a successor's in-degree
// counter. The old word then tells at once whether this push removes u: its
// counter went from one to zero and the other had not reached zero before (which
// would have removed u already).
#if TRIM_MODES & 16
using PushWord = unsigned long long;
__device__ __forceinline__ PushWord push(const Dev& D, uint32_t u, uint32_t dir) {
  return atomicAdd(&D.cnt_io[u], dir ? 0ull - (1ull << 32) : ~0ull);
}
__device__ __forceinline__ bool push_removes(PushWord old, uint32_t dir) {
  const uint32_t o = (uint32_t)old, i = (uint32_t)(old >> 32);
  return dir ? i == 1u && o != 0u : o == 1u && i != 0u;
}
// the row of a vertex removed by pushes of direction dir, whose entries get pushes of the same one
__device__ __forceinline__ const uint32_t* push_off(const Dev& D, uint32_t dir) {
  return dir ? D.off : D.ioff;
}
__device__ __forceinline__ const uint32_t* push_tgt(const Dev& D, uint32_t dir) {
  return dir ? D.tgt : D.itgt;
}
// stats runs: the in-edges and out-edges of a removed vertex
__device__ __forceinline__ void count_rows(const Dev& D, bool removed, uint32_t u, Counters& K) {
  if (!(D.flags & F_STATS) || !removed) return;
  K.pushed += __ldg(&D.ioff[u + 1]) - __ldg(&D.ioff[u]);
  K.edges += __ldg(&D.off[u + 1]) - __ldg(&D.off[u]);
}
#else
using PushWord = uint32_t;
__device__ __forceinline__ PushWord push(const Dev& D, uint32_t u, uint32_t) {
  return atomicSub(&D.cnt[u], 1u);
}
__device__ __forceinline__ bool push_removes(PushWord old, uint32_t) { return old == 1u; }
__device__ __forceinline__ const uint32_t* push_off(const Dev& D, uint32_t) { return D.ioff; }
__device__ __forceinline__ const uint32_t* push_tgt(const Dev& D, uint32_t) { return D.itgt; }
#endif

// Warp-collective: copies this warp's slices to global memory at the given bases.
__device__ __forceinline__ void copy_slices(const Dev& D, const Cta& B, const WarpSlice& w,
                                            unsigned warp, uint32_t* live_out) {
  const unsigned lane = lane_id();
  const uint32_t* sl = slice(warp, 0);
  const uint32_t* sr = w4_rows(B, warp);
  const uint32_t* se = slice(warp, 2);
  const uint32_t* sv = slice(warp, 3);
  for (uint32_t i = lane; i < w.nlog; i += 32) D.log[w.log_base + i] = sl[i];
  for (uint32_t i0 = 0; i0 < w.nw4; i0 += 32) {  // warp-uniform loop: mark_chunks is collective
    const uint32_t i = i0 + lane;
    const bool has = i < w.nw4;
    uint32_t eo = 0, ee = 0;
    if (has) {
      eo = w.edge_base + se[i];
      ee = w.edge_base + (i + 1 < w.nw4 ? se[i + 1] : w.nedge);
      D.w4_row[w.w4_base + i] = sr[i];
      D.w4_eoff[w.w4_base + i] = eo;
      if (MODES & M_INOUT) D.w4_dir[w.w4_base + i] = sl[i];  // in+out: the row's direction
    }
    mark_chunks(D, has, w.w4_base + i, eo, ee);
  }
  for (uint32_t i = lane; i < w.nlive; i += 32) live_out[w.live_base + i] = sv[i];
}

// Warp-collective: a slice is full; the warp reserves global space on its own.
__device__ __noinline__ void warp_flush(uint32_t r, uint32_t* live_out) {
  const Dev& D = cta_dev;
  Cta& B = cta_state;
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  WarpSlice& w = B.ws[warp];
  // three lanes reserve at once; removals that are only counted (nlog = 0)
  // wait for the CTA flush
  if (lane == 0 && w.nlog) {
    w.log_base = atomicAdd(&D.C->log_len, w.nlog + w.ncount);
    if (w.log_base + w.nlog + w.ncount > D.n) { set_error(D, TRIM_ERR_STATE, 0xD1); w.nlog = 0; }
    w.ncount = 0;
  }
  if (lane == 1 && w.nw4) {
    const unsigned long long o = atomicAdd(
        &D.C->w4, (unsigned long long)w.nw4 | ((unsigned long long)w.nedge << 32));
    w.w4_base = (uint32_t)o;
    w.edge_base = (uint32_t)(o >> 32);
    // (the words of in+out trimming stop a second removal of a vertex only if
    // G^T is the transpose of G)
    if ((MODES & M_INOUT) && w.w4_base + w.nw4 > D.n) {
      set_error(D, TRIM_ERR_STATE, 0xD7);
      w.nw4 = 0;
    }
  }
  if (lane == 2 && w.nlive) {
    w.live_base = atomicAdd(&D.C->rs[r & 3].live_count, w.nlive);
    if (w.live_base + w.nlive > D.n) { set_error(D, TRIM_ERR_STATE, 0xD3); w.nlive = 0; }
  }
  __syncwarp();
  const WarpSlice c = w;
  copy_slices(D, B, c, warp, live_out);
  __syncwarp();
  if (lane == 0) w.nlog = w.nw4 = w.nedge = w.nlive = 0;
  __syncwarp();
}

// Warp-collective: lanes with pred are removed in round r: level[u] = r and u
// joins F_r in the dead log; if it has in-edges (and AC-4 may run) it also
// joins the AC-4 work list with its G^T row and in-degree. With pre, the caller
// has already loaded u's G^T row start (prow) and in-degree (pdin). dout is u's
// out-degree where the caller knows it (AC-3/AC-6 scans; 0 for AC-4, which
// never loads it): it only feeds the scheduler's live-edge count without G^T.
__device__ __forceinline__ void append_dead(const Dev& D, Cta& B, bool pred, uint32_t u,
                                            uint32_t r, uint32_t* live_out,
                                            bool initial = false, bool pre = false,
                                            uint32_t prow = 0, uint32_t pdin = 0,
                                            uint32_t dout = 0) {
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  const unsigned mask = __ballot_sync(FULL, pred);
  if (mask == 0u) return;
  const bool feats = feats_on(D, B.S);
  const bool live_edges = feats || (D.flags & F_LIVE_EDGES);
  // whenever the run may use AC-4, every flavour keeps its work list complete
  const bool track = D.ioff != nullptr && ((D.flags & F_AC4_POSSIBLE) || feats);
  uint32_t row = 0, din = 0;
  if (!pred) dout = 0;
  if (pred && track) {
    if (pre) {
      row = prow;
      din = pdin;
    } else {
      row = __ldg(&D.ioff[u]);
      din = __ldg(&D.ioff[u + 1]) - row;
    }
  }
  const bool w = pred && din > 0u && (D.flags & F_AC4_POSSIBLE);
  const unsigned wmask = __ballot_sync(FULL, w);
  const unsigned lt = (1u << lane) - 1u;
  const unsigned k = __popc(mask), kw = __popc(wmask);
  const unsigned ew = w ? din : 0u;
  const unsigned eincl = warp_incl_scan(ew);
  const unsigned esum = __shfl_sync(FULL, eincl, 31);
  WarpSlice& ws = B.ws[warp];
  const unsigned kl = initial ? 0u : k;  // F_0 is only counted: no variant reads it back
  if (ws.nlog + kl > LW || ws.nw4 + kw > w4_cap(B)) warp_flush(r, live_out);
  const uint32_t pl = ws.nlog, pw = ws.nw4, pe = ws.nedge;
  if (pred && !initial) {
    slice(warp, 0)[pl + __popc(mask & lt)] = u;
    D.level[u] = r;
  }
  unsigned mdin = 0;
  if (wmask) {
    mdin = __reduce_max_sync(FULL, ew);
    if (w) {
      const unsigned at = pw + __popc(wmask & lt);
      w4_rows(B, warp)[at] = row;
      slice(warp, 2)[at] = pe + eincl - ew;
    }
  }
  unsigned s_in = 0, s_out = 0;
  unsigned h0 = 0, h1 = 0;
  if (live_edges) s_out = __reduce_add_sync(FULL, dout);
  if (feats) {
    s_in = __reduce_add_sync(FULL, din);
    h0 = __popc(__ballot_sync(FULL, pred && din < 8u));
    h1 = __popc(__ballot_sync(FULL, pred && din >= 8u && din < 256u));
  }
  __syncwarp();
  if (lane == 0) {
    ws.nlog = pl + kl;
    ws.ncount += k - kl;
    ws.nw4 = pw + kw;
    ws.nedge = pe + esum;
    ws.max_din = max(ws.max_din, mdin);
    if (live_edges) ws.sum_out += s_out;
    if (feats) {
      ws.sum_in += s_in;
      ws.hist[0] += h0;
      ws.hist[1] += h1;
      ws.hist[2] += k - h0 - h1;
    }
  }
  __syncwarp();
}

// Warp-collective append of survivors to the AC-3 output live list.
__device__ __forceinline__ void append_live(const Dev& D, Cta& B, bool pred, uint32_t v,
                                            uint32_t r, uint32_t* out_list) {
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  const unsigned mask = __ballot_sync(FULL, pred);
  if (mask == 0u) return;
  const unsigned k = __popc(mask);
  WarpSlice& ws = B.ws[warp];
  if (ws.nlive + k > LW) warp_flush(r, out_list);
  const uint32_t pv = ws.nlive;
  if (pred) slice(warp, 3)[pv + __popc(mask & ((1u << lane) - 1u))] = v;
  __syncwarp();
  if (lane == 0) ws.nlive = pv + k;
  __syncwarp();
}

#if TRIM_LOCAL && !TRIM_AC6_ONLY && !TRIM_AC3_ONLY
// Warp-collective: lanes with pred add a work-list entry (row start, length; in+out
// trimming: and direction) of a vertex that is already removed and counted.
__device__ __forceinline__ void append_w4(const Dev& D, Cta& B, bool pred, uint32_t row,
                                          uint32_t din, uint32_t r, uint32_t dir) {
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  const bool w = pred && din > 0u;
  const unsigned wmask = __ballot_sync(FULL, w);
  if (wmask == 0u) return;
  const unsigned kw = __popc(wmask);
  const unsigned ew = w ? din : 0u;
  const unsigned eincl = warp_incl_scan(ew);
  const unsigned esum = __shfl_sync(FULL, eincl, 31);
  WarpSlice& ws = B.ws[warp];
  if (ws.nw4 + kw > w4_cap(B)) warp_flush(r, D.live0);
  const uint32_t pw = ws.nw4, pe = ws.nedge;
  const unsigned mdin = __reduce_max_sync(FULL, ew);
  if (w) {
    const unsigned at = pw + __popc(wmask & ((1u << lane) - 1u));
    w4_rows(B, warp)[at] = row;
    slice(warp, 2)[at] = pe + eincl - ew;
    if (MODES & M_INOUT) slice(warp, 0)[at] = dir;
  }
  __syncwarp();
  if (lane == 0) {
    ws.nw4 = pw + kw;
    ws.nedge = pe + esum;
    ws.max_din = max(ws.max_din, mdin);
  }
  __syncwarp();
}

#if TRIM_MODES & 16
// Warp-collective, in+out trimming: lanes with pred were removed in this round
// (their level is already set) by pushes of direction dir; each joins the work list with
// its row of that direction. Removals are only counted in the dead log, never
// written: no variant of this flavour reads it.
__device__ __forceinline__ void append_dead_io(const Dev& D, Cta& B, bool pred, uint32_t r,
                                               uint32_t row, uint32_t len, uint32_t dir) {
  const unsigned mask = __ballot_sync(FULL, pred);
  if (mask == 0u) return;
  append_w4(D, B, pred, row, len, r, dir);
  if (lane_id() == 0) B.ws[threadIdx.x >> 5].ncount += __popc(mask);
  __syncwarp();
}
#endif

// Warp-collective, local rounds: lanes with pred remove u in round r (its G^T
// row start and in-degree already loaded). A removal with at most LQ_DMAX
// in-edges that fits this CTA's queue (buffer b) stays local: its G^T row is
// copied into the queue now, all of the warp's rows at once (each lane loads
// entries of the flattened rows, so the loads overlap). Everything else takes
// the global path of an ordinary round (dead log, work list) and marks the
// round as overflowing.
__device__ __forceinline__ void local_append(const Dev& D, Cta& B, bool pred, uint32_t u,
                                             uint32_t r, uint32_t row, uint32_t din,
                                             uint32_t b, uint32_t dir, uint32_t cap) {
  const unsigned lane = lane_id();
  const unsigned mask = __ballot_sync(FULL, pred);
  if (mask == 0u) return;
  if (pred) D.level[u] = r;
  const bool want = pred && din > 0u && din <= LQ_DMAX;
  const unsigned wm = __ballot_sync(FULL, want);
  bool ovf = pred && din > LQ_DMAX;
  if (wm) {
    const unsigned ew = want ? din : 0u;
    const unsigned eincl = warp_incl_scan(ew);
    const unsigned esum = __shfl_sync(FULL, eincl, 31);
    const unsigned excl = eincl - ew;
    const unsigned k = __popc(wm);
    unsigned long long old = 0;
    if (lane == 0)
      old = atomicAdd(&B.lq_cnt[b], (unsigned long long)k | ((unsigned long long)esum << 32));
    old = __shfl_sync(FULL, old, 0);
    const uint32_t be = (uint32_t)old, bd = (uint32_t)(old >> 32);
    if (be + k <= LQ_ENTRIES && bd + esum <= cap) {  // warp-uniform
      if (lane == 0) atomicMax(&B.lq_vend[b], be + k);
      if (want) {
        const uint32_t slot = be + __popc(wm & ((1u << lane) - 1u));
        B.lq_row[b][slot] = row;
        B.lq_din[b][slot] = din | (dir << 31);
      }
      // predecessors: element j of the flattened rows belongs to the lane with
      // the largest exclusive prefix <= j; four loads in flight per lane
      for (uint32_t j0 = 0; j0 < esum; j0 += 128u) {
        uint32_t t[4], to[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint32_t j = j0 + (uint32_t)q * 32u + lane;
          const unsigned o = owner_of(excl, j);
          const uint32_t ro = __shfl_sync(FULL, row, o), xo = __shfl_sync(FULL, excl, o);
          to[q] = (MODES & M_INOUT) ? __shfl_sync(FULL, dir, o) : 0u;
          t[q] = j < esum ? __ldg(&push_tgt(D, to[q])[ro + (j - xo)]) : 0u;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint32_t j = j0 + (uint32_t)q * 32u + lane;
          if (j < esum) B.lq_ids[b][bd + j] = t[q];
#if TRIM_MODES & 16
          if (j < esum) B.lq_dir[b][bd + j] = (uint8_t)to[q];
#endif
        }
      }
    } else {
      ovf = ovf || want;
    }
  }
  const unsigned om = __ballot_sync(FULL, ovf);
  if (lane == 0) {
    atomicAdd(&B.lq_k, (unsigned)__popc(mask & ~om));
    if (om) B.lq_ovf = 1u;
  }
#if TRIM_MODES & 16
  append_dead_io(D, B, ovf, r, row, din, dir);
#else
  append_dead(D, B, ovf, u, r, D.live0, false, true, row, din);
#endif
}
#endif

// End of round r: moves every warp slice of the CTA to global memory with one
// global atomic per counter (all threads of the CTA). The (up to three) space
// reservations are issued by three lanes at once, so they cost one round trip.
__device__ void flush_round(const Dev& D, Cta& B, uint32_t r, uint32_t* live_out) {
  __syncthreads();
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (warp == 0) {
    // exclusive prefix of the per-warp counts (lane i holds warp i)
    const bool has = lane < nw;
    const uint32_t a = has ? B.ws[lane].nlog + B.ws[lane].ncount : 0u,
                   b = has ? B.ws[lane].nw4 : 0u, c = has ? B.ws[lane].nedge : 0u,
                   d = has ? B.ws[lane].nlive : 0u;
    const uint32_t ia = warp_incl_scan(a), ib = warp_incl_scan(b), ic = warp_incl_scan(c),
                   id = warp_incl_scan(d);
    const uint32_t ta = __shfl_sync(FULL, ia, 31), tb = __shfl_sync(FULL, ib, 31),
                   tc = __shfl_sync(FULL, ic, 31), td = __shfl_sync(FULL, id, 31);
    RoundStat* rs = &D.C->rs[r & 3];
    unsigned long long got = 0;
    if (lane == 0 && ta) got = atomicAdd(&D.C->log_len, ta);
    if (lane == 1 && tb)
      got = atomicAdd(&D.C->w4, (unsigned long long)tb | ((unsigned long long)tc << 32));
    if (lane == 2 && td) got = atomicAdd(&rs->live_count, td);
    uint32_t lb = (uint32_t)__shfl_sync(FULL, got, 0);
    const unsigned long long w4o = __shfl_sync(FULL, got, 1);
    uint32_t vb = (uint32_t)__shfl_sync(FULL, got, 2);
    const uint32_t wb = (uint32_t)w4o, eb = (uint32_t)(w4o >> 32);
    if (ta && lb + ta > D.n) {
      if (lane == 0) set_error(D, TRIM_ERR_STATE, 0xD5);
      lb = 0xFFFFFFFFu;
    }
    if (td && vb + td > D.n) {
      if (lane == 0) set_error(D, TRIM_ERR_STATE, 0xD6);
      vb = 0xFFFFFFFFu;
    }
    const bool feats = feats_on(D, B.S);
    if (feats || (D.flags & F_LIVE_EDGES)) {
      const uint32_t s_out = __reduce_add_sync(FULL, has ? B.ws[lane].sum_out : 0u);
      if (lane == 4 && s_out) atomicAdd(&rs->sum_out, (unsigned long long)s_out);
    }
    {
      const uint32_t md = __reduce_max_sync(FULL, has ? B.ws[lane].max_din : 0u);
      if (lane == 8 && md) atomicMax(&rs->max_din, md);
    }
    if (feats) {
      const uint32_t s_in = __reduce_add_sync(FULL, has ? B.ws[lane].sum_in : 0u);
      uint32_t h[3];
      for (int i = 0; i < 3; ++i) h[i] = __reduce_add_sync(FULL, has ? B.ws[lane].hist[i] : 0u);
      // independent reductions from separate lanes (no return value: no wait)
      if (lane == 3 && s_in) atomicAdd(&rs->sum_in, (unsigned long long)s_in);
      if (lane >= 5 && lane < 8 && h[lane - 5]) atomicAdd(&rs->hist[lane - 5], h[lane - 5]);
    }
    if (has) {
      WarpSlice& w = B.ws[lane];
      w.log_base = lb + ia - a;
      w.w4_base = wb + ib - b;
      w.edge_base = eb + ic - c;
      w.live_base = vb + id - d;
      if (lb == 0xFFFFFFFFu) w.nlog = 0;
      if ((MODES & M_INOUT) && wb + tb > D.n) {  // as in warp_flush
        set_error(D, TRIM_ERR_STATE, 0xD7);
        w.nw4 = 0;
      }
      if (vb == 0xFFFFFFFFu) w.nlive = 0;
    }
  }
  __syncthreads();
  const WarpSlice c = B.ws[warp];
  copy_slices(D, B, c, warp, live_out);
  __syncwarp();
  if (lane == 0) {
    WarpSlice& w = B.ws[warp];
    w.nlog = w.nw4 = w.nedge = w.nlive = w.ncount = 0;
    w.sum_in = w.sum_out = 0;
    w.hist[0] = w.hist[1] = w.hist[2] = 0;
    w.max_din = 0;
  }
}

// ------------------------------------------------------------------ grid barrier

// Grid-wide barrier: each CTA adds one arrival to a monotone counter and waits
// until all gridDim.x arrivals of this epoch are in (counted from the value the
// counter had when this kernel started: a resumed segment continues it). The
// wait is bounded by spin_limit_ns; past it the run stops with
// TRIM_ERR_TIMEOUT. Returns false if the run must stop (any error flag).
// With read_err false the error flag is not read here: the round loop reads it
// in advance(), together with the round's counters (one memory round trip less).
__device__ bool grid_barrier(const Dev& D, Cta& B, bool read_err = true) {
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned target = B.bar_base + (++B.epoch) * gridDim.x;
    fence_acq_rel();
    red_relaxed_add(&D.C->bar, 1u);
    const uint64_t t0 = globaltimer();
    // relaxed polls, then one acquiring load once every arrival is in (an
    // acquiring load per poll would invalidate this SM's L1 every time)
    while ((int)(ld_relaxed(&D.C->bar) - target) < 0) {
      if (globaltimer() - t0 > D.spin_limit_ns) {
        set_error(D, TRIM_ERR_TIMEOUT, 1);
        B.err = TRIM_ERR_TIMEOUT;
        break;
      }
    }
    (void)ld_acquire(&D.C->bar);
    if (read_err) B.err = ld_relaxed(&D.C->err);
  }
  __syncthreads();
  return B.err == 0u;
}

// Warp-collective: adds this warp's counters to the run totals (stats runs only).
// The CTA's totals stay in shared memory for the whole launch and reach the
// global counters once, when the kernel ends (stats_publish): no global
// atomics per warp and round.
__device__ __forceinline__ void stats_flush(const Dev& D, Cta& B, const Counters& K) {
  if (!(D.flags & F_STATS)) return;
  // (a warp's counts since the last call: below 2^32, see Counters)
  const unsigned e = __reduce_add_sync(FULL, K.edges), p = __reduce_add_sync(FULL, K.pushed),
                 c = __reduce_add_sync(FULL, K.cand), s = __reduce_add_sync(FULL, K.swept);
  if (lane_id() == 0) {
    if (e) atomicAdd(&B.kstat[0], (unsigned long long)e);
    if (p) atomicAdd(&B.kstat[1], (unsigned long long)p);
    if (c) atomicAdd(&B.kstat[2], (unsigned long long)c);
    if (s) atomicAdd(&B.kstat[3], (unsigned long long)s);
  }
}

__device__ __forceinline__ void stats_publish(const Dev& D, Cta& B) {
  if (!(D.flags & F_STATS)) return;
  __syncthreads();
  if (threadIdx.x < 4 && B.kstat[threadIdx.x]) atomicAdd(&D.C->stats[threadIdx.x], B.kstat[threadIdx.x]);
}

// ------------------------------------------------------------------ scans

// Thread-level forward scan of v's successors from position i (row start s,
// length d): returns the first position whose target is not removed before
// round r, or d. At most `batches` x 4 edges; *resolved tells whether it ended.
__device__ __forceinline__ uint32_t scan_thread(const Dev& D, uint32_t v, uint32_t s, uint32_t d,
                                                uint32_t i, uint32_t r, int batches,
                                                bool& resolved, Counters& K) {
  for (int b = 0; b < batches; ++b) {
    if (i >= d) { resolved = true; return d; }
    const uint32_t nb = min(4u, d - i);
    uint32_t t[4], lv[4];
#if TRIM_MODES & 32
#pragma unroll
    for (int q = 0; q < 4; ++q) t[q] = (q < (int)nb) ? row_target(D, v, s, i + q) : 0u;
#else
    // four targets on a 16-byte boundary (of the address: a caller's array may
    // start anywhere) come with one load
    if (nb == 4u && (reinterpret_cast<uintptr_t>(D.tgt + s + i) & 15u) == 0u) {
      const uint4 x = __ldg(reinterpret_cast<const uint4*>(D.tgt + s + i));
      t[0] = x.x; t[1] = x.y; t[2] = x.z; t[3] = x.w;
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) t[q] = (q < (int)nb) ? __ldg(&D.tgt[s + i + q]) : 0u;
    }
#endif
#pragma unroll
    for (int q = 0; q < 4; ++q) lv[q] = (q < (int)nb) ? ldcg(&D.level[t[q]]) : 0u;
    K.edges += nb;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < (int)nb && lv[q] >= r) { resolved = true; return i + q; }
    i += nb;
  }
  resolved = (i >= d);
  return i;
}

// Warp-collective: finishes the scans of lanes with !resolved, one lane at a
// time, 32 successors per step (ballot picks the first live one).
__device__ __forceinline__ void scan_warp_finish(const Dev& D, bool& resolved, uint32_t v,
                                                 uint32_t s, uint32_t d, uint32_t& i, uint32_t r,
                                                 Counters& K) {
  const unsigned lane = lane_id();
  unsigned pend = __ballot_sync(FULL, !resolved);
  while (pend) {
    const int src = __ffs(pend) - 1;
    pend &= pend - 1;
    const uint32_t ss = __shfl_sync(FULL, s, src), dd = __shfl_sync(FULL, d, src);
    const uint32_t vv = __shfl_sync(FULL, v, src);
    uint32_t ii = __shfl_sync(FULL, i, src);
    uint32_t found = dd;
    while (ii < dd) {
      const uint32_t k = ii + lane;
      bool live = false;
      if (k < dd) live = ldcg(&D.level[row_target(D, vv, ss, k)]) >= r;
      const unsigned b = __ballot_sync(FULL, live);
      if (lane == 0) K.edges += min(32u, dd - ii);
      if (b) { found = ii + __ffs(b) - 1; break; }
      ii += 32;
    }
    if ((int)lane == src) { i = found; resolved = true; }
  }
}

// ------------------------------------------------------------------ scheduler

__device__ __forceinline__ float log2p1(float x) { return log2f(1.0f + x); }

// Cost rule of TRIM_SCHED_HEURISTIC: the work each variant would do in round
// r+1, in units of one random memory access, with one-time entry costs spread
// over a horizon of H rounds (a greedy rule that charged them to one round
// would never leave a variant whose cost recurs every round).
//   AC-4: pushes every in-edge of the removed vertices it has not processed yet
//         (the backlog beyond the newest frontier is a one-time cost).
//   AC-3: sweeps its live list (all n vertices the first time), every round.
//   AC-6: while it runs, re-scans about one supporting-set member per removed
//         vertex; entering it rebuilds the sets of all live vertices.
__device__ uint32_t heuristic_choice(const Dev& D, const Sched& L, uint32_t nF, uint32_t n_live,
                                     uint32_t w_end, uint32_t e_end) {
  constexpr float H = 4.0f;
  const float inf = 3.0e38f;
  const float eF = (float)(e_end - L.e_end);          // in-edges of the newest frontier
  const float backlog = (float)(e_end - L.e_c4);      // in-edges not yet pushed
  const float items = (float)(w_end - L.c4w);
  float c4 = (L.variant == TRIM_AC4_PUSH) ? eF + 0.25f * items
                                           : (backlog - eF) / H + eF + 0.25f * items;
  const float sweep = (L.ac3_list == NIL) ? (float)D.n : (float)L.live_in_len;
  float c3 = 2.0f * sweep;
  float c6 = (L.variant == TRIM_AC6_SUPPORT)
                 ? 4.0f * (float)nF
                 : (3.0f * (float)n_live + (float)D.n) / H + 4.0f * (float)nF;
  c4 *= D.heur_push_ratio;
  c6 *= D.heur_ac6_ratio;
  if (!(D.flags & F_AC4_POSSIBLE) || D.ioff == nullptr) c4 = inf;
  if (!(D.flags & F_AC6_POSSIBLE)) c6 = inf;
  if (!(D.flags & F_AC3_POSSIBLE)) c3 = inf;
  if (c4 <= c3 && c4 <= c6) return TRIM_AC4_PUSH;
  if (c6 <= c3) return TRIM_AC6_SUPPORT;
  return TRIM_AC3_PULL;
}

// Warp-collective MLP 12 -> 32 -> 32 -> 3 (ReLU) read from the model blob in
// global memory (W1[32][12] b1[32] W2[32][32] b2[32] W3[3][32] b3[3] mean[12]
// istd[12] lo[12] hi[12]; 16-byte aligned): lane j computes hidden unit j of
// each layer from row j of W1 and W2 (float4 loads). It runs only in rounds
// after which the scheduler is consulted, so the model stays out of shared
// memory. Returns the argmax class among the available variants, its softmax
// probability, and whether every feature lies in the model's training range.
__device__ uint32_t mlp_choice(const Dev& D, const float* f, bool* in_range,
                               float* confidence) {
  const unsigned lane = lane_id();
  const float* M = D.model;
  bool ok = true;
  float x[NFEAT];
#pragma unroll
  for (int i = 0; i < NFEAT; ++i) {
    const float mean = __ldg(M + 1571 + i), istd = __ldg(M + 1583 + i);
    const float lo = __ldg(M + 1595 + i), hi = __ldg(M + 1607 + i);
    ok = ok && f[i] >= lo && f[i] <= hi;
    x[i] = (f[i] - mean) * istd;
  }
  const float4* w1 = reinterpret_cast<const float4*>(M + lane * NFEAT);
  float h1 = __ldg(M + 384 + lane);
#pragma unroll
  for (int q = 0; q < NFEAT / 4; ++q) {
    const float4 w = __ldg(w1 + q);
    h1 = fmaf(w.x, x[4 * q], h1);
    h1 = fmaf(w.y, x[4 * q + 1], h1);
    h1 = fmaf(w.z, x[4 * q + 2], h1);
    h1 = fmaf(w.w, x[4 * q + 3], h1);
  }
  h1 = fmaxf(h1, 0.0f);
  const float4* w2 = reinterpret_cast<const float4*>(M + 416 + lane * 32);
  float acc[4] = {__ldg(M + 1440 + lane), 0.0f, 0.0f, 0.0f};  // four independent chains
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const float4 w = __ldg(w2 + q);
    acc[0] = fmaf(w.x, __shfl_sync(FULL, h1, 4 * q), acc[0]);
    acc[1] = fmaf(w.y, __shfl_sync(FULL, h1, 4 * q + 1), acc[1]);
    acc[2] = fmaf(w.z, __shfl_sync(FULL, h1, 4 * q + 2), acc[2]);
    acc[3] = fmaf(w.w, __shfl_sync(FULL, h1, 4 * q + 3), acc[3]);
  }
  const float h2 = fmaxf((acc[0] + acc[1]) + (acc[2] + acc[3]), 0.0f);
  float z[3];
#pragma unroll
  for (int o = 0; o < 3; ++o)
    z[o] = warp_sum(__ldg(M + 1472 + o * 32 + lane) * h2) + __ldg(M + 1568 + o);
  if (D.ioff == nullptr || !(D.flags & F_AC4_POSSIBLE)) z[TRIM_AC4_PUSH] = -3.0e38f;
  if (!(D.flags & F_AC6_POSSIBLE)) z[TRIM_AC6_SUPPORT] = -3.0e38f;
  if (!(D.flags & F_AC3_POSSIBLE)) z[TRIM_AC3_PULL] = -3.0e38f;
  uint32_t best = 0;
  if (z[1] > z[best]) best = 1;
  if (z[2] > z[best]) best = 2;
  // softmax probability of the choice among the available variants
  float den = 0.0f;
#pragma unroll
  for (int o = 0; o < 3; ++o) den += expf(z[o] - z[best]);
  *confidence = 1.0f / den;
  *in_range = ok;
  return best;
}

// Warp 0 of every CTA, after the barrier that ends round r (r = 0: the initial
// sink pass): closes round r in the CTA's copy of the schedule and prepares
// round r+1. Reads only values that are final for every CTA at this point, so
// all copies take the same decisions. CTA 0 also publishes results and logs.
__device__ ROUND_FN void advance(const Dev& D, Cta& B) {
  const unsigned lane = lane_id();
  Ctrl* C = D.C;
  Sched L = B.S;
  const uint32_t r = L.round;
  const RoundStat* rs = &C->rs[r & 3];
  // the scheduler chooses round r+1 unless a committed stretch covers it
  const bool consult = (MODES & M_SCHED) && B.mode > TRIM_AC3_PULL &&
                       !(L.cstop != 0u && r < L.cstop);
  const bool feats = feats_on(D, L);
  const bool logged = (D.flags & F_ROUND_LOG) && D.rlog != nullptr && r >= 1 && r - 1 < D.rlog_cap;
  // every value this step reads from the control block, issued together
  const uint32_t err = ld_relaxed(&C->err);
  // removals so far: logged ones plus those counted only by local rounds
  const uint32_t len = ld_relaxed(&C->log_len) + L.skew;
  const unsigned long long w4 = ld_relaxed64(&C->w4);
  const uint32_t live_count = ld_relaxed(&rs->live_count);
  const uint32_t max_din = ld_relaxed(&rs->max_din);
  unsigned long long sum_in = 0, sum_out = 0, t_r = 0, t_rm1 = 0, local_edges = 0;
  uint32_t h0 = 0, h1 = 0, h2 = 0;
  const bool live_edges = feats || (D.flags & F_LIVE_EDGES);
  // with G^T and a complete AC-4 work list the live-edge count follows from
  // running totals (the scheduler flavours keep it without F_LIVE_EDGES)
  const bool by_counts = D.ioff != nullptr && (D.flags & F_AC4_POSSIBLE) &&
                         ((MODES & M_SCHED) || live_edges);
  if (live_edges) sum_out = ld_relaxed64(&rs->sum_out);
  if (by_counts) local_edges = ld_relaxed64(&C->local_edges);
  if (feats) {
    sum_in = ld_relaxed64(&rs->sum_in);
    h0 = ld_relaxed(&rs->hist[0]);
    h1 = ld_relaxed(&rs->hist[1]);
    h2 = ld_relaxed(&rs->hist[2]);
    t_rm1 = ld_relaxed64(&C->t_round[(r - 1) & 3]);
  }
  if (feats || logged) t_r = ld_relaxed64(&C->t_round[r & 3]);
  const uint32_t w_end = (uint32_t)w4, e_end = (uint32_t)(w4 >> 32);
  const uint32_t nF = len - L.fe;  // |F_r|
  const bool cta0 = blockIdx.x == 0 && lane == 0;
  if (r >= 1) {
    if (L.variant <= 2u) L.vcount[L.variant] += 1;
    if (cta0) {
      if (L.variant <= 2u) C->vcount[L.variant] = L.vcount[L.variant];
      if (logged) {
        trim_round_rec_t* rec = &D.rlog[r - 1];
        rec->round = r;
        rec->variant = L.variant;
        rec->frontier = L.fe - L.fb;
        rec->removed = nF;
        rec->t_start_ns = t_r;
        rec->t_end_ns = globaltimer();
        rec->t_work_ns = ld_relaxed64(&C->t_work[r & 3]);
        rec->t_flush_ns = ld_relaxed64(&C->t_flush[r & 3]);
        for (int i = 0; i < NFEAT; ++i) rec->features[i] = L.feat[i];
        C->rlog_len = r;
      }
    }
    if (L.variant == TRIM_AC4_PUSH) {  // pushed every work-list entry that existed before round r
      L.c4w = L.w_end;
      L.e_c4 = L.e_end;
      L.bmax = 0;
    }
    if (L.variant == TRIM_AC3_PULL) {
      L.ac3_list = L.live_out;
      L.live_in_len = live_count;
    }
    // the first AC-6 or AC-3 round wrote the support position of every vertex
    // still live (both sweep all live vertices when they first run)
    if (L.variant == TRIM_AC6_SUPPORT || L.variant == TRIM_AC3_PULL) L.supp_valid = 1u;
  }
  L.bmax = max(L.bmax, max_din);  // the entries of F_r join the AC-4 backlog
  if (cta0) {
    C->rounds = nF ? r + 1 : r;
    C->n_dead = len;
  }
  // live-edge count. With G^T and a complete AC-4 work list: edges between live
  // vertices = m minus the in-edges of removed vertices (a removed vertex has
  // only removed successors, so every edge that touches one ends in one).
  // Otherwise: with G^T, the same from the in-degree sums; without it, out-edges
  // of live vertices (AC-3/AC-6 know each removed vertex's degree).
  // (in-edges pushed from local queues belong to removed vertices without
  // work-list entries)
  if (by_counts) L.m_live = (unsigned long long)D.m - e_end - local_edges;
  else if (live_edges) L.m_live -= (D.ioff != nullptr) ? sum_in : sum_out;
  if (nF == 0) {
    L.done = 1;
  } else {
    const uint32_t n_live = D.n - len;
    float f[NFEAT];
    for (int i = 0; i < NFEAT; ++i) f[i] = 0.0f;
    if (feats) {
      f[0] = log2p1((float)nF);
      f[1] = log2p1((float)sum_in);
      f[2] = log2p1((float)(e_end - L.e_c4));  // in-edges AC-4 has not pushed yet
      f[3] = log2p1((float)n_live);
      f[4] = log2p1((float)L.m_live);
      f[5] = (float)nF / (float)max(1u, n_live);
      f[6] = (float)sum_in / (float)max(1ull, L.m_live);
      f[7] = (float)h0 / (float)nF;
      f[8] = (float)h1 / (float)nF;
      f[9] = (float)h2 / (float)nF;
      // time of round r-1 per vertex of its frontier (CTA 0's clock, published to all)
      f[10] = (r >= 2) ? log2p1((float)(t_r - t_rm1) / (float)max(1u, L.fprev)) : 0.0f;
      f[11] = (r >= 1) ? (float)L.variant : -1.0f;  // the variant whose state is current
    }
    uint32_t next;
    bool confident = false;  // the learned scheduler may commit at once
    if (!(MODES & M_SCHED) || B.mode <= TRIM_AC3_PULL) {
      next = B.mode;
    } else if (!consult) {
      next = L.variant;  // inside a committed stretch
    } else if (B.mode == TRIM_SCHED_SCRIPTED) {
      next = D.script_len ? D.script[r % D.script_len] : 0u;
      if (next > 2u) next = TRIM_AC3_PULL;
      if (next == TRIM_AC4_PUSH && D.ioff == nullptr) next = TRIM_AC3_PULL;
    } else {
      next = heuristic_choice(D, L, nF, n_live, w_end, e_end);
      if (B.mode == TRIM_SCHED_LEARNED && D.model != nullptr) {
        bool in_range = false;
        float conf = 0.0f;
#if TRIM_MODES & 8
        const uint32_t learned = mlp_choice(D, f, &in_range, &conf);
#else
        const uint32_t learned = next;
#endif
        if (in_range) {
          next = learned;
          confident = D.commit_confidence > 0.0f && conf >= D.commit_confidence;
        }
      }
    }
    // rounds in a row with an unchanged choice. After commit_after of them
    // (or a learned choice at or above commit_confidence) the run commits: the
    // next recheck_rounds rounds (doubling while the same commit repeats) run
    // the variant without consulting the scheduler or gathering features, and
    // the count stays one short of a commit, so that the first consulted round
    // after the stretch re-commits if the scheduler keeps the variant.
    if (!consult) {
      L.stable = D.commit_after ? D.commit_after - 1u : 0u;
    } else {
      L.stable = (r >= 1 && next == L.variant) ? L.stable + 1u : 1u;
      if (confident) L.stable = max(L.stable, D.commit_after);
      L.cstop = 0u;
      if (D.commit_after != 0u && L.stable >= D.commit_after) {
        const uint32_t p0 = D.recheck_rounds ? D.recheck_rounds : 1u;
        const uint32_t p = (next == L.clast && L.cperiod) ? min(L.cperiod * 2u, 1u << 30) : p0;
        L.cperiod = p;
        L.clast = next;
        const unsigned long long stop = (unsigned long long)r + 1u + p;
        L.cstop = stop > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)stop;
        L.stable = D.commit_after - 1u;
        if (cta0 && r == 0u) C->commit_round0 = 1u;
      }
      if (cta0) C->consults += 1u;
    }
    L.prev_variant = (r >= 1) ? L.variant : NIL;
    L.fprev = L.fe - L.fb;  // frontier of round r, for the timing feature two rounds on
    L.variant = next;
    if (next != TRIM_AC4_PUSH) L.mixed = 1;
    L.round = r + 1;
    L.fb = L.fe;
    L.fe = len;
    L.w_end = w_end;
    L.e_end = e_end;
    if (next == TRIM_AC3_PULL) L.live_out = (L.ac3_list == NIL) ? 0u : (L.ac3_list ^ 1u);
    for (int i = 0; i < NFEAT; ++i) L.feat[i] = f[i];
  }
  __syncwarp();
  if (lane == 0) {
    B.S = L;
    B.err = err;
  }
}

// CTA 0, start of round k: timestamp, and zero the accumulator slot of round k+2.
__device__ __forceinline__ void start_round(const Dev& D, uint32_t k) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    D.C->t_round[k & 3] = globaltimer();
    RoundStat* z = &D.C->rs[(k + 2) & 3];
    z->sum_in = 0; z->sum_out = 0;
    z->hist[0] = z->hist[1] = z->hist[2] = 0;
    z->live_count = 0;
    z->max_din = 0;
  }
}

// ------------------------------------------------------------------ AC-4

// AC-4 push: decrement the counters of the predecessors of every removed vertex
// not yet pushed, i.e. the in-edges [e_c4, e_end) of the work list. The edges are
// cut into 32-edge chunks and each warp takes an equal run of chunks, so a hub's
// in-edges spread over many warps. The owner of a chunk's first edge comes from
// chunk_first; the next 31 work-list entries own the rest of the chunk (every
// entry has at least one edge), and a shuffle search finds each lane's owner.
// Rows are read once and leave the L2 first, so that more of the counters stay
// (4,096 packed graphs, 25 million counters, 1.6 million pushes a round near the
// DRAM's rate: kernel 1,984 us per run without that, 1,940 with; the same for the work
// list and the removed vertices' offsets was slower, 2,005 and 1,998, as they are
// read soon or again; in the asynchronous tail 6,355 against 6,619).
__device__ ROUND_FN void ac4_round(const Dev& D, Cta& B, const Sched& S, uint32_t gwarp,
                                   uint32_t nwarps) {
  constexpr int U = 4;  // chunks in flight per warp
  Counters K;
  const unsigned lane = lane_id();
  const uint32_t r = S.round;
  // a vertex whose counter reaches zero is still live unless another variant
  // ran (also in the AC-4-only flavour: a committed stretch of a scheduled run
  // may follow AC-6 or AC-3 rounds, whose removals AC-4 has not yet pushed)
  const bool check = S.mixed;
  const uint32_t ea = S.e_c4, eb = S.e_end, ia = S.c4w, ib = S.w_end;
  if (eb <= ea) return;
  // A small round (at most one entry and one 32-edge chunk per warp) whose
  // entries all have few in-edges gives each warp one work-list entry: its row
  // and edge range come with one load, no chunk-owner lookup, and the warp
  // walks the entry's in-edges 32 at a time (at most 8 steps).
  if (ib - ia <= nwarps && eb - ea <= 32u * nwarps && S.bmax <= 256u) {
    // warp w of CTA c takes entry w * grid + c: a small round's entries (and
    // the memory requests they cause) spread over every SM
    const uint32_t j = ia + (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    if (j < ib) {
      const uint32_t row = ldcg(&D.w4_row[j]);
      const uint32_t eo = ldcg(&D.w4_eoff[j]);
      const uint32_t ee = (j + 1u < ib) ? ldcg(&D.w4_eoff[j + 1u]) : eb;
      for (uint32_t k0 = eo; k0 < ee; k0 += 32u) {
        const uint32_t e = k0 + lane;
        const bool valid = e < ee;
        const uint32_t u = valid ? ld_stream(&D.itgt[row + (e - eo)]) : 0u;
        const uint32_t old = valid ? atomicSub(&D.cnt[u], 1u) : 0u;
        K.pushed += valid ? 1 : 0;
        bool pred = valid && old == 1u;
        if (pred && check) pred = ldcg(&D.level[u]) == LIVE;
        append_dead(D, B, pred, u, r, D.live0);
      }
    }
    stats_flush(D, B, K);
    return;
  }
  const uint32_t c0 = ea >> 5, c1 = (eb + 31u) >> 5;
  const uint32_t per = (c1 - c0 + nwarps - 1) / nwarps;
  const uint32_t cb = c0 + gwarp * per, ce = min(c1, cb + per);
  uint32_t cfb = 0;
  for (uint32_t c = cb; c < ce; c += U) {
    const uint32_t k = (c - cb) & 31u;
    if (k == 0u) cfb = (c + lane < ce) ? ldcg(&D.chunk_first[c + lane]) : 0u;
    uint32_t wrow[U], weo[U], u[U], old[U];
    bool valid[U];
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const uint32_t first = max(__shfl_sync(FULL, cfb, (k + q) & 31u), ia);
      const uint32_t ii = first + lane;
      const bool in = c + q < ce && ii < ib;
      wrow[q] = in ? ldcg(&D.w4_row[ii]) : 0u;
      weo[q] = in ? ldcg(&D.w4_eoff[ii]) : 0xFFFFFFFFu;
    }
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const uint32_t e = ((c + q) << 5) + lane;
      valid[q] = c + q < ce && e >= ea && e < eb;
      const unsigned j = owner_of(weo[q], e);
      const uint32_t idx = __shfl_sync(FULL, wrow[q], j) + (e - __shfl_sync(FULL, weo[q], j));
      u[q] = valid[q] ? ld_stream(&D.itgt[idx]) : 0u;
    }
#pragma unroll
    for (int q = 0; q < U; ++q) old[q] = valid[q] ? atomicSub(&D.cnt[u[q]], 1u) : 0u;
#pragma unroll
    for (int q = 0; q < U; ++q) {
      K.pushed += valid[q] ? 1 : 0;
      bool pred = valid[q] && old[q] == 1u;
      if (pred && check) pred = ldcg(&D.level[u[q]]) == LIVE;
      append_dead(D, B, pred, u[q], r, D.live0);
    }
  }
  stats_flush(D, B, K);
}

#if TRIM_LOCAL
// ------------------------------------------------------------------ local AC-4 rounds

#if !TRIM_AC6_ONLY && !TRIM_AC3_ONLY
// End of a local stretch that returns to ordinary rounds (all threads): the
// queued vertices of round r (buffer b) become work-list entries, and the round
// ends like an ordinary one (flush, grid barrier, advance). A rare path, out of
// line in the scheduler flavour so that its flush and scheduler code add no
// registers to the local rounds.
#if TRIM_MODES & 8
__device__ __noinline__
#else
__device__ __forceinline__
#endif
void local_leave(uint32_t b, uint32_t r) {
  const Dev& D = cta_dev;
  Cta& B = cta_state;
  const unsigned lane = lane_id();
  const uint32_t ne = B.lq_vend[b];
  for (uint32_t i0 = (threadIdx.x >> 5) * 32u; i0 < ne; i0 += blockDim.x) {
    const uint32_t i = i0 + lane;
    const bool has = i < ne;
    const uint32_t len = has ? B.lq_din[b][i] : 0u;  // (in+out: direction in the top bit)
    append_w4(D, B, has, has ? B.lq_row[b][i] : 0u, len & 0x7FFFFFFFu, r, len >> 31);
  }
  flush_round(D, B, r, D.live0);
  if ((D.flags & F_ROUND_LOG) && blockIdx.x == 0 && threadIdx.x == 0)
    D.C->t_flush[r & 3] = globaltimer();
  if (!grid_barrier(D, B, false)) return;
  if (threadIdx.x < 32) advance(D, B);
  __syncthreads();
}
#endif

// Does round S.round start a stretch of local rounds? Its pending work-list
// entries (the stretch's first round gives each warp whole entries) must have
// at most local_edges_max in-edges in all, none more than 256.
__device__ __forceinline__ bool local_start(const Dev& D, const Sched& S) {
#if TRIM_AC3_ONLY
  return D.local_edges_max != 0u;  // from the first round to the last
#elif TRIM_AC6_ONLY
  // AC-6: the sets were built, and the last round's removals are at most one to a
  // warp (kernel ms, with up to one / two / four / eight: deep cascades of 2^20 vertices
  // with 7,340 to a level 1.387 / 1.428 / 1.428 / 1.429, with 14,680 0.826 / 0.826 /
  // 1.046 / 1.043; planted graphs of 300,000 vertices 0.229 / 0.246 / 0.247 / 0.247, of
  // 1,000,000 0.287 / 0.288 / 0.292 / 0.461)
  return S.prev_variant == TRIM_AC6_SUPPORT && S.variant == TRIM_AC6_SUPPORT &&
         S.fe - S.fb <= min(D.local_edges_max, gridDim.x * (blockDim.x >> 5));
#else
  if (D.local_edges_max == 0u || S.variant != TRIM_AC4_PUSH) return false;
  // with the schedulers: inside a committed stretch only, whose last round
  // (the one the scheduler reads features of) runs as an ordinary round
  if ((MODES & M_SCHED) && !(S.cstop != 0u && S.round + 1u < S.cstop)) return false;
  // In+out trimming takes one entry to a warp in a stretch's first round, so it starts one
  // with at most two each; wider rounds are better spread by inout_round (kernel us with any
  // number / with this bound: R-MAT of 2^22 vertices 149 and 145, of 2^23 269 and 258, 80
  // packed graphs 289 and 278, planted 4,000,000 362 and 349; deep cascades the same).
  if ((MODES & M_INOUT) && S.w_end - S.c4w > 2u * gridDim.x * (blockDim.x >> 5)) return false;
  const uint32_t edges = S.e_end - S.e_c4;
  return edges <= D.local_edges_max && S.bmax <= 256u;
#endif
}

// Thread 0: closes local round L.round, in which nF vertices were removed, all
// of them counted only by the local barrier (the schedule step of advance()
// for a round of the AC-4-only flavour, without reading the control block).
__device__ void local_close(const Dev& D, Cta& B, uint32_t nF) {
  Sched& L = B.S;
  const uint32_t r = L.round;
  constexpr uint32_t variant = TRIM_AC6_ONLY   ? TRIM_AC6_SUPPORT
                               : TRIM_AC3_ONLY ? TRIM_AC3_PULL
                                               : TRIM_AC4_PUSH;
  L.vcount[variant] += 1u;
  L.c4w = L.w_end;  // the stretch's first round pushed every pending entry
  L.e_c4 = L.e_end;
  L.bmax = 0u;
  if (!TRIM_AC6_ONLY) L.skew += nF;  // (those are in the log)
  if (blockIdx.x == 0) {
    Ctrl* C = D.C;
    if (nF == 0u) {  // (a stretch that goes on or leaves publishes later)
      C->vcount[variant] = L.vcount[variant];
      C->rounds = r;
      C->n_dead = L.fe;
      C->local_rounds = L.lround;
    }
    if ((D.flags & F_ROUND_LOG) && D.rlog != nullptr && r >= 1u && r - 1u < D.rlog_cap) {
      trim_round_rec_t* rec = &D.rlog[r - 1u];
      rec->round = r;
      rec->variant = variant;
      rec->frontier = L.fe - L.fb;
      rec->removed = nF;
      rec->t_start_ns = C->t_round[r & 3];
      rec->t_end_ns = globaltimer();
      rec->t_work_ns = C->t_work[r & 3];
      rec->t_flush_ns = rec->t_work_ns;  // a local round moves nothing to global lists
      for (int i = 0; i < NFEAT; ++i) rec->features[i] = L.feat[i];  // that chose round r
      C->rlog_len = r;
    }
  }
  // round r+1 is chosen without the scheduler (a committed or fixed variant;
  // a flavour without the schedulers never sets features)
  if (MODES & M_SCHED)
    for (int i = 0; i < NFEAT; ++i) L.feat[i] = 0.0f;
  if (nF == 0u) {
    L.done = 1u;
    return;
  }
  L.stable = D.commit_after ? D.commit_after - 1u : 0u;  // as advance() in this flavour
  L.prev_variant = variant;
  L.fprev = L.fe - L.fb;
  L.round = r + 1u;
  L.fb = L.fe;
  L.fe += nF;
}

#if TRIM_ASYNC
// The asynchronous tail (see below) takes a level's vertices one to a warp, so it starts once there are
// about as many workers as vertices. Measured on deep cascades (ms, tail from
// round 128 against rounds; 4,560 workers): 4,096 chains of 2,867 6.8 against
// 13.2, 5,872 of 2,000 7.6 against 10.2, but 7,000 of 300 1.88 against 1.63 and
// 11,744 of 1,000 7.4 against 6.2.
__device__ __forceinline__ uint32_t async_workers() { return gridDim.x * ((blockDim.x >> 5) - 1u); }
__device__ __forceinline__ bool async_few(uint32_t vertices) {
  return 10ull * vertices <= 13ull * async_workers();
}
#endif

// End of local round r (all threads): one arrival per CTA on the barrier word
// of this round's parity, carrying 2^48 + 2^32 * (overflowed) + the CTA's local
// removals; the wait ends when the word has grown by gridDim.x arrivals since
// its value after its previous round (lbase), and that growth is the round's
// totals. A slot is reused two rounds later, when every CTA has read it. The
// wait is bounded like grid_barrier's. Thread 0 then decides how the stretch
// goes on (B.lq_next: LQ_GO on, LQ_DONE the run is over, both after closing
// the round; LQ_LEAVE back to ordinary rounds). Returns false on a timeout.
constexpr uint32_t LQ_GO = 0, LQ_DONE = 1, LQ_LEAVE = 2;
__device__ bool local_barrier(const Dev& D, Cta& B, uint32_t b, uint32_t r) {
  __syncthreads();
  if (threadIdx.x == 0) {
    Sched& S = B.S;
    const uint32_t slot = S.lround & 1u;
    if (((MODES & M_SCHED) || (D.flags & F_LIVE_EDGES)) && B.lq_pushed)
      atomicAdd(&D.C->local_edges, (unsigned long long)B.lq_pushed);
    const unsigned long long add =
        (1ull << 48) | ((unsigned long long)B.lq_ovf << 32) | (unsigned long long)B.lq_k;
    const unsigned long long base = S.lbase[slot];
    // AC-6 rounds hand levels, records and list heads to other CTAs, AC-3 rounds levels.
    if (TRIM_AC6_ONLY || TRIM_AC3_ONLY) fence_acq_rel();
    // Otherwise no fence before the arrival: across a local barrier CTAs exchange nothing
    // through plain memory, only counter decrements, and every decrement of
    // this round has returned its value (it is performed at L2) before this
    // arrival is issued. Levels written here are read after the kernel or
    // after an ordinary (fenced) barrier.
    red_relaxed_add64(&D.C->lbar[slot], add);
    // the next round fills the buffer this round read
#if TRIM_AC3_ONLY
    B.live_n[b ^ 1u] = 0u;
#endif
    B.lq_cnt[b ^ 1u] = 0ull;
    B.lq_vend[b ^ 1u] = 0u;
    B.lq_k = 0u;
    B.lq_ovf = 0u;
    B.lq_pushed = 0u;
    // the stretch ends before the last round of a committed stretch (the
    // scheduler reads its features) and, where the asynchronous tail may take
    // over (asked every ASYNC_RETRY rounds), as it starts from the work list
    const bool last = (MODES & M_SCHED) && r + 1u >= S.cstop;
#if TRIM_ASYNC
    const bool ask = D.async_edges_max != 0u && !(D.flags & F_ROUND_LOG) && !S.mixed &&
                     r + 1u >= ASYNC_MIN_ROUND && r + 1u >= S.async_from &&
                     (r + 1u) % ASYNC_RETRY == 0u;
#endif
    const uint64_t t0 = globaltimer();
    // relaxed polls: an acquiring load would also invalidate this SM's L1 on
    // every iteration, and nothing read after this barrier needs it
    unsigned long long cur = ld_relaxed64(&D.C->lbar[slot]);
    while ((uint32_t)((cur - base) >> 48) != gridDim.x) {
      if (globaltimer() - t0 > D.spin_limit_ns) {
        set_error(D, TRIM_ERR_TIMEOUT, 2);
        B.err = TRIM_ERR_TIMEOUT;
        break;
      }
      cur = ld_relaxed64(&D.C->lbar[slot]);
    }
    if (TRIM_AC6_ONLY || TRIM_AC3_ONLY) fence_acq_rel();
    const unsigned long long d = cur - base;
    S.lbase[slot] = cur;
    S.lround += 1u;
    const uint32_t nF = (uint32_t)d, n_ovf = (uint32_t)(d >> 32) & 0xFFFFu;
#if TRIM_ASYNC
    const bool stop = last || (ask && async_few(nF));
#else
    const bool stop = last;
#endif
    if (n_ovf == 0u && (nF == 0u || !stop)) {
      local_close(D, B, nF);  // every removal of the round is in the queues
      B.lq_next = nF ? LQ_GO : LQ_DONE;
    } else {
      S.skew += nF;  // advance() closes the round after the work-list handover
      if (blockIdx.x == 0) D.C->local_rounds = S.lround;
      B.lq_next = LQ_LEAVE;
    }
  }
  __syncthreads();
  return B.err == 0u;
}

#if !TRIM_AC6_ONLY && !TRIM_AC3_ONLY
// Runs local rounds from round B.S.round on: the first pushes the pending
// work-list entries (one per warp), later ones the predecessors in the CTA's
// queue. A removed vertex's row bounds are loaded once its counter has reached
// zero, not alongside every decrement: one more dependent load per round, but
// one random access per push instead of two, and large rounds are bound by
// those (kernel ms, rounds only, late against alongside: in+out of 2^23
// vertices 6.73 and 7.25, AC-4 of 2^24 12.4 and 12.8, of 2^20 1.205 and 1.222, of
// 2^16 1.005 and 1.015). Up to LQ_LATE_MIN vertices the offsets stay in every
// SM's L1, and the bounds come alongside (1,000 vertices: 0.0539 against 0.0549).
// The stretch ends when a round removes nothing (the run is done),
// when a round overflowed the queues, or (with the schedulers) before the last
// round of the committed stretch; in the last
// two cases the queued vertices join the global work list and the round ends
// like an ordinary one (flush, grid barrier, advance). Returns false on a
// timeout.
__device__ __noinline__ bool local_stretch() {
  const Dev& D = cta_dev;
  Cta& B = cta_state;
  Counters K;
  const unsigned lane = lane_id();
  // A CTA may queue LQ_SKEW times the stretch's mean load at its start: past that
  // every round waits for the fullest CTAs (a removal goes to the CTA that pushed
  // last, often one that lags), and the ordinary round that an overflow brings
  // (about 12 us) spreads the work evenly again. Kernel ms, with the bound and
  // with queues filled to LQ_EDGES: in+out of 2^23 vertices 6.73 and 7.52, of 2^20
  // 1.354 and 1.510; AC-4 of 2^24 (rounds only) 12.4 and 13.2, of 2^20 1.205 and
  // 1.283. Multiples of 3 / 4 / 6: in+out of 5,000,011 4.15 / 4.21 / 4.52, of 2^20 1.049 /
  // 1.045 / 1.083, 200 packed graphs 0.581 / 0.554 / 0.537. Where few edges are pending a
  // full queue is cheaper than leaving, so the bound has a floor: kernel us with 256 / 512 /
  // 768 / 1,024, packed graphs, 64 402 / 350 / 348 / 356, 80 462 / 405 / 396 / 400, 256 570 / 556 /
  // 552 / 552; in+out of 2^20 1,055 / 1,049 / 1,145 / 1,202, of 5,000,011 4,218 / 4,218 / 4,575 /
  // 4,835.
  const float mean = __fdividef((float)(B.S.e_end - B.S.e_c4), (float)gridDim.x);
  const uint32_t cap = min(LQ_EDGES, max(LQ_FLOOR, (uint32_t)((float)LQ_SKEW * mean)));
  const bool late = D.n > LQ_LATE_MIN;
  bool first = true;
  while (true) {
    const uint32_t r = B.S.round;
    const uint32_t b = B.S.lround & 1u;
    [[maybe_unused]] const bool check = B.S.mixed;
    start_round(D, r);
    if (first) {
      const uint32_t ia = B.S.c4w, ib = B.S.w_end, eb = B.S.e_end;
      const uint32_t nw = gridDim.x * (blockDim.x >> 5);
      // G entries to a warp (one where there are enough warps), their edges end to
      // end: a stretch may begin with many more entries than warps. 4,096 packed
      // graphs, kernel us: 1,990 against 2,041 with one entry after the other.
      // (In+out keeps one: it starts with at most two entries to a warp.)
      constexpr bool kOne = (MODES & M_INOUT) != 0;
      const uint32_t G = kOne ? 1u : min(32u, (ib - ia + nw - 1u) / nw);
      auto of = [&](uint32_t x, unsigned o) { return kOne ? x : __shfl_sync(FULL, x, o); };
      for (uint32_t j0 = ia + ((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * G; j0 < ib;
           j0 += nw * G) {
        const uint32_t ne = min(G, ib - j0), j = kOne ? j0 : j0 + lane;
        const bool in = kOne || lane < ne;
        const uint32_t row = in ? ldcg(&D.w4_row[j]) : 0u;
        const uint32_t eo = in ? ldcg(&D.w4_eoff[j]) : 0xFFFFFFFFu;
        const uint32_t ee = (j0 + ne < ib) ? ldcg(&D.w4_eoff[j0 + ne]) : eb;
        const uint32_t dir = (MODES & M_INOUT) ? ldcg(&D.w4_dir[j]) : 0u;
        for (uint32_t k0 = of(eo, 0); k0 < ee; k0 += 32u) {
          const uint32_t e = k0 + lane;
          const bool valid = e < ee;
          const unsigned o = kOne || G == 1u ? 0u : owner_of(eo, e);
          const uint32_t at = of(row, o) + (e - of(eo, o));
          const uint32_t u = valid ? __ldg(&push_tgt(D, dir)[at]) : 0u;
          uint32_t p0 = 0u, p1 = 0u;
          if (valid && !late) {
            p0 = __ldg(&push_off(D, dir)[u]);
            p1 = __ldg(&push_off(D, dir)[u + 1u]);
          }
          const PushWord old = valid ? push(D, u, dir) : 0u;
          bool pred = valid && push_removes(old, dir);
#if TRIM_MODES & 16
          count_rows(D, pred, u, K);
#else
          K.pushed += valid ? 1u : 0u;
          if (pred && check) pred = ldcg(&D.level[u]) == LIVE;
#endif
          if (pred && late) {
            p0 = __ldg(&push_off(D, dir)[u]);
            p1 = __ldg(&push_off(D, dir)[u + 1u]);
          }
          local_append(D, B, pred, u, r, p0, p1 - p0, b, dir, cap);
        }
      }
    } else {
      const uint32_t qb = b ^ 1u;
      const uint32_t qe = (uint32_t)(B.lq_cnt[qb] >> 32);
      for (uint32_t base = 0; base < qe; base += 2u * blockDim.x) {  // CTA-uniform
        uint32_t u[2], p0[2], p1[2], dir[2];
        PushWord old[2];
        bool valid[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const uint32_t k = base + (uint32_t)q * blockDim.x + threadIdx.x;
          valid[q] = k < qe;
          u[q] = valid[q] ? B.lq_ids[qb][k] : 0u;
          dir[q] = 0u;
#if TRIM_MODES & 16
          dir[q] = valid[q] ? B.lq_dir[qb][k] : 0u;
#endif
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          p0[q] = p1[q] = 0u;
          if (valid[q] && !late) {
            p0[q] = __ldg(&push_off(D, dir[q])[u[q]]);
            p1[q] = __ldg(&push_off(D, dir[q])[u[q] + 1u]);
          }
          old[q] = valid[q] ? push(D, u[q], dir[q]) : 0u;
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          if (q && base + blockDim.x >= qe) break;  // CTA-uniform
          bool pred = valid[q] && push_removes(old[q], dir[q]);
#if TRIM_MODES & 16
          count_rows(D, pred, u[q], K);
#else
          K.pushed += valid[q] ? 1u : 0u;
          if (pred && check) pred = ldcg(&D.level[u[q]]) == LIVE;
#endif
          if (pred && late) {
            p0[q] = __ldg(&push_off(D, dir[q])[u[q]]);
            p1[q] = __ldg(&push_off(D, dir[q])[u[q] + 1u]);
          }
          local_append(D, B, pred, u[q], r, p0[q], p1[q] - p0[q], b, dir[q], cap);
        }
      }
      if (threadIdx.x == 0) B.lq_pushed = qe;
    }
    if ((D.flags & F_ROUND_LOG) && blockIdx.x == 0) {
      __syncthreads();
      if (threadIdx.x == 0) D.C->t_work[r & 3] = globaltimer();
    }
    if (!local_barrier(D, B, b, r)) break;
    const uint32_t next = B.lq_next;
    if (next == LQ_DONE) break;
    if (next == LQ_GO) {
      first = false;
      continue;
    }
    local_leave(b, r);
    break;
  }
  stats_flush(D, B, K);
  return B.err == 0u;
}
#endif

#endif  // TRIM_LOCAL
#if TRIM_ASYNC
// ------------------------------------------------------- asynchronous AC-4 tail
//
// A vertex's level is one more than the top level among its successors
// (Definition 2: round r removes the vertices whose successors were all
// removed before round r, the last of them in round r - 1). The pushes can
// carry that maximum, and then the rest of an AC-4 run needs no rounds at all.
// Every vertex gets a 16-byte record: a 64-bit word (top level pushed so far
// << 32 | live-successor counter) and its G^T row (start, length). The push
// from a removed vertex of level l replaces the word by (max(top, l) << 32 |
// counter - 1) in one compare-and-swap, and the push that takes the counter to
// zero removes the vertex with level max(top, l) + 1: every successor has
// pushed by then, so the maximum is over all of them, whatever the order of
// the pushes.
//
// What bounds it is the chain of dependent memory accesses per level, so no
// warp waits for another. Each worker warp loops on its own over a batch of up
// to 32 pushes held in registers, the G^T row of one removed vertex: it loads
// the records (word and row come with one sector), issues the compare-and-swaps,
// and while these are under way loads the row of a vertex whose counter it saw
// at one; if the swaps went as foreseen (nearly always), that row is its next
// batch. A level then costs two dependent accesses to memory.
//
// A removed vertex's row stays with the warp whose push removed it, the warp of
// the last of its successors to go: work drifts towards the warps that lag, and
// every level waits for the slowest warp. So a batch that removes several
// vertices hands all but one of them on at once: to idle workers of the CTA (a
// claim, a mailbox, a wake-up: no lock, nobody polls), else to the CTA's ring.
// Rows over 32 in-edges go the same way in pieces of 32; rows over AQ_LOCAL_DMAX
// in-edges, or that the ring has no room for, to a global list of pieces of at
// most kAsyncPiece. One warp of each CTA, the control warp, gives pieces of the
// ring to workers that became idle, and while there is none sends them, one
// each, to CTAs with idle workers (channels, see async_control).
//
// Measured (ms per trim, kernel only; chains of 2,867 and 10,000 levels): the
// deep cascade 2^24 6.45, the large mixed graph 20.5. As one step per CTA, two
// pushes per thread, with a rebalance of all CTAs when a queue grew: 11.3 and
// 36.1 (a level paid for the word, the swap, the row and two CTA barriers in
// turn). With batches of several rows (first build, one row 6.7 and 21.0), up to 32
// pushes: 8.9 and 29.4; 16: 7.8 and 25.1.
//
// Rows in the global pieces, or a ring half full, need a rebalance: every CTA's
// workers stop after their batch, write what they hold (entries of their batch,
// pieces of the ring) to global lists, and after a grid barrier each CTA takes
// an even slice of those and of the pieces written since the last rebalance; a
// second barrier closes the rebalance (counts published, the lists' counters
// ready for the next). The tail ends when no CTA has work: a token count holds
// one token per CTA with work; a CTA releases its token when its workers and
// ring are empty and its rows sent are acknowledged, and a count of zero (with
// no rebalance asked for) ends the run.
//
// What it gains it gains where a batch removes one vertex, whose row stays in its warp
// (chains). Where batches remove several or none, rows change hands all the time, and they
// gather in few CTAs, as every row stays where the last of its vertex's successors went;
// where a level has many more vertices than there are workers, every row waits for one.
// Rounds are faster there, so the tail looks at itself: a CTA that has handed on more than a
// row for every four batches, or whose ring stays crowded, asks for a rebalance, and that
// compares the totals. If the tail does not pay, it goes on up to the top level removed so
// far only; vertices of the next level are parked in the AC-4 work list, and once no CTA has
// work, the counters return to their array and ordinary rounds go on from that list
// (async_leave). A later tail waits ASYNC_WAIT rounds, twice as long each time.
//
// Measured (ms per trim; rounds only / tail as one step per CTA / without leaving / as
// here): 3,000 levels of 100 vertices with three random successors each in the level below 8.8 /
// 12.3 / 30.1 / 8.6; 400 levels of 3,000 with 40 8.0 / 17.6 / 28.6 / 8.3; 1,000 chains of 200
// below 40 levels of 300,000 1.6 / 2.9 / 6.9 / 1.9; 1,000 chains of 2,000 6.1 / 5.8 / 3.0 / 3.1. The look
// costs chains 1 to 2 per cent. Rows over AQ_LOCAL_DMAX in-edges at every other level bring a
// rebalance each, slower than a round: ASYNC_CLOSE of those in a row end the tail as well (800
// levels, every other one a vertex with 2,000 predecessors: 5.3 / 6.4 / 8.2 / 7.1).
//
// It takes over at the start of an AC-4 round r (r >= ASYNC_MIN_ROUND) whose
// pending work-list entries are exactly the vertices removed in round r - 1,
// at most async_edges_max in-edges, and runs the rest of the run or until it leaves (with
// the schedulers: it starts only inside a committed stretch). Rounds before ASYNC_MIN_ROUND stay rounds (local ones
// where they can): on graphs that peel in fewer rounds they were faster.
__device__ __forceinline__ bool async_start(const Dev& D, const Sched& S) {
  if (D.async_edges_max == 0u || S.variant != TRIM_AC4_PUSH || S.mixed) return false;
  if ((D.flags & F_ROUND_LOG) || S.round < ASYNC_MIN_ROUND || S.round < S.async_from) return false;
  if (S.prev_variant != TRIM_AC4_PUSH) return false;
  if ((MODES & M_SCHED) && D.mode > TRIM_AC3_PULL && !(S.cstop != 0u && S.round < S.cstop))
    return false;
  const uint32_t edges = S.e_end - S.e_c4;
  return edges <= min(D.async_edges_max, 32u * async_workers()) && S.bmax <= 256u &&
         async_few(S.w_end - S.c4w);
}

constexpr uint32_t AS_STEP = 0, AS_DONE = 1, AS_REBALANCE = 2;

// The CTA's ring of row pieces (dynamic shared memory): row starts | lengths |
// levels, a power of two of pieces each (1 to 2 per thread). With the pieces
// that its warps hold there are never more than kAsyncRows per thread.
__device__ __forceinline__ uint32_t async_ring_cap() {
  return 1u << (31 - __clz(2 * (int)blockDim.x));
}
// ... behind it each worker's mailbox (3 x 32 words) ...
__device__ __forceinline__ uint32_t* async_mail(uint32_t warp) {
  return dyn_smem + 3u * async_ring_cap() + warp * 96u;
}

// What a worker warp holds between batches: the batch (lane i < cnt: push to
// predecessor p with level l), a row piece being worked off (warp-uniform),
// its next work-list entry, its removals and top level not yet added to the
// CTA's, the phase of its wake-up barrier, and whether parts of the last
// rebalance's share may be unclaimed. (aw, itgt and level are copies of the
// pointers in Dev, kept in registers)
struct AsyncWarp {
  uint4* aw;
  const uint32_t* itgt;
  uint32_t* level;
  uint32_t p, l, cnt;
  uint32_t pr, pl, pv;
  uint32_t wj;
  uint32_t removed, top;
  uint32_t cap;
  uint32_t phase;
  bool share;
};

__device__ __forceinline__ uint32_t vol(const uint32_t& x) {
  return *reinterpret_cast<const volatile uint32_t*>(&x);
}
// Warp-collective: lane 0's reading of x, the same for every lane (the lanes may
// read at different times, and what follows is warp-collective)
__device__ __forceinline__ uint32_t warp_vol(const uint32_t& x) {
  return __shfl_sync(FULL, vol(x), 0);
}
__device__ __forceinline__ void set_vol(uint32_t& x, uint32_t v) {
  *reinterpret_cast<volatile uint32_t*>(&x) = v;
}
__device__ __forceinline__ ulonglong2 ld_relaxed_v2(const uint4* p) {
  ulonglong2 v;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];"
               : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// Idle workers sleep on a barrier of their own and have a bit in a_idle. Whoever
// clears a bit has claimed that worker: it writes rows to the worker's mailbox
// (n of them) and wakes it with the one arrival its barrier waits for. Nobody
// polls shared memory and nothing takes a lock: a worker that hands rows over
// goes on with its own batch at once.
// One thread: claims an idle worker; its number, or 32 if there is none.
__device__ __forceinline__ uint32_t async_claim(Cta& B) {
  while (true) {
    const uint32_t m = vol(B.a_idle);
    if (m == 0u) return 32u;
    const uint32_t w = (uint32_t)__ffs(m) - 1u;
    if (atomicAnd(&B.a_idle, ~(1u << w)) >> w & 1u) return w;
  }
}
__device__ __forceinline__ void async_wake(Cta& B, uint32_t w, uint32_t n) {
  set_vol(B.w_rows[w], n);
  __threadfence_block();
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&B.w_bar[w])) : "memory");
}

// Warp-collective: the rows (row, len > 0, lev) that lanes hold go to idle
// workers of this CTA, a batch's worth each, in the order of the lanes. Lanes
// whose row (or what is left of it) found no idle worker keep it: len stays > 0.
__device__ __forceinline__ void async_give(Cta& B, uint32_t& row, uint32_t& len, uint32_t lev) {
  const unsigned lane = lane_id();
  unsigned m = __ballot_sync(FULL, len != 0u);
  uint32_t w = 32u, n = 0, e = 0;  // the claimed worker, its rows and their edges so far
  while (m) {
    const int j = __ffs(m) - 1;
    const uint32_t rj = __shfl_sync(FULL, row, j), nj = __shfl_sync(FULL, len, j);
    const uint32_t vj = __shfl_sync(FULL, lev, j);
    const uint32_t c = min(nj, 32u);
    if (w < 32u && e + c > 32u) {  // this worker has its batch
      if (lane == 0) async_wake(B, w, n);
      w = 32u;
    }
    if (w >= 32u) {
      if (lane == 0) w = async_claim(B);
      w = __shfl_sync(FULL, w, 0);
      if (w >= 32u) break;
      n = e = 0u;
    }
    if (lane == 0) {
      uint32_t* box = async_mail(w);
      box[n] = rj;
      box[32u + n] = c;
      box[64u + n] = vj;
    }
    ++n;
    e += c;
    if ((int)lane == j) {
      row += c;
      len -= c;
    }
    if (nj <= 32u) m &= m - 1u;
  }
  __syncwarp();
  if (w < 32u && lane == 0) async_wake(B, w, n);
  __syncwarp();
}

// Warp-collective: the rows that lanes hold go to the ring in pieces of
// AQ_PIECE, all or (where they do not fit) none: len becomes 0 if they did. A
// piece is there once its length is; only the control warp takes pieces out.
__device__ __forceinline__ void async_ring(Cta& B, uint32_t row, uint32_t& len, uint32_t lev) {
  const uint32_t nd = (len + AQ_PIECE - 1u) / AQ_PIECE;
  const uint32_t nincl = warp_incl_scan(nd);
  const uint32_t ND = __shfl_sync(FULL, nincl, 31);
  const uint32_t QR = async_ring_cap();
  uint32_t base = 0, ok = 0;
  if (lane_id() == 0) {
    uint32_t t = vol(B.r_tail);
    while (ND <= QR && t - vol(B.r_head) <= QR - ND) {
      const uint32_t seen = atomicCAS(&B.r_tail, t, t + ND);
      if (seen == t) {
        ok = 1u;
        break;
      }
      t = seen;
    }
    base = t;
  }
  ok = __shfl_sync(FULL, ok, 0);
  if (!ok) return;
  uint32_t at = __shfl_sync(FULL, base, 0) + nincl - nd;
  for (uint32_t i = 0; i < nd; ++i, ++at) {
    const uint32_t k = at & (QR - 1u);
    dyn_smem[k] = row + i * AQ_PIECE;
    dyn_smem[2u * QR + k] = lev;
    __threadfence_block();
    set_vol(dyn_smem[QR + k], min(AQ_PIECE, len - i * AQ_PIECE));
  }
  len = 0u;
  __syncwarp();
}

// Warp-collective: lanes with ovf set removed a vertex (G^T row start row,
// in-degree din, level lev) whose row goes to the global list of pieces, cut
// into pieces of at most kAsyncPiece in-edges; the CTA then asks for a
// rebalance. The pieces are read only after the rebalance's grid barrier.
__device__ __noinline__ void async_spill(bool ovf, uint32_t row,
                                         uint32_t din, uint32_t lev) {
  const Dev& D = cta_dev;
  Cta& B = cta_state;
  const unsigned lane = lane_id();
  const uint32_t np = ovf ? (din + kAsyncPiece - 1u) / kAsyncPiece : 0u;
  const uint32_t incl = warp_incl_scan(np);
  const uint32_t tot = __shfl_sync(FULL, incl, 31);
  uint32_t s = 0;
  if (lane == 0) {
    s = atomicAdd(&D.C->oq_res, tot);
    set_vol(B.a_want, 1u);
  }
  s = __shfl_sync(FULL, s, 0);
  // (cannot fail: every removal adds at most ceil(din / kAsyncPiece) pieces)
  if ((uint64_t)s + tot > D.oq_cap) {
    if (lane == 0) set_error(D, TRIM_ERR_STATE, 5);
    return;
  }
  if (ovf) {
    const uint32_t at = s + incl - np;
    for (uint32_t i = 0; i < np; ++i) {
      D.oq_row[at + i] = row + i * kAsyncPiece;
      D.oq_len[at + i] = min(kAsyncPiece, din - i * kAsyncPiece);
      D.oq_lev[at + i] = lev;
    }
  }
}

// Warp-collective: the G^T rows (row, len) that the lanes hold, laid end to end
// with exclusive prefix excl: element lane - at of them (at <= lane < at +
// total) becomes this lane's push, with its row's level.
__device__ __forceinline__ void async_take(AsyncWarp& A, uint32_t at, uint32_t total,
                                           uint32_t excl, uint32_t row, uint32_t lev) {
  const uint32_t j = lane_id() - at;
  const unsigned o = owner_of(excl, j);
  const uint32_t ro = __shfl_sync(FULL, row, o), xo = __shfl_sync(FULL, excl, o);
  const uint32_t lo = __shfl_sync(FULL, lev, o);
  if (j < total) {
    A.p = __ldg(&A.itgt[ro + (j - xo)]);
    A.l = lo;
  }
}

// Warp-collective: lanes in `rows` hold the G^T row of a removed vertex. The
// first, or with `many` all that fit, join this warp's next batch, of which
// `total` lanes are taken: their pushes are loaded (A.p, A.l). Returns the lanes
// whose row is left over. (All of them while the last rebalance's share is
// unclaimed: the share comes first, so that a warp asked to stop can.)
__device__ __forceinline__ unsigned async_pick(AsyncWarp& A, unsigned rows, uint32_t row,
                                               uint32_t len, uint32_t lev, bool many,
                                               uint32_t& total) {
  if (A.share) return rows;
  unsigned left = 0;
  const uint32_t k0 = lane_id() - total;
  uint32_t at = 0, sum = 0;
  while (rows) {  // (seldom more than three rows)
    const int j = __ffs(rows) - 1;
    const uint32_t rj = __shfl_sync(FULL, row, j), nj = __shfl_sync(FULL, len, j);
    const uint32_t vj = __shfl_sync(FULL, lev, j);
    if (nj <= 32u - total - sum && (many || total + sum == 0u)) {
      const uint32_t k = k0 - sum;
      if (k < nj) {
        at = rj + k;
        A.l = vj;
      }
      sum += nj;
    } else {
      left |= 1u << j;
    }
    rows &= rows - 1u;
  }
  if (k0 < sum) A.p = __ldg(&A.itgt[at]);
  total += sum;
  return left;
}

// Warp-collective: rows left over by async_pick go to idle workers, one each,
// else to the ring, else (rows over AQ_LOCAL_DMAX in-edges at once) to the
// global pieces. A row of a batch or less is placed by its own lane.
__device__ __forceinline__ void async_surplus(const Dev& D, Cta& B, unsigned left, uint32_t row,
                                              uint32_t len, uint32_t lev) {
  const bool mine = left >> lane_id() & 1u;
  uint32_t el = mine ? len : 0u;
  if (mine && el <= 32u) {
    const uint32_t w = async_claim(B);
    if (w < 32u) {
      uint32_t* box = async_mail(w);
      box[0] = row;
      box[32] = el;
      box[64] = lev;
      async_wake(B, w, 1u);
      el = 0u;
    }
  }
  __syncwarp();
  if (!__any_sync(FULL, el != 0u)) return;
  const bool ovf = el > AQ_LOCAL_DMAX;
  if (ovf) el = 0u;
  if (__any_sync(FULL, el > 32u)) async_give(B, row, el, lev);
  if (__any_sync(FULL, el != 0u)) async_ring(B, row, el, lev);
  if (__any_sync(FULL, ovf || el != 0u))
    async_spill(ovf || el != 0u, row, ovf ? len : el, lev);
}

// Warp-collective: a worker that found nothing to do adds its counts to the
// CTA's, sets its idle bit and sleeps until it is claimed; the rows it is given
// become its batch. (The wait ends: the control warp, whose own waits are
// bounded, claims every idle worker when it ends the stretch.)
__device__ __forceinline__ void async_idle(const Dev& D, Cta& B, AsyncWarp& A) {
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  A.top = __reduce_max_sync(FULL, A.top);
  uint32_t n = 0;
  if (lane == 0) {
    if (A.removed) {
      atomicAdd(&B.a_removed, A.removed);
      atomicMax(&B.a_maxlev, A.top);
    }
    __threadfence_block();
    atomicOr(&B.a_idle, 1u << warp);
    __threadfence_block();
    if (vol(B.a_next) != AS_STEP && (atomicAnd(&B.a_idle, ~(1u << warp)) >> warp & 1u)) {
      // (claimed itself: the control warp may have passed this bit by)
    } else {
      uint32_t done = 0;
      while (!done) {
        asm volatile(
            "{\n .reg .pred p;\n"
            " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
            " selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done) : "r"(smem_addr(&B.w_bar[warp])), "r"(A.phase & 1u), "r"(10000u) : "memory");
        if (!done && vol(B.a_next) == AS_DONE) break;  // (nobody wakes it any more)
      }
      if (done) n = vol(B.w_rows[warp]) | 0x80000000u;
    }
  }
  n = __shfl_sync(FULL, n, 0);
  A.removed = 0u;
  A.top = 0u;
  if (n >> 31) A.phase ^= 1u;
  n &= 0x7FFFFFFFu;
  if (n) {
    __threadfence_block();
    const uint32_t* box = async_mail(warp);
    const bool in = lane < n;
    const uint32_t row = in ? box[lane] : 0u, len = in ? box[32u + lane] : 0u;
    const uint32_t lev = in ? box[64u + lane] : 0u;
    const uint32_t incl = warp_incl_scan(len);
    A.cnt = __shfl_sync(FULL, incl, 31);  // (at most 32)
    async_take(A, 0u, A.cnt, incl - len, row, lev);
  }
}

// Warp-collective: fills the batch's free lanes from the piece being worked
// off; a warp without any work claims a part of the last rebalance's share (32
// entries, a row or a piece) or a pending work-list entry first.
__device__ __forceinline__ void async_fill(const Dev& D, Cta& B, AsyncWarp& A, uint32_t nwork) {
  const unsigned lane = lane_id();
  if (A.cnt == 0u && A.pl == 0u && A.share) {
    const size_t par = (size_t)((B.a_gen - 1u) & 1u);
    uint32_t e = 0, r = 0, q = 0;
    if (lane == 0) e = atomicAdd(&B.sh_elo, 32u);
    e = __shfl_sync(FULL, e, 0);
    if (e < B.sh_ehi) {
      A.cnt = min(32u, B.sh_ehi - e);
      if (lane < A.cnt) {
        A.p = ldcg(&D.ae_id[par * D.ae_cap + e + lane]);
        A.l = ldcg(&D.ae_lev[par * D.ae_cap + e + lane]);
      }
    } else {
      if (lane == 0) {
        atomicSub(&B.sh_elo, 32u);  // (the cursor stays near its end)
        r = atomicAdd(&B.sh_rlo, 1u);
        q = r < B.sh_rhi ? 0xFFFFFFFFu : atomicAdd(&B.sh_plo, 1u);
      }
      r = __shfl_sync(FULL, r, 0);
      q = __shfl_sync(FULL, q, 0);
      if (r < B.sh_rhi) {
        A.pr = ldcg(&D.er_row[par * D.er_cap + r]);
        A.pl = ldcg(&D.er_len[par * D.er_cap + r]);
        A.pv = ldcg(&D.er_lev[par * D.er_cap + r]);
      } else if (q < B.sh_phi) {
        A.pr = ldcg(&D.oq_row[q]);
        A.pl = ldcg(&D.oq_len[q]);
        A.pv = ldcg(&D.oq_lev[q]);
      } else if (A.wj < B.S.w_end) {
        const uint32_t eo = ldcg(&D.w4_eoff[A.wj]);
        const uint32_t ee = (A.wj + 1u < B.S.w_end) ? ldcg(&D.w4_eoff[A.wj + 1u]) : B.S.e_end;
        A.pr = ldcg(&D.w4_row[A.wj]);
        A.pl = ee - eo;
        A.pv = B.S.round - 1u;
        A.wj += nwork;
      }
    }
    // what no warp has claimed yet (a claimed part is its warp's to finish)
    A.share = vol(B.sh_elo) < B.sh_ehi || vol(B.sh_rlo) < B.sh_rhi || vol(B.sh_plo) < B.sh_phi ||
              A.wj < B.S.w_end;
    A.share = __any_sync(FULL, A.share);
  }
  if (A.pl != 0u && A.cnt < 32u) {
    const uint32_t k = min(32u - A.cnt, A.pl), j = lane - A.cnt;
    if (j < k) {
      A.p = __ldg(&A.itgt[A.pr + j]);
      A.l = A.pv;
    }
    A.pr += k;
    A.pl -= k;
    A.cnt += k;
  }
}

// Warp-collective: lanes with park removed a vertex of the level after the tail's last one:
// its row (row start, length) joins the AC-4 work list, for the round after that level.
__device__ __noinline__ void async_park(bool park, uint32_t row, uint32_t len) {
  const Dev& D = cta_dev;
  const unsigned lane = lane_id(), m = __ballot_sync(FULL, park);
  const uint32_t ew = park ? len : 0u, incl = warp_incl_scan(ew);
  const uint32_t longest = __reduce_max_sync(FULL, ew);
  unsigned long long o = 0;
  if (lane == 31) {
    o = atomicAdd(&D.C->w4, ((unsigned long long)incl << 32) | __popc(m));
    atomicMax(&D.C->a_bmax, longest);
  }
  o = __shfl_sync(FULL, o, 31);
  const uint32_t at = (uint32_t)o + __popc(m & ((1u << lane) - 1u));
  const uint32_t eo = (uint32_t)(o >> 32) + incl - ew;
  if (park) {
    D.w4_row[at] = row;
    D.w4_eoff[at] = eo;
  }
  mark_chunks(D, park, at, eo, eo + ew);
}

// Warp-collective: one batch. The compare-and-swaps are issued before the rows
// of the vertices they should remove are loaded, and checked after: the row
// accesses do not wait for them. A word whose counter is zero belongs to a
// vertex that is not live (masked): it is left alone.
__device__ __forceinline__ void async_batch(const Dev& D, Cta& B, AsyncWarp& A, Counters& K) {
  const unsigned lane = lane_id();
  const bool valid = lane < A.cnt;
  const uint32_t p = A.p, l = A.l;
  ulonglong2 a = make_ulonglong2(0ull, 0ull);
  if (valid) a = ld_relaxed_v2(&A.aw[p]);
  unsigned long long* word = reinterpret_cast<unsigned long long*>(&A.aw[p]);
  const uint32_t cnt = (uint32_t)a.x, row = (uint32_t)a.y, len = (uint32_t)(a.y >> 32);
  const bool live = valid && cnt != 0u;
  uint32_t lev = max((uint32_t)(a.x >> 32), l);
  K.pushed += valid ? 1u : 0u;
  unsigned long long prev = a.x;
  if (live) prev = atomicCAS(word, a.x, ((unsigned long long)lev << 32) | (cnt - 1u));
  uint32_t total = 0;
  const unsigned seen = __ballot_sync(FULL, live && cnt == 1u && len != 0u && lev < A.cap);
  // One row per batch: a warp that keeps several is slower (it waits for the
  // latest of more accesses), and every level waits for the slowest. Only where
  // rows pile up in the ring (more than there are warps for) are batches filled.
  const bool many = (seen & (seen - 1u)) != 0u &&
                    __shfl_sync(FULL, vol(B.r_tail) - vol(B.r_head), 0) >= (blockDim.x >> 5);
  unsigned left = async_pick(A, seen, row, len, lev + 1u, many, total);
  bool pend = live && prev != a.x;
  bool removed = live && !pend && cnt == 1u;
  const bool clean = !__any_sync(FULL, pend);
  if (!clean) {
    // a failed compare-and-swap means another push on the same word succeeded,
    // so the loop ends; the bound only guards against a broken invariant
    for (uint32_t it = 0; pend; ++it) {
      const unsigned long long w = prev;
      if ((uint32_t)w == 0u) break;
      if (it == (1u << 22)) {
        set_error(D, TRIM_ERR_TIMEOUT, 6);
        break;
      }
      lev = max((uint32_t)(w >> 32), l);
      prev = atomicCAS(word, w, ((unsigned long long)lev << 32) | ((uint32_t)w - 1u));
      if (prev == w) {
        removed = (uint32_t)w == 1u;
        pend = false;
      }
    }
    __syncwarp();
  }
  const unsigned rm = __ballot_sync(FULL, removed);
  if (!clean) {
    // not all as foreseen: rows of vertices that another push removed leave the
    // batch, rows of vertices removed after all join it
    const unsigned rows = __ballot_sync(FULL, removed && len != 0u && lev < A.cap);
    if (seen & ~rows) {
      total = 0u;
      left = async_pick(A, rows, row, len, lev + 1u, many, total);
    } else if (rows & ~seen) {
      left |= async_pick(A, rows & ~seen, row, len, lev + 1u, many, total);
    }
  }
  if (rm) {
    if (removed) {
      A.level[p] = lev + 1u;
      A.top = max(A.top, lev + 1u);
    }
    A.removed += __popc(rm);
  }
  A.cnt = total;
  if (left != 0u || A.cap != NIL) {
    const bool park = removed && len != 0u && lev >= A.cap;
    if (left) {
      // rows beyond the batch's first (a single one that is too long, or that makes way for
      // the last rebalance's share, tells nothing of the graph)
      const uint32_t more = (uint32_t)__popc(left) - (total == 0u ? 1u : 0u);
      if (lane == 0 && more) atomicAdd(&B.a_hand, more);
      async_surplus(D, B, left, row, len, lev + 1u);
    }
    if (__any_sync(FULL, park)) async_park(park, row, len);
  }
}

// A worker warp: batches until the control warp ends the stretch (and the last
// rebalance's share is claimed).
__device__ __forceinline__ void async_work(const Dev& D, Cta& B, AsyncWarp& A, uint32_t nwork,
                                           Counters& K) {
  while (true) {
    const uint32_t next = warp_vol(B.a_next);
    if (next == AS_DONE || (next != AS_STEP && !A.share)) break;
    async_fill(D, B, A, nwork);
    if (A.cnt == 0u) {
      if (!A.share) async_idle(D, B, A);
      continue;
    }
    async_batch(D, B, A, K);
    if (lane_id() == 0) atomicAdd(&B.a_prog, 1u);
  }
}

// One thread: publishes this CTA's removals and top level; releases its token after
// that (CTA 0 reads the totals once the token count is zero).
__device__ __forceinline__ void async_publish(const Dev& D, Cta& B) {
  Ctrl* C = D.C;
  if (B.a_removed) {
    atomicAdd(&C->a_removed, B.a_removed);
    atomicMax(&C->a_maxlev, B.a_maxlev);
    B.a_removed = 0u;
    B.a_maxlev = 0u;
  }
}
__device__ __forceinline__ void async_release(const Dev& D, Cta& B) {
  Ctrl* C = D.C;
  async_publish(D, B);
  fence_acq_rel();  // the counts before the release
  atomicSub(&C->a_tokens, 1u);
  B.a_token = 0u;
}

// Rows on their way to another CTA travel on channels: lane i of a control warp
// sends to the CTA async_offset(i) further on, one row at a time, and receives
// from the one as far back. A channel is a 16-byte message in the receiver's
// line (row start, length and a tag; level and the tag again: each 64-bit half
// says by itself whether it has arrived, so no fence is needed) and the tag it
// acknowledged in the sender's line.
__device__ __forceinline__ uint32_t async_offset(uint32_t i) {
  return gridDim.x > 32u ? 1u + i * ((gridDim.x - 1u) / 32u) : i + 1u;
}
struct AsyncChannel {
  uint32_t to, from;      // CTAs (to == this one: no channel)
  uint32_t sent, taken;   // tags of the last message sent and received
};

// The control warp: receives and dispatches rows, and watches until the stretch
// ends, then sets a_next and wakes the idle workers.
// Rows that arrive go to idle workers or the ring. Pieces in the ring go to
// idle workers, and where there are none to CTAs that have some. Rows in the global pieces, or a
// ring half full, ask for a rebalance. A CTA without work and
// with every row it sent acknowledged publishes its counts, releases its token,
// and waits until rows arrive, a rebalance is asked for or
// the token count is zero (the run is over). Every wait is bounded:
// spin_limit_ns without a heartbeat from a working CTA (or, with work, without
// a batch of its own workers) ends the run with TRIM_ERR_TIMEOUT.
__device__ __noinline__ void async_control() {
  const Dev& D = cta_dev;
  Cta& B = cta_state;
  Ctrl* C = D.C;
  const unsigned lane = lane_id();
  const uint32_t QR = async_ring_cap(), nwk = (blockDim.x >> 5) - 1u, all = (1u << nwk) - 1u;
  const uint32_t G = gridDim.x, off = async_offset(lane);
  AsyncChannel ch;
  ch.to = off < G ? (blockIdx.x + off) % G : blockIdx.x;
  ch.from = off < G ? (blockIdx.x + G - off) % G : blockIdx.x;
  ch.sent = B.ch_sent[lane];
  ch.taken = B.ch_taken[lane];
  const ulonglong2* in = &D.ch_msg[32u * blockIdx.x + lane];
  uint64_t t0 = globaltimer(), tb = t0;
  uint32_t beat = ld_relaxed(&C->a_beat), prog = vol(B.a_prog), next = AS_STEP;
  uint32_t load = 0xFFFFFFFFu, crowded = 0;
  for (uint32_t turn = 0; next == AS_STEP; ++turn) {
    // everything this turn looks at, under way together
    unsigned long long m0, m1;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(m0), "=l"(m1) : "l"(in) : "memory");
    const uint32_t ack = ld_relaxed(&D.ch_ack[32u * blockIdx.x + lane]);
    // (a CTA with hardly any work looks for requests every turn: others wait for it)
    const bool watch = (turn & 3u) == 0u || __shfl_sync(FULL, B.a_token, 0) == 0u ||
                       __popc(warp_vol(B.a_idle)) + 2u >= nwk;
    uint32_t err = 0, req = 0, tok = 0, bt = 0;
    if (watch && lane == 0) {
      err = ld_relaxed(&C->err);
      req = ld_relaxed(&C->a_req);
      tok = ld_relaxed(&C->a_tokens);
      bt = ld_relaxed(&C->a_beat);
    }
    // rows that arrived
    const uint32_t tag = ch.taken + 1u;
    const bool here = (uint32_t)(m1 >> 32) == tag && (uint32_t)(m0 >> 40) == (tag & 0xFFFFFFu);
    const unsigned hm = __ballot_sync(FULL, here);
    if (hm) {
      uint32_t row = (uint32_t)m0, len = here ? (uint32_t)(m0 >> 32) & 0xFFu : 0u;
      const uint32_t lev = (uint32_t)m1;
      async_give(B, row, len, lev);
      if (__any_sync(FULL, len != 0u)) async_ring(B, row, len, lev);
      // (a row that even the ring has no room for stays where it is)
      const bool took = here && len == 0u;
      // a CTA without a token takes one before it acknowledges: until then the
      // sender's covers the row
      uint32_t tokens = 1u;
      if (lane == 0 && B.a_token == 0u) {
        B.a_token = 1u;
        tokens = atomicAdd(&C->a_tokens, 1u);
      }
      tokens = __shfl_sync(FULL, tokens, 0);
      if (took && tokens != 0u) {  // (0: never, the sender holds one; the test waits for the addition)
        ch.taken = tag;
        st_relaxed(&D.ch_ack[32u * ch.from + lane], tag);
      }
      __syncwarp();
    }
    // pieces in the ring (all workers idle before it is seen empty: then
    // nothing but this warp adds to it, and there is no work at all)
    const uint32_t mask = warp_vol(B.a_idle);
    __threadfence_block();
    const uint32_t head = __shfl_sync(FULL, B.r_head, 0), rows = warp_vol(B.r_tail) - head;
    const bool idle = mask == all && rows == 0u && !__any_sync(FULL, ack != ch.sent);
    crowded = rows > 2u * nwk ? crowded + 1u : 0u;
    const uint32_t now_load = nwk - __popc(mask) + min(rows, 255u);
    if (now_load != load) {
      load = now_load;
      if (lane == 0) st_relaxed(&D.ch_load[blockIdx.x], load);
    }
    if (rows != 0u) {
      const uint32_t k = (head + lane) & (QR - 1u);
      uint32_t len = vol(dyn_smem[QR + k]);  // (0: not there yet)
      const unsigned rm = __ballot_sync(FULL, len != 0u);
      const uint32_t n = rm == FULL ? 32u : (uint32_t)__ffs(~rm) - 1u;  // leading pieces
      if (n) {
        __threadfence_block();
        if (lane >= n) len = 0u;
        uint32_t row = dyn_smem[k];
        const uint32_t lev = dyn_smem[2u * QR + k];
        async_give(B, row, len, lev);
        const unsigned left = __ballot_sync(FULL, len != 0u);
        uint32_t done = left ? (uint32_t)__ffs(left) - 1u : n;
        if (left && rows > 1u) {  // (a single row waits for a worker here)
          // the i-th lane whose channel is free and leads to idle workers
          // sends the i-th piece left; nearly idle CTAs first
          const uint32_t their = ld_relaxed(&D.ch_load[ch.to]);
          const bool can = ch.to != blockIdx.x && ack == ch.sent && their < nwk;
          const unsigned lo = __ballot_sync(FULL, can && their <= nwk / 2u);
          const unsigned cm = lo ? lo : __ballot_sync(FULL, can);
          const uint32_t from = done + __popc(cm & ((1u << lane) - 1u));
          const bool send = (cm >> lane & 1u) && from < n;
          const uint32_t sr = __shfl_sync(FULL, row, from & 31u), sv = __shfl_sync(FULL, lev, from & 31u);
          const uint32_t sl = __shfl_sync(FULL, len, from & 31u);
          const uint32_t ns = __popc(__ballot_sync(FULL, send));
          if (send) {
            ch.sent += 1u;
            const unsigned long long s0 = (unsigned long long)sr | ((unsigned long long)sl << 32) |
                                          ((unsigned long long)(ch.sent & 0xFFFFFFu) << 40);
            const unsigned long long s1 = (unsigned long long)sv | ((unsigned long long)ch.sent << 32);
            asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(&D.ch_msg[32u * ch.to + lane]),
                         "l"(s0), "l"(s1) : "memory");
          }
          done += ns;
        }
        if (lane < done) set_vol(dyn_smem[QR + k], 0u);
        __threadfence_block();
        __syncwarp();
        if (lane == 0) set_vol(B.r_head, head + done);
      }
    }
    __syncwarp();
    if (lane == 0 && (watch || idle)) {
      const uint64_t now = globaltimer();
      const uint32_t pr = vol(B.a_prog), hand = vol(B.a_hand);
      if (err != 0u) {
        B.err = err;
        next = AS_DONE;
      } else if (vol(B.a_want) || rows > QR / 2u ||
                 (B.a_cap == NIL && ((hand >= B.a_look && hand > (pr - B.a_prog0) / 4u) ||
                                     crowded >= B.a_patience))) {
        atomicMax(&C->a_req, B.a_gen + 1u);
        next = AS_REBALANCE;
      } else if (watch && (int)(req - B.a_gen) > 0) {
        next = AS_REBALANCE;
      } else if (B.a_token) {
        if (idle) {
          async_release(D, B);
          t0 = now;
        } else if (pr != prog) {
          prog = pr;
          t0 = now;
          if (now - tb > 100000u) {  // a heartbeat every 100 us
            tb = now;
            red_relaxed_add(&C->a_beat, 1u);
          }
        }
      } else if (watch && tok == 0u) {
        // (a CTA that asks for a rebalance holds its token until the
        // rebalance, so a zero count means no rebalance can come)
        next = AS_DONE;
      } else if (watch && bt != beat) {
        beat = bt;
        t0 = now;
      }
      if (next == AS_STEP && now > t0 && now - t0 > D.spin_limit_ns) {
        set_error(D, TRIM_ERR_TIMEOUT, 4);
        B.err = TRIM_ERR_TIMEOUT;
        next = AS_DONE;
      }
    }
    next = __shfl_sync(FULL, next, 0);
    // (polls and sends take from the workers: 6.7 ms on the deep cascade with
    // 1,600 ns and two rows, 9.2 with 200 ns and two, 10.6 with 200 ns and one)
    if (next == AS_STEP) __nanosleep(1600);
  }
  B.ch_sent[lane] = ch.sent;
  B.ch_taken[lane] = ch.taken;
  __syncwarp();
  if (lane == 0) {
    set_vol(B.a_next, next);
    __threadfence_block();
    // (a worker that sets its bit after this sees a_next and does not sleep)
    for (uint32_t w = async_claim(B); w < 32u; w = async_claim(B)) async_wake(B, w, 0u);
  }
  __syncwarp();
}

// All threads, every CTA (generation g = B.a_gen): writes the workers' entries
// and pieces and the ring's pieces to the global lists of parity g & 1; after
// a grid barrier every CTA takes an even slice of those and of the pieces
// written since the last rebalance; tokens follow the new shares and CTA 0
// clears the other parity's counters (last read after rebalance g - 1, by every
// CTA before this rebalance's first barrier); a second barrier publishes both
// before any CTA writes to the lists again. Returns false on an error.
__device__ __forceinline__ bool async_rebalance(const Dev& D, Cta& B, AsyncWarp& A) {
  Ctrl* C = D.C;
  const unsigned lane = lane_id();
  const uint32_t par = B.a_gen & 1u;
  const uint32_t QR = async_ring_cap();
  uint32_t eo = 0, ro = 0;
  A.top = __reduce_max_sync(FULL, A.top);
  if (lane == 0) {
    if (A.cnt) eo = atomicAdd(&B.a_ne, A.cnt);
    if (A.pl) ro = atomicAdd(&B.a_nr, 1u);
    if (A.removed) {
      atomicAdd(&B.a_removed, A.removed);
      atomicMax(&B.a_maxlev, A.top);
    }
  }
  eo = __shfl_sync(FULL, eo, 0);
  A.removed = 0u;
  A.top = 0u;
  __syncthreads();
  const uint32_t head = B.r_head, nring = B.r_tail - head, ne = B.a_ne, nr = B.a_nr + nring;
  if (threadIdx.x == 0) {
    async_publish(D, B);
    if (B.a_hand) atomicAdd(&C->a_hand, B.a_hand);
    B.a_hand = 0u;
    B.a_prog0 = B.a_prog;
    B.a_ebase = ne ? atomicAdd(&C->e_n[par], ne) : 0u;
    B.a_rbase = nr ? atomicAdd(&C->er_n[par], nr) : 0u;
    // (cannot fail: the lists hold what every CTA can hold)
    if ((uint64_t)B.a_ebase + ne > D.ae_cap || (uint64_t)B.a_rbase + nr > D.er_cap)
      set_error(D, TRIM_ERR_STATE, 7);
  }
  __syncthreads();
  if ((uint64_t)B.a_ebase + ne <= D.ae_cap && (uint64_t)B.a_rbase + nr <= D.er_cap) {
    const size_t e0 = (size_t)par * D.ae_cap + B.a_ebase, r0 = (size_t)par * D.er_cap + B.a_rbase;
    if (lane < A.cnt) {
      D.ae_id[e0 + eo + lane] = A.p;
      D.ae_lev[e0 + eo + lane] = A.l;
    }
    for (uint32_t i = threadIdx.x; i < nring; i += blockDim.x) {
      const uint32_t k = (head + i) & (QR - 1u);
      D.er_row[r0 + i] = dyn_smem[k];
      D.er_len[r0 + i] = dyn_smem[QR + k];
      D.er_lev[r0 + i] = dyn_smem[2u * QR + k];
      dyn_smem[QR + k] = 0u;
    }
    if (lane == 0 && A.pl) {
      D.er_row[r0 + nring + ro] = A.pr;
      D.er_len[r0 + nring + ro] = A.pl;
      D.er_lev[r0 + nring + ro] = A.pv;
    }
  }
  A.cnt = 0u;
  A.pl = 0u;
  A.share = true;
  if (!grid_barrier(D, B)) return false;
  if (threadIdx.x == 0) {
    const uint64_t G = gridDim.x, b = blockIdx.x;
    const uint64_t tE = ld_relaxed(&C->e_n[par]), tR = ld_relaxed(&C->er_n[par]);
    const uint32_t p_hi = ld_relaxed(&C->oq_res);
    const uint64_t tP = p_hi - B.a_plo;
    B.sh_elo = (uint32_t)(b * tE / G);
    B.sh_ehi = (uint32_t)((b + 1u) * tE / G);
    B.sh_rlo = (uint32_t)(b * tR / G);
    B.sh_rhi = (uint32_t)((b + 1u) * tR / G);
    B.sh_plo = B.a_plo + (uint32_t)(b * tP / G);
    B.sh_phi = B.a_plo + (uint32_t)((b + 1u) * tP / G);
    B.a_plo = p_hi;
    if (B.a_cap == NIL) {  // (the same decision in every CTA)
      const uint32_t removed = ld_relaxed(&C->a_removed), hand = ld_relaxed(&C->a_hand);
      const uint32_t dr = removed - B.a_seen_removed, dh = hand - B.a_seen_hand;
      const uint32_t top = max(ld_relaxed(&C->a_maxlev), B.S.round - 1u);
      B.a_close = top - B.a_seen_top <= 4u ? B.a_close + 1u : 0u;
      if (tR + tP > async_workers() || (dh >= ASYNC_LOOK && dh > dr / 4u) ||
          B.a_close >= ASYNC_CLOSE)
        B.a_cap = top;
      B.a_seen_top = top;
      B.a_seen_removed = removed;
      B.a_seen_hand = hand;
      B.a_look = min(2u * B.a_look, 1u << 20);
      B.a_patience = min(2u * B.a_patience, 1u << 20);
    }
    B.r_head = B.r_tail;  // the ring went to the list
    B.a_ne = 0u;
    B.a_nr = 0u;
    B.a_want = 0u;
    B.a_gen += 1u;
    B.a_next = AS_STEP;
    const bool busy = B.sh_ehi > B.sh_elo || B.sh_rhi > B.sh_rlo || B.sh_phi > B.sh_plo;
    // (a CTA left without work releases its token later, if it may)
    if (busy && !B.a_token) {
      atomicAdd(&C->a_tokens, 1u);
      B.a_token = 1u;
    }
    if (blockIdx.x == 0) {
      C->e_n[par ^ 1u] = 0u;
      C->er_n[par ^ 1u] = 0u;
      C->a_rebalances = B.a_gen;
    }
  }
  const bool ok = grid_barrier(D, B);
  A.cap = B.a_cap;
  return ok;
}

// End of a tail whose last level was a_cap (all threads): the counters go back to their
// array, and the schedule goes on with round a_cap + 2, which pushes the vertices of level
// a_cap + 1, parked in the work list; where nothing was parked the run has ended (B.S stays
// as it was). Returns false on an error.
__device__ __noinline__ bool async_leave() {
  const Dev& D = cta_dev;
  Cta& B = cta_state;
  Ctrl* C = D.C;
  const uint32_t stride = gridDim.x * blockDim.x;
  unsigned long long pushed = 0;  // by the tail, for vertices without work-list entries
  for (uint64_t v = blockIdx.x * blockDim.x + threadIdx.x; v < D.n; v += stride) {
    const uint4 x = __ldcg(&D.aw[v]);
    D.cnt[v] = x.x;
    if (MODES & M_SCHED) {
      const uint32_t l = ldcg(&D.level[v]);
      pushed += l >= B.S.round && l <= B.a_cap ? x.w : 0u;
    }
  }
  if (MODES & M_SCHED) {
    pushed = warp_sum(pushed);
    if (lane_id() == 0 && pushed) atomicAdd(&C->local_edges, pushed);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    // the next rounds' accumulators (rounds cleared them two ahead)
    for (int k = 0; k < 4; ++k) {
      RoundStat* z = &C->rs[k];
      z->sum_in = 0; z->sum_out = 0;
      z->hist[0] = z->hist[1] = z->hist[2] = 0;
      z->live_count = 0;
      z->max_din = 0;
    }
  }
  if (!grid_barrier(D, B)) return false;
  const unsigned long long w4 = ld_relaxed64(&C->w4);
  if (threadIdx.x == 0 && (uint32_t)w4 != B.S.w_end) {
    Sched& S = B.S;
    const uint32_t removed = ld_relaxed(&C->a_removed) - B.a_base, next = B.a_cap + 2u;
    S.vcount[TRIM_AC4_PUSH] += next - S.round;
    S.prev_variant = TRIM_AC4_PUSH;
    S.fprev = S.fe - S.fb;
    S.round = next;
    S.fe += removed;
    S.fb = S.fe - ((uint32_t)w4 - S.w_end);  // (those with in-edges)
    S.skew += removed;
    S.c4w = S.w_end;
    S.e_c4 = S.e_end;
    S.w_end = (uint32_t)w4;
    S.e_end = (uint32_t)(w4 >> 32);
    S.bmax = ld_relaxed(&C->a_bmax);
    S.stable = D.commit_after ? D.commit_after - 1u : 0u;
    if (MODES & M_SCHED)
      for (int i = 0; i < NFEAT; ++i) S.feat[i] = 0.0f;
    S.async_wait = S.async_wait ? min(2u * S.async_wait, 1u << 20) : ASYNC_WAIT;
    S.async_from = next + S.async_wait;
    if (blockIdx.x == 0) {
      C->vcount[TRIM_AC4_PUSH] = S.vcount[TRIM_AC4_PUSH];
      C->rounds = next;
      C->n_dead = S.fe;
    }
  }
  __syncthreads();
  return true;
}

// Runs the rest of the run asynchronously from round B.S.round = r0 (all
// threads): every vertex's record is set from its counter and its G^T row, and
// the workers push the pending work-list entries (level r0 - 1) and what
// follows from them until the token count is zero. CTA 0 then publishes the
// run's totals: alpha = top level + 1 (r0 if the tail removed nothing), and
// one AC-4 round for each of rounds r0 .. alpha; or, where the tail left (see async_leave),
// rounds go on. Returns false on an error.
__device__ __noinline__ bool async_tail() {
  const Dev& D = cta_dev;
  Cta& B = cta_state;
  Counters K;
  Ctrl* C = D.C;
  const unsigned warp = threadIdx.x >> 5, nwk = (blockDim.x >> 5) - 1u;  // the last warp controls
  const uint32_t r0 = B.S.round, nwork = gridDim.x * nwk;
  {
    constexpr int U = 4;  // records in flight per thread
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t v0 = blockIdx.x * blockDim.x + threadIdx.x; v0 < D.n; v0 += U * stride) {
      uint32_t c[U], s[U], e[U];
#pragma unroll
      for (int q = 0; q < U; ++q) {
        const uint64_t v = (uint64_t)v0 + (uint64_t)q * stride;
        const bool has = v < D.n;
        c[q] = has ? ldcg(&D.cnt[v]) : 0u;
        s[q] = has ? __ldg(&D.ioff[v]) : 0u;
        e[q] = has ? __ldg(&D.ioff[v + 1u]) : 0u;
      }
#pragma unroll
      for (int q = 0; q < U; ++q) {
        const uint64_t v = (uint64_t)v0 + (uint64_t)q * stride;
        if (v < D.n) D.aw[v] = make_uint4(c[q], 0u, s[q], e[q] - s[q]);
      }
    }
  }
  for (uint32_t i = threadIdx.x; i < async_ring_cap(); i += blockDim.x)
    dyn_smem[async_ring_cap() + i] = 0u;
  if (threadIdx.x < 32u) {
    B.ch_sent[threadIdx.x] = B.ch_taken[threadIdx.x] = 0u;
    D.ch_msg[32u * blockIdx.x + threadIdx.x] = make_ulonglong2(0ull, 0ull);
    D.ch_ack[32u * blockIdx.x + threadIdx.x] = 0u;
  }
  if (threadIdx.x == 0) {
    B.r_head = B.r_tail = 0u;
    B.a_idle = 0u;
    for (uint32_t w = 0; w < MAX_WARPS; ++w)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&B.w_bar[w])) : "memory");
    B.a_next = AS_STEP;
    B.sh_elo = B.sh_ehi = B.sh_rlo = B.sh_rhi = B.sh_plo = B.sh_phi = 0u;
    B.a_removed = 0u;
    B.a_maxlev = 0u;
    B.a_ne = B.a_nr = 0u;
    B.a_token = 1u;
    B.a_want = 0u;
    // (what an earlier tail of the run left: nothing changes it between tails)
    B.a_plo = ld_relaxed(&C->oq_res);
    B.a_base = B.a_seen_removed = ld_relaxed(&C->a_removed);
    B.a_seen_hand = ld_relaxed(&C->a_hand);
    B.a_seen_top = r0 - 1u;
    B.a_close = 0u;
    B.a_prog = B.a_prog0 = 0u;
    B.a_cap = NIL;
    B.a_hand = 0u;
    B.a_look = ASYNC_LOOK;
    B.a_patience = ASYNC_PATIENCE;
    D.ch_load[blockIdx.x] = nwk;
    if (blockIdx.x == 0) {
      C->a_tokens = gridDim.x;
      C->a_bmax = 0u;
      if (C->a_round == 0u) C->a_round = r0;
    }
  }
  if (!grid_barrier(D, B, false)) return false;
  AsyncWarp A;
  A.aw = D.aw;
  A.itgt = D.itgt;
  A.level = D.level;
  A.p = A.l = A.cnt = 0u;
  A.pr = A.pl = A.pv = 0u;
  A.wj = warp < nwk ? B.S.c4w + warp * gridDim.x + blockIdx.x : B.S.w_end;
  A.removed = A.top = 0u;
  A.cap = NIL;
  A.phase = 0u;
  A.share = true;
  bool ok = true;
  while (true) {
    if (warp < nwk) async_work(D, B, A, nwork, K);
    else async_control();
    __syncthreads();
    if (B.a_next == AS_DONE) break;
    if (!async_rebalance(D, B, A)) {
      ok = false;
      break;
    }
  }
  stats_flush(D, B, K);
  __syncthreads();
  if (threadIdx.x == 0)  // (the next tail initialises them again)
    for (uint32_t w = 0; w < MAX_WARPS; ++w)
      asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_addr(&B.w_bar[w])) : "memory");
  if (ok && B.err == 0u && B.a_cap != NIL && !async_leave()) return false;
  if (threadIdx.x == 0 && B.S.round == r0) {  // (not handed back to rounds)
    if (blockIdx.x == 0 && ok && B.err == 0u) {
      fence_acq_rel();  // every CTA published its counts before its last release
      const uint32_t removed = ld_relaxed(&C->a_removed) - B.a_base;
      const uint32_t top = ld_relaxed(&C->a_maxlev);
      Sched& S = B.S;
      const uint32_t alpha = removed ? max(r0, top + 1u) : r0;
      S.vcount[TRIM_AC4_PUSH] += alpha - r0 + 1u;
      C->vcount[TRIM_AC4_PUSH] = S.vcount[TRIM_AC4_PUSH];
      C->rounds = alpha;
      C->n_dead = S.fe + removed;
    }
    B.S.done = 1u;
  }
  __syncthreads();
  return ok && B.err == 0u;
}
#endif

#if TRIM_MODES & 16
// ------------------------------------------------------------------ in+out

// In+out round r (Section 4's remark: with G^T loaded a vertex also needs a
// live incoming edge). A vertex whose out-degree counter reached zero has only
// removed successors left, so its G row has no live vertex and only its G^T row is
// pushed (the predecessors' out-degree counters); one whose in-degree counter
// reached zero has only removed predecessors, and only its G row is pushed (the
// successors' in-degree counters). So every work-list entry has one row and its direction,
// half the pushes of walking both. A counter that reaches zero removes its
// vertex in round r unless the other counter had removed it before: both are in
// one word, and the push sees both. Edges are balanced over the warps in
// 32-edge chunks as in ac4_round.
//
// Measured (kernel ms, deep cascades of 5,000,011 vertices and 1,001 rounds / 2^20
// and 251 / R-MAT 2^22 / 2^23): 4.21 / 1.05 / 0.139 / 0.251; with both rows pushed, a
// compare-and-swap of the level and every round through the global lists 8.32 /
// 2.02 / 0.155 / 0.268.
__device__ ROUND_FN void inout_round(const Dev& D, Cta& B, const Sched& S, uint32_t gwarp,
                                     uint32_t nwarps) {
  constexpr int U = 4;
  Counters K;
  const unsigned lane = lane_id();
  const uint32_t r = S.round;
  const uint32_t ea = S.e_c4, eb = S.e_end, ia = S.c4w, ib = S.w_end;
  if (eb <= ea) return;
  const uint32_t c0 = ea >> 5, c1 = (eb + 31u) >> 5;
  const uint32_t per = (c1 - c0 + nwarps - 1) / nwarps;
  const uint32_t cb = c0 + gwarp * per, ce = min(c1, cb + per);
  uint32_t cfb = 0;
  for (uint32_t c = cb; c < ce; c += U) {
    const uint32_t k = (c - cb) & 31u;
    if (k == 0u) cfb = (c + lane < ce) ? ldcg(&D.chunk_first[c + lane]) : 0u;
    uint32_t wrow[U], weo[U], wdir[U], u[U];
    PushWord old[U];
    bool valid[U];
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const uint32_t first = max(__shfl_sync(FULL, cfb, (k + q) & 31u), ia);
      const uint32_t ii = first + lane;
      const bool in = c + q < ce && ii < ib;
      wrow[q] = in ? ldcg(&D.w4_row[ii]) : 0u;
      weo[q] = in ? ldcg(&D.w4_eoff[ii]) : 0xFFFFFFFFu;
      wdir[q] = in ? ldcg(&D.w4_dir[ii]) : 0u;
    }
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const uint32_t e = ((c + q) << 5) + lane;
      valid[q] = c + q < ce && e >= ea && e < eb;
      const unsigned j = owner_of(weo[q], e);
      const uint32_t at = __shfl_sync(FULL, wrow[q], j) + (e - __shfl_sync(FULL, weo[q], j));
      wdir[q] = __shfl_sync(FULL, wdir[q], j);
      u[q] = valid[q] ? __ldg(&push_tgt(D, wdir[q])[at]) : 0u;
    }
#pragma unroll
    for (int q = 0; q < U; ++q) old[q] = valid[q] ? push(D, u[q], wdir[q]) : 0u;
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const bool pred = valid[q] && push_removes(old[q], wdir[q]);
      uint32_t row = 0, len = 0;
      if (pred) {
        row = __ldg(&push_off(D, wdir[q])[u[q]]);
        len = __ldg(&push_off(D, wdir[q])[u[q] + 1u]) - row;
        D.level[u[q]] = r;
      }
      count_rows(D, pred, u[q], K);
      append_dead_io(D, B, pred, r, row, len, wdir[q]);
    }
  }
  stats_flush(D, B, K);
}
#endif

// ------------------------------------------------------------------ AC-3

__device__ ROUND_FN void ac3_round(const Dev& D, Cta& B, const Sched& S, uint32_t gwarp,
                                   uint32_t nwarps) {
  Counters K;
  const unsigned lane = lane_id();
  const uint32_t r = S.round;
  const bool all = (S.ac3_list == NIL);
  const uint32_t* Lin = (S.ac3_list == 1u) ? D.live1 : D.live0;
  uint32_t* Lout = S.live_out ? D.live1 : D.live0;
  const uint32_t N = all ? D.n : S.live_in_len;
  for (uint32_t base = gwarp * 32; base < N; base += nwarps * 32) {
    const uint32_t idx = base + lane;
    const bool has = idx < N;
    const uint32_t v = has ? (all ? idx : ldcg(&Lin[idx])) : 0u;
    const bool alive = has && ldcg(&D.level[v]) == LIVE;
    uint32_t s = 0, d = 0, i0 = 0, i = 0;
    bool resolved = true;
    if (alive) {
      row_bounds(D, v, s, d);
      i0 = S.supp_valid ? ldcg(&D.supp[v]) : 0u;  // no support position yet: the row start
      i = scan_thread(D, v, s, d, i0, r, 2, resolved, K);
    }
    scan_warp_finish(D, resolved, v, s, d, i, r, K);
    const bool dies = alive && i >= d;
    const bool stays = alive && !dies;
    if (stays && (i != i0 || !S.supp_valid)) D.supp[v] = i;
    K.swept += has ? 1 : 0;
    append_dead(D, B, dies, v, r, Lout, false, false, 0, 0, d);
    append_live(D, B, stays, v, r, Lout);
  }
  stats_flush(D, B, K);
}

#if TRIM_LOCAL && TRIM_AC3_ONLY
// A run of AC-3 alone, from round 1 to the end: each CTA sweeps its own vertices
// (every block of 32 in turn, so that the vertices of a level, often neighbours, are
// spread over the CTAs) and keeps its survivors in its own part of the live lists. A round needs no shared list, no space
// reservation, no dead log and no read of the control block; it ends at a fenced
// local barrier that carries the removals. A list entry has all that a sweep needs:
// the vertex, its support, the support's position and the row's end; while the
// support lives, that is the entry and one level. Returns false on a timeout.
//
// Small rounds are bound by their fixed parts (flush and reservations 1.1 us,
// barrier and schedule step 3, the level of every live vertex one more
// dependent load), large ones by the rows. Kernel us per run, through the shared
// lists / with lists per CTA of vertices alone / as here: planted graphs of 1,000
// vertices (17 rounds) 95 / 59 / 59, 100,000 (22) 164 / 116 / 90, 1,000,000 (31) 582 / 446 /
// 275; deep cascade of 2^20 (301) 7,663 / 4,224 / 2,640; R-MAT of 2^22 (4) 231 / 207 / 136.
__device__ __noinline__ bool local_stretch() {
  const Dev& D = cta_dev;
  Cta& B = cta_state;
  Counters K;
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
  const uint32_t n = D.n, blocks = (n + 31u) / 32u;
  // first entry of the CTA's part, and its blocks
  const uint32_t turns = blocks / gridDim.x, left = blocks % gridDim.x;
  const uint32_t part = 32u * (turns * blockIdx.x + min(left, blockIdx.x));
  const uint32_t own = turns + (blockIdx.x < left ? 1u : 0u);
  bool first = true;
  while (true) {
    const uint32_t r = B.S.round;
    const uint32_t b = B.S.lround & 1u;
    const uint4* in = (b ? D.s_rec : D.s_heads) + part;  // written in the last round
    uint4* out = (b ? D.s_heads : D.s_rec) + part;
    start_round(D, r);
    const uint32_t N = first ? own * 32u : B.live_n[b ^ 1u];
    for (uint32_t base = warp * 32u; base < N; base += blockDim.x) {
      const uint32_t k = base + lane;
      bool alive = k < N, stays = false;
      uint4 x = make_uint4(0u, 0u, 0u, 0u);
      if (first) {
        x.x = 32u * (base / 32u * gridDim.x + blockIdx.x) + lane;
        alive = x.x < n;
        K.swept += alive ? 1 : 0;
        alive = alive && ldcg(&D.level[x.x]) == LIVE;
        if (alive) {
          uint32_t s, d;
          row_bounds(D, x.x, s, d);
          x.z = s;
          x.w = s + d;
        }
      } else if (alive) {
        x = __ldcg(&in[k]);
        stays = ldcg(&D.level[x.y]) >= r;
        K.swept += 1;
        K.edges += 1;
      }
      if (__any_sync(FULL, alive && !stays)) {
        const bool scan = alive && !stays;
        uint32_t i = x.z + (first ? 0u : 1u);
        bool resolved = true;
        if (scan) i = scan_thread(D, x.x, 0u, x.w, i, r, 2, resolved, K);
        scan_warp_finish(D, resolved, x.x, 0u, x.w, i, r, K);
        if (scan && i < x.w) {
          stays = true;
          x.y = row_target(D, x.x, 0u, i);
          x.z = i;
        } else if (scan) {
          D.level[x.x] = r;
        }
      }
      const unsigned gone = __ballot_sync(FULL, alive && !stays);
      const unsigned kept = __ballot_sync(FULL, stays);
      uint32_t at = 0;
      if (lane == 0) {
        if (gone) atomicAdd(&B.lq_k, (uint32_t)__popc(gone));
        if (kept) at = atomicAdd(&B.live_n[b], (uint32_t)__popc(kept));
      }
      at = __shfl_sync(FULL, at, 0);
      if (stays) out[at + __popc(kept & ((1u << lane) - 1u))] = x;
    }
    if ((D.flags & F_ROUND_LOG) && blockIdx.x == 0) {
      __syncthreads();
      if (threadIdx.x == 0) D.C->t_work[r & 3] = globaltimer();
    }
    stats_flush(D, B, K);
    K = Counters();
    if (!local_barrier(D, B, b, r)) break;
    if (B.lq_next != LQ_GO) break;  // done (a round cannot overflow)
    first = false;
  }
  return B.err == 0u;
}
#endif

// ------------------------------------------------------------------ AC-6

#if !TRIM_AC6_ONLY
// Warp-collective re-scan of members of a supporting set whose owner was
// removed in round r-1: scan forward from the position after the lost support;
// on success join the new support's set (intrusive list), else remove.
__device__ __forceinline__ void ac6_rescan(const Dev& D, Cta& B, bool valid, uint32_t v,
                                           uint32_t r, Counters& K) {
  const bool alive = valid && ldcg(&D.level[v]) == LIVE;
  uint32_t s = 0, d = 0, i = 0;
  bool resolved = true;
  if (alive) {
    row_bounds(D, v, s, d);
    i = scan_thread(D, v, s, d, ldcg(&D.supp[v]) + 1u, r, 2, resolved, K);
  }
  scan_warp_finish(D, resolved, v, s, d, i, r, K);
  const bool dies = alive && i >= d;
  if (alive && !dies) {
    D.supp[v] = i;
    const uint32_t t = row_target(D, v, s, i);
    D.s_next[v] = atomicExch(&D.s_head[t], v);
  }
  K.cand += valid ? 1 : 0;
  append_dead(D, B, dies, v, r, D.live0, false, false, 0, 0, d);
}

#endif

// Block-wide exclusive scan of one value per thread (blockDim.x <= 1024).
__device__ unsigned block_excl_scan(unsigned x, unsigned* total) {
  __shared__ unsigned wsum[33];
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const unsigned incl = warp_incl_scan(x);
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const unsigned t = lane < nw ? wsum[lane] : 0u;
    const unsigned ti = warp_incl_scan(t);
    wsum[lane] = ti - t;
    if (lane == 31) wsum[32] = ti;
  }
  __syncthreads();
  const unsigned res = incl - x + wsum[warp];
  *total = wsum[32];
  __syncthreads();
  return res;
}

__device__ unsigned block_sum(unsigned x) {
  __shared__ unsigned ws[32];
  const unsigned lane = lane_id(), warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  x = warp_sum(x);
  if (lane == 0) ws[warp] = x;
  __syncthreads();
  unsigned t = 0;
  if (warp == 0) {
    t = lane < nw ? ws[lane] : 0u;
    t = warp_sum(t);
    if (lane == 0) ws[0] = t;
  }
  __syncthreads();
  t = ws[0];
  __syncthreads();
  return t;
}

#if TRIM_AC6_ONLY
// The counters of the entry's counting sort are contended: on skewed graphs with
// sorted rows the first successors of most vertices are a few hubs, and the atomics on
// the hottest line alone took most of the pass. So each CTA counts in a table in
// shared memory first (a slot belongs to the first support that hashes there;
// others go to the global counter) and adds its totals to the global counters at
// the end. A vertex keeps its rank (in its CTA's table, or globally), so the
// scatter needs no atomics. The table lies in append slices that AC-6 does not use:
// keys, counts, and the CTA's first rank of each support.
constexpr uint32_t AC6_HEADS = 4;
// Rows in host memory come over the link, entry by entry as they are needed: after the
// first build a record then holds UNREAD instead of the next successor (ids are below 2^31),
// and row bounds are read once there. (Later re-scans, far fewer, read ahead as elsewhere;
// the check there cost AC-6 of packed graphs 0.7 per cent.) AC-6 of R-MAT of 2^22 vertices
// read in place, call us: 785 with all next successors read ahead, 567 so (574 before the
// records), 2^20 242, 189 (212).
constexpr uint32_t UNREAD = 0xFFFFFFFEu;
__device__ __forceinline__ bool rows_far(const Dev& D) {
  return !(MODES & M_IMPLICIT) && (D.flags & F_ROWS_FAR) != 0u;
}
__device__ __forceinline__ uint32_t* set_head(const Dev& D, uint32_t w, uint32_t q) {
  return reinterpret_cast<uint32_t*>(&D.s_heads[w]) + q;
}
__device__ __forceinline__ uint32_t sort_slots() { return (blockDim.x >> 5) * LW; }
__device__ __forceinline__ uint32_t sort_slot(uint32_t t) {
  return __umulhi(t * 0x9E3779B1u, sort_slots());
}
__device__ __forceinline__ uint32_t* sort_word(uint32_t slot, int which) {
  return &slice(slot / LW, which)[slot % LW];
}

// First pass of the entry in the flavours that run AC-6 alone: every live vertex
// looks for its support, is counted there and gets its record, or is removed. Each
// lane has four vertices in flight, and checks their rows' first successors; the
// vertices that must scan on (about one in eight) wait in a list until they
// fill a warp.
__device__ __forceinline__ void ac6_supports(const Dev& D, Cta& B, uint32_t r, uint32_t gwarp,
                                             uint32_t nwarps) {
  constexpr int U = 4;
  Counters K;
  const unsigned lane = lane_id();
  const uint32_t n = D.n;
  const bool far = rows_far(D);
  for (uint32_t e = threadIdx.x; e < sort_slots(); e += blockDim.x) {
    *sort_word(e, 1) = NIL;
    *sort_word(e, 2) = 0u;
  }
  __syncthreads();
  // counts v's support t: v's rank in the CTA's table or globally
  auto count = [&](uint32_t t) -> uint32_t {
    const uint32_t e = sort_slot(t);
    uint32_t key = *const_cast<volatile uint32_t*>(sort_word(e, 1));
    if (key == NIL) key = atomicCAS(sort_word(e, 1), NIL, t);
    return atomicAdd(key == NIL || key == t ? sort_word(e, 2) : &D.s_cnt[t], 1u);
  };
  // (the support is parked in the link until the scatter)
  auto store = [&](uint32_t v, uint32_t t, uint32_t rank, uint32_t after, uint32_t pos,
                   uint32_t end) {
    D.s_rec[v] = make_uint4(t, after, pos, end);
    D.s_rank[v] = rank;
  };
  uint32_t* list = slice(threadIdx.x >> 5, 3);  // at most 31 + 32 * U entries
  uint32_t nl = 0;
  for (uint32_t base = gwarp * (32u * U);; base += nwarps * (32u * U)) {
    const bool last = base >= n;
    if (!last) {
      uint32_t s[U], d[U], t[U], after[U], x[U];
      bool alive[U];
#pragma unroll
      for (int q = 0; q < U; ++q) {
        const uint32_t v = base + q * 32u + lane;
        alive[q] = v < n && ldcg(&D.level[v]) == LIVE;
        s[q] = d[q] = 0u;
#if !(TRIM_MODES & 32)
        if (v < n) row_bounds(D, v, s[q], d[q]);
#endif
        K.swept += v < n ? 1 : 0;
      }
#pragma unroll
      for (int q = 0; q < U; ++q) {  // (a live vertex has a successor)
        const uint32_t v = base + q * 32u + lane;
#if TRIM_MODES & 32
        if (alive[q]) row_bounds(D, v, s[q], d[q]);
#endif
        t[q] = alive[q] ? row_target(D, v, s[q], 0u) : 0u;
        after[q] = !(alive[q] && d[q] > 1u) ? NIL : far ? UNREAD : row_target(D, v, s[q], 1u);
      }
#pragma unroll
      for (int q = 0; q < U; ++q) {
        x[q] = alive[q] ? ldcg(&D.level[t[q]]) : 0u;
        K.edges += alive[q] ? 1 : 0;
      }
#pragma unroll
      for (int q = 0; q < U; ++q) {
        const bool slow = alive[q] && x[q] < r;
        const unsigned mask = __ballot_sync(FULL, slow);
        if (slow) list[nl + __popc(mask & ((1u << lane) - 1u))] = base + q * 32u + lane;
        if (slow && far) D.s_rec[base + q * 32u + lane] = make_uint4(s[q], d[q], 0u, 0u);
        nl += __popc(mask);
        alive[q] = alive[q] && !slow;
        x[q] = alive[q] ? count(t[q]) : 0u;
      }
#pragma unroll
      for (int q = 0; q < U; ++q)
        if (alive[q])
          store(base + q * 32u + lane, t[q], x[q], after[q], s[q] + 1u, s[q] + d[q]);
      __syncwarp();
    }
    while (nl >= 32u || (last && nl)) {
      const uint32_t take = min(32u, nl);
      const bool has = lane < take;
      const uint32_t v = has ? list[nl - take + lane] : 0u;
      __syncwarp();
      nl -= take;
      uint32_t s = 0, d = 0, i = 0;
      bool resolved = true;
      if (has && far) {  // (its bounds, not to read them again)
        const uint4 x = __ldcg(&D.s_rec[v]);
        s = x.x;
        d = x.y;
      } else if (has) {
        row_bounds(D, v, s, d);
      }
      if (has) i = scan_thread(D, v, s, d, 1u, r, 2, resolved, K);
      scan_warp_finish(D, resolved, v, s, d, i, r, K);
      const bool found = has && i < d;
      if (found) {
        const uint32_t t = row_target(D, v, s, i);
        store(v, t, count(t), i + 1u >= d ? NIL : far ? UNREAD : row_target(D, v, s, i + 1u),
              s + i + 1u, s + d);
      } else if (has) {
        D.s_heads[v] = make_uint4(NIL, NIL, NIL, NIL);
      }
      append_dead(D, B, has && !found, v, r, D.live0);
    }
    if (last) break;
  }
  __syncthreads();
  for (uint32_t e = threadIdx.x; e < sort_slots(); e += blockDim.x) {
    const uint32_t k = *sort_word(e, 2);
    *sort_word(e, 3) = k ? atomicAdd(&D.s_cnt[*sort_word(e, 1)], k) : 0u;
  }
  stats_flush(D, B, K);
}
#else
__device__ __forceinline__ void ac6_supports(const Dev& D, Cta& B, const Sched& S, uint32_t gwarp,
                                             uint32_t nwarps) {
  Counters K;
  const unsigned lane = lane_id();
  const uint32_t r = S.round, n = D.n;
  for (uint32_t base = gwarp * 32; base < n; base += nwarps * 32) {
    const uint32_t v = base + lane;
    const bool has = v < n;
    if (has) D.s_head[v] = NIL;
    const bool alive = has && ldcg(&D.level[v]) == LIVE;
    uint32_t s = 0, d = 0, i0 = 0, i = 0;
    bool resolved = true;
    if (alive) {
      row_bounds(D, v, s, d);
      i0 = S.supp_valid ? ldcg(&D.supp[v]) : 0u;  // no support position yet: the row start
      i = scan_thread(D, v, s, d, i0, r, 2, resolved, K);
    }
    scan_warp_finish(D, resolved, v, s, d, i, r, K);
    const bool dies = alive && i >= d;
    if (alive && !dies) {
      if (i != i0 || !S.supp_valid) D.supp[v] = i;
      const uint32_t t = row_target(D, v, s, i);
      D.s_next[v] = t;  // parked here until the scatter below
      atomicAdd(&D.s_cnt[t], 1u);
    }
    K.swept += has ? 1 : 0;
    append_dead(D, B, dies, v, r, D.live0, false, false, 0, 0, d);
  }
  stats_flush(D, B, K);
}
#endif

// AC-6 entry (the first AC-6 round, or the first after another variant ran):
// every live vertex re-checks its support position, joins the bulk supporting
// set of the support it keeps (a counting sort by support: count, grid-wide
// scan, scatter), or is removed. Three internal grid barriers.
//
// Measured (R-MAT of 2^22 vertices, 1.8 million of them live, kernel us with AC-6
// alone): 168 before, with every count and rank an atomic on the global counter and
// one vertex per lane in flight; 124 now (four in flight alone 197 with the records,
// the counting table 164, scans on in full warps 160, list heads written once 130).
__device__ ROUND_FN bool ac6_entry(const Dev& D, Cta& B, const Sched& S, uint32_t gwarp,
                                   uint32_t nwarps) {
  const unsigned lane = lane_id();
  const uint32_t n = D.n;
#if TRIM_AC6_ONLY
  ac6_supports(D, B, S.round, gwarp, nwarps);
#else
  ac6_supports(D, B, S, gwarp, nwarps);
#endif
  if (!grid_barrier(D, B)) return false;
  // grid-wide exclusive scan of s_cnt into s_off, four entries per thread and step
  const uint32_t chunk = ((n + gridDim.x - 1) / gridDim.x + 31) & ~31u;
  const uint32_t c0 = min(n, blockIdx.x * chunk), c1 = min(n, c0 + chunk);
  auto counts = [&](uint32_t i) -> uint4 {  // entries i .. i+3, i a multiple of 4
    if (i + 3u < c1) return __ldcg(reinterpret_cast<const uint4*>(&D.s_cnt[i]));
    uint4 x = make_uint4(0u, 0u, 0u, 0u);
    if (i < c1) x.x = ldcg(&D.s_cnt[i]);
    if (i + 1u < c1) x.y = ldcg(&D.s_cnt[i + 1u]);
    if (i + 2u < c1) x.z = ldcg(&D.s_cnt[i + 2u]);
    return x;
  };
  {
    unsigned acc = 0;
    for (uint32_t i = c0 + 4u * threadIdx.x; i < c1; i += 4u * blockDim.x) {
      const uint4 x = counts(i);
      acc += x.x + x.y + x.z + x.w;
    }
    acc = block_sum(acc);
    if (threadIdx.x == 0) D.bsum[blockIdx.x] = acc;
  }
  if (!grid_barrier(D, B)) return false;
  {
    unsigned pre = 0;
    for (uint32_t j = threadIdx.x; j < blockIdx.x; j += blockDim.x) pre += ldcg(&D.bsum[j]);
    pre = block_sum(pre);
    for (uint32_t t0 = c0; t0 < c1; t0 += 4u * blockDim.x) {
      const uint32_t i = t0 + 4u * threadIdx.x;
      const uint4 x = i < c1 ? counts(i) : make_uint4(0u, 0u, 0u, 0u);
      unsigned tot;
      const unsigned ex = pre + block_excl_scan(x.x + x.y + x.z + x.w, &tot);
      const uint4 o = make_uint4(ex, ex + x.x, ex + x.x + x.y, ex + x.x + x.y + x.z);
      if (i + 3u < c1) {
        *reinterpret_cast<uint4*>(&D.s_off[i]) = o;
      } else {
        if (i < c1) D.s_off[i] = o.x;
        if (i + 1u < c1) D.s_off[i + 1u] = o.y;
        if (i + 2u < c1) D.s_off[i + 2u] = o.z;
      }
#if TRIM_AC6_ONLY
      // (the counters are zero between builds)
      if (i + 3u < c1) {
        *reinterpret_cast<uint4*>(&D.s_cnt[i]) = make_uint4(0u, 0u, 0u, 0u);
      } else {
        for (uint32_t j = i; j < c1; ++j) D.s_cnt[j] = 0u;
      }
#endif
      pre += tot;
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) D.s_off[n] = pre;
  }
  if (!grid_barrier(D, B)) return false;
  constexpr int U = 4;
  for (uint32_t base = gwarp * (32u * U); base < n; base += nwarps * (32u * U)) {
    uint32_t t[U], off[U], pos[U];
    bool alive[U];
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const uint32_t v = base + q * 32u + lane;
      alive[q] = v < n && ldcg(&D.level[v]) == LIVE;
    }
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const uint32_t v = base + q * 32u + lane;
#if TRIM_AC6_ONLY
      t[q] = alive[q] ? ldcg(&D.s_rec[v].x) : 0u;
      pos[q] = alive[q] ? ldcg(&D.s_rank[v]) : 0u;
#else
      t[q] = alive[q] ? ldcg(&D.s_next[v]) : 0u;
#endif
    }
#pragma unroll
    for (int q = 0; q < U; ++q) {
      off[q] = alive[q] ? ldcg(&D.s_off[t[q]]) : 0u;
#if !TRIM_AC6_ONLY
      pos[q] = alive[q] ? atomicSub(&D.s_cnt[t[q]], 1u) - 1u : 0u;  // (back to zero)
#endif
    }
#pragma unroll
    for (int q = 0; q < U; ++q) {
      if (!alive[q]) continue;
      const uint32_t v = base + q * 32u + lane;
#if TRIM_AC6_ONLY
      const uint32_t e = sort_slot(t[q]);
      if (*sort_word(e, 1) == t[q]) pos[q] += *sort_word(e, 3);
      D.s_heads[v] = make_uint4(NIL, NIL, NIL, NIL);
#endif
      pos[q] += off[q];
      if (pos[q] >= n) set_error(D, TRIM_ERR_STATE, 0xD2);  // counts out of step
      else D.s_list[pos[q]] = v;
    }
  }
  return true;
}

#if TRIM_AC6_ONLY
// AC-6 rounds of the flavours that run nothing else. What bounds a deep run is the
// chain of dependent random accesses in each round, so every vertex with a support
// has a record of 16 bytes: the next member of its list, the successor to try when
// its support goes (already read from the row, NIL at the row's end), that successor's
// position and the row's end. A walk of a set finds all a re-scan needs in one
// access per hop, and the vertex that dies (no successor left) needs no other. A
// member that moves checks the successor's level, and reads its row's next entry
// for the new record meanwhile. A vertex has four list heads, and members go to the
// one that a hash of their id gives: the hops down a set run side by side (sets
// of some tens of members in the first rounds of a deep graph).
//
// Measured (kernel ms per run, before: one list head, members' level, position and row
// loaded one after the other, every round through the global lists): deep
// cascades of 1,000,003 vertices and 1,503 rounds 16.7 and now 10.2, of 2^20 and 2,802
// rounds 33.2 and 19.1, of 2^16 and 302 rounds 3.4 and 2.08. On the way: local rounds
// without the records 13.7 (one head 17.3, two 14.6, sixteen 12.3), with records and
// one general walk for all rounds 13.1, with the short walk and queues per CTA 10.6. A
// round is now 6.4 us: about 3.5 of it a walk and a move (a warp alone
// on its scheduler takes 5 cycles an instruction, an access 400, an atomic 800), 0.65
// the fence, 1.1 the barrier.

// Warp-collective, local rounds: space in the dead log for the lanes of mask (lane 0's
// atomic, under way until log_removed).
__device__ __forceinline__ uint32_t log_space(const Dev& D, Cta& B, unsigned mask) {
  uint32_t at = 0;
  if (mask && lane_id() == 0) {
    at = atomicAdd(&D.C->log_len, (uint32_t)__popc(mask));
    atomicAdd(&B.lq_k, (uint32_t)__popc(mask));
  }
  return at;
}
__device__ __forceinline__ void log_removed(const Dev& D, unsigned mask, uint32_t at, uint32_t u,
                                            uint32_t r) {
  if (mask == 0u) return;
  at = __shfl_sync(FULL, at, 0);
  if (at + __popc(mask) > D.n) {
    if (lane_id() == 0) set_error(D, TRIM_ERR_STATE, 0xD8);
  } else if (mask >> lane_id() & 1u) {
    D.log[at + __popc(mask & ((1u << lane_id()) - 1u))] = u;
    D.level[u] = r;
  }
}

// Warp-collective re-scan of members v of sets whose owner was removed in round
// r - 1, from their records (next successor t at position pos of a row that
// ends at end): the first live successor from there on takes them into its set,
// without one they are removed.
template <bool LOCAL>
__device__ __forceinline__ void ac6_rescan(const Dev& D, Cta& B, bool valid, uint32_t v, uint32_t t,
                                           uint32_t pos, uint32_t end, uint32_t r, Counters& K) {
  if (!(MODES & M_IMPLICIT) && valid && t == UNREAD) t = row_target(D, v, 0u, pos);
  const bool cand = valid && t != NIL;
  // members without a successor left die: their log space is asked for first
  const unsigned now = __ballot_sync(FULL, valid && !cand);
  const uint32_t at = LOCAL ? log_space(D, B, now) : 0u;
  uint32_t lv = 0, after = NIL;
  if (cand) {
    lv = ldcg(&D.level[t]);
    if (pos + 1u < end) after = row_target(D, v, 0u, pos + 1u);
    K.edges += 1;
  }
  bool found = cand && lv >= r;
  const unsigned scan = __ballot_sync(FULL, cand && !found);
  if (scan) {  // the rare case: scan on
    uint32_t i = pos + 1u;
    bool resolved = !(cand && !found);
    // one or two rows: the whole warp scans each, 32 successors in one step; more of
    // them: each lane its own first, four successors in a step
    if (__popc(scan) > 2 && !resolved) i = scan_thread(D, v, 0u, end, i, r, 2, resolved, K);
    scan_warp_finish(D, resolved, v, 0u, end, i, r, K);
    if (cand && !found && i < end) {
      found = true;
      pos = i;
      t = row_target(D, v, 0u, i);
      after = i + 1u < end ? row_target(D, v, 0u, i + 1u) : NIL;
    }
  }
  if (found) {
    const uint32_t next = atomicExch(set_head(D, t, (v * 0x9E3779B1u) >> 30), v);
    D.s_rec[v] = make_uint4(next, after, pos + 1u, end);
  }
  K.cand += valid ? 1 : 0;
  if (LOCAL) {
    log_removed(D, now, at, v, r);
    const unsigned late = __ballot_sync(FULL, cand && !found);  // after a scan
    if (late) log_removed(D, late, log_space(D, B, late), v, r);
  } else {
    append_dead(D, B, valid && !found, v, r, D.live0);
  }
}

// Warp-collective: re-scans the supporting sets of up to 32 removed vertices,
// the w of lanes < G with has. Members are staged with their records, up to 64, in
// an append slice that AC-6 does not use.
__device__ __forceinline__ void ac6_sets(const Dev& D, Cta& B, bool has, uint32_t w, uint32_t G,
                                         uint32_t r, Counters& K) {
  const unsigned lane = lane_id();
  uint4* st = reinterpret_cast<uint4*>(slice(threadIdx.x >> 5, 1));
  // bulk members of S(w): contiguous, spread over the lanes
  uint32_t ss = 0, sd = 0;
  if (has) {
    ss = ldcg(&D.s_off[w]);
    sd = ldcg(&D.s_off[w + 1]) - ss;
  }
  uint32_t kb = 0, total = 0, excl = 0;
  unsigned nbuf = 0;
  for (unsigned q0 = 0; q0 < G * AC6_HEADS; q0 += 32) {
    // members that joined S(w) during the epoch: 32 lists at a time
    const unsigned j = (q0 + lane) / AC6_HEADS;  // below 32, as G is at most 32
    const uint32_t wj = __shfl_sync(FULL, w, j);
    const bool hj = __shfl_sync(FULL, has ? 1 : 0, j) != 0 && j < G;
    uint32_t cur = hj ? ldcg(set_head(D, wj, lane % AC6_HEADS)) : NIL;
    if (q0 == 0) {
      const unsigned incl = warp_incl_scan(sd);
      total = __shfl_sync(FULL, incl, 31);
      excl = incl - sd;
    }
    unsigned steps = 0;
    // bulk members, then the lists' (all walkers hop in step), are staged; re-scans
    // run 32 at a time. A member's record is read before it can be re-scanned
    // (and move to another set).
    while (true) {
      const unsigned wm = __ballot_sync(FULL, cur != NIL);
      bool stage = false, hop = false;
      uint32_t v = 0, at = nbuf + lane;
      if (kb < total) {
        const uint32_t k = kb + lane;
        const unsigned o = G == 1 ? 0u : owner_of(excl, k);
        const unsigned so = __shfl_sync(FULL, ss, o), eo = __shfl_sync(FULL, excl, o);
        stage = k < total;
        if (stage) v = ldcg(&D.s_list[so + (k - eo)]);
        nbuf += min(32u, total - kb);
        kb += 32u;
      } else if (wm) {
        if (++steps > D.n) {  // a set holds at most n members: longer means a broken list
          if (lane == 0) set_error(D, TRIM_ERR_STATE, 0xD4);
          return;
        }
        stage = hop = cur != NIL;
        v = cur;
        at = nbuf + __popc(wm & ((1u << lane) - 1u));
        nbuf += __popc(wm);
      } else if (nbuf == 0u) {
        break;
      }
      if (stage) {
        const uint4 x = __ldcg(&D.s_rec[v]);
        if (hop) cur = x.x;
        st[at] = make_uint4(v, x.y, x.z, x.w);
      }
      __syncwarp();
      const bool more = __any_sync(FULL, cur != NIL) || kb < total;
      while (nbuf >= 32u || (!more && nbuf > 0u)) {
        const unsigned take = min(32u, nbuf);
        const bool valid = lane < take;
        const uint4 m = st[valid ? nbuf - take + lane : 0u];
        __syncwarp();
        nbuf -= take;
        ac6_rescan<false>(D, B, valid, m.x, m.y, m.z, m.w, r, K);
      }
    }
  }
}

// The same for the set of one removed vertex w in a local round. A warp that runs
// alone on its scheduler pays for every instruction as well: this is the short form.
__device__ __forceinline__ void ac6_set(const Dev& D, Cta& B, uint32_t w, uint32_t r, Counters& K) {
  const unsigned lane = lane_id();
  uint4* st = reinterpret_cast<uint4*>(slice(threadIdx.x >> 5, 1));
  uint32_t cur = lane < AC6_HEADS ? ldcg(set_head(D, w, lane)) : NIL;
  const uint32_t ss = ldcg(&D.s_off[w]), total = ldcg(&D.s_off[w + 1]) - ss;
  uint32_t kb = 0, steps = 0;
  unsigned nbuf = 0, wm = __ballot_sync(FULL, cur != NIL);
  while (wm || kb < total) {
    if (kb < total) {
      if (kb + lane < total) {
        const uint32_t v = ldcg(&D.s_list[ss + kb + lane]);
        const uint4 x = __ldcg(&D.s_rec[v]);
        st[nbuf + lane] = make_uint4(v, x.y, x.z, x.w);
      }
      nbuf += min(32u, total - kb);
      kb += 32u;
    } else {
      if (cur != NIL) {
        const uint4 x = __ldcg(&D.s_rec[cur]);
        st[nbuf + __popc(wm & ((1u << lane) - 1u))] = make_uint4(cur, x.y, x.z, x.w);
        cur = x.x;
      }
      nbuf += __popc(wm);
      wm = __ballot_sync(FULL, cur != NIL);
      if (++steps > D.n) {  // a set holds at most n members: longer means a broken list
        if (lane == 0) set_error(D, TRIM_ERR_STATE, 0xD4);
        return;
      }
    }
    __syncwarp();
    while (nbuf >= 32u || (nbuf && !wm && kb >= total)) {
      const unsigned take = min(32u, nbuf);
      const bool valid = lane < take;
      const uint4 m = st[valid ? nbuf - take + lane : 0u];
      __syncwarp();
      nbuf -= take;
      ac6_rescan<true>(D, B, valid, m.x, m.y, m.z, m.w, r, K);
    }
  }
}

__device__ ROUND_FN bool ac6_round(const Dev& D, Cta& B, const Sched& S, uint32_t gwarp,
                                   uint32_t nwarps) {
  if (S.prev_variant != TRIM_AC6_SUPPORT) return ac6_entry(D, B, S, gwarp, nwarps);
  Counters K;
  const unsigned lane = lane_id();
  const uint32_t r = S.round;
  const uint32_t N = S.fe - S.fb;
  const uint32_t G = min(32u, max(1u, (N + nwarps - 1) / nwarps));
  for (uint32_t base = S.fb + gwarp * G; base < S.fe; base += nwarps * G) {
    const uint32_t item = base + lane;
    const bool has = lane < G && item < S.fe;
    const uint32_t w = has ? ldcg(&D.log[item - S.skew]) : 0u;  // (as in the other ac6_round)
    ac6_sets(D, B, has, w, G, r, K);
  }
  stats_flush(D, B, K);
  return true;
}

// Local AC-6 rounds, from round B.S.round on: the removals of the last round, in the
// dead log, are spread over all warps, and a warp writes what its set removes to the
// log at once. A round needs no slices, no flush and no read of the control block; it
// ends at a fenced local barrier that carries its totals (the fence covers the
// log, levels, records and heads). The stretch ends when nothing was removed (the
// run is done), or with more removals than warps, for ordinary rounds.
// Returns false on a timeout.
//
// One log for all CTAs, an atomic and a load more per round than a queue in each:
// a vertex stays with the set it leaves last, so the queues of few CTAs filled up
// (175 to 229 of 304 CTAs had none) and had to be spread again by ordinary rounds. Kernel
// ms with those queues / with the log: 1,000,003 vertices in 1,503 rounds 10.6 / 10.2, 2^20 in
// 301 3.09 / 2.49, planted 100,000 0.187 / 0.158.
__device__ __noinline__ bool local_stretch() {
  const Dev& D = cta_dev;
  Cta& B = cta_state;
  Counters K;
  const uint32_t nw = gridDim.x * (blockDim.x >> 5);
  while (true) {
    const uint32_t r = B.S.round;
    start_round(D, r);
    const uint32_t from = B.S.fb - B.S.skew, N = B.S.fe - B.S.fb;
    for (uint32_t k = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; k < N; k += nw)
      ac6_set(D, B, ldcg(&D.log[from + k]), r, K);
    if ((D.flags & F_ROUND_LOG) && blockIdx.x == 0) {
      __syncthreads();
      if (threadIdx.x == 0) D.C->t_work[r & 3] = globaltimer();
    }
    if (!local_barrier(D, B, B.S.lround & 1u, r)) break;
    if (B.lq_next != LQ_GO || B.S.fe - B.S.fb > nw) break;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) D.C->local_rounds = B.S.lround;
  stats_flush(D, B, K);
  return B.err == 0u;
}
#else
__device__ ROUND_FN bool ac6_round(const Dev& D, Cta& B, const Sched& S, uint32_t gwarp,
                                   uint32_t nwarps) {
  if (S.prev_variant != TRIM_AC6_SUPPORT) return ac6_entry(D, B, S, gwarp, nwarps);
  Counters K;
  const unsigned lane = lane_id();
  const uint32_t r = S.round;
  const uint32_t N = S.fe - S.fb;
  const uint32_t G = min(32u, max(1u, (N + nwarps - 1) / nwarps));
  uint32_t* wb = B.wbuf[threadIdx.x >> 5];
  for (uint32_t base = S.fb + gwarp * G; base < S.fe; base += nwarps * G) {
    const uint32_t item = base + lane;
    const bool has = lane < G && item < S.fe;
    // F_{r-1} was logged by an AC-6 round: its entries sit `skew` positions
    // below their counts (removals counted only by local rounds are not logged)
    const uint32_t w = has ? ldcg(&D.log[item - S.skew]) : 0u;
    uint32_t cur = has ? ldcg(&D.s_head[w]) : NIL;
    // bulk members of S(w): contiguous, spread over the lanes
    uint32_t ss = 0, sd = 0;
    if (has) {
      ss = ldcg(&D.s_off[w]);
      sd = ldcg(&D.s_off[w + 1]) - ss;
    }
    const unsigned incl = warp_incl_scan(sd);
    const unsigned total = __shfl_sync(FULL, incl, 31);
    const unsigned excl = incl - sd;
    for (unsigned k0 = 0; k0 < total; k0 += 32) {
      const unsigned k = k0 + lane;
      const bool valid = k < total;
      const unsigned j = G == 1 ? 0u : owner_of(excl, k);
      const unsigned sj = __shfl_sync(FULL, ss, j), ej = __shfl_sync(FULL, excl, j);
      const uint32_t v = valid ? ldcg(&D.s_list[sj + (k - ej)]) : 0u;
      ac6_rescan(D, B, valid, v, r, K);
    }
    // members that joined S(w) during the epoch (intrusive lists): all walkers
    // hop in step and stage the members; re-scans run 32 at a time. A member's
    // next pointer is read before it can be re-scanned (and move to another set).
    unsigned nbuf = 0, steps = 0;
    while (true) {
      const bool walking = cur != NIL;
      const unsigned wm = __ballot_sync(FULL, walking);
      if (wm == 0u && nbuf == 0u) break;
      if (wm) {
        if (++steps > D.n) {  // a set holds at most n members: longer means a broken list
          if (lane == 0) set_error(D, TRIM_ERR_STATE, 0xD4);
          break;
        }
        if (walking) {
          const uint32_t v = cur;
          cur = ldcg(&D.s_next[v]);
          wb[nbuf + __popc(wm & ((1u << lane) - 1u))] = v;
        }
        nbuf += __popc(wm);
        __syncwarp();
      }
      const bool more = __any_sync(FULL, cur != NIL);
      while (nbuf >= 32u || (!more && nbuf > 0u)) {
        const unsigned take = min(32u, nbuf);
        const bool valid = lane < take;
        const uint32_t v = valid ? wb[nbuf - take + lane] : 0u;
        __syncwarp();
        nbuf -= take;
        ac6_rescan(D, B, valid, v, r, K);
      }
    }
  }
  stats_flush(D, B, K);
  return true;
}
#endif

// ------------------------------------------------------------------ init (round 0)

// Each warp takes U blocks of 32 consecutive vertices at a time and issues all
// their offset loads (and G^T offsets, needed for the sinks' work-list entries)
// before using any: the pass is bound by memory parallelism, not by bandwidth.
__device__ ROUND_FN void init_round(const Dev& D, Cta& B, uint32_t gwarp, uint32_t nwarps) {
  constexpr int U = 4;
  const unsigned lane = lane_id();
  const uint32_t n = D.n;
  [[maybe_unused]] const bool w4 = (D.flags & F_AC4_POSSIBLE) != 0;
  const bool rows = D.ioff != nullptr;
#if TRIM_MODES & 16
  Counters K;
#endif
  for (uint32_t base = gwarp * (32u * U); base < n; base += nwarps * (32u * U)) {
    uint32_t o0[U], o1[U], i0[U], i1[U];
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const uint32_t v = base + q * 32u + lane;
      const bool has = v < n;
#if TRIM_MODES & 32
      o0[q] = 0u;
      o1[q] = has ? ig_degree(D, v) : 0u;
#else
      o0[q] = has ? __ldg(&D.off[v]) : 0u;
      o1[q] = has ? __ldg(&D.off[v + 1]) : 0u;
#endif
#if TRIM_MODES & 16
      // in+out needs every vertex's in-degree
      i0[q] = (has && rows) ? __ldg(&D.ioff[v]) : 0u;
      i1[q] = (has && rows) ? __ldg(&D.ioff[v + 1]) : 0u;
#endif
    }
#if !(TRIM_MODES & 16)
    // one-sided: only the vertices removed here (no out-edge) need their G^T
    // row, for their work-list entry; the loads of all four blocks go out together
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const bool sink = base + q * 32u + lane < n && o1[q] == o0[q];
      i0[q] = (sink && rows) ? __ldg(&D.ioff[base + q * 32u + lane]) : 0u;
      i1[q] = (sink && rows) ? __ldg(&D.ioff[base + q * 32u + lane + 1]) : 0u;
    }
#endif
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const uint32_t v = base + q * 32u + lane;
      const bool has = v < n;
      const uint32_t d = o1[q] - o0[q];
#if TRIM_MODES & 16
      // in+out: no out-edge or no in-edge removes the vertex in round 0
      const uint32_t din = i1[q] - i0[q];
      if (has) {
        D.level[v] = (d && din) ? LIVE : 0u;
        D.cnt_io[v] = ((unsigned long long)din << 32) | d;
      }
      const bool dies = has && (d == 0u || din == 0u);
      if (dies) K.pushed += din, K.edges += d;
      append_dead_io(D, B, dies, 0u, d ? o0[q] : i0[q], d ? d : din, d ? 1u : 0u);
#else
      if (has) {
        D.level[v] = d ? LIVE : 0u;
        if (w4) D.cnt[v] = d;
      }
      append_dead(D, B, has && d == 0u, v, 0u, D.live0, true, true, i0[q], i1[q] - i0[q]);
#endif
    }
  }
#if TRIM_MODES & 16
  stats_flush(D, B, K);
#endif
}

#if !(TRIM_MODES & 48)
// Initial pass with a dead mask (vertex sampling, Section 9): a masked vertex
// is DEAD from the start: level 0 (removed before round 1 for every variant),
// counter 0 (a decrement can never return 1), never on the work list, not
// counted. An unmasked vertex counts its unmasked successors: with none it is
// removed in round 0, else it is LIVE with that count as its AC-4 counter.
// With AC-4 every edge of an unmasked vertex is counted: each warp takes 32
// vertices and walks their edges laid end to end, 32 per step with four
// steps' loads in flight; a vertex's count in a step is the popcount of the
// step's unmasked-target ballot over the lanes that hold its edges. Rows with
// more than kMaskHeavy edges wait until the end, when a warp takes each of them
// or, with more than kMaskGiant, the whole CTA. A run
// without AC-4 needs only whether one unmasked successor exists, so each lane
// scans its own row and stops at the first one (rows longer than 32: the
// whole warp).
__device__ __forceinline__ uint32_t lane_range(uint32_t a, uint32_t b) {  // bits [a, b), b <= 32
  const uint32_t hi = b >= 32u ? 0xFFFFFFFFu : ((1u << b) - 1u);
  const uint32_t lo = a >= 32u ? 0xFFFFFFFFu : ((1u << a) - 1u);
  return hi & ~lo;
}

constexpr uint32_t kMaskHeavy = 512;
constexpr uint32_t kMaskGiant = 2048;
constexpr uint32_t kMaskHeavyCap = LW - MAX_WARPS;  // list + per-warp sums in one slice
constexpr uint32_t kMaskOnce = 1u << 21;  // from here on targets pass by the L1

// The mask comes as one bit per vertex: the pass is bound by the look-ups of the
// targets' marks (random accesses), and the bits of the targets that skewed graphs
// keep asking for stay in the L1, which the streamed targets pass by where the bits fill
// it (from kMaskOnce vertices on; below, the targets' next sectors are worth keeping).
// There, blocks of 32 vertices go to the CTAs in turn, so that a small graph of long rows
// has all SMs at work. Kernel us, a byte per vertex and rows over 1,024 by the CTA / bits,
// always passing by and blocks next to each other / as here: R-MAT of 3,000,017 vertices,
// half of them masked, 264 / 194 / 186, 1,000,000 118 / 82 / 79, 1,000,000 vertices with 16
// random successors 50 / 55 / 44, 20,000 with 800 161 / 235 / 34.
// kMaskHeavy of 256 / 512 / 1,024: R-MAT of 3,000,017 201 / 191 / 191, 20,000 with 800 34 / 34 / 149;
// kMaskGiant of 2,048 / 4,096 / 16,384: R-MAT 186 / 191 / 223, 5,000 vertices with 3,000 33 / 41 / 41.
__device__ __forceinline__ bool is_masked(const Dev& D, uint32_t v) {
  return __ldg(&D.mask[v >> 5]) >> (v & 31u) & 1u;
}
__device__ __forceinline__ uint32_t ld_once(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

__device__ ROUND_FN void init_round_masked(const Dev& D, Cta& B) {
  const unsigned lane = lane_id();
  const uint32_t n = D.n;
  const uint32_t nwarps = gridDim.x * (blockDim.x >> 5);
  const bool once = n >= kMaskOnce;
  const uint32_t gwarp = once ? blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)
                              : (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const bool w4 = (D.flags & F_AC4_POSSIBLE) != 0;
  // the CTA's deferred heavy rows and its reduction scratch: warp 0's live-list
  // slice, which no append of this pass uses (its work-list slices stay in
  // buffers 1 and 2: w4_wide is 0 here)
  uint32_t* heavy = slice(0, 3);
  uint32_t* wsum = heavy + kMaskHeavyCap;
  if (threadIdx.x == 0) B.lq_scratch = 0u;
  __syncthreads();
  // the next 32 vertices' mark, row and G^T row are loaded while the last are counted
  uint32_t next[5];
  auto load = [&](uint32_t v) {
    const bool in = v < n;
    next[0] = in && is_masked(D, v) ? 1u : 0u;
    next[1] = in ? __ldg(&D.off[v]) : 0u;
    next[2] = in ? __ldg(&D.off[v + 1]) : 0u;
    next[3] = in && w4 ? __ldg(&D.ioff[v]) : 0u;
    next[4] = in && w4 ? __ldg(&D.ioff[v + 1]) : 0u;
  };
  load(gwarp * 32u + lane);
  for (uint32_t base = gwarp * 32u; base < n; base += nwarps * 32u) {
    const uint32_t v = base + lane;
    const bool has = v < n;
    const bool masked = next[0] != 0u;
    const uint32_t s = next[1], d = next[2] - next[1];
    const uint32_t irow = next[3], din = next[4] - next[3];
    load(min(base + nwarps * 32u, n) + lane);
    uint32_t c = 0;
    bool deferred = false;
    if (w4 && !masked && d > kMaskHeavy) {
      const uint32_t at = atomicAdd(&B.lq_scratch, 1u);
      if (at < kMaskHeavyCap) {
        heavy[at] = v;
        deferred = true;
      }
    }
    if (w4) {
      const uint32_t dd = (masked || deferred) ? 0u : d;
      const uint32_t incl = warp_incl_scan(dd), excl = incl - dd;
      const uint32_t total = __shfl_sync(FULL, incl, 31);
      for (uint32_t k0 = 0; k0 < total; k0 += 128u) {  // warp-uniform
        uint32_t at[4], t[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint32_t k = k0 + (uint32_t)q * 32u + lane;
          const unsigned o = owner_of(excl, k);
          const uint32_t so = __shfl_sync(FULL, s, o), xo = __shfl_sync(FULL, excl, o);
          at[q] = so + (k - xo);
        }
        if (once) {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            t[q] = k0 + (uint32_t)q * 32u + lane < total ? ld_once(&D.tgt[at[q]]) : 0u;
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            t[q] = k0 + (uint32_t)q * 32u + lane < total ? __ldg(&D.tgt[at[q]]) : 0u;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint32_t cs = k0 + (uint32_t)q * 32u;  // flattened index of lane 0
          const bool live = cs + lane < total && !is_masked(D, t[q]);
          const uint32_t bal = __ballot_sync(FULL, live);
          const uint32_t a = excl <= cs ? 0u : min(excl - cs, 32u);
          const uint32_t e = excl + dd;
          const uint32_t b = e <= cs ? 0u : min(e - cs, 32u);
          c += __popc(bal & lane_range(a, b));
        }
      }
    } else {
      const bool own = has && !masked && d <= 32u;  // scanned by its own lane
      for (uint32_t k0 = 0; k0 < (own ? d : 0u) && c == 0u; k0 += 4u) {
        uint32_t tq[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) tq[q] = (k0 + q < d) ? __ldg(&D.tgt[s + k0 + q]) : 0u;
#pragma unroll
        for (int q = 0; q < 4; ++q) c += (k0 + q < d && !is_masked(D, tq[q])) ? 1u : 0u;
      }
      unsigned big = __ballot_sync(FULL, has && !masked && d > 32u);
      while (big) {
        const int j = __ffs(big) - 1;
        big &= big - 1u;
        const uint32_t sj = __shfl_sync(FULL, s, j), dj = __shfl_sync(FULL, d, j);
        uint32_t part = 0;
        for (uint32_t k0 = 0; k0 < dj; k0 += 128u) {  // warp-uniform
          uint32_t tq[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint32_t k = k0 + (uint32_t)q * 32u + lane;
            tq[q] = k < dj ? __ldg(&D.tgt[sj + k]) : 0u;
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint32_t k = k0 + (uint32_t)q * 32u + lane;
            part += (k < dj && !is_masked(D, tq[q])) ? 1u : 0u;
          }
          if (__any_sync(FULL, part != 0u)) break;
        }
        part = __reduce_add_sync(FULL, part);
        if ((int)lane == j) c = part;
      }
    }
    // (a deferred row is counted below; every lane takes part in append_dead,
    // a warp-collective call)
    if (has && !deferred) {
      D.level[v] = (masked || c == 0u) ? 0u : LIVE;
      if (w4) D.cnt[v] = masked ? 0u : c;
    }
    append_dead(D, B, has && !masked && !deferred && c == 0u, v, 0u, D.live0, true, w4, irow, din);
  }
  __syncthreads();
  const uint32_t nh = min(B.lq_scratch, kMaskHeavyCap);
  const unsigned warp = threadIdx.x >> 5;
  for (uint32_t h = warp; h < nh; h += blockDim.x >> 5) {  // a warp to a row
    const uint32_t v = heavy[h];
    const uint32_t s = __ldg(&D.off[v]), e = __ldg(&D.off[v + 1]);
    if (e - s > kMaskGiant) continue;
    uint32_t part = 0;
    const uint32_t d = e - s;
    for (uint32_t k0 = lane; k0 < d; k0 += 256u) {
      uint32_t tq[8];
#pragma unroll
      for (int q = 0; q < 8; ++q)
        tq[q] = k0 + q * 32u < d ? ld_once(&D.tgt[s + k0 + q * 32u]) : 0u;
#pragma unroll
      for (int q = 0; q < 8; ++q)
        part += (k0 + q * 32u < d && !is_masked(D, tq[q])) ? 1u : 0u;
    }
    part = __reduce_add_sync(FULL, part);
    if (lane == 0) {
      D.level[v] = part ? LIVE : 0u;
      D.cnt[v] = part;
    }
    append_dead(D, B, lane == 0 && part == 0u, v, 0u, D.live0, true);
  }
  for (uint32_t h = 0; h < nh; ++h) {  // block-uniform
    const uint32_t v = heavy[h];
    const uint32_t s = __ldg(&D.off[v]), e = __ldg(&D.off[v + 1]);
    if (e - s <= kMaskGiant) continue;
    uint32_t part = 0;
    for (uint32_t k0 = s; k0 < e; k0 += 4u * blockDim.x) {
      uint32_t tq[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t k = k0 + (uint32_t)q * blockDim.x + threadIdx.x;
        tq[q] = k < e ? __ldg(&D.tgt[k]) : 0u;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t k = k0 + (uint32_t)q * blockDim.x + threadIdx.x;
        part += (k < e && !is_masked(D, tq[q])) ? 1u : 0u;
      }
    }
    part = __reduce_add_sync(FULL, part);
    if (lane == 0) wsum[warp] = part;
    __syncthreads();
    if (warp == 0) {
      uint32_t c = lane < (blockDim.x >> 5) ? wsum[lane] : 0u;
      c = __reduce_add_sync(FULL, c);
      if (lane == 0) {
        D.level[v] = c ? LIVE : 0u;
        D.cnt[v] = c;
      }
      append_dead(D, B, lane == 0 && c == 0u, v, 0u, D.live0, true);
    }
    __syncthreads();
  }
}
#endif

}  // namespace

#ifndef TRIM_MIN_BLOCKS
#define TRIM_MIN_BLOCKS 2
#endif
__global__ void __launch_bounds__(512, TRIM_MIN_BLOCKS) TRIM_KERNEL(const __grid_constant__ Dev P) {
  Cta& B = cta_state;
  {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(&P);
    uint32_t* dst = reinterpret_cast<uint32_t*>(&cta_dev);
    for (unsigned i = threadIdx.x; i < sizeof(Dev) / 4; i += blockDim.x) dst[i] = src[i];
  }
  const uint32_t wpb = blockDim.x >> 5;
  const uint32_t nwarps = gridDim.x * wpb;
  const uint32_t gwarp = blockIdx.x * wpb + (threadIdx.x >> 5);
  if (P.flags & F_CONTINUE) {
    // enqueued behind a run's first segment: resume the run if that segment
    // handed it over; else (the run is over or failed) return at once
    if (threadIdx.x == 0) {
      const volatile Ctrl* C = P.C;
      B.skip = (C->err == 0u && C->resume != 0u) ? 0u : 1u;
    }
    __syncthreads();
    if (B.skip) return;  // every CTA read the same control block: all return
  }
  if (threadIdx.x == 0) {
    Sched& S = B.S;
    if (P.flags & F_CONTINUE) {
      B.resume = 1u;
      B.bar_base = ((const volatile Ctrl*)P.C)->bar;
    } else {
      B.resume = P.resume;
      B.bar_base = P.bar_base;
    }
    B.mode = P.mode;
    if (blockIdx.x == 0) P.C->segments += 1u;
    S.round = 0; S.fb = 0; S.fe = 0;
    S.variant = NIL; S.prev_variant = NIL;
    S.c4w = 0; S.e_c4 = 0; S.w_end = 0; S.e_end = 0;
    S.ac3_list = NIL; S.live_in_len = 0; S.live_out = 0;
    S.done = 0; S.fprev = 0; S.mixed = 0;
    S.vcount[0] = S.vcount[1] = S.vcount[2] = 0;
    S.stable = 0;
    S.cstop = 0; S.cperiod = 0; S.clast = NIL;
    S.bmax = 0;
    S.m_live = P.m;
    for (int i = 0; i < NFEAT; ++i) S.feat[i] = 0.0f;
    S.skew = 0;
    S.supp_valid = 0;
    S.lround = 0;
    S.lbase[0] = S.lbase[1] = 0;
    S.async_from = S.async_wait = 0;

    for (int w = 0; w < MAX_WARPS; ++w) {
      WarpSlice& x = B.ws[w];
      x.nlog = x.nw4 = x.nedge = x.nlive = x.ncount = 0;
      x.sum_in = x.sum_out = 0;
      x.max_din = 0;
      x.hist[0] = x.hist[1] = x.hist[2] = 0;
    }
    B.epoch = 0;
    B.err = 0;
    B.w4_wide = 0;
    B.kstat[0] = B.kstat[1] = B.kstat[2] = B.kstat[3] = 0;
#if TRIM_LOCAL
    B.lq_cnt[0] = B.lq_cnt[1] = 0;
    B.lq_vend[0] = B.lq_vend[1] = 0;
    B.lq_k = B.lq_ovf = B.lq_pushed = 0;
#if TRIM_ASYNC
    B.a_gen = 0;
#endif
#if TRIM_AC3_ONLY
    B.live_n[0] = B.live_n[1] = 0;
#endif
#endif
  }
  if (threadIdx.x == 0 && B.resume) {
    // continue a run that an earlier segment left at the start of round saved.round
    const volatile uint32_t* w = reinterpret_cast<const volatile uint32_t*>(&P.C->saved);
    uint32_t* dst = reinterpret_cast<uint32_t*>(&B.S);
    for (unsigned i = 0; i < sizeof(Sched) / 4; ++i) dst[i] = w[i];
  }
  __syncthreads();
#if TRIM_MODES == 15
  const Dev& D = cta_dev;  // round functions are not inlined here
#else
  const Dev& D = P;
#endif
  bool ok = true;
  if (!B.resume) {
    start_round(D, 0);
    // (the initial pass with a dead mask keeps buffer 3 for its heavy rows)
    if (threadIdx.x == 0) B.w4_wide = ((MODES & M_INOUT) || D.mask != nullptr) ? 0u : 1u;
    __syncthreads();
#if !(TRIM_MODES & 48)
    if (D.mask != nullptr) init_round_masked(D, B);
    else
#endif
      init_round(D, B, gwarp, nwarps);
    flush_round(D, B, 0, D.live0);
    ok = grid_barrier(D, B, false);
    // every warp's copy finished before the barrier; the __syncthreads after
    // advance() publishes this before any work-list append
    if (threadIdx.x == 0) B.w4_wide = 0;
  }
  bool fresh = !B.resume;  // a resumed segment starts with its round already chosen
  while (ok) {
    if (fresh && threadIdx.x < 32) advance(D, B);  // also reads the error flag
    fresh = true;
    __syncthreads();
    if (B.err) break;
    const Sched& S = B.S;  // changes only in advance(), between barriers
    if (S.done) {
      if (blockIdx.x == 0 && threadIdx.x == 0) D.C->resume = 0;
      break;
    }
    const bool have = (S.variant == TRIM_AC4_PUSH && (MODES & M_AC4)) ||
                      (S.variant == TRIM_AC6_SUPPORT && (MODES & M_AC6)) ||
                      (S.variant == TRIM_AC3_PULL && (MODES & M_AC3));
    // This kernel lacks the variant chosen for this round: it saves the
    // schedule state and hands the run over at the start of the round (every
    // CTA takes the decision from the same state, so all stop here); the
    // kernel that has the variant resumes it.
    if (!have) {
      if (blockIdx.x == 0 && threadIdx.x == 0) {
        volatile uint32_t* w = reinterpret_cast<volatile uint32_t*>(&D.C->saved);
        const uint32_t* src = reinterpret_cast<const uint32_t*>(&B.S);
        for (unsigned i = 0; i < sizeof(Sched) / 4; ++i) w[i] = src[i];
        D.C->resume_variant = S.variant;
        if (D.C->first_exit_round == 0u) D.C->first_exit_round = S.round;
        __threadfence();
        D.C->resume = 1;
      }
      break;
    }
#if TRIM_LOCAL
#if TRIM_ASYNC
    if (async_start(D, S)) {
      if (!async_tail()) break;
      fresh = false;  // done: the tail ran the rest of the run
      continue;
    }
#endif
    if (local_start(D, S)) {
      if (!local_stretch()) break;
      fresh = false;  // done, or the stretch's last round already ran advance()
      continue;
    }
#endif
    start_round(D, S.round);
#if TRIM_MODES & 16
    inout_round(D, B, S, gwarp, nwarps);
#else
    if ((MODES & M_AC4) && S.variant == TRIM_AC4_PUSH) {
      ac4_round(D, B, S, gwarp, nwarps);
    } else if ((MODES & M_AC6) && S.variant == TRIM_AC6_SUPPORT) {
      if (!ac6_round(D, B, S, gwarp, nwarps)) break;
    } else if (MODES & M_AC3) {
      ac3_round(D, B, S, gwarp, nwarps);
    }
#endif
    const bool stamp = (D.flags & F_ROUND_LOG) && blockIdx.x == 0 && threadIdx.x == 0;
    if (stamp) D.C->t_work[S.round & 3] = globaltimer();
    flush_round(D, B, S.round, S.live_out ? D.live1 : D.live0);
    if (stamp) D.C->t_flush[S.round & 3] = globaltimer();
    ok = grid_barrier(D, B, false);
  }
  stats_publish(D, B);  // every exit of the loop is taken by the whole CTA
}

// ---------------------------------------------------------------- helpers


#if TRIM_MODES == 34
// Edge count of an implicit graph: the sum of its degrees (one pass, n draws).
__global__ void trim_implicit_degree_sum_kernel(Dev D, unsigned long long* m) {
  unsigned long long acc = 0;
  for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < D.n; v += gridDim.x * blockDim.x)
    acc += ig_degree(D, v);
  acc = warp_sum(acc);
  if (lane_id() == 0 && acc) atomicAdd(m, acc);
}
#endif
