// trim_scc.cu -- the SCC decomposition that trimming feeds (Section 1: FW-BW
// with trimming, as in ISPAN), in one cooperative launch behind the in+out
// trimming that finds the size-1 components: size-2 trimming, trimming passes,
// and forward-backward steps until no vertex is open. The host driver is
// trim_run_scc in trim_api.cu.
//
// State: comp[v] = the smallest vertex id of v's component once known, else
// SCC_OPEN. The open vertices stand in a list that every step shortens.
//
// The first step is one forward-backward search from a pivot, the open vertex
// with the largest min(in-degree, out-degree): in a graph with a giant component
// that vertex is nearly always in it, and two searches that touch most edges
// not at all close it. (Searches from every vertex at once, as below, would
// walk the giant component's edges several times.) Every later step works on every open
// vertex at once: its forward part labels each open vertex with the smallest
// open vertex that reaches it (label propagation along G, i.e. forward searches
// from every vertex at once, each vertex keeping the smallest source); a vertex
// r whose label is r itself is reached by no smaller open vertex, and the
// backward search from r inside label r (through G^T) collects exactly r's
// component: every member reaches r and is reached from r, so it carries label
// r, and r, reached by no smaller vertex, is its smallest member. Each step
// closes at least the component of the smallest open vertex, and disconnected
// parts of the graph (separate graphs of a batch) progress together.
//
// A level of a search is bound by latency when it is small (a grid barrier, not
// a launch and a host round trip, ends it) and by random accesses when it is
// large; rows are spread over the warps up to 32 vertices at a time laid end to end,
// and rows over kSccHeavy edges, cut into pieces and those laid end to end, over the
// whole grid (one warp on a hub's row was what a level waited for).
//
// Measured (ms per call, in+out trimming included; before: one launch and one host
// read per level and pass, a warp per row, searches from every vertex in every step):
// R-MAT scale 20 0.34 (6.3), 22 0.71 (17.4); 1,024 packed planted graphs 5.1 (15.2); a
// planted graph of 100,000 0.43 (0.95); 20 dense parts joined in a row 20 (42).
#include "trim_internal.cuh"

using namespace trimk;

namespace {
constexpr uint32_t SCC_OPEN = 0xFFFFFFFFu;
constexpr uint32_t NONE = 0xFFFFFFFFu;
constexpr uint32_t CLOSED = 0xFFFFFFFFu;  // search mark of a vertex with a component
constexpr unsigned FULL = 0xFFFFFFFFu;
// (20 parts of 2,000 vertices with 1,500 / 1,000 edges each, ms: kSccHeavy of 512, 1,024, 4,096
// 0.93 / 0.76, 0.93 / 1.00, 1.28 / 0.94, 2,000 hubs of 3,000 leaves 1.43, 1.43, 2.30; kSccChunk of
// 128, 256, 1,024 0.92 / 0.99, 0.93 / 1.00, 1.18 / 1.07, R-MAT 2^20 0.333, 0.343, 0.414)
constexpr uint32_t kSccHeavy = 1024;   // longer rows go to the whole grid ...
constexpr uint32_t kSccChunk = 256;    // ... in pieces of this many edges
constexpr uint32_t kBuf = 256;         // entries staged per warp before a flush
constexpr int kMaxWarps = 16;

// Per-CTA state: the warps' append buffers, and the barrier's progress.
struct Scc {
  uint32_t buf[kMaxWarps][kBuf];
  unsigned epoch;
  unsigned err;
  unsigned phase;
};

__device__ __forceinline__ uint32_t gwarp() {
  return blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
}
__device__ __forceinline__ uint32_t nwarps() { return gridDim.x * (blockDim.x >> 5); }

// A warp in a long phase shows that it goes on: one increment of the heartbeat every
// kPace steps of its row loops (some 100 us).
constexpr uint32_t kPace = 256;
__device__ __forceinline__ void pace(const SccArgs& A, uint32_t& steps, uint32_t k) {
  steps += k;
  if (steps >= kPace) {
    steps = 0u;
    if (lane_id() == 0) atomicAdd(&A.C->beat, 1u);
  }
}

// Grid-wide barrier: a phase ends. The wait is bounded by spin_limit_ns without any
// progress (an arrival or a heartbeat): how long a phase takes depends on the graph
// (one warp may have a row of millions of edges to itself). Phase p
// counts into slot p & 3, which is read in phase p + 1; the slot of phase p + 2
// was last read in phase p - 1 and is cleared by CTA 0 at the start of phase p.
// Returns false when the run must stop.
__device__ bool scc_sync(const SccArgs& A, Scc& S) {
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned target = (++S.epoch) * gridDim.x;
    __threadfence();
    atomicAdd(&A.C->bar, 1u);
    uint64_t t0 = globaltimer();
    bool looked = false;
    unsigned seen = 0;
    while ((int)(ld_relaxed(&A.C->bar) - target) < 0) {
      if (globaltimer() - t0 > A.spin_limit_ns) {
        const unsigned cur = ld_relaxed(&A.C->bar) + ld_relaxed(&A.C->beat);  // both only grow
        if (looked && cur == seen) {
          atomicCAS(&A.C->err, 0u, (unsigned)TRIM_ERR_TIMEOUT);
          break;
        }
        looked = true;
        seen = cur;
        t0 = globaltimer();
      }
    }
    (void)ld_acquire(&A.C->bar);
    S.err = ld_relaxed(&A.C->err);
    S.phase += 1u;
    if (blockIdx.x == 0) {
      SccSlot* z = &A.C->slot[(S.phase + 2u) & 3u];
      z->n = z->hits = 0u;
      z->heavy = 0ull;
    }
  }
  __syncthreads();
  return S.err == 0u;
}
__device__ __forceinline__ SccSlot* now(const SccArgs& A, const Scc& S) {
  return &A.C->slot[S.phase & 3u];
}
__device__ __forceinline__ const SccSlot* before(const SccArgs& A, const Scc& S) {
  return &A.C->slot[(S.phase - 1u) & 3u];
}

// Vertices that a warp takes at a time out of `count`: few if there are few, as it looks
// through long rows one after the other (4 parts of 1,500 vertices with 1,300 edges each:
// 0.98 ms with 32).
__device__ __forceinline__ uint32_t group(uint32_t count) {
  return min(32u, max(1u, (count + nwarps() - 1u) / nwarps()));
}

// Appends to a global list, staged in the warp's buffer: one atomic per flush.
struct Out {
  uint32_t* list;
  unsigned* count;
  uint32_t have;
};
__device__ __forceinline__ void flush(Scc& S, Out& o) {
  if (o.have == 0u) return;
  const uint32_t* b = S.buf[threadIdx.x >> 5];
  __syncwarp();
  uint32_t at = 0;
  if (lane_id() == 0) at = atomicAdd(o.count, o.have);
  at = __shfl_sync(FULL, at, 0);
  for (uint32_t i = lane_id(); i < o.have; i += 32u) o.list[at + i] = b[i];
  __syncwarp();
  o.have = 0u;
}
// Warp-collective: lanes with pred append v.
__device__ __forceinline__ void put(Scc& S, Out& o, bool pred, uint32_t v) {
  const unsigned m = __ballot_sync(FULL, pred);
  if (m == 0u) return;
  if (o.have + 32u > kBuf) flush(S, o);
  if (pred) S.buf[threadIdx.x >> 5][o.have + __popc(m & ((1u << lane_id()) - 1u))] = v;
  o.have += __popc(m);
}
// Adds a count per lane to a counter (warp-collective).
__device__ __forceinline__ void add(unsigned* c, unsigned x) {
  x = __reduce_add_sync(FULL, x);
  if (lane_id() == 0 && x) atomicAdd(c, x);
}

// All warps: f(u, w, valid) (warp-collective) for the edges u -> w of the rows of
// list[0..count): a warp takes up to 32 vertices, their rows laid end to end,
// four loads in flight per lane. Rows over kSccHeavy edges go to the heavy list
// for heavy_edges, in the next phase: one atomic of the warp reserves their entries
// and their pieces, so that the entries' first pieces rise along the list.
template <class F>
__device__ __forceinline__ void list_edges(const SccArgs& A, const Scc& S, const uint32_t* off,
                                           const uint32_t* tgt, const uint32_t* list,
                                           uint32_t count, F f) {
  const unsigned lane = lane_id();
  const uint32_t nw = nwarps(), G = group(count);
  uint32_t steps = 0;
  for (uint32_t base = gwarp() * G; base < count; base += nw * G) {  // warp-uniform
    const bool has = lane < G && base + lane < count;
    const uint32_t u = has ? ldcg(&list[base + lane]) : 0u;
    const uint32_t s = has ? __ldg(&off[u]) : 0u;
    uint32_t d = has ? __ldg(&off[u + 1u]) - s : 0u;
    const bool big = d > kSccHeavy;
    const unsigned bm = __ballot_sync(FULL, big);
    if (bm) {
      const uint32_t np = big ? (d - 1u) / kSccChunk + 1u : 0u, pincl = warp_incl_scan(np);
      unsigned long long o = 0;
      if (lane == 31)
        o = atomicAdd(&now(A, S)->heavy, ((unsigned long long)pincl << 32) | __popc(bm));
      o = __shfl_sync(FULL, o, 31);
      if (big) {
        const uint32_t at = (uint32_t)o + __popc(bm & ((1u << lane) - 1u));
        A.heavy[at] = u;
        A.hpos[at] = (uint32_t)(o >> 32) + pincl - np;
        d = 0u;
      }
    }
    const uint32_t incl = warp_incl_scan(d), excl = incl - d;
    const uint32_t total = __shfl_sync(FULL, incl, 31);
    pace(A, steps, 1u + total / 128u);  // (at most 32 rows of kSccHeavy)
    for (uint32_t k0 = 0; k0 < total; k0 += 128u) {
      uint32_t uu[4], w[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t k = k0 + (uint32_t)q * 32u + lane;
        const unsigned o = owner_of(excl, k);
        const uint32_t so = __shfl_sync(FULL, s, o), xo = __shfl_sync(FULL, excl, o);
        uu[q] = __shfl_sync(FULL, u, o);
        w[q] = k < total ? __ldg(&tgt[so + (k - xo)]) : 0u;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) f(uu[q], w[q], k0 + (uint32_t)q * 32u + lane < total);
    }
  }
}
// The rows of the heavy list (`heavy`: its entries, and its pieces << 32), their
// pieces laid end to end: every warp takes an equal run of them, and finds the row
// of its first one by a search over the entries' first pieces, 32 ways a step.
// (20 parts of 2,000 vertices with 1,500 edges each, joined by single edges: 697 ms
// with the rows one after the other, each from the first warp on; a warp per row and
// launch per level, before that, 42 ms.)
template <class F>
__device__ __forceinline__ void heavy_edges(const SccArgs& A, const uint32_t* off,
                                            const uint32_t* tgt, unsigned long long heavy, F f) {
  const unsigned lane = lane_id();
  const uint32_t rows = (uint32_t)heavy, pieces = (uint32_t)(heavy >> 32), nw = nwarps();
  const uint32_t per = (pieces + nw - 1u) / nw;
  // (neighbouring runs on different SMs)
  uint32_t p = ((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * per;
  const uint32_t p1 = min(pieces, p + per);
  if (p >= p1) return;  // warp-uniform
  uint32_t h = 0, steps = 0;
  for (uint32_t len = rows; len > 1u;) {
    const uint32_t step = (len + 31u) / 32u, r = lane * step;
    const unsigned b = __ballot_sync(FULL, r < len && ldcg(&A.hpos[h + r]) <= p);
    const uint32_t skip = (31u - __clz(b)) * step;  // (b has lane 0)
    h += skip;
    len = min(step, len - skip);
  }
  for (; p < p1; ++h) {  // warp-uniform
    const uint32_t u = ldcg(&A.heavy[h]), first = ldcg(&A.hpos[h]);
    const uint32_t s = __ldg(&off[u]), e = __ldg(&off[u + 1u]);
    const uint32_t end = min(p1, first + (e - s - 1u) / kSccChunk + 1u);
    for (; p < end; ++p) {
      pace(A, steps, kSccChunk / 128u);
      const uint64_t k0 = s + (uint64_t)(p - first) * kSccChunk;
#pragma unroll
      for (uint32_t i = 0; i < kSccChunk; i += 128u) {
        uint32_t w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint64_t k = k0 + i + (uint32_t)q * 32u + lane;
          w[q] = k < e ? __ldg(&tgt[k]) : 0u;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) f(u, w[q], k0 + i + (uint32_t)q * 32u + lane < e);
      }
    }
  }
}

// Does the row [s, s + d) hold an entry for which hit(w) is true? Warp-collective
// for the lanes with want: four entries per lane at a time, up to 32 of a row;
// what is left of longer rows is looked through by the whole warp.
template <class H>
__device__ __forceinline__ bool row_any(const SccArgs& A, const uint32_t* tgt, uint32_t s,
                                        uint32_t d, bool want, uint32_t& steps, H hit) {
  const unsigned lane = lane_id();
  bool found = false;
  uint32_t i = 0;
  while (want && !found && i < d && i < 32u) {
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = i + q < d ? __ldg(&tgt[s + i + q]) : 0u;
    bool h[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) h[q] = i + q < d && hit(w[q]);
    found = h[0] || h[1] || h[2] || h[3];
    i += 4u;
  }
  __syncwarp();
  unsigned big = __ballot_sync(FULL, want && !found && d > 32u);
  while (big) {
    const int j = __ffs(big) - 1;
    big &= big - 1u;
    const uint32_t sj = __shfl_sync(FULL, s, j), dj = __shfl_sync(FULL, d, j);
    bool any = false;
    for (uint32_t k0 = 32u; k0 < dj && !any; k0 += 128u) {  // warp-uniform
      pace(A, steps, 1u);
      uint32_t w[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t k = k0 + (uint32_t)q * 32u + lane;
        w[q] = k < dj ? __ldg(&tgt[sj + k]) : 0u;
      }
      bool h = false;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t k = k0 + (uint32_t)q * 32u + lane;
        h = h || (k < dj && hit(w[q]));
      }
      any = __any_sync(FULL, h);
    }
    if ((int)lane == j) found = any;
  }
  return found;
}

// Open entries of the row [s, s + d) for the lanes with want: those other than
// `self` counted up to 2 (oth, the first one in *first) and all of them up to 3.
__device__ __forceinline__ void row_count(const SccArgs& A, const uint32_t* tgt, uint32_t s,
                                          uint32_t d, bool want, uint32_t self, uint32_t& steps,
                                          uint32_t& oth, uint32_t& all, uint32_t& first) {
  const unsigned lane = lane_id();
  oth = all = 0u;
  first = NONE;
  for (uint32_t i = 0; want && d <= 32u && i < d && (oth < 2u || all < 3u); i += 4u) {
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = i + q < d ? __ldg(&tgt[s + i + q]) : 0u;
    bool o[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) o[q] = i + q < d && ldcg(&A.comp[w[q]]) == SCC_OPEN;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (!o[q]) continue;
      ++all;
      if (w[q] != self) {
        if (first == NONE) first = w[q];
        ++oth;
      }
    }
  }
  __syncwarp();
  unsigned big = __ballot_sync(FULL, want && d > 32u);
  while (big) {
    const int j = __ffs(big) - 1;
    big &= big - 1u;
    const uint32_t sj = __shfl_sync(FULL, s, j), dj = __shfl_sync(FULL, d, j);
    const uint32_t vj = __shfl_sync(FULL, self, j);
    uint32_t o = 0, a = 0, f = NONE;
    for (uint32_t k0 = 0; k0 < dj && (o < 2u || a < 3u); k0 += 32u) {  // warp-uniform
      pace(A, steps, 1u);
      const uint32_t k = k0 + lane;
      const uint32_t w = k < dj ? __ldg(&tgt[sj + k]) : 0u;
      const bool open = k < dj && ldcg(&A.comp[w]) == SCC_OPEN;
      const unsigned om = __ballot_sync(FULL, open && w != vj);
      if (om && f == NONE) f = __shfl_sync(FULL, w, __ffs(om) - 1);
      o += __popc(om);
      a += __popc(__ballot_sync(FULL, open));
    }
    if ((int)lane == j) {
      oth = o;
      all = a;
      first = f;
    }
  }
  oth = min(oth, 2u);
  all = min(all, 3u);
}

// The open vertices of list[0..count) go to `to` (one phase; its count is in the
// phase's slot).
__device__ __forceinline__ void keep_open(const SccArgs& A, Scc& S, const uint32_t* list,
                                          uint32_t count, uint32_t* to) {
  Out o{to, &now(A, S)->n, 0u};
  for (uint32_t base = gwarp() * 32u; base < count; base += nwarps() * 32u) {
    const uint32_t i = base + lane_id();
    const uint32_t v = i < count ? ldcg(&list[i]) : 0u;
    put(S, o, i < count && ldcg(&A.comp[v]) == SCC_OPEN, v);
  }
  flush(S, o);
}

__device__ __forceinline__ void close_vertex(const SccArgs& A, uint32_t v, uint32_t c) {
  A.comp[v] = c;
  A.fw[v] = CLOSED;
  A.bw[v] = CLOSED;
}

// Search from the frontier in A.fa (k vertices, marked with `stamp`) along
// (off, tgt), whose transpose is (roff, rtgt), among the open vertices in
// `allow` (where given: those whose mark there is allowed). A small frontier
// offers its rows; once it is large, the vertices not yet marked look for a
// marked neighbour instead (usually within a few entries; large from 1/4, 1/16, 1/64 of
// them on: R-MAT 2^20 0.597, 0.343, 0.342 ms, dense parts 0.94, 0.93, 1.16). Returns false on an
// error.
__device__ bool search(const SccArgs& A, Scc& S, const uint32_t* off, const uint32_t* tgt,
                       const uint32_t* roff, const uint32_t* rtgt, uint32_t* mark, uint32_t stamp,
                       const uint32_t* allow, uint32_t allowed, const uint32_t* open, uint32_t n_open,
                       uint32_t k, uint32_t& levels) {
  const unsigned lane = lane_id();
  uint32_t *fa = A.fa, *fb = A.fb;
  uint32_t left = n_open - min(n_open, k);  // not marked yet (at most)
  while (k > 0u) {
    ++levels;
    Out o{fb, &now(A, S)->n, 0u};
    if ((uint64_t)k * 16u > left) {
      const uint32_t G = group(n_open);
      uint32_t steps = 0;
      for (uint32_t base = gwarp() * G; base < n_open; base += nwarps() * G) {
        const uint32_t i = base + lane;
        const bool in = lane < G && i < n_open;
        const uint32_t v = in ? ldcg(&open[i]) : 0u;
        const bool want = in && ldcg(&mark[v]) < stamp &&
                          (allow == nullptr || ldcg(&allow[v]) == allowed);
        const uint32_t s = want ? __ldg(&roff[v]) : 0u;
        const uint32_t d = want ? __ldg(&roff[v + 1u]) - s : 0u;
        pace(A, steps, 1u);
        const bool hit = row_any(A, rtgt, s, d, want, steps, [&](uint32_t w) { return ldcg(&mark[w]) == stamp; });
        if (hit) mark[v] = stamp;
        put(S, o, hit, v);
      }
      flush(S, o);
      if (!scc_sync(A, S)) return false;
      k = ldcg(&before(A, S)->n);
    } else {
      auto visit = [&](uint32_t, uint32_t w, bool valid) {
        const bool take = valid && ldcg(&mark[w]) < stamp &&
                          (allow == nullptr || ldcg(&allow[w]) == allowed) &&
                          atomicMax(&mark[w], stamp) < stamp;
        put(S, o, take, w);
      };
      list_edges(A, S, off, tgt, fa, k, visit);
      flush(S, o);
      if (!scc_sync(A, S)) return false;
      const unsigned long long heavy = __ldcg(&before(A, S)->heavy);
      k = ldcg(&before(A, S)->n);
      if (heavy) {  // (their finds join the same list, behind those of the phase before)
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&now(A, S)->n, k);
        o.count = &now(A, S)->hits;
        o.list = fb + k;
        heavy_edges(A, off, tgt, heavy, visit);
        flush(S, o);
        if (!scc_sync(A, S)) return false;
        k = ldcg(&before(A, S)->n) + ldcg(&before(A, S)->hits);
      }
    }
    left -= min(left, k);
    uint32_t* t = fa;
    fa = fb;
    fb = t;
  }
  return true;
}

// Trimming passes: an open vertex without an open successor, or without an open
// predecessor, is a component of its own (its other neighbours are in components
// already complete, so no cycle through it remains).
__device__ bool trim_passes(const SccArgs& A, Scc& S, const uint32_t* open, uint32_t n_open,
                            unsigned& trimmed) {
  const unsigned lane = lane_id();
  for (int pass = 0; pass < 1024; ++pass) {
    unsigned gone = 0;
    const uint32_t G = group(n_open);
    uint32_t steps = 0;
    for (uint32_t base = gwarp() * G; base < n_open; base += nwarps() * G) {
      const uint32_t i = base + lane;
      const bool in_list = lane < G && i < n_open;
      const uint32_t v = in_list ? ldcg(&open[i]) : 0u;
      const bool is = in_list && ldcg(&A.comp[v]) == SCC_OPEN;
      auto hit = [&](uint32_t w) { return ldcg(&A.comp[w]) == SCC_OPEN; };
      const uint32_t s = is ? __ldg(&A.off[v]) : 0u, d = is ? __ldg(&A.off[v + 1u]) - s : 0u;
      pace(A, steps, 1u);
      const bool out = row_any(A, A.tgt, s, d, is, steps, hit);
      const uint32_t t = out ? __ldg(&A.ioff[v]) : 0u, e = out ? __ldg(&A.ioff[v + 1u]) - t : 0u;
      const bool in = row_any(A, A.itgt, t, e, out, steps, hit);
      if (is && !in) {
        close_vertex(A, v, v);
        ++gone;
      }
    }
    add(&now(A, S)->hits, gone);
    if (!scc_sync(A, S)) return false;
    const unsigned k = ldcg(&before(A, S)->hits);
    trimmed += k;
    if (k == 0u) break;
  }
  return true;
}

}  // namespace

__global__ void __launch_bounds__(512, 2) trim_scc_kernel(SccArgs A) {
  __shared__ Scc S;
  const unsigned lane = lane_id();
  const uint32_t n = A.n;
  if (threadIdx.x == 0) {
    S.epoch = S.err = S.phase = 0u;
  }
  // in+out trimming failed: its error is the run's
  if (ld_relaxed(&A.run->err) != 0u) return;
  __syncthreads();
  // size-1 components from in+out trimming; the others are open
  {
    Out o{A.open0, &now(A, S)->n, 0u};
    for (uint32_t base = gwarp() * 32u; base < n; base += nwarps() * 32u) {
      const uint32_t v = base + lane;
      const bool open = v < n && A.level[v] == LIVE;
      if (v < n) {
        A.comp[v] = open ? SCC_OPEN : v;
        A.fw[v] = A.bw[v] = open ? 0u : CLOSED;
      }
      put(S, o, open, v);
    }
    flush(S, o);
  }
  if (!scc_sync(A, S)) return;
  uint32_t *open = A.open0, *spare = A.open1;
  uint32_t n_open = ldcg(&before(A, S)->n);
  // Size-2 trimming: for every open vertex its only open successor other than
  // itself (out1) and its only open predecessor other than itself (in1),
  // parallel edges counted separately, NONE when there is none or more than
  // one; a vertex with a self-loop, which is a component of its own, is never
  // paired. `more` is true for a self-loop and for three or more open
  // successors; the second pass over G^T is for the few others.
  const uint32_t G = group(n_open);
  uint32_t steps2 = 0;
  for (uint32_t base = gwarp() * G; base < n_open; base += nwarps() * G) {
    const uint32_t i = base + lane;
    const bool is = lane < G && i < n_open;
    const uint32_t v = is ? ldcg(&open[i]) : 0u;
    const uint32_t s = is ? __ldg(&A.off[v]) : 0u, d = is ? __ldg(&A.off[v + 1u]) - s : 0u;
    uint32_t oth = 0, all = 0, o1 = NONE, ioth = 0, iall = 0, i1 = NONE;
    pace(A, steps2, 1u);
    row_count(A, A.tgt, s, d, is, v, steps2, oth, all, o1);
    const bool more = all > oth;
    const bool back = is && !more;
    const uint32_t t = back ? __ldg(&A.ioff[v]) : 0u, e = back ? __ldg(&A.ioff[v + 1u]) - t : 0u;
    row_count(A, A.itgt, t, e, back, v, steps2, ioth, iall, i1);
    if (is) {
      A.fa[v] = (!more && oth == 1u) ? o1 : NONE;
      A.fb[v] = (!more && ioth == 1u) ? i1 : NONE;
    }
  }
  if (!scc_sync(A, S)) return;
  // v and u = out1[v] with out1[u] = v are each other's only open successors, so
  // {u, v} is a component (a closed 2-cycle); the same with predecessors. Both
  // members write the same label.
  {
    unsigned pairs = 0;
    for (uint32_t base = gwarp() * 32u; base < n_open; base += nwarps() * 32u) {
      const uint32_t i = base + lane;
      if (i < n_open) {
        const uint32_t v = ldcg(&open[i]);
        const uint32_t o = ldcg(&A.fa[v]), p = ldcg(&A.fb[v]);
        uint32_t u = NONE;
        if (o != NONE && ldcg(&A.fa[o]) == v) u = o;
        else if (p != NONE && ldcg(&A.fb[p]) == v) u = p;
        if (u != NONE) {
          close_vertex(A, v, min(u, v));
          pairs += v < u ? 1u : 0u;
        }
      }
    }
    add(&now(A, S)->hits, pairs);
  }
  if (!scc_sync(A, S)) return;
  const unsigned size2 = ldcg(&before(A, S)->hits);
  unsigned trimmed = 0;
  uint32_t steps = 0, levels = 0, stamp = 0;
  while (true) {
    if (!trim_passes(A, S, open, n_open, trimmed)) return;
    keep_open(A, S, open, n_open, spare);
    if (!scc_sync(A, S)) return;
    n_open = ldcg(&before(A, S)->n);
    uint32_t* t = open;
    open = spare;
    spare = t;
    if (n_open == 0u) break;  // every vertex has its component
    if (steps == 0u) {
      // a forward-backward search from one pivot
      unsigned long long best = 0ull;
      for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_open;
           i += gridDim.x * blockDim.x) {
        const uint32_t v = ldcg(&open[i]);
        const uint32_t d = min(__ldg(&A.off[v + 1u]) - __ldg(&A.off[v]),
                               __ldg(&A.ioff[v + 1u]) - __ldg(&A.ioff[v]));
        const unsigned long long key = ((unsigned long long)d << 32) | (0xFFFFFFFFu - v);
        best = key > best ? key : best;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long x = __shfl_xor_sync(FULL, best, o);
        best = x > best ? x : best;
      }
      if (lane == 0 && best) atomicMax(&A.C->best, best);
      if (!scc_sync(A, S)) return;
      const uint32_t pivot = 0xFFFFFFFFu - (uint32_t)ld_acquire64(&A.C->best);
      const uint32_t f = ++stamp, b = ++stamp;
      if (blockIdx.x == 0 && threadIdx.x == 0) {
        A.fa[0] = pivot;
        A.fw[pivot] = f;
        A.bw[pivot] = b;
      }
      if (!scc_sync(A, S)) return;
      if (!search(A, S, A.off, A.tgt, A.ioff, A.itgt, A.fw, f, nullptr, 0u, open, n_open, 1u, levels))
        return;
      if (blockIdx.x == 0 && threadIdx.x == 0) A.fa[0] = pivot;
      if (!scc_sync(A, S)) return;
      if (!search(A, S, A.ioff, A.itgt, A.off, A.tgt, A.bw, b, A.fw, f, open, n_open, 1u, levels))
        return;
      uint32_t least = NONE;
      for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_open;
           i += gridDim.x * blockDim.x) {
        const uint32_t v = ldcg(&open[i]);
        if (ldcg(&A.bw[v]) == b) least = min(least, v);
      }
      least = __reduce_min_sync(FULL, least);
      if (lane == 0 && least != NONE) atomicMin(&A.C->least, least);
      if (!scc_sync(A, S)) return;
      const uint32_t c = ld_relaxed(&A.C->least);
      for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_open;
           i += gridDim.x * blockDim.x) {
        const uint32_t v = ldcg(&open[i]);
        if (ldcg(&A.bw[v]) == b) close_vertex(A, v, c);
      }
    } else {
      // labels: every open vertex starts with its own id and joins the first frontier
      uint32_t *fa = A.fa, *fb = A.fb;
      for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_open;
           i += gridDim.x * blockDim.x) {
        const uint32_t v = ldcg(&open[i]);
        A.label[v] = v;
        fa[i] = v;
      }
      if (!scc_sync(A, S)) return;
      // every frontier vertex offers its label to its open successors; one whose
      // label drops joins the next frontier (once per level: fw holds its stamp)
      uint32_t k = n_open;
      while (k > 0u) {
        ++levels;
        const uint32_t st = ++stamp;
        Out o{fb, &now(A, S)->n, 0u};
        auto offer = [&](uint32_t u, uint32_t w, bool valid) {
          bool take = false;
          if (valid && ldcg(&A.comp[w]) == SCC_OPEN) {
            const uint32_t lu = ldcg(&A.label[u]);
            take = ldcg(&A.label[w]) > lu && atomicMin(&A.label[w], lu) > lu &&
                   atomicExch(&A.fw[w], st) != st;
          }
          put(S, o, take, w);
        };
        list_edges(A, S, A.off, A.tgt, fa, k, offer);
        flush(S, o);
        if (!scc_sync(A, S)) return;
        const unsigned long long heavy = __ldcg(&before(A, S)->heavy);
        k = ldcg(&before(A, S)->n);
        if (heavy) {
          o.count = &now(A, S)->hits;
          o.list = fb + k;
          heavy_edges(A, A.off, A.tgt, heavy, offer);
          flush(S, o);
          if (!scc_sync(A, S)) return;
          k += ldcg(&before(A, S)->hits);
        }
        uint32_t* x = fa;
        fa = fb;
        fb = x;
      }
      // roots: open vertices that kept their own label start the backward searches
      const uint32_t st = ++stamp;
      {
        Out o{fa, &now(A, S)->n, 0u};
        for (uint32_t base = gwarp() * 32u; base < n_open; base += nwarps() * 32u) {
          const uint32_t i = base + lane;
          const uint32_t v = i < n_open ? ldcg(&open[i]) : 0u;
          const bool root = i < n_open && ldcg(&A.label[v]) == v;
          if (root) A.bw[v] = st;
          put(S, o, root, v);
        }
        flush(S, o);
      }
      if (!scc_sync(A, S)) return;
      k = ldcg(&before(A, S)->n);
      while (k > 0u) {  // through G^T, inside the label
        ++levels;
        Out o{fb, &now(A, S)->n, 0u};
        auto visit = [&](uint32_t u, uint32_t w, bool valid) {
          const bool take = valid && ldcg(&A.bw[w]) < st &&
                            ldcg(&A.label[w]) == ldcg(&A.label[u]) && atomicMax(&A.bw[w], st) < st;
          put(S, o, take, w);
        };
        list_edges(A, S, A.ioff, A.itgt, fa, k, visit);
        flush(S, o);
        if (!scc_sync(A, S)) return;
        const unsigned long long heavy = __ldcg(&before(A, S)->heavy);
        k = ldcg(&before(A, S)->n);
        if (heavy) {
          o.count = &now(A, S)->hits;
          o.list = fb + k;
          heavy_edges(A, A.ioff, A.itgt, heavy, visit);
          flush(S, o);
          if (!scc_sync(A, S)) return;
          k += ldcg(&before(A, S)->hits);
        }
        uint32_t* x = fa;
        fa = fb;
        fb = x;
      }
      // an open vertex that the backward search from its label's root reached
      // belongs to that root's component
      for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_open;
           i += gridDim.x * blockDim.x) {
        const uint32_t v = ldcg(&open[i]);
        if (ldcg(&A.bw[v]) == st) close_vertex(A, v, ldcg(&A.label[v]));
      }
    }
    if (!scc_sync(A, S)) return;
    ++steps;
  }
  // number of components: vertices that label their own component
  unsigned k = 0;
  for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
    k += ldcg(&A.comp[v]) == v ? 1u : 0u;
  add(&A.C->components, k);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    A.C->size2 = size2;
    A.C->trimmed = trimmed;
    A.C->steps = steps;
    A.C->levels = levels;
    A.C->done = 1u;
  }
}
