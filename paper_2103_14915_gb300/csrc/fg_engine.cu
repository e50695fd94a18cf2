// Buffered fork-processing engine (Alg. 2) as one persistent cooperative kernel.
//
// One launch runs every round of the buffered loop for a batch of queries:
//
//   INIT      InitBuffers: each query's seed operation <q, src, 0> (PPR: residual 1)
//             goes to the buffer of (partition(src), q)                   (Alg. 2, Sec. 3.2)
//   loop (one round per iteration, device-wide barrier between phases):
//     SCAN-A  per-block totals of buffered operations / non-empty buffers
//     SCAN-B  exclusive scan -> one work item per non-empty (partition, query)
//             buffer ("Consolidate": operations grouped by query, Sec. 4.2,
//             App. B.1 with K = |Q| buckets); ScheduleNextPart (Sec. 5.2):
//             FIFO takes every non-empty buffer, PRIORITY the ones whose best
//             value is within a window of their query's best pending value
//     SCATTER move this round's operations from the append arena into bins
//             ordered by (partition, query)
//     PROCESS IntraPartProcess: each warp claims a work item, stages the
//             query's slice of the partition's state in shared memory, applies
//             the buffered operations, relaxes / pushes inside the partition
//             until done or until a yield heuristic fires (Sec. 5.1), writes the
//             slice back and appends operations for other partitions to the
//             arena (Alg. 2, "send operations to neighbor partitions")
//   until no buffer holds an operation (Alg. 2 loop condition).
//
// A work item is owned by exactly one warp per round, so the query's state
// slice of that partition has a single writer (the atomic-free consolidation
// of Sec. 4.2, here at warp granularity). Operations to other partitions are
// filtered by a plain read of the target's committed value (SSSP/BFS).
#include <algorithm>
#include <cstdio>

#include "fg_device.cuh"

namespace fg {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr uint32_t kMaxVisitSteps = 1u << 22;  // relax/push steps of one visit before the watchdog fires
constexpr uint32_t kBlockChunk = 16;            // work items a block claims at once
constexpr uint32_t kTailChunk = 2;              // ... once fewer than 4 full chunks per block are left
constexpr uint32_t kArenaChunk = 64;            // arena slots a warp reserves at once (>= 32)
constexpr int kUnroll = 4;                      // steps of 32 arcs with their loads in flight together
constexpr uint32_t kMoreArcs = 0x8000u;         // of a queue entry
constexpr int kExt = 64;                        // candidates for other partitions a warp gathers before it sends them

// Per-warp counters. visits and edges are lane-uniform; spills and yields are
// summed over the lanes when flushed.
struct Counters {
  unsigned long long visits = 0, edges = 0, spills = 0, yields = 0;
};

// Per-warp shared memory of a PPR visit: the residuals and four bitmaps of S bits.
struct WarpSmem {
  uint32_t *d;      // [S] residuals (f32 bits)
  uint32_t *cur;    // [nw] frontier being expanded
  uint32_t *nxt;    // [nw] frontier of the next step
  uint32_t *carry;  // [nw] left for a later visit (yield / spill)
  uint32_t *pfx;    // [nw] exclusive popcount prefix of cur
};

// Per-warp shared memory of an SSSP / BFS visit: the distances, a queue of the
// vertices to expand, and four bitmaps of S bits.
struct DistSmem {
  uint32_t *d;      // [S] distances
  uint16_t *ring;   // [S] queue of vertices to expand, each at most once; kMoreArcs: may have more than four arcs
  uint32_t *inq;    // [nw] vertices in the queue
  uint32_t *far;    // [nw] values at or beyond the in-visit window T when marked
  uint32_t *carry;  // [nw] values at or beyond the visit's bound Ty when marked
  uint32_t *spill;  // [nw] vertices whose candidates for other partitions did not fit
  uint32_t *ext;    // [3 * kExt] candidates for other partitions: target, value, source
};

// Per-warp area in words, rounded up to 16 bytes so every warp's slice is
// 16-byte aligned (the dynamic shared memory base is). Up to 1,024 vertices a
// partition three blocks fit an SM; with 2,048 two of an SSSP or BFS visit do (three
// without the ring), which costs less than the ring gives but on strips: 1024^2
// grid, 256 sources, SSSP 95 -> 68 ms, BFS 57 -> 40 in grown partitions; in
// partitions of two grid rows 284 -> 329 and 314 -> 377.
__host__ __device__ inline size_t warp_smem_words(bool ppr, int S) {
  const size_t nw = (size_t)(S / 32);
  const size_t words = ppr ? (size_t)S + 4u * nw : (size_t)S + (size_t)S / 2u + 4u * nw + 3u * (size_t)kExt;
  return (words + 3u) & ~(size_t)3u;
}



// ---------------------------------------------------------------------------
// Warp-collective append of at most one operation per lane to the arena.
// Per-buffer counts (and best value for priority scheduling) are aggregated
// across lanes that target the same buffer (__match_any_sync). Returns false
// for lanes whose operation did not fit (the caller spills it); lanes without
// an operation return true.
//
// Slots come from the warp's ArenaSlots: the warp reserves kArenaChunk slots
// of the arena at a time, so the device-wide cursor is touched once per chunk
// rather than once per append (a returning atomic on one address that every
// warp of the grid shares). Reserved slots a warp does not fill become holes
// (kInvalidKey) that SCATTER skips. An arena too small for a few chunks of every
// busy warp is reserved slot by slot (a.arena_chunk, launch_engine): a visit that
// sends five operations must not keep 59 others from theirs, who would take the
// same vertices up again in the next round. Without ArenaSlots (seeding), each call
// reserves exactly what it appends.
// ---------------------------------------------------------------------------
struct ArenaSlots {
  unsigned long long pos = 0, end = 0;  // lane-uniform: [pos, end) reserved, not yet written
  unsigned long long seen = 0;          // device-wide cursor as of the last reservation
};

// Arena pressure: once a quarter of the arena is left, visits stop at their
// next step and unvisited items are carried to the next round, so a round's
// appends stay within the arena instead of spilling. (A spilled relaxation
// re-marks its source vertex, and re-expanding a vertex of high degree round
// after round multiplies the work.)
__device__ __forceinline__ bool arena_pressed(const EngineArgs &a, unsigned long long cursor) {
  return cursor >= a.e_cap - (a.e_cap >> 2);
}

__device__ __forceinline__ void release_slots(const EngineArgs &a, ArenaSlots &sl) {
  const int lane = lane_id();
  const unsigned long long lim = sl.end < a.e_cap ? sl.end : a.e_cap;
  for (unsigned long long s = sl.pos + (unsigned long long)lane; s < lim; s += 32ull) a.e_key[s] = kInvalidKey;
  sl.pos = sl.end;
}

__device__ __forceinline__ bool emit_ops(const EngineArgs &a, bool has, uint32_t key, uint32_t lv,
                                         uint32_t val, bool track_prio, ArenaSlots *sl = nullptr) {
  const unsigned m = __ballot_sync(kFull, has);
  if (m == 0) return true;
  const int lane = lane_id();
  const unsigned n = (unsigned)__popc(m);
  unsigned long long base = 0;
  if (sl != nullptr) {
    if (sl->pos + n > sl->end) {
      release_slots(a, *sl);
      const unsigned take = max(n, a.arena_chunk);
      if (lane == 0) base = atomicAdd(&a.ctrl->e_cursor, (unsigned long long)take);
      base = __shfl_sync(kFull, base, 0);
      sl->pos = base;
      sl->end = base + take;
      sl->seen = sl->end;
    }
    base = sl->pos;
    sl->pos += n;
  } else {
    const int leader = __ffs(m) - 1;
    if (lane == leader) base = atomicAdd(&a.ctrl->e_cursor, (unsigned long long)n);
    base = __shfl_sync(kFull, base, leader);
  }
  const unsigned long long slot = base + (unsigned long long)__popc(m & ((1u << lane) - 1u));
  const bool fits = has && slot < a.e_cap;
  if (fits) {
    a.e_key[slot] = key;
    a.e_op[slot] = make_uint2(lv, val);
  }
  const unsigned fm = __ballot_sync(kFull, fits);
  if (fits) {
    const unsigned grp = __match_any_sync(fm, key);
    const int gl = __ffs(grp) - 1;
    if (track_prio) {
      const uint32_t mn = __reduce_min_sync(grp, val);
      if (lane == gl) atomicMin(&a.prio[key], mn);
    }
    if (lane == gl) atomicAdd(&a.cnt[key], (unsigned)__popc(grp));
  }
  return !has || fits;
}

// Grid-stride fill of count 32-bit words with 16-byte stores for the aligned body.
__device__ __forceinline__ void fill_u32(uint32_t *p, uint64_t count, uint32_t val, uint64_t tid, uint64_t nthr) {
  const uint64_t mis = (reinterpret_cast<uintptr_t>(p) & 15u) >> 2;
  const uint64_t head = mis ? umin64(count, 4u - mis) : 0u;
  if (tid < head) p[tid] = val;
  const uint64_t body = (count - head) / 4u;
  uint4 *q = reinterpret_cast<uint4 *>(p + head);
  const uint4 v4 = make_uint4(val, val, val, val);
  for (uint64_t i = tid; i < body; i += nthr) q[i] = v4;
  const uint64_t tail0 = head + body * 4u;
  if (tid < count - tail0) p[tail0 + tid] = val;
}

// Lane `lane` owns the words [w0, w1) of an nw-word bitmap.
struct WordRange {
  int w0, w1;
  __device__ WordRange(int nw, int lane) {
    const int per = (nw + 31) >> 5;
    w0 = min(nw, lane * per);
    w1 = min(nw, w0 + per);
  }
};

// Build the exclusive popcount prefix of cur; returns the frontier size.
__device__ __forceinline__ uint32_t frontier_prefix(const WarpSmem &w, const WordRange &r) {
  uint32_t tot = 0;
  for (int wd = r.w0; wd < r.w1; ++wd) {
    w.pfx[wd] = tot;
    tot += __popc(w.cur[wd]);
  }
  const uint32_t incl = warp_incl_scan(tot);
  const uint32_t ex = incl - tot;
  for (int wd = r.w0; wd < r.w1; ++wd) w.pfx[wd] += ex;
  __syncwarp();
  return __shfl_sync(kFull, incl, 31);
}

// idx-th set bit of cur (0-based), using the prefix array.
__device__ __forceinline__ uint32_t frontier_select(const WarpSmem &w, int nw, uint32_t idx) {
  int lo = 0, hi = nw - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (w.pfx[mid] <= idx) lo = mid; else hi = mid - 1;
  }
  const uint32_t word = w.cur[lo];
  const uint32_t r = idx - w.pfx[lo];
  const int bit = __fns(word, 0, (int)r + 1);
  return (uint32_t)lo * 32u + (uint32_t)bit;
}

// Query state is kept in partition-major (internal) vertex order, so a
// partition's slice of one query is a contiguous run of S values.
__device__ __forceinline__ void load_slice(uint32_t *dst, const uint32_t *src, int Sp, int lane) {
  if (((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15u) == 0 && (Sp & 3) == 0) {
    const uint4 *s4 = reinterpret_cast<const uint4 *>(src);
    uint4 *d4 = reinterpret_cast<uint4 *>(dst);
    for (int i = lane; i < (Sp >> 2); i += 32) d4[i] = __ldcg(s4 + i);
  } else {
    for (int i = lane; i < Sp; i += 32) dst[i] = __ldcg(src + i);
  }
}

__device__ __forceinline__ void store_slice(uint32_t *dst, const uint32_t *src, int Sp, int lane) {
  if (((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15u) == 0 && (Sp & 3) == 0) {
    uint4 *d4 = reinterpret_cast<uint4 *>(dst);
    const uint4 *s4 = reinterpret_cast<const uint4 *>(src);
    for (int i = lane; i < (Sp >> 2); i += 32) __stcg(d4 + i, s4[i]);
  } else {
    for (int i = lane; i < Sp; i += 32) __stcg(dst + i, src[i]);
  }
}

// The resident partition's CSR: prp = rp + partition base, indexed by the
// local vertex id, holding absolute arc offsets into g.adj / g.wt.
// A vertex's arc range must lie inside the arc arrays (never index outside them).
__device__ __forceinline__ bool arcs_in_range(const DevGraph &g, uint32_t e0, uint32_t deg) {
  return (uint64_t)e0 + deg <= g.m;
}

// The arc after the `step` from j on, or tot: tot may be any number below 2^32,
// so j + step must not pass it.
__device__ __forceinline__ uint32_t next_arcs(uint32_t j, uint32_t tot, uint32_t step) {
  return tot - j > step ? j + step : tot;
}

// The visit's queue: positions head .. tail - 1 of the ring (modulo S).
struct Queue {
  uint32_t head = 0, tail = 0;  // the same in every lane
};

// Shared-memory atomics with a result under a predicate (no branch): the old
// value, or `none` where on is false.
__device__ __forceinline__ uint32_t shared_min_if(bool on, uint32_t addr, uint32_t x, uint32_t none) {
  uint32_t old = none;
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %3, 0;\n\t@q atom.shared.min.u32 %0, [%1], %2;\n\t}"
               : "+r"(old) : "r"(addr), "r"(x), "r"((uint32_t)on) : "memory");
  return old;
}
__device__ __forceinline__ uint32_t shared_or_if(bool on, uint32_t addr, uint32_t x, uint32_t none) {
  uint32_t old = none;
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %3, 0;\n\t@q atom.shared.or.b32 %0, [%1], %2;\n\t}"
               : "+r"(old) : "r"(addr), "r"(x), "r"((uint32_t)on) : "memory");
  return old;
}

// K arcs a lane: from values dv to targets u (kInf: none; bit 31 = the target
// has more than four arcs) over weights wt. A target in this partition is
// lowered, marked in its set -- queue (nd < T), far window ([T, Ty)) or later
// visit -- and, if it was not in it yet, put into the queue. A far or carry bit
// stays when its vertex is lowered into the queue: the sets are held against
// the values when they are read. out[k] = the target lies in another
// partition. Every lane calls it.
//
// A step of a visit is one chain of dependent operations, and a branch of its
// own for each arc would put the arcs' chains one after another; so the arcs go
// side by side, predicated, with one vote each at the end.
template <int QT, int K>
__device__ __forceinline__ void relax_arcs(const EngineArgs &a, const DistSmem &w, Queue &qu, const uint32_t (&u)[K],
                                           const uint32_t (&wt)[K], const uint32_t (&dv)[K], uint32_t p, uint32_t T,
                                           uint32_t Ty, uint32_t (&nd)[K], bool (&out)[K]) {
  const uint32_t S1 = (uint32_t)(a.g.S - 1), lt = (1u << lane_id()) - 1u;
  const uint32_t s_d = smem_addr(w.d), s_inq = smem_addr(w.inq), s_far = smem_addr(w.far), s_carry = smem_addr(w.carry);
  uint32_t old[K], was[K];
  bool over = false;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    nd[k] = dv[k] + (QT == Q_BFS ? 1u : wt[k]);
    over |= u[k] != kInf && (nd[k] < dv[k] || nd[k] == kInf);
  }
  if (over) {  // 2^32 - 1 reached: saturate and report
    atomicCAS(&a.ctrl->status, 0, (int)FG_ERR_OVERFLOW);
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (nd[k] < dv[k] || nd[k] == kInf) nd[k] = kInf - 1u;
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const bool in = ((u[k] & 0x7FFFFFFFu) >> a.g.slog2) == p;
    out[k] = u[k] != kInf && !in;
    old[k] = shared_min_if(u[k] != kInf && in, s_d + (u[k] & S1) * 4u, nd[k], 0u);
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const uint32_t lu = u[k] & S1, set = nd[k] < T ? s_inq : (nd[k] < Ty ? s_far : s_carry);
    was[k] = shared_or_if(nd[k] < old[k], set + (lu >> 5) * 4u, 1u << (lu & 31), kFull);
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const uint32_t lu = u[k] & S1;
    const bool push = ((was[k] >> (lu & 31)) & 1u) == 0u && nd[k] < T;
    const unsigned m = __ballot_sync(kFull, push);
    if (push) w.ring[(qu.tail + (uint32_t)__popc(m & lt)) & S1] = (uint16_t)(lu | ((u[k] >> 31) << 15));
    qu.tail += (uint32_t)__popc(m);
  }
}

// Put the set bits of a lane's word of inq into the queue. Every lane calls it.
__device__ __forceinline__ void queue_bits(const DistSmem &w, Queue &qu, uint32_t bits, uint32_t first, uint32_t S1) {
  const uint32_t c = (uint32_t)__popc(bits), incl = warp_incl_scan(c);
  uint32_t at = qu.tail + incl - c;
  for (; bits; bits &= bits - 1u) w.ring[at++ & S1] = (uint16_t)((first + (uint32_t)__ffs(bits) - 1u) | kMoreArcs);
  qu.tail += __shfl_sync(kFull, incl, 31);
}

// ---------------------------------------------------------------------------
// Candidates for other partitions. An arc that leaves the partition needs the
// target's committed value, a read from L2 or HBM, and on a road-like graph
// one arc in twenty leaves: read on the spot, it would add its latency to
// most steps of the visit's chain. So a visit puts such candidates (target,
// value, source vertex) into the warp's list in shared memory and sends them
// 32 at a time: drop those that do not lower the target, append the others to
// the arena, and mark the source of one that does not fit for a later visit.
// ---------------------------------------------------------------------------
struct ExtList {
  uint32_t n = 0;  // held, the same in every lane, < 32 between calls
};

__device__ __forceinline__ void ext_send(const EngineArgs &a, const DistSmem &w, ExtList &x, uint32_t cnt, uint32_t q,
                                         Counters &ctr, ArenaSlots &sl) {
  const int lane = lane_id();
  __syncwarp();
  const bool mine = (uint32_t)lane < cnt;
  const uint32_t u = mine ? w.ext[lane] : 0u, nd = mine ? w.ext[kExt + lane] : kInf,
                 v = mine ? w.ext[2 * kExt + lane] : 0u;
  const bool has = mine && nd < a.dist[(size_t)q * (size_t)a.g.n + u];
  if (!emit_ops(a, has, (u >> a.g.slog2) * (uint32_t)a.nq + q, u & (uint32_t)(a.g.S - 1), nd, true, &sl)) {
    atomicOr(&w.spill[v >> 5], 1u << (v & 31));
    ctr.spills++;
  }
  const uint32_t left = x.n - cnt;  // < 32
  uint32_t m0 = 0u, m1 = 0u, m2 = 0u;
  if ((uint32_t)lane < left) {
    m0 = w.ext[cnt + lane];
    m1 = w.ext[kExt + cnt + lane];
    m2 = w.ext[2 * kExt + cnt + lane];
  }
  __syncwarp();
  if ((uint32_t)lane < left) {
    w.ext[lane] = m0;
    w.ext[kExt + lane] = m1;
    w.ext[2 * kExt + lane] = m2;
  }
  x.n = left;
  __syncwarp();
}

// Every lane calls it; lanes with `on` have a candidate.
__device__ __forceinline__ void ext_add(const EngineArgs &a, const DistSmem &w, ExtList &x, bool on, uint32_t u,
                                        uint32_t nd, uint32_t v, uint32_t q, Counters &ctr, ArenaSlots &sl) {
  const unsigned m = __ballot_sync(kFull, on);
  if (m == 0u) return;
  if (on) {
    const uint32_t at = x.n + (uint32_t)__popc(m & ((1u << lane_id()) - 1u));
    w.ext[at] = u;
    w.ext[kExt + at] = nd;
    w.ext[2 * kExt + at] = v;
  }
  x.n += (uint32_t)__popc(m);
  if (x.n >= 32u) ext_send(a, w, x, 32u, q, ctr, sl);
}

// ---------------------------------------------------------------------------
// SSSP / BFS visit of one (partition, query) buffer. On a road-like graph a
// visit expands few vertices at a time (some eleven of four arcs on the
// 1024^2 grid) one after another, so its time is the length of the dependent
// chain of a step, not its arcs. Vertices to expand wait in a first-in
// first-out queue; a step takes up to 32 from its head, in one of two forms:
//   PAIRS  graphs whose out-degrees are at most kPairSlots: the arcs of a
//          vertex stand in a record of fixed size (g.pairs), read without
//          offsets, scan or search. Two lanes take a vertex, two arcs each
//          with one 16-byte load; the few vertices of more than four arcs
//          take a second load. 16 vertices a step. (The three figures below
//          in the other form: 67.0, 20.9 and 0.61 ms.)
//   else   the arcs of 32 vertices are spread evenly over the lanes, kUnroll
//          runs of 32 with their loads in flight together.
// What a step spends is mostly warp-wide operations (35-65 cycles each for a
// vote, a shuffle, a warp barrier, as for a shared-memory read) and branches, so
// the queue is a list in shared memory rather than bitmaps searched with scans,
// arcs go side by side (relax_arcs), and whatever is rare stands behind one
// branch. On the 1024^2 grid (GB300; with bitmaps, two reads behind the offsets
// and 32 arcs after another before): SSSP, 256 sources 82.0 -> 58.1 ms; BFS on
// 701 x 1113, 100 sources 29.8 -> 17.9; one source on 41 x 48 0.92 -> 0.45. A
// round ends with its longest visit: warps wait 60 % of their time there.
// ---------------------------------------------------------------------------
template <int QT, bool PAIRS>
__device__ void visit_dist(const EngineArgs &a, const DistSmem &w, uint4 item, uint32_t qbound, const uint32_t *prp,
                           Counters &ctr, ArenaSlots &sl) {
  const DevGraph &g = a.g;
  const int lane = lane_id();
  const uint32_t key = item.x, off = item.y, cnt = item.z, flags = item.w;
  const uint32_t nq = (uint32_t)a.nq;
  const uint32_t p = key / nq, q = key - p * nq;
  const int S = g.S, nw = S >> 5;
  const uint32_t S1 = (uint32_t)(S - 1);
  const uint32_t base = p << g.slog2;
  const int Sp = min(S, g.n - (int)base);
  uint32_t *drow = a.dist + (size_t)q * (size_t)g.n;
  Queue qu;
  ExtList xl;

  // 1. stage the query's slice of this partition (bypassing L1)
  load_slice(w.d, drow + base, Sp, lane);
  for (int i = Sp + lane; i < S; i += 32) w.d[i] = kInf;
  uint32_t *pend = a.pend + (size_t)key * (size_t)nw;
  for (int wd = lane; wd < nw; wd += 32) {
    // 2. vertices deferred by an earlier visit
    uint32_t b = 0u;
    if (flags & 1u) {
      b = __ldcg(pend + wd);
      pend[wd] = 0u;
    }
    w.inq[wd] = b; w.far[wd] = 0u; w.carry[wd] = 0u; w.spill[wd] = 0u;
  }
  __syncwarp();
  // 3. apply buffered operations; an operation is live iff it improves the value
  const uint2 *ops = a.b_op + off;
  for (uint32_t j = lane; j < cnt; j += 32) {
    const uint2 o = __ldcg(ops + j);
    if (o.y < atomicMin(&w.d[o.x], o.y)) atomicOr(&w.inq[o.x >> 5], 1u << (o.x & 31));
  }
  __syncwarp();
  for (int wd = lane; wd - lane < nw; wd += 32) queue_bits(w, qu, wd < nw ? w.inq[wd] : 0u, (uint32_t)wd * 32u, S1);
  __syncwarp();
  // 4. in-visit windows: values >= Ty wait for a later visit (yield heuristic 2);
  //    values in [T, Ty) wait for the window to advance (near/far order).
  uint32_t fmin = kInf;
  for (uint32_t i = lane; i < qu.tail; i += 32) fmin = min(fmin, w.d[w.ring[i] & ~kMoreArcs]);
  fmin = warp_min_u32(fmin);
  if (fmin == kInf) return;  // every operation was stale: the slice is unchanged
  ctr.visits++;
  // values at or beyond Ty stay buffered for a later visit: the yield window
  // (first value + delta) and, under priority scheduling, the query's round
  // bound (best pending value + window), i.e. Delta-stepping across partitions
  const uint32_t Ty = min(a.delta ? sat_add_u32(fmin, a.delta) : kInf, qbound);
  uint32_t T = a.bucket ? min(sat_add_u32(fmin, a.bucket), Ty) : Ty;
  if (T != kInf) {
    const uint32_t n0 = qu.tail;  // at most S entries, from position 0: kept ones move to the front
    qu.tail = 0;
    for (uint32_t b0 = 0; b0 < n0; b0 += 32) {
      const uint32_t i = b0 + (uint32_t)lane;
      const uint32_t v = i < n0 ? w.ring[i] & ~kMoreArcs : 0u;
      const uint32_t d = i < n0 ? w.d[v] : kInf;
      __syncwarp();
      const bool keep = i < n0 && d < T;
      if (i < n0 && !keep) {
        const uint32_t bit = 1u << (v & 31);
        atomicAnd(&w.inq[v >> 5], ~bit);
        atomicOr(&(d < Ty ? w.far : w.carry)[v >> 5], bit);
      }
      const unsigned m = __ballot_sync(kFull, keep);
      if (keep) w.ring[qu.tail + (uint32_t)__popc(m & ((1u << lane) - 1u))] = (uint16_t)(v | kMoreArcs);
      qu.tail += (uint32_t)__popc(m);
    }
    __syncwarp();
  }

  // Yield heuristic 1 is asked each time the vertices that were queued when it
  // was asked last have been taken: a step takes 16 or 32 of them, and a visit
  // that stops among them leaves the rest of a frontier to another round (256^2
  // grid, 64 SSSP sources, yield_edges 64: 115 ms asked every step, 29 so).
  const bool a_yields = a.yield_edges != 0;
  uint32_t turn = 0;  // queue position
  uint32_t steps = 0;
  uint32_t arcs = 0;        // PAIRS: of this lane, at most four a step
  uint64_t warp_arcs = 0;   // else: of the warp; hubs taken again and again pass 2^32
  auto scanned = [&]() -> uint64_t { return PAIRS ? (uint64_t)__reduce_add_sync(kFull, arcs) : warp_arcs; };
  static_assert(32ull * 4ull * kMaxVisitSteps < 1ull << 32, "the arcs of a PAIRS visit are counted in 32 bits");
  for (;;) {
    // everything but taking a step stands behind one branch
    if ((qu.head == qu.tail) | (++steps % 256u == 0u) | (a_yields & ((int32_t)(qu.head - turn) >= 0)) |
        arena_pressed(a, sl.seen)) {
      // bounded loop: a visit can never spin forever
      if (steps > kMaxVisitSteps) {
        raise_status(a.ctrl, FG_ERR_TIMEOUT, kSiteVisit);
        break;
      }
      if (steps % 256u == 0u && ld_volatile_i32(&a.ctrl->abort)) break;
      if (qu.head == qu.tail) {
        // advance the in-visit window to the smallest far value; a vertex whose
        // value fell below the window since it was marked has been queued then
        uint32_t fm = kInf;
        if (a.bucket) {
          for (int wd = lane; wd < nw; wd += 32) {
            uint32_t b = w.far[wd], drop = 0u;
            while (b) {
              const int t = __ffs(b) - 1;
              b &= b - 1;
              const uint32_t d = w.d[wd * 32 + t];
              if (d < T) drop |= 1u << t;
              else fm = min(fm, d);
            }
            w.far[wd] &= ~drop;
          }
          fm = warp_min_u32(fm);
        }
        if (fm == kInf) break;
        T = min(sat_add_u32(fm, a.bucket), Ty);
        for (int wd = lane; wd - lane < nw; wd += 32) {
          uint32_t mv = 0u;
          if (wd < nw) {
            for (uint32_t b = w.far[wd]; b; b &= b - 1) {
              const int t = __ffs(b) - 1;
              if (w.d[wd * 32 + t] < T) mv |= 1u << t;
            }
            w.far[wd] &= ~mv;
            w.inq[wd] |= mv;
          }
          queue_bits(w, qu, mv, (uint32_t)wd * 32u, S1);
        }
        __syncwarp();
        continue;
      }
      // yield heuristic 1, or arena pressure: leave the rest to a later visit
      if (a_yields && (int32_t)(qu.head - turn) >= 0) {
        if (scanned() >= a.yield_edges) break;
        turn = qu.tail;
      }
      if (arena_pressed(a, sl.seen)) break;
    }
    const uint32_t F = min(qu.tail - qu.head, PAIRS ? 16u : 32u);
    // A vertex leaves the queue before its value is read, so that a later fall
    // queues it again.
    if (PAIRS) {
      const uint32_t i = (uint32_t)lane >> 1;
      uint32_t v = 0, dv = 0;
      uint4 r = make_uint4(kInf, 0u, kInf, 0u), r2 = r;
      bool more = false;
      if (i < F) {
        const uint32_t en = w.ring[(qu.head + i) & S1];
        v = en & ~kMoreArcs;
        more = (en & kMoreArcs) != 0u;
        const uint4 *rec = reinterpret_cast<const uint4 *>(g.pairs) + (size_t)(base + v) * (kPairSlots / 2) + (lane & 1);
        r = __ldg(rec);
        if (more) r2 = __ldg(rec + 2);
        if (!(lane & 1)) atomicAnd(&w.inq[v >> 5], ~(1u << (v & 31)));
      }
      qu.head += F;
      const bool four = __any_sync(kFull, more);
      __syncwarp();  // both lanes of a vertex read its value after it has left the queue
      if (i < F) dv = w.d[v];
      const uint32_t u[2] = {r.x, r.z}, wt[2] = {r.y, r.w}, from[2] = {dv, dv};
      uint32_t nd[2], nd2[2] = {kInf, kInf};
      bool out[2], out2[2] = {false, false};
      arcs += (r.x != kInf ? 1u : 0u) + (r.z != kInf ? 1u : 0u);
      relax_arcs<QT, 2>(a, w, qu, u, wt, from, p, T, Ty, nd, out);
      const uint32_t u2[2] = {r2.x, r2.z}, wt2[2] = {r2.y, r2.w};
      if (four) {
        arcs += (r2.x != kInf ? 1u : 0u) + (r2.z != kInf ? 1u : 0u);
        relax_arcs<QT, 2>(a, w, qu, u2, wt2, from, p, T, Ty, nd2, out2);
      }
      if (__any_sync(kFull, out[0] || out[1] || out2[0] || out2[1])) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          ext_add(a, w, xl, out[k], u[k] & 0x7FFFFFFFu, nd[k], v, q, ctr, sl);
          ext_add(a, w, xl, out2[k], u2[k] & 0x7FFFFFFFu, nd2[k], v, q, ctr, sl);
        }
      }
    } else {
      uint32_t v = 0, dv = 0, a0 = 0, deg = 0;
      if ((uint32_t)lane < F) {
        v = w.ring[(qu.head + (uint32_t)lane) & S1] & ~kMoreArcs;
        a0 = prp[v];
        deg = prp[v + 1] - a0;
        if (deg > g.max_deg || !arcs_in_range(g, a0, deg)) {  // inconsistent view: skip
          raise_status(a.ctrl, FG_ERR_CUDA, kSiteDegree);
          deg = 0;
        }
        atomicAnd(&w.inq[v >> 5], ~(1u << (v & 31)));
      }
      qu.head += F;
      __syncwarp();
      if ((uint32_t)lane < F) dv = w.d[v];
      const uint32_t incl = warp_incl_scan(deg);
      const uint32_t exd = incl - deg;
      const uint32_t tot = __shfl_sync(kFull, incl, 31);
      warp_arcs += tot;
      for (uint32_t j = 0; j < tot; j = next_arcs(j, tot, 32u * kUnroll)) {
        const uint32_t left = tot - j;
        uint32_t u[kUnroll], wt[kUnroll], own[kUnroll];
#pragma unroll
        for (int k = 0; k < kUnroll; ++k) {
          u[k] = kInf;
          wt[k] = 1u;
          own[k] = 0u;
          if (32u * (uint32_t)k < left) {  // warp-uniform
            const uint32_t t = j + 32u * (uint32_t)k + (uint32_t)lane;
            const bool has = 32u * (uint32_t)k + (uint32_t)lane < left;
            const int L = owner_lane(exd, has ? t : 0u);
            const uint32_t eL = __shfl_sync(kFull, a0, L) + (t - __shfl_sync(kFull, exd, L));
            own[k] = (uint32_t)L;
            if (has) {
              u[k] = g.adj[eL];
              if (QT != Q_BFS && g.wt != nullptr) wt[k] = g.wt[eL];
            }
          }
        }
        uint32_t du[kUnroll], nd[kUnroll];
        bool out[kUnroll];
#pragma unroll
        for (int k = 0; k < kUnroll; ++k) du[k] = __shfl_sync(kFull, dv, (int)own[k]);
        relax_arcs<QT, kUnroll>(a, w, qu, u, wt, du, p, T, Ty, nd, out);
        bool any_out = false;
#pragma unroll
        for (int k = 0; k < kUnroll; ++k) any_out |= out[k];
        if (__any_sync(kFull, any_out)) {
#pragma unroll
          for (int k = 0; k < kUnroll; ++k)
            ext_add(a, w, xl, out[k], u[k], nd[k], __shfl_sync(kFull, v, (int)own[k]), q, ctr, sl);
        }
      }
    }
    __syncwarp();  // the queue's new entries are read by the next step
  }
  ctr.edges += scanned();
  if (xl.n > 0u) ext_send(a, w, xl, xl.n, q, ctr, sl);
  __syncwarp();

  // 5. leftovers -> pending bitmap of this buffer: what is still queued (the
  // visit stopped early), values beyond the bounds, spilled vertices. A carry
  // bit whose value has fallen below Ty since went through the queue, a far
  // one below T as well.
  uint32_t cmin = kInf;
  bool any = false;
  for (int wd = lane; wd < nw; wd += 32) {
    uint32_t b = w.inq[wd] | w.spill[wd];
    uint32_t late = (w.carry[wd] | w.far[wd]) & ~b;
    for (uint32_t x = b | late; x; x &= x - 1) {
      const int t = __ffs(x) - 1;
      const uint32_t bit = 1u << t, d = w.d[wd * 32 + t];
      if ((late & bit) && d < T) continue;
      b |= bit;
      cmin = min(cmin, d);
    }
    if (b) {
      any = true;
      pend[wd] = b;
    }
  }
  any = __any_sync(kFull, any);
  cmin = warp_min_u32(cmin);
  if (any && lane == 0) {
    a.dirty[key] = 1u;
    atomicMin(&a.prio[key], cmin);
    ctr.yields++;
  }
  // 6. write the slice back
  __syncwarp();
  store_slice(drow + base, w.d, Sp, lane);
}

// ---------------------------------------------------------------------------
// PPR forward-push visit of one (partition, query) buffer.
// Residuals of the slice live in shared memory; estimates and their Kahan
// compensation are updated in global memory (single writer per slice).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float ppr_thr(const uint32_t *prp, float eps, uint32_t v_local) {
  const uint32_t d = prp[v_local + 1] - prp[v_local];
  return eps * (float)(d > 0u ? d : 1u);
}

// Targets of arcs j + 32 k + lane of a batch of vertices (exd: arcs before a
// lane's vertex, of which it has deg from a0 on; none: one to the source), kInf
// beyond the `left` that there are from j on, and the lanes of their vertices. A round lasts as long as its
// longest visit, and a visit with a hub as long as the chain over the hub's arcs:
// so the loads of kUnroll steps are in flight together, and steps within one
// vertex take their owner once. R-MAT 2^18, 64 sources, per batch: 4.55 ms with one
// step at a time, 3.90 so.
// Only for pass 2. The count decides when a batch reserves its room: with hubs
// quicker there, a round that fills the arena carries small batches over instead
// of hubs (3,600 of them, not 800, and 2.7 ms), and the pushes come in another
// order, which moves estimates by ten times what two runs differ by.
__device__ __forceinline__ void ppr_targets(const DevGraph &g, uint32_t src, uint32_t exd, uint32_t deg, uint32_t a0,
                                            uint32_t j, uint32_t left, uint32_t (&u)[kUnroll],
                                            uint32_t (&own)[kUnroll]) {
  const uint32_t last = j + (min(32u * kUnroll, left) - 1u);
  const int ends = owner_lane(exd, (lane_id() & 1) ? last : j);
  const int L = __shfl_sync(kFull, ends, 0);
  if (L == __shfl_sync(kFull, ends, 1)) {
    const uint32_t degL = __shfl_sync(kFull, deg, L);
    const uint32_t e = __shfl_sync(kFull, a0, L) + (j - __shfl_sync(kFull, exd, L));
#pragma unroll
    for (int k = 0; k < kUnroll; ++k) {
      const uint32_t t = 32u * k + (uint32_t)lane_id();
      own[k] = (uint32_t)L;
      u[k] = t < left ? (degL > 0u ? __ldg(g.adj + e + t) : src) : kInf;
    }
    return;
  }
#pragma unroll
  for (int k = 0; k < kUnroll; ++k) {
    const uint32_t t = j + 32u * k + (uint32_t)lane_id();
    const bool has = 32u * k + (uint32_t)lane_id() < left;
    own[k] = (uint32_t)owner_lane(exd, has ? t : 0u);
    const uint32_t degL = __shfl_sync(kFull, deg, (int)own[k]);
    const uint32_t e = __shfl_sync(kFull, a0, (int)own[k]) + (t - __shfl_sync(kFull, exd, (int)own[k]));
    u[k] = has ? (degL > 0u ? __ldg(g.adj + e) : src) : kInf;
  }
}

__device__ void visit_ppr(const EngineArgs &a, const WarpSmem &w0, uint4 item, const uint32_t *prp, Counters &ctr,
                          ArenaSlots &sl) {
  const DevGraph &g = a.g;
  const int lane = lane_id();
  const uint32_t key = item.x, off = item.y, cnt = item.z, flags = item.w;
  const uint32_t nq = (uint32_t)a.nq;
  const uint32_t p = key / nq, q = key - p * nq;
  const int S = g.S, nw = S >> 5;
  const uint32_t base = p << g.slog2;
  const int Sp = min(S, g.n - (int)base);
  const size_t row = (size_t)q * (size_t)g.n;
  float *rrow = a.pr_r + row;
  float *prow = a.pr_p + row;
  float *crow = a.pr_c + row;
  WarpSmem w = w0;
  float *rs = reinterpret_cast<float *>(w.d);
  const WordRange wr(nw, lane);
  const float alpha = a.alpha, eps = a.eps;
  const float beta = 1.0f - alpha;
  const uint32_t src_int = g.intl ? (uint32_t)g.intl[a.src[q]] : (uint32_t)a.src[q];

  load_slice(w.d, reinterpret_cast<const uint32_t *>(rrow + base), Sp, lane);
  for (int i = Sp + lane; i < S; i += 32) rs[i] = 0.f;
  for (int wd = lane; wd < nw; wd += 32) {
    w.cur[wd] = 0u; w.nxt[wd] = 0u; w.carry[wd] = 0u;
  }
  uint32_t *pend = a.pend + (size_t)key * (size_t)nw;
  if (flags & 1u) {
    for (int wd = lane; wd < nw; wd += 32) {
      w.cur[wd] = __ldcg(pend + wd);
      pend[wd] = 0u;
    }
  }
  __syncwarp();
  const uint2 *ops = a.b_op + off;
  for (uint32_t j = lane; j < cnt; j += 32) {
    const uint2 o = __ldcg(ops + j);
    const float inc = __uint_as_float(o.y);
    const float thr = ppr_thr(prp, eps, o.x);
    const float old = atomicAdd(&rs[o.x], inc);
    if (old < thr && __fadd_rn(old, inc) >= thr) atomicOr(&w.cur[o.x >> 5], 1u << (o.x & 31));
  }
  __syncwarp();

  uint64_t vis_edges = 0;
  bool stopped = false, touched = (cnt > 0) || (flags & 1u);
  uint32_t steps = 0;
  for (;;) {
    if (++steps > kMaxVisitSteps || ((steps & 255u) == 0 && ld_volatile_i32(&a.ctrl->abort))) {
      if (steps > kMaxVisitSteps) raise_status(a.ctrl, FG_ERR_TIMEOUT, kSiteVisit);
      stopped = true;
      break;
    }
    const uint32_t F = frontier_prefix(w, wr);
    if (F == 0) break;
    if (a.yield_edges && vis_edges >= a.yield_edges) {
      stopped = true;
      break;
    }
    for (uint32_t b0 = 0; b0 < F; b0 += 32) {
      const uint32_t idx = b0 + (uint32_t)lane;
      const bool valid = idx < F;
      uint32_t v = 0, a0 = 0, deg = 0;
      if (valid) {
        v = frontier_select(w, nw, idx);
        a0 = prp[v];
        deg = prp[v + 1] - a0;
        if (deg > g.max_deg || !arcs_in_range(g, a0, deg)) {  // inconsistent view: skip
          raise_status(a.ctrl, FG_ERR_CUDA, kSiteDegree);
          deg = 0;
        }
      }
      // arcs this lane's vertex contributes (a dangling vertex sends one
      // operation back to the source)
      const uint32_t arcs = valid ? (deg > 0u ? deg : 1u) : 0u;
      const uint32_t incl = warp_incl_scan(arcs);
      const uint32_t exd = incl - arcs;
      const uint32_t tot = __shfl_sync(kFull, incl, 31);
      // pass 1: count operations for other partitions and reserve them at once
      uint32_t n_ext = 0;
      for (uint32_t j = 0; j < tot; j += 32) {
        const uint32_t t = j + (uint32_t)lane;
        const bool has = t < tot;
        const int L = owner_lane(exd, has ? t : 0u);
        const uint32_t degL = __shfl_sync(kFull, deg, L);
        const uint32_t eL = __shfl_sync(kFull, a0, L) + (t - __shfl_sync(kFull, exd, L));
        bool ext = false;
        if (has) {
          const uint32_t u = degL > 0u ? g.adj[eL] : src_int;
          ext = (u >> g.slog2) != p;
        }
        n_ext += __popc(__ballot_sync(kFull, ext));
      }
      // reserve the batch's cross-partition increments together, from the
      // warp's own arena chunk (a new chunk of at least kArenaChunk slots
      // when it runs short)
      unsigned long long rbase = 0;
      if (n_ext) {
        if (sl.pos + n_ext > sl.end) {
          release_slots(a, sl);
          const unsigned long long want = n_ext > kArenaChunk ? (unsigned long long)n_ext : kArenaChunk;
          unsigned long long b = 0;
          if (lane == 0) b = atomicAdd(&a.ctrl->e_cursor, want);
          b = __shfl_sync(kFull, b, 0);
          sl.pos = b;
          sl.end = b + want;
          sl.seen = sl.end;
        }
        rbase = sl.pos;
        sl.pos += n_ext;
      }
      if (n_ext && rbase + n_ext > a.e_cap) {
        // does not fit this round: keep these vertices for a later visit
        if (n_ext > a.e_cap) raise_status(a.ctrl, FG_ERR_BIN_OVERFLOW, kSiteArena);
        for (unsigned long long s = rbase + lane; s < a.e_cap && s < rbase + n_ext; s += 32)
          a.e_key[s] = kInvalidKey;
        if (valid) atomicOr(&w.carry[v >> 5], 1u << (v & 31));
        if (lane == 0) ctr.spills++;
        __syncwarp();
        continue;
      }
      // take the residuals and move alpha * rho into the estimates (Kahan)
      float rho = 0.f, inc_l = 0.f;
      if (valid) {
        rho = atomicExch(&rs[v], 0.f);
        const uint32_t gi = base + v;
        const float pe = __ldcg(prow + gi), ce = __ldcg(crow + gi);
        const float y = __fsub_rn(__fmul_rn(alpha, rho), ce);
        const float tsum = __fadd_rn(pe, y);
        __stcg(crow + gi, __fsub_rn(__fsub_rn(tsum, pe), y));
        __stcg(prow + gi, tsum);
        inc_l = deg > 0u ? __fdiv_rn(__fmul_rn(beta, rho), (float)deg) : __fmul_rn(beta, rho);
      }
      vis_edges += tot;
      // pass 2: spread (1 - alpha) rho
      uint32_t run = 0;
      for (uint32_t j = 0; j < tot; j = next_arcs(j, tot, 32u * kUnroll)) {
        uint32_t u[kUnroll], own[kUnroll];
        ppr_targets(g, src_int, exd, deg, a0, j, tot - j, u, own);
#pragma unroll
        for (int k = 0; k < kUnroll; ++k) {
          const float inc = __shfl_sync(kFull, inc_l, (int)own[k]);
          const bool ext = u[k] != kInf && (u[k] >> g.slog2) != p;
          const uint32_t lu = u[k] & (uint32_t)(S - 1);
          if (u[k] != kInf && !ext) {
            const float thr = ppr_thr(prp, eps, lu);
            const float old = atomicAdd(&rs[lu], inc);
            if (old < thr && __fadd_rn(old, inc) >= thr) atomicOr(&w.nxt[lu >> 5], 1u << (lu & 31));
          }
          const unsigned em = __ballot_sync(kFull, ext);
          if (ext) {
            const unsigned long long slot = rbase + run + __popc(em & ((1u << lane) - 1u));
            const uint32_t pk = (u[k] >> g.slog2) * nq + q;
            a.e_key[slot] = pk;
            a.e_op[slot] = make_uint2(lu, __float_as_uint(inc));
            const unsigned grp = __match_any_sync(em, pk);
            if (lane == __ffs(grp) - 1) atomicAdd(&a.cnt[pk], (unsigned)__popc(grp));
          }
          run += __popc(em);
        }
      }
      __syncwarp();
    }
    for (int wd = wr.w0; wd < wr.w1; ++wd) w.cur[wd] = 0u;
    __syncwarp();
    uint32_t *tmp = w.cur; w.cur = w.nxt; w.nxt = tmp;
  }
  ctr.edges += vis_edges;
  if (touched) ctr.visits++;

  bool any = false;
  for (int wd = wr.w0; wd < wr.w1; ++wd) {
    uint32_t b = w.carry[wd];
    if (stopped) b |= w.cur[wd] | w.nxt[wd];
    if (b) {
      any = true;
      pend[wd] = b;
    }
  }
  any = __any_sync(kFull, any);
  if (any && lane == 0) {
    a.dirty[key] = 1u;
    ctr.yields++;
  }
  __syncwarp();
  store_slice(reinterpret_cast<uint32_t *>(rrow + base), w.d, Sp, lane);
}

// Coin of the random scheduler: a 32-bit mix of (key, round) (the finalizer
// of MurmurHash3, Appleby 2011).
__device__ __forceinline__ uint32_t sched_coin(uint32_t key, uint32_t round) {
  uint32_t x = key * 0x9E3779B1u ^ (round + 1u) * 0x85EBCA77u;
  x ^= x >> 16;
  x *= 0x85EBCA6Bu;
  x ^= x >> 13;
  x *= 0xC2B2AE35u;
  x ^= x >> 16;
  return x;
}

// Buffer skipped by priority scheduling this round (SSSP/BFS). No warp stages
// this (partition, query) slice in the current round, so its operations are
// applied directly to the query's state with atomicMin and the improved
// vertices join the buffer's pending bitmap; the buffer stays non-empty.
__device__ void carry_item(const EngineArgs &a, uint4 item, uint32_t item_prio) {
  const DevGraph &g = a.g;
  const int lane = lane_id();
  const uint32_t key = item.x, off = item.y, cnt = item.z;
  const uint32_t nq = (uint32_t)a.nq;
  const uint32_t p = key / nq, q = key - p * nq;
  const uint32_t base = p << g.slog2;
  const int nw = g.S >> 5;
  uint32_t *drow = a.dist + (size_t)q * (size_t)g.n;
  uint32_t *pend = a.pend + (size_t)key * (size_t)nw;
  bool any = false;
  for (uint32_t j = lane; j < cnt; j += 32) {
    const uint2 o = __ldcg(a.b_op + off + j);
    const uint32_t old = atomicMin(drow + base + o.x, o.y);
    if (o.y < old) {
      atomicOr(pend + (o.x >> 5), 1u << (o.x & 31));
      any = true;
    }
  }
  any = __any_sync(kFull, any) || (item.w & 1u);
  if (any && lane == 0) {
    a.dirty[key] = 1u;
    atomicMin(&a.prio[key], item_prio);
  }
}

// ---------------------------------------------------------------------------
// Block-wide exclusive scan of one u64 per thread.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long block_excl_scan(unsigned long long x, unsigned long long *s_warp,
                                                              unsigned long long &total) {
  const int lane = lane_id(), wid = threadIdx.x >> 5;
  const unsigned long long incl = warp_incl_scan(x);
  if (lane == 31) s_warp[wid] = incl;
  block_sync();
  if (wid == 0) {
    unsigned long long v = lane < kWarps ? s_warp[lane] : 0ull;
    const unsigned long long vi = warp_incl_scan(v);
    if (lane < kWarps) s_warp[lane] = vi - v;
    if (lane == kWarps - 1) s_warp[kWarps] = vi;
  }
  block_sync();
  const unsigned long long ex = s_warp[wid] + incl - x;
  total = s_warp[kWarps];
  block_sync();
  return ex;
}

// Block-level work claiming. *claim packs (end << 32 | next) for the block's
// current chunk of item indices; the one warp that draws next == end refills
// the chunk from the device-wide counter, warps that draw past the end wait
// for the refill. Chunks are consecutive items (ordered by partition, then
// query), so the warps of one block mostly visit the same partition and read
// its CSR through the SM's L1. Called by one lane; returns an index >= tot
// when the round has no work left for this block.
__device__ uint32_t claim_item(Ctrl *c, unsigned long long *claim, volatile int *done, uint32_t tot,
                               uint64_t watchdog_ns) {
  uint64_t t0 = 0;
  unsigned spins = 0;
  for (;;) {
    if (*done) return kInvalidKey;
    const unsigned long long old = atomicAdd(claim, 1ull);
    const uint32_t pos = (uint32_t)old, end = (uint32_t)(old >> 32);
    if (pos < end) return pos;
    if (pos == end) {
      // full chunks while plenty of work is left; near the end of the round
      // small ones, so that no block takes several visits per warp into the tail
      const uint32_t seen = *reinterpret_cast<volatile uint32_t *>(&c->item_next);
      const uint32_t left = seen < tot ? tot - seen : 0u;
      const uint32_t chunk = left > 4u * kBlockChunk * gridDim.x ? kBlockChunk : kTailChunk;
      uint32_t b = atomicAdd(&c->item_next, chunk);
      if (ld_volatile_i32(&c->abort)) b = tot;
      if (b >= tot) {
        *done = 1;
        return kInvalidKey;
      }
      const uint32_t e = min(tot, b + chunk);
      atomicExch(claim, ((unsigned long long)e << 32) | (unsigned long long)(b + 1u));
      return b;
    }
    // another warp is refilling: wait until the chunk end moves (bounded)
    while ((uint32_t)(*reinterpret_cast<volatile unsigned long long *>(claim) >> 32) == end && !*done) {
      if ((++spins & 63u) == 0) {
        const uint64_t t = global_ns();
        if (t0 == 0) t0 = t;
        else if (t - t0 > watchdog_ns) {
          raise_status(c, FG_ERR_TIMEOUT, kSiteClaim);
          *done = 1;
          return kInvalidKey;
        }
      }
      __nanosleep(32);
    }
  }
}

template <int QT, bool PAIRS>
__global__ void __launch_bounds__(kThreads, 3) engine_kernel(EngineArgs a) {
  extern __shared__ __align__(16) uint32_t smem_dyn[];
  __shared__ unsigned long long s_scan[kWarps + 1];
  __shared__ unsigned long long s_pre[4];
  __shared__ unsigned long long s_hv[kWarps];
  __shared__ unsigned long long s_claim;  // block's chunk of work items (claim_item)
  __shared__ int s_claim_done;
  constexpr bool kPPR = (QT == Q_PPR);

  const int lane = lane_id(), wid = threadIdx.x >> 5;
  const int S = a.g.S, nw = S >> 5;
  WarpSmem w;   // PPR
  DistSmem wd;  // SSSP, BFS
  {
    uint32_t *b = smem_dyn + (size_t)wid * warp_smem_words(kPPR, S);
    if (kPPR) {
      w.d = b;
      w.cur = b + S;
      w.nxt = w.cur + nw;
      w.carry = w.nxt + nw;
      w.pfx = w.carry + nw;
    } else {
      wd.d = b;
      wd.ring = reinterpret_cast<uint16_t *>(b + S);
      wd.inq = b + S + S / 2;
      wd.far = wd.inq + nw;
      wd.carry = wd.far + nw;
      wd.spill = wd.carry + nw;
      wd.ext = wd.spill + nw;
    }
  }
  Ctrl *c = a.ctrl;
  // every block reads the generation before its first arrival, so all agree
  unsigned gen = barrier_generation(c);
  Counters ctr;
  // phase clock of block 0 (device time between device-wide barriers)
  uint64_t t_prev = (blockIdx.x == 0 && threadIdx.x == 0) ? global_ns() : 0ull;
  unsigned long long ph[6] = {0ull, 0ull, 0ull, 0ull, 0ull, 0ull};
#define FG_PHASE(k)                                             \
  do {                                                          \
    if (blockIdx.x == 0 && threadIdx.x == 0) {                  \
      const uint64_t t_now = global_ns();                       \
      ph[k] += t_now - t_prev;                                  \
      t_prev = t_now;                                           \
    }                                                           \
  } while (0)
  const uint64_t K = (uint64_t)a.g.nparts * (uint64_t)a.nq;
  const uint64_t per_blk = (K + gridDim.x - 1) / gridDim.x;
  const uint64_t k0 = umin64(K, (uint64_t)blockIdx.x * per_blk);
  const uint64_t k1 = umin64(K, k0 + per_blk);
  const uint32_t gwarp = blockIdx.x * kWarps + wid, nwarps = gridDim.x * kWarps;

  // ---- K0: state tiles and per-buffer counters (InitBuffers, first half) ----
  {
    const uint64_t rows = (uint64_t)a.nq * (uint64_t)a.g.n;
    const uint64_t tid = (uint64_t)blockIdx.x * kThreads + threadIdx.x, nthr = (uint64_t)gridDim.x * kThreads;
    if (kPPR) {
      fill_u32(reinterpret_cast<uint32_t *>(a.pr_p), rows, 0u, tid, nthr);
      fill_u32(reinterpret_cast<uint32_t *>(a.pr_r), rows, 0u, tid, nthr);
      fill_u32(reinterpret_cast<uint32_t *>(a.pr_c), rows, 0u, tid, nthr);
    } else {
      fill_u32(a.dist, rows, kInf, tid, nthr);
      fill_u32(a.prio, K, kInf, tid, nthr);
      fill_u32(a.qbest, 2u * (uint64_t)a.nq, kInf, tid, nthr);
    }
    fill_u32(a.cnt, K, 0u, tid, nthr);
    fill_u32(a.dirty, K, 0u, tid, nthr);
  }
  if (!grid_barrier(c, gen, a.watchdog_ns)) goto done;
  FG_PHASE(0);

  // ---- INIT: seed operations (InitBuffers, second half) ----
  for (uint32_t q0 = gwarp * 32u; q0 < (uint32_t)a.nq; q0 += nwarps * 32u) {
    const uint32_t q = q0 + lane;
    bool has = q < (uint32_t)a.nq;
    uint32_t key = 0, lv = 0;
    if (has && (a.src[q] < 0 || a.src[q] >= a.g.n)) {
      raise_status(c, FG_ERR_INVALID_ARG, kSiteSource);  // source id out of range
      has = false;
    }
    if (has) {
      const int32_t s = a.src[q];
      const uint32_t v = a.g.intl ? (uint32_t)a.g.intl[s] : (uint32_t)s;
      key = (v >> a.g.slog2) * (uint32_t)a.nq + q;
      lv = v & (uint32_t)(S - 1);
    }
    const uint32_t val0 = kPPR ? __float_as_uint(1.0f) : 0u;
    const bool ok = emit_ops(a, has, key, lv, val0, !kPPR);
    if (!ok) raise_status(c, FG_ERR_BIN_OVERFLOW, kSiteArena);
  }
  if (!grid_barrier(c, gen, a.watchdog_ns)) goto done;
  FG_PHASE(1);

  for (uint32_t round = 0;; ++round) {
    // best pending value per query: written in SCAN-A, read in SCAN-B and PROCESS,
    // and the other half is cleared in SCATTER for the next round
    uint32_t *qb_cur = a.qbest + (size_t)(round & 1u) * (size_t)a.nq;
    uint32_t *qb_nxt = a.qbest + (size_t)((round + 1u) & 1u) * (size_t)a.nq;
    // ---- SCAN-A: per-block totals ----
    {
      unsigned long long loc = 0, hv = 0;
      uint32_t mx = 0;  // largest buffer of the round (max-operations scheduling)
#pragma unroll 4
      for (uint64_t k = k0 + threadIdx.x; k < k1; k += kThreads) {
        const uint32_t n_ops = __ldcg(a.cnt + k);
        const bool dk = __ldcg(a.dirty + k) != 0u;
        const bool act = n_ops > 0u || dk;
        loc += ((unsigned long long)n_ops << 32) | (act ? 1ull : 0ull);
        hv += dk ? 1ull : 0ull;
        if (!kPPR && act && a.sched == FG_SCHED_PRIORITY)
          atomicMin(&qb_cur[(uint32_t)k % (uint32_t)a.nq], __ldcg(a.prio + k));
        if (!kPPR && a.sched == FG_SCHED_MAXOPS) mx = n_ops > mx ? n_ops : mx;
      }
      if (!kPPR && a.sched == FG_SCHED_MAXOPS) {
        mx = __reduce_max_sync(kFull, mx);
        if (lane == 0 && mx > 0u) atomicMax(&c->max_ops[round & 1u], mx);
      }
      loc = warp_sum(loc);
      hv = warp_sum(hv);
      if (lane == 0) { s_scan[wid] = loc; s_hv[wid] = hv; }
      block_sync();
      if (threadIdx.x == 0) {
        unsigned long long t = 0, th = 0;
        for (int i = 0; i < kWarps; ++i) { t += s_scan[i]; th += s_hv[i]; }
        a.blocksum[blockIdx.x] = t;
        a.blocksum[gridDim.x + blockIdx.x] = th;
      }
    }
    if (!grid_barrier(c, gen, a.watchdog_ns)) goto done;
    FG_PHASE(2);
    // ---- SCAN-B: work items, bin offsets, buffer reset ----
    unsigned long long tot_ops, tot_items, emitted;
    {
      unsigned long long pre = 0, all = 0, preh = 0, allh = 0;
      for (int i = threadIdx.x; i < (int)gridDim.x; i += kThreads) {
        const unsigned long long v = __ldcg(a.blocksum + i);
        const unsigned long long vh = __ldcg(a.blocksum + gridDim.x + i);
        all += v;
        allh += vh;
        if (i < (int)blockIdx.x) { pre += v; preh += vh; }
      }
      pre = warp_sum(pre);
      all = warp_sum(all);
      preh = warp_sum(preh);
      allh = warp_sum(allh);
      if (lane == 0) { s_hv[wid] = preh; }
      block_sync();
      if (threadIdx.x == 0) {
        unsigned long long t = 0;
        for (int i = 0; i < kWarps; ++i) t += s_hv[i];
        s_pre[2] = t;
      }
      block_sync();
      if (lane == 0) { s_hv[wid] = allh; }
      block_sync();
      if (threadIdx.x == 0) {
        unsigned long long t = 0;
        for (int i = 0; i < kWarps; ++i) t += s_hv[i];
        s_pre[3] = t;
      }
      block_sync();
      if (lane == 0) s_scan[wid] = pre;
      block_sync();
      if (threadIdx.x == 0) {
        unsigned long long t = 0;
        for (int i = 0; i < kWarps; ++i) t += s_scan[i];
        s_pre[0] = t;
      }
      block_sync();
      if (lane == 0) s_scan[wid] = all;
      block_sync();
      if (threadIdx.x == 0) {
        unsigned long long t = 0;
        for (int i = 0; i < kWarps; ++i) t += s_scan[i];
        s_pre[1] = t;
      }
      block_sync();
      pre = s_pre[0];
      all = s_pre[1];
      tot_ops = all >> 32;
      tot_items = all & 0xFFFFFFFFull;
      emitted = umin64(*reinterpret_cast<volatile unsigned long long *>(&c->e_cursor), a.e_cap);
      block_sync();
      if (tot_items == 0) break;
      if (round >= a.max_rounds) {
        if (threadIdx.x == 0) raise_status(c, FG_ERR_TIMEOUT, kSiteRounds);
        break;
      }
      unsigned long long run_ops = pre >> 32, run_items = pre & 0xFFFFFFFFull, run_h = s_pre[2];
      const unsigned long long H = s_pre[3];
      const uint32_t window = a.sched_window;
      // tiles of kThreads keys; the next tile's counters are loaded while the
      // current one is scanned and written (the block scan synchronises)
      const bool by_window = !kPPR && a.sched == FG_SCHED_PRIORITY;
      const uint32_t round_max = (!kPPR && a.sched == FG_SCHED_MAXOPS)
                                     ? *reinterpret_cast<volatile unsigned *>(&c->max_ops[round & 1u])
                                     : 0u;
      uint32_t nx_ops = 0, nx_dirty = 0, nx_prio = kInf, nx_qb = kInf;
      {
        const uint64_t k = k0 + threadIdx.x;
        if (k < k1) {
          nx_ops = __ldcg(a.cnt + k);
          nx_dirty = __ldcg(a.dirty + k);
          if (!kPPR) nx_prio = __ldcg(a.prio + k);
          if (by_window) nx_qb = __ldcg(qb_cur + (uint32_t)k % (uint32_t)a.nq);
        }
      }
      for (uint64_t t0 = k0; t0 < k1; t0 += kThreads) {
        const uint64_t k = t0 + threadIdx.x;
        const uint32_t n_ops = nx_ops, dflag = nx_dirty, pr = nx_prio, qb = nx_qb;
        const bool act = k < k1 && (n_ops > 0u || dflag != 0u);
        {
          const uint64_t kn = k + kThreads;
          nx_ops = 0u;
          nx_dirty = 0u;
          nx_prio = kInf;
          nx_qb = kInf;
          if (kn < k1) {
            nx_ops = __ldcg(a.cnt + kn);
            nx_dirty = __ldcg(a.dirty + kn);
            if (!kPPR) nx_prio = __ldcg(a.prio + kn);
            if (by_window) nx_qb = __ldcg(qb_cur + (uint32_t)kn % (uint32_t)a.nq);
          }
        }
        const bool heavy = act && dflag != 0u;
        const unsigned long long x = ((unsigned long long)n_ops << 32) | (act ? 1ull : 0ull) | (heavy ? (1ull << 16) : 0ull);
        unsigned long long tile_tot;
        const unsigned long long ex = block_excl_scan(x, s_scan, tile_tot);
        if (act) {
          const unsigned long long I = run_items + (ex & 0xFFFFull), J = run_h + ((ex >> 16) & 0xFFFFull);
          const uint32_t item_idx = (uint32_t)(heavy ? J : H + I - J);
          const uint32_t off = (uint32_t)(run_ops + (ex >> 32));
          uint32_t fl = dflag ? 1u : 0u;
          if (!kPPR) {
            if (by_window && pr > sat_add_u32(qb, window)) fl |= 2u;
            // Max-#ops and Random (Tab. 4A) in round form: a buffer without
            // carried-over work waits one round when it holds under a quarter
            // of the round's largest buffer, or when a coin drawn from (key,
            // round) says so; it then carries its work and is taken next round
            if (dflag == 0u && a.sched == FG_SCHED_MAXOPS && 4ull * (unsigned long long)n_ops < round_max)
              fl |= 2u;
            if (dflag == 0u && a.sched == FG_SCHED_RANDOM && (sched_coin((uint32_t)k, round) & 1u)) fl |= 2u;
            a.prio[k] = kInf;
          }
          a.items[item_idx] = make_uint4((uint32_t)k, off, n_ops, fl);
          if (!kPPR) a.iprio[item_idx] = pr;
          a.cur[k] = off;
          a.cnt[k] = 0u;
          a.dirty[k] = 0u;
        }
        run_ops += tile_tot >> 32;
        run_items += tile_tot & 0xFFFFull;
        run_h += (tile_tot >> 16) & 0xFFFFull;
      }
      if (blockIdx.x == 0 && threadIdx.x == 0) {
        c->rounds += 1ull;
        c->ops += tot_ops;
        if (tot_ops > c->max_round_ops) c->max_round_ops = tot_ops;
      }
    }
    if (!grid_barrier(c, gen, a.watchdog_ns)) goto done;
    FG_PHASE(3);
    // ---- SCATTER: arena -> bins ordered by (partition, query) ----
    {
      if (blockIdx.x == 0 && threadIdx.x == 0) {
        c->e_cursor = 0ull;
        c->item_next = 0u;
        c->max_ops[(round + 1u) & 1u] = 0u;
      }
      if (threadIdx.x == 0) {  // visible to the block after the barrier below
        s_claim = 0ull;
        s_claim_done = 0;
      }
      if (!kPPR && a.sched == FG_SCHED_PRIORITY)
        for (uint32_t i = blockIdx.x * kThreads + threadIdx.x; i < (uint32_t)a.nq; i += gridDim.x * kThreads)
          qb_nxt[i] = kInf;
      const unsigned long long n_emit = emitted;
      for (unsigned long long i0 = (unsigned long long)gwarp * 32ull; i0 < n_emit; i0 += (unsigned long long)nwarps * 32ull) {
        const unsigned long long i = i0 + lane;
        const bool has0 = i < n_emit;
        uint32_t key = kInvalidKey;
        uint2 o = make_uint2(0u, 0u);
        if (has0) {
          key = __ldcg(a.e_key + i);
          o = __ldcg(a.e_op + i);
        }
        const bool has = has0 && key != kInvalidKey;
        const unsigned m = __ballot_sync(kFull, has);
        if (has) {
          const unsigned grp = __match_any_sync(m, key);
          const int gl = __ffs(grp) - 1;
          uint32_t pos = 0;
          if (lane == gl) pos = atomicAdd(&a.cur[key], (unsigned)__popc(grp));
          pos = __shfl_sync(grp, pos, gl) + __popc(grp & ((1u << lane) - 1u));
          a.b_op[pos] = o;
        }
      }
      (void)tot_ops;
    }
    if (!grid_barrier(c, gen, a.watchdog_ns)) goto done;
    FG_PHASE(4);
    // ---- PROCESS: IntraPartProcess of every work item ----
    // Items are handed out by claim_item (block-level chunks). The resident
    // partition lives in L1/L2: the graph and the round's active state slices
    // fit in L2. No block-level synchronisation here.
    {
      ArenaSlots sl;
      for (;;) {
        uint32_t idx = 0;
        if (lane == 0) idx = claim_item(c, &s_claim, &s_claim_done, (uint32_t)tot_items, a.watchdog_ns);
        idx = __shfl_sync(kFull, idx, 0);
        if (idx >= (uint32_t)tot_items) break;
        const uint4 it = __ldcg(a.items + idx);
        const uint32_t p = it.x / (uint32_t)a.nq;
        const uint32_t *prp = a.g.rp + ((size_t)p << a.g.slog2);
        bool defer = !kPPR && (it.w & 2u);
        if (!kPPR && !defer) {
          unsigned long long cursor = 0;
          if (lane == 0) cursor = *reinterpret_cast<volatile unsigned long long *>(&c->e_cursor);
          cursor = __shfl_sync(kFull, cursor, 0);
          defer = arena_pressed(a, cursor > sl.seen ? cursor : sl.seen);
        }
        if (defer) {
          carry_item(a, it, __ldcg(a.iprio + idx));
        } else if (kPPR) {
          visit_ppr(a, w, it, prp, ctr, sl);
        } else {
          const uint32_t q = it.x - p * (uint32_t)a.nq;
          const uint32_t qbound =
              a.sched == FG_SCHED_PRIORITY ? sat_add_u32(__ldcg(qb_cur + q), a.sched_window) : kInf;
          visit_dist<QT, PAIRS>(a, wd, it, qbound, prp, ctr, sl);
        }
      }
      release_slots(a, sl);  // before the barrier: SCATTER reads every reserved slot
    }
    if (!grid_barrier(c, gen, a.watchdog_ns)) goto done;
    FG_PHASE(5);
  }
done:
#undef FG_PHASE
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const uint64_t t_now = global_ns();
    ph[3] += t_now - t_prev;  // the final scan that found no work
    for (int k = 0; k < 6; ++k) atomicAdd(&c->phase_ns[k], ph[k]);
  }
  {
    const unsigned long long sp = warp_sum(ctr.spills), yl = warp_sum(ctr.yields);
    if (lane == 0) {
      atomicAdd(&c->visits, ctr.visits);
      atomicAdd(&c->edges, ctr.edges);
      atomicAdd(&c->arcs_read, ctr.edges);
      atomicAdd(&c->spills, sp);
      atomicAdd(&c->yields, yl);
    }
  }
}

// ---------------------------------------------------------------------------
// Per-query mass check (PPR): fold the Kahan compensation into the estimate
// (p_out = p - c, FP32) and accumulate sum(p_out) + sum(r) in FP64.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) ppr_finalize_kernel(const float *p, const float *cmp, const float *r,
                                                           float *p_out, float *r_out, const int32_t *orig, int64_t n,
                                                           int64_t chunks, double *mass) {
  __shared__ double s_red[8];
  const int64_t q = blockIdx.x / chunks, ch = blockIdx.x % chunks;
  const int64_t per = (n + chunks - 1) / chunks;
  const int64_t i0 = ch * per, i1 = i0 + per < n ? i0 + per : n;
  const float *prow = p + q * n;
  const float *crow = cmp + q * n;
  const float *rrow = r + q * n;
  float *porow = p_out + q * n;
  float *rorow = r_out ? r_out + q * n : nullptr;
  double acc = 0.0;
  for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    const float pf = __fsub_rn(prow[i], crow[i]);
    const float rf = rrow[i];
    const int64_t o = orig ? (int64_t)orig[i] : i;
    porow[o] = pf;
    if (rorow && rorow != rrow) rorow[o] = rf;
    acc += (double)pf + (double)rf;
  }
  if (mass) {
    acc = warp_sum(acc);
    if (lane_id() == 0) s_red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += s_red[i];
      atomicAdd(mass + q, t);
    }
  }
}

// Query-major state in internal order -> caller's output in original order.
__global__ void __launch_bounds__(256) permute_out_kernel(const uint32_t *state, uint32_t *out, const int32_t *orig,
                                                          int64_t n, int64_t rows) {
  const int64_t total = n * rows;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t q = t / n, i = t - q * n;
    out[q * n + orig[i]] = state[t];
  }
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
// The arc records of a graph whose out-degrees are at most kPairSlots: left
// packed, the rest kInf; bit 31 of a target = it has more than four arcs itself
// (its record's second half is then read with the first).
__global__ void __launch_bounds__(256) pair_records_kernel(DevGraph g, uint2 *out) {
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  const int64_t v = i / kPairSlots;
  const uint32_t k = (uint32_t)(i % kPairSlots);
  if (v >= (int64_t)g.nparts * g.S) return;
  uint2 r = make_uint2(kInf, 0u);
  if (v < g.n) {
    const uint32_t e = g.rp[v], deg = g.rp[v + 1] - e;
    if (k < deg) {
      const uint32_t u = g.adj[e + k];
      r = make_uint2(u | (g.rp[u + 1] - g.rp[u] > 4u ? 0x80000000u : 0u), g.wt ? g.wt[e + k] : 1u);
    }
  }
  out[i] = r;
}

cudaError_t launch_pair_records(const DevGraph &g, uint2 *out, cudaStream_t s) {
  const int64_t total = (int64_t)g.nparts * g.S * kPairSlots;
  pair_records_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(g, out);
  return cudaGetLastError();
}

static const void *engine_fn(int qtype, bool pairs) {
  switch (qtype) {
    case Q_SSSP: return pairs ? (const void *)engine_kernel<Q_SSSP, true> : (const void *)engine_kernel<Q_SSSP, false>;
    case Q_BFS: return pairs ? (const void *)engine_kernel<Q_BFS, true> : (const void *)engine_kernel<Q_BFS, false>;
    default: return (const void *)engine_kernel<Q_PPR, false>;
  }
}

// Lets a kernel be launched with any dynamic shared memory the device has: the
// limit belongs to the kernel, not to a graph, and graphs of different
// partition sizes are in use at once.
cudaError_t allow_dynamic_smem(const void *fn) {
  cudaFuncAttributes at;
  int dev = 0, optin = 0;
  cudaError_t e = cudaFuncGetAttributes(&at, fn);
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)at.sharedSizeBytes);
}

cudaError_t engine_grid_size(int qtype, bool pairs, int S, int *blocks, int *threads, size_t *smem) {
  const void *fn = engine_fn(qtype, pairs);
  *threads = kThreads;
  *smem = (size_t)kWarps * warp_smem_words(qtype == Q_PPR, S) * sizeof(uint32_t);
  cudaError_t e = allow_dynamic_smem(fn);
  if (e != cudaSuccess) return e;
  int per_sm = 0, dev = 0, sms = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kThreads, *smem);
  if (e != cudaSuccess) return e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  *blocks = per_sm * sms;
  return cudaSuccess;
}

cudaError_t launch_engine(const EngineArgs &a, int blocks, int threads, size_t smem, cudaStream_t s) {
  EngineArgs copy = a;
  // SSSP / BFS: whole chunks while the arena holds four of every warp that can be
  // busy. A visit sends what leaves its partition at its end, so with fewer the
  // first visits to end would take the arena (64 sources, 256^2 grid: 512 slots
  // 4.2 s with chunks, 1.8 without; 4,096 slots 490 and 207 ms; 32,768 slots 102 and 46).
  const uint64_t busy = std::min<uint64_t>((uint64_t)a.g.nparts * (uint64_t)a.nq, (uint64_t)blocks * kWarps);
  copy.arena_chunk = a.e_cap < 4ull * kArenaChunk * busy ? 1u : kArenaChunk;
  void *args[] = {(void *)&copy};
  return cudaLaunchCooperativeKernel(engine_fn(a.qtype, a.g.pairs != nullptr), dim3(blocks), dim3(threads), args, smem, s);
}

cudaError_t launch_ppr_finalize(const EngineArgs &a, double *mass, float *p_out, float *r_out, cudaStream_t s) {
  const int64_t n = a.g.n;
  const int64_t chunks = (n + 4095) / 4096;
  const int64_t grid = chunks * (int64_t)a.nq;
  if (grid <= 0) return cudaSuccess;
  ppr_finalize_kernel<<<(unsigned)grid, 256, 0, s>>>(a.pr_p, a.pr_c, a.pr_r, p_out, r_out, a.g.orig, n, chunks, mass);
  return cudaGetLastError();
}

cudaError_t launch_permute_out(const uint32_t *state, uint32_t *out, const int32_t *orig, int64_t n, int64_t rows,
                               cudaStream_t s) {
  const int64_t total = n * rows;
  if (total <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const int64_t want = (total + 255) / 256;
  const unsigned grid = (unsigned)(want < (int64_t)sms * 16 ? want : (int64_t)sms * 16);
  permute_out_kernel<<<grid, 256, 0, s>>>(state, out, orig, n, rows);
  return cudaGetLastError();
}

}  // namespace fg
