// Arcs that lie on no shortest path, found once per graph for the group
// engine's SSSP batches.
//
// An arc (v, u) of weight w is on some shortest path only if w = d(v, u). So
// when a walk from v to u shorter than w is known, the arc can be left out and
// every distance from every source stays the same: the arcs of a shortest path
// all satisfy w = d and are never left out. Walks through a few hubs are enough
// to see most of them on a power-law graph with spread weights: with R[v][k] =
// the length of a walk from v to hub k and F[u][k] = of one from hub k to u,
// the arc goes when min over k of R[v][k] + F[u][k] < w. (A walk that uses the
// arc itself is at least w long, so it never counts against it.)
//
// Eight hubs of largest out-degree are used. On R-MAT graphs with weights
// 1..255 they leave 9-12 % of the arcs (2^13 to 2^16 vertices, edge factor 16,
// both directions; 16 hubs: 0.3 points fewer; the arcs with w = d exactly: 8 %
// at 2^14), and 21 % at edge factor 4.
//
// R and F come from rounds over all arcs on a table T[v][16] (lanes 0-7 = R,
// 8-15 = F): one 64-byte line per end of an arc, half a warp per 128 arcs, so
// that hubs are spread over many warps. R[v] takes the minimum over v's arcs in
// a register, F[u] is lowered with atomicMin. Values only fall and every value
// is the length of a walk, whatever the order and however stale a read, so any
// number of rounds gives valid bounds; the rounds stop when one changes nothing
// (each launch looks at its predecessor's flag), 8 to 11 on R-MAT.
//
// What it gives (GB300, R-MAT 2^20 vertices, 31.4 M arcs, weights 1..255): the
// marks take 7.6 ms once per graph; a batch of 256 SSSP queries reads 51.6 M
// arcs instead of 769.5 M and takes 8.8 ms instead of 55.8 by this alone (directed, 300,007
// vertices, 6.5 M arcs, 97 queries: 3.1 instead of 10.1; 7.5 and 2.2 with the group engine's later steps). The rounds are bound
// by the random 64-byte lines of T (64 MB here, mostly in L2).
#include <cstdint>

#include "fg_device.cuh"

namespace fg {
namespace {

constexpr int kRedThreads = 256;
constexpr int kRedArcs = 128;  // arcs per half warp (rounds)
constexpr int kMarkArcs = 64;  // arcs per lane group of eight (marks): two words of bits

// Largest vertex v with rp[v] <= e (e < rp[n]): the owner of arc e.
__device__ __forceinline__ uint32_t arc_owner(const uint32_t *rp, int32_t n, uint32_t e) {
  uint32_t lo = 0, hi = (uint32_t)n;
  while (hi - lo > 1u) {
    const uint32_t mid = lo + (hi - lo) / 2u;
    if (__ldg(rp + mid) <= e) lo = mid; else hi = mid;
  }
  return lo;
}

__global__ void __launch_bounds__(kRedThreads) reduce_init(uint32_t *T, int64_t n, HubSet h, unsigned *flags) {
  const int64_t i = (int64_t)blockIdx.x * kRedThreads + threadIdx.x;
  if (i <= kReduceRounds) flags[i] = i == 0 ? 1u : 0u;
  if (i >= n * 16) return;
  T[i] = h.v[i & 7] == (uint32_t)(i >> 4) ? 0u : kInf;
}

__global__ void __launch_bounds__(kRedThreads) reduce_round(DevGraph g, uint32_t *T, const unsigned *before,
                                                            unsigned *changed) {
  if (*before == 0u) return;  // the round before changed nothing
  const int64_t half = ((int64_t)blockIdx.x * kRedThreads + threadIdx.x) >> 4;
  const uint64_t first = (uint64_t)half * kRedArcs;
  if (first >= g.m) return;
  const int lane = threadIdx.x & 15;
  const unsigned mask = 0xFFFFu << (threadIdx.x & 16);
  // (offsets within the piece: arc numbers near 2^32 have no room for a step past the end)
  const uint32_t e0 = (uint32_t)first, len = (uint32_t)umin64(g.m - first, kRedArcs);
  uint32_t v = arc_owner(g.rp, g.n, e0), next = __ldg(g.rp + v + 1);
  uint32_t tv = T[(size_t)v * 16 + lane], best = tv;
  bool moved = false;
  for (uint32_t o = 0; o < len; o += 16u) {
    const uint32_t eb = e0 + o, cnt = min(len - o, 16u);
    const uint32_t xa = (uint32_t)lane < cnt ? __ldg(g.adj + eb + lane) : 0u;
    const uint32_t wa = (uint32_t)lane < cnt ? __ldg(g.wt + eb + lane) : 0u;
    uint32_t t[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const uint32_t x = __shfl_sync(mask, xa, j, 16);
      t[j] = (uint32_t)j < cnt ? T[(size_t)x * 16 + lane] : kInf;
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const uint32_t w = __shfl_sync(mask, wa, j, 16), x = __shfl_sync(mask, xa, j, 16);
      if ((uint32_t)j >= cnt) continue;
      while (eb + (uint32_t)j >= next) {  // on to the owner of this arc
        if (best < tv) {
          atomicMin(T + (size_t)v * 16 + lane, best);
          moved = true;
        }
        ++v;
        next = __ldg(g.rp + v + 1);
        tv = T[(size_t)v * 16 + lane];
        best = tv;
      }
      const uint32_t from = lane < 8 ? t[j] : tv;
      const uint32_t c = from + w;
      if (c < from || from == kInf || c == kInf) continue;
      if (lane < 8) {
        best = c < best ? c : best;
      } else if (c < t[j]) {
        atomicMin(T + (size_t)x * 16 + lane, c);
        moved = true;
      }
    }
  }
  if (best < tv) {
    atomicMin(T + (size_t)v * 16 + lane, best);
    moved = true;
  }
  if (__any_sync(mask, moved) && lane == 0) *changed = 1u;
}

// Bit e of bits = arc e stays.
__global__ void __launch_bounds__(kRedThreads) reduce_mark(DevGraph g, const uint32_t *__restrict__ T, uint2 *bits) {
  const int64_t grp = ((int64_t)blockIdx.x * kRedThreads + threadIdx.x) >> 3;
  const uint64_t first = (uint64_t)grp * kMarkArcs;
  if (first >= g.m) return;
  const int lane = threadIdx.x & 7;
  const unsigned mask = 0xFFu << (threadIdx.x & 24);
  const uint32_t e0 = (uint32_t)first, len = (uint32_t)umin64(g.m - first, kMarkArcs);
  uint32_t v = arc_owner(g.rp, g.n, e0), next = __ldg(g.rp + v + 1);
  uint32_t rv = __ldg(T + (size_t)v * 16 + lane);
  uint64_t keep = 0ull;
  for (uint32_t o = 0; o < len; o += 8u) {
    const uint32_t eb = e0 + o, cnt = min(len - o, 8u);
    const uint32_t xa = (uint32_t)lane < cnt ? __ldg(g.adj + eb + lane) : 0u;
    const uint32_t wa = (uint32_t)lane < cnt ? __ldg(g.wt + eb + lane) : 0u;
    uint32_t f[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t x = __shfl_sync(mask, xa, j, 8);
      f[j] = (uint32_t)j < cnt ? __ldg(T + (size_t)x * 16 + 8 + lane) : kInf;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t w = __shfl_sync(mask, wa, j, 8);
      if ((uint32_t)j >= cnt) continue;
      while (eb + (uint32_t)j >= next) {
        ++v;
        next = __ldg(g.rp + v + 1);
        rv = __ldg(T + (size_t)v * 16 + lane);
      }
      uint32_t s = sat_add_u32(rv, f[j]);  // kInf + anything stays kInf
      s = min(s, __shfl_xor_sync(mask, s, 1, 8));
      s = min(s, __shfl_xor_sync(mask, s, 2, 8));
      s = min(s, __shfl_xor_sync(mask, s, 4, 8));
      if (s >= w) keep |= 1ull << (o + (uint32_t)j);
    }
  }
  if (lane == 0) bits[grp] = make_uint2((uint32_t)keep, (uint32_t)(keep >> 32));
}

}  // namespace

cudaError_t mark_useful_arcs(const DevGraph &g, const HubSet &hubs, uint32_t *table, unsigned *flags, uint32_t *bits,
                             cudaStream_t s) {
  const int64_t init = ((int64_t)g.n * 16 + kRedThreads - 1) / kRedThreads;
  reduce_init<<<(unsigned)init, kRedThreads, 0, s>>>(table, g.n, hubs, flags);
  cudaError_t e = cudaGetLastError();
  const int64_t halves = (int64_t)((g.m + kRedArcs - 1) / kRedArcs), groups = (int64_t)((g.m + kMarkArcs - 1) / kMarkArcs);
  const unsigned rb = (unsigned)((halves * 16 + kRedThreads - 1) / kRedThreads);
  for (int r = 0; r < kReduceRounds && e == cudaSuccess; ++r) {
    reduce_round<<<rb, kRedThreads, 0, s>>>(g, table, flags + r, flags + r + 1);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return e;
  reduce_mark<<<(unsigned)((groups * 8 + kRedThreads - 1) / kRedThreads), kRedThreads, 0, s>>>(
      g, table, reinterpret_cast<uint2 *>(bits));
  return cudaGetLastError();
}

}  // namespace fg
