// Sweep cuts over PPR vectors: the conductance step of the network community
// profile (NCP) application, which runs PPRs from a random sample of seed
// vertices (Sec. 1; Sec. 6.1 seeds 0.01% of the vertices). For query q the
// vertices with p(v) > 0 are ordered by the FP32 key p(v) / max(d(v), 1),
// largest first, ties by smaller original id; for each prefix S_k of the first
// `top` of them the kernel writes the conductance
//     phi(S_k) = cut(S_k) / min(vol(S_k), vol(V) - vol(S_k)),
// vol = sum of out-degrees, cut = arcs from S_k to the rest; and, across all
// queries of the call, the profile NCP(k) = min over queries of phi(S_k).
//
// The sort key of a vertex is 64 bits (~key bits << 32 | id), unique, ascending =
// key descending then id ascending. Five kernels, each spread over as many
// blocks as its work has room for:
//   sample   a histogram over 4,096 bins of the key bits (exponent and four
//            bits of mantissa) of one row chunk in sixteen (of all chunks up to
//            2^16 vertices), and from it a bin edge that the `top`-th key lies
//            above for all but certain, with about 1.4 times as many keys above
//            it as are wanted;
//   filter   one pass over the row: the sort keys of the vertices at or above the
//            edge go to the row's list, and the vertices with p > 0 are counted.
//            A vertex whose key must round below the edge is skipped before the
//            division (an FP32 test with a stated bound);
//   order    a block per row sorts the list and keeps the first `top`. A row whose
//            list is too long, or shorter than it has to be (the sample says
//            nothing about the rows of an adversary, or about ties), is streamed
//            instead through a buffer in shared memory that is cut back to the
//            `top` smallest keys whenever it fills: the kept set is the same;
//   inside   the neighbours ranked before each kept vertex: a shared-memory hash
//            from internal id to rank, the arcs of a block's vertices spread
//            evenly over its threads;
//   scan     prefix sums of d(v) - 2 * inside(v) and of d(v) give cut and vol
//            exactly in int64; phi = cut / den in FP64.
// The row read (p from HBM, 4 B per vertex; the degree table, shared by all
// queries, mostly from L2) is the traffic and bounds the filter; the others work
// on shared memory and the kept vertices' adjacency. R-MAT 2^20, 105 rows, top
// 4,096 (GB300): sample 16 us, edge 4, filter 116 (440 MB at 3.8 TB/s, and as
// much again of degrees from L2), order 55, inside 100, scan 18, and 0.33 ms for
// the call. One block per row doing all of it took 1.94 ms: 105 blocks leave a
// third of the SMs idle, and the threshold that its buffer finds on the way lets
// five times as many keys in. Rows of few vertices take one
// block, and few rows with a small `top` two kernels (below).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <mutex>

#include "fg_host.h"

namespace fg {
namespace {

constexpr int kThreads = 512;                   // 16 warps
constexpr int kWarps = kThreads / 32;
constexpr int kMaxTop = FG_NCP_MAX_TOP;         // 4096
constexpr int kCap = 2 * kMaxTop;               // candidate buffer (64-bit entries)
constexpr int kHash = 2 * kMaxTop;              // hash slots (load <= 1/2)
constexpr int kHashLog2 = 13;
constexpr uint32_t kEmpty = 0xFFFFFFFFu;
static_assert(kHash == (1 << kHashLog2), "hash size");

// dynamic shared memory of the order kernel: the candidate buffer (kBytesA) and,
// where a row is streamed, the copy of a cut
constexpr size_t kBytesA = (size_t)kCap * 8;
constexpr size_t kSmem = kBytesA + (size_t)kMaxTop * 8;

struct NcpArgs {
  const float *p = nullptr;        // [nq][n] original order
  const uint32_t *deg = nullptr;   // [n] out-degree, original order
  const uint32_t *rp = nullptr;    // [n+1] internal order
  const uint32_t *adj = nullptr;   // [m] internal ids
  const int32_t *intl = nullptr;   // original -> internal, or null (identity)
  int64_t n = 0;
  uint64_t m = 0;
  int32_t top = 0;
  int32_t *order = nullptr;        // [nq][top] or null
  double *phi = nullptr;           // [nq][top] or null
  int32_t *count = nullptr;        // [nq] or null
  unsigned long long *ncp = nullptr;  // [top] encoded profile, or null
  // scratch of the rows of one launch
  uint32_t *hist = nullptr;           // [rows][kBins] sampled keys per bin
  uint32_t *edge = nullptr;           // [rows] encoded key the list starts at
  unsigned long long *list = nullptr; // [rows][kCap] sort keys at or above it
  uint32_t *listed = nullptr;         // [rows] their number (beyond kCap: not all are there)
  uint32_t *positive = nullptr;       // [rows] vertices with p > 0
  unsigned long long *part = nullptr; // [min(rows, kStreamSlots)][parts][top] a streamed row's keys by parts
  uint32_t *kept = nullptr;           // [rows] min(top, positive)
  uint32_t *ids = nullptr;            // [rows][top] internal ids in sweep order
  uint32_t *first = nullptr;          // [rows][top + 1] arcs of the kept vertices before each (exclusive sums)
  int32_t *gain = nullptr;            // [rows][top] d - 2 * inside
};

// Sort key of a vertex: FP32 bit pattern of p / max(d, 1) plus one (bit
// patterns of non-negative floats order as the floats do); 0 = not a
// candidate (p not > 0, which also rejects NaN).
__device__ __forceinline__ uint32_t key_enc(float p, uint32_t d) {
  if (!(p > 0.f)) return 0u;
  const float k = __fdiv_rn(p, __uint2float_rn(d > 0u ? d : 1u));
  return __float_as_uint(k) + 1u;
}

// Order-preserving map of a double onto uint64 (for atomicMin), and back.
__device__ __forceinline__ unsigned long long dbl_enc(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double dbl_dec(unsigned long long e) {
  const unsigned long long b = (e >> 63) ? (e & 0x7FFFFFFFFFFFFFFFull) : ~e;
  return __longlong_as_double((long long)b);
}

// Profile: accumulate ? encode the caller's value : start from +inf (encoded).
enum class ProfileBegin { kNone, kFresh, kAccumulate };
__device__ __forceinline__ void profile_begin(unsigned long long *ncp, int i, bool accumulate) {
  const double x = accumulate ? __longlong_as_double((long long)ncp[i]) : __longlong_as_double(0x7FF0000000000000ll);
  ncp[i] = dbl_enc(x);
}

// Inclusive prefix sum within a warp.
template <typename T>
__device__ __forceinline__ T warp_prefix_incl(T x, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

constexpr int kVecPerTile = 1;                    // float4 row loads per thread per tile
constexpr int kSlots = 4 * kVecPerTile;            // row elements per thread per tile
constexpr int kTile = kThreads * kSlots;           // row elements per tile
// After a cut the buffer holds `top` <= kMaxTop keys; the room left above that
// decides how often the buffer is cut (a cut is a radix select over it).
static_assert(kCap - kTile >= kMaxTop + kTile, "after a cut, at least one full tile of admissions fits before the next");

// Row elements of tile t held by this thread: slot e. Vector form (n a
// multiple of 4): float4 / uint4 loads, element
// 4 * (t * kVecPerTile * kThreads + (e / 4) * kThreads + tid) + e % 4; scalar
// form: t * kTile + e * kThreads + tid. Each warp's addresses are contiguous.
template <bool VEC>
__device__ __forceinline__ int64_t slot_index(int64_t t, int e) {
  if (VEC) return 4 * (t * kVecPerTile * kThreads + (int64_t)(e >> 2) * kThreads + threadIdx.x) + (e & 3);
  return t * kTile + (int64_t)e * kThreads + threadIdx.x;
}

template <bool VEC>
__device__ __forceinline__ void load_tile(const float *prow, const uint32_t *deg, int64_t n, int64_t t,
                                          float (&pv)[kSlots], uint32_t (&dv)[kSlots]) {
  if (VEC) {
#pragma unroll
    for (int h = 0; h < kVecPerTile; ++h) {
      const int64_t v = slot_index<true>(t, 4 * h);
      float4 p4 = make_float4(0.f, 0.f, 0.f, 0.f);
      uint4 d4 = make_uint4(0u, 0u, 0u, 0u);
      if (v < n) {  // n is a multiple of 4: the whole vector is in the row
        p4 = __ldg(reinterpret_cast<const float4 *>(prow + v));
        d4 = __ldg(reinterpret_cast<const uint4 *>(deg + v));
      }
      pv[4 * h] = p4.x; pv[4 * h + 1] = p4.y; pv[4 * h + 2] = p4.z; pv[4 * h + 3] = p4.w;
      dv[4 * h] = d4.x; dv[4 * h + 1] = d4.y; dv[4 * h + 2] = d4.z; dv[4 * h + 3] = d4.w;
    }
  } else {
#pragma unroll
    for (int e = 0; e < kSlots; ++e) {
      const int64_t v = slot_index<false>(t, e);
      pv[e] = v < n ? __ldg(prow + v) : 0.f;
      dv[e] = v < n ? __ldg(deg + v) : 0u;
    }
  }
}

// Sort key of a candidate: ascending order = key descending, id ascending.
// Unique per vertex, so "the top smallest sort keys" is exact with no ties.
__device__ __forceinline__ unsigned long long sort_key(uint32_t enc, uint32_t v) {
  return ((unsigned long long)(~enc) << 32) | v;
}

struct Stream {
  unsigned long long *buf;  // [kCap] candidates
  unsigned long long *tmp;  // [kMaxTop]
  uint32_t *h;              // [256] digit histogram
  uint32_t *wsum;           // [kWarps]
  uint32_t *n_buf;          // candidates held
  uint32_t *n_tmp;
  unsigned long long *thr;  // keys >= thr cannot rank among the top any more
  uint32_t *sel;            // [2] bucket of the top-th key, keys below that bucket
};

// Cut the buffer back to its T smallest keys (block-wide; B = held > T).
// Radix select over the eight 8-bit digits of the 64-bit keys, from the top:
// each pass narrows the prefix of the T-th smallest key; after the last one
// the prefix is that key itself (keys are unique). The buffer keeps the keys
// <= it, and from then on the stream admits only keys below it.
__device__ void cut_back(const Stream &st, uint32_t T) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t B = *st.n_buf;
  unsigned long long prefix = 0;
  uint32_t below = 0;
  for (int shift = 56; shift >= 0; shift -= 8) {
    for (int i = tid; i < 256; i += kThreads) st.h[i] = 0u;
    __syncthreads();
    // the leading digits of the held keys fall into few bins: lanes with the
    // same bin add their count through one atomic (else they serialise)
    for (uint32_t base = 0; base < B; base += kThreads) {
      const uint32_t i = base + tid;
      uint32_t bin = 0xFFFFFFFFu;
      if (i < B) {
        const unsigned long long k = st.buf[i];
        if (shift == 56 || (k >> (shift + 8)) == prefix) bin = (uint32_t)((k >> shift) & 255u);
      }
      const unsigned grp = __match_any_sync(0xFFFFFFFFu, bin);
      if (bin != 0xFFFFFFFFu && lane == __ffs(grp) - 1) atomicAdd(&st.h[bin], (uint32_t)__popc(grp));
    }
    __syncthreads();
    // inclusive prefix over the 256 bins (threads 0..255, warps 0..7)
    uint32_t c = tid < 256 ? st.h[tid] : 0u;
    uint32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31 && warp < 8) st.wsum[warp] = incl;
    __syncthreads();
    if (tid < 256) {
      uint32_t off = below;
      for (int w = 0; w < warp; ++w) off += st.wsum[w];
      const uint32_t hi = off + incl, lo = hi - c;
      if (lo < T && hi >= T) {
        st.sel[0] = (uint32_t)tid;
        st.sel[1] = lo;
      }
    }
    __syncthreads();
    prefix = (prefix << 8) | st.sel[0];
    below = st.sel[1];
    __syncthreads();  // sel and h are rewritten by the next digit
  }
  const unsigned long long kth = prefix;  // the T-th smallest key
  if (tid == 0) *st.n_tmp = 0u;
  __syncthreads();
  for (uint32_t i = tid; i < B; i += kThreads) {
    const unsigned long long k = st.buf[i];
    if (k <= kth) {
      const uint32_t pos = atomicAdd(st.n_tmp, 1u);
      if (pos < (uint32_t)kMaxTop) st.tmp[pos] = k;
    }
  }
  __syncthreads();
  const uint32_t kept = min(*st.n_tmp, (uint32_t)kMaxTop);
  for (uint32_t i = tid; i < kept; i += kThreads) st.buf[i] = st.tmp[i];
  if (tid == 0) {
    *st.n_buf = kept;
    *st.thr = kth;
  }
  __syncthreads();
}

// Admission of one tile (block-wide): each thread offers up to kSlots keys
// (bit e of `mask` set = key[e] is below the threshold); admitted keys are
// appended to the buffer, and the barrier that ends the tile decides,
// uniformly, whether the buffer must be cut before the next tile.
__device__ __forceinline__ void admit_tile(const Stream &st, uint32_t T, const unsigned long long (&key)[kSlots],
                                           unsigned mask) {
  const int lane = threadIdx.x & 31;
  uint32_t held_after = 0;  // lane 0: the count right after this warp's last append
  if (__any_sync(0xFFFFFFFFu, mask != 0u)) {  // most tiles admit nothing once the buffer is full
#pragma unroll
    for (int e = 0; e < kSlots; ++e) {
      const bool take = (mask >> e) & 1u;
      const unsigned bal = __ballot_sync(0xFFFFFFFFu, take);
      if (bal) {
        uint32_t pos = 0;
        if (lane == 0) {
          pos = atomicAdd(st.n_buf, (uint32_t)__popc(bal));
          held_after = max(held_after, pos + (uint32_t)__popc(bal));
        }
        pos = __shfl_sync(0xFFFFFFFFu, pos, 0) + (uint32_t)__popc(bal & ((1u << lane) - 1u));
        if (take && pos < (uint32_t)kCap) st.buf[pos] = key[e];
      }
    }
  }
  // The last append of the tile saw the final count. (Reading the count after
  // a plain barrier would race with the next tile's appends.)
  if (__syncthreads_or(held_after > (uint32_t)(kCap - kTile))) cut_back(st, T);
}

__device__ __forceinline__ void stream_begin(const Stream &st) {
  if (threadIdx.x == 0) {
    *st.n_buf = 0u;
    *st.thr = ~0ull;  // every key is admitted until the first cut (real keys are below 2^64 - 2^32)
  }
  __syncthreads();
}

// The FP32 key value of the threshold (0 while every key is admitted).
__device__ __forceinline__ float thr_key(unsigned long long thr) {
  if (thr == ~0ull) return 0.f;
  const uint32_t enc = ~(uint32_t)(thr >> 32);
  return __uint_as_float(enc - 1u);
}

// Tiles [tlo, thi) of a row: every vertex whose sort key may
// still be among the T smallest is kept (the buffer holds at most T after the
// final cut). Tiles are visited in a scrambled order: step i takes tile
// tlo + (i * odd) mod P, P = the range rounded up to a power of two (a
// bijection; steps past the range load nothing), so keys that drift along the
// vertex ids (degree correlates with id in R-MAT numbering) do not keep
// beating the threshold.
//
// Most vertices end far below the threshold key K, and the exact key needs an
// IEEE division. A vertex is skipped without it when p < (K (1 - 2^-20)) * d
// in FP32 (three roundings of at most 2^-24 each: the conversion of d and the
// two products, so p / d < K (1 - 2^-21) and the rounded key is below K); the
// test is used only while the products are normal and finite. Every other
// vertex gets its exact key.
template <bool VEC>
__device__ void stream_row(const NcpArgs &a, const float *prow, const Stream &st, uint32_t T, int64_t tlo,
                           int64_t thi) {
  const int64_t n = a.n;
  int64_t P = 1;
  while (P < thi - tlo) P <<= 1;
  auto tile_at = [P, tlo](int64_t i) {
    return tlo + (int64_t)(((uint64_t)i * 0x9E3779B97F4A7C15ull) & (uint64_t)(P - 1));
  };
  const int64_t hi_elem = thi * kTile;  // elements of tiles >= thi belong to another segment
  float pc[kSlots];
  uint32_t dc[kSlots];
  load_tile<VEC>(prow, a.deg, n, tile_at(0) < thi ? tile_at(0) : (n + kTile) / kTile + 1, pc, dc);
  for (int64_t i = 0; i < P; ++i) {
    const int64_t t = tile_at(i);
    float pn[kSlots] = {};
    uint32_t dn[kSlots] = {};
    if (i + 1 < P) {
      const int64_t tn = tile_at(i + 1);
      if (tn < thi) load_tile<VEC>(prow, a.deg, n, tn, pn, dn);  // in flight while tile t is filtered
    }
    const unsigned long long thr = *st.thr;
    // Kc = K (1 - 2^-20), rounded; used only while it is a normal number, so
    // that Kc * d (d >= 1) is normal too (the products stay finite: checked)
    const float Kc = __fmul_rn(thr_key(thr), 0x1.ffffe0p-1f);
    const bool filt = Kc >= 1.17549435e-38f;  // FLT_MIN
    unsigned long long key[kSlots];
    unsigned mask = 0;  // slots of this thread that are admitted
#pragma unroll
    for (int e = 0; e < kSlots; ++e) {
      const int64_t v = slot_index<VEC>(t, e);
      key[e] = ~0ull;
      if (t >= thi || v >= hi_elem || !(pc[e] > 0.f)) continue;
      if (filt) {
        const float lim = __fmul_rn(Kc, __uint2float_rn(dc[e] > 0u ? dc[e] : 1u));
        if (lim <= 3.40282347e+38f && pc[e] < lim) continue;
      }
      const uint32_t enc = key_enc(pc[e], dc[e]);
      key[e] = sort_key(enc, (uint32_t)v);
      if (key[e] < thr) mask |= 1u << e;
    }
    admit_tile(st, T, key, mask);
#pragma unroll
    for (int e = 0; e < kSlots; ++e) {
      pc[e] = pn[e];
      dc[e] = dn[e];
    }
  }
  if (*st.n_buf > T) cut_back(st, T);
}

// Stream `count` keys (parts' survivors, ~0 = padding) through the same buffer;
// at most T are held afterwards.
__device__ void stream_keys(const unsigned long long *keys, int64_t count, const Stream &st, uint32_t T) {
  for (int64_t base = 0; base < count; base += kTile) {
    const unsigned long long thr = *st.thr;
    unsigned long long key[kSlots];
    unsigned mask = 0;
#pragma unroll
    for (int e = 0; e < kSlots; ++e) {
      const int64_t i = base + (int64_t)e * kThreads + threadIdx.x;
      key[e] = i < count ? __ldcg(keys + i) : ~0ull;
      if (key[e] < thr) mask |= 1u << e;
    }
    admit_tile(st, T, key, mask);
  }
  if (*st.n_buf > T) cut_back(st, T);
}

// ---- sample -----------------------------------------------------------------
constexpr int kBinsLog2 = 12, kBins = 1 << kBinsLog2, kBinShift = 19;  // bins of the key's FP32 bits
constexpr int kChunk = 128;                     // row elements of a chunk (a float4 a lane)
constexpr int kSampleEvery = 16;                // one chunk of so many, for rows of more than kSampleAll elements
constexpr int64_t kSampleAll = 1 << 16;
constexpr int kSampleChunks = 128;              // chunks a block samples

__device__ __forceinline__ uint32_t chunk_hash(uint32_t c) {
  c *= 0x9E3779B1u;
  return c ^ (c >> 15);
}

// Encoded keys of the elements of a row's sampled chunk c, four a lane.
template <bool VEC>
__device__ __forceinline__ void sample_chunk(const NcpArgs &a, const float *prow, int64_t c, int every,
                                             uint32_t (&enc)[4]) {
  const int lane = threadIdx.x & 31;
  const int64_t v0 = (c * every + (every > 1 ? chunk_hash((uint32_t)c) % (uint32_t)every : 0u)) * kChunk;
  float p[4] = {0.f, 0.f, 0.f, 0.f};
  uint32_t d[4] = {1u, 1u, 1u, 1u};
  if (VEC) {
    const int64_t v = v0 + 4 * lane;
    if (v < a.n) {
      const float4 p4 = __ldg(reinterpret_cast<const float4 *>(prow + v));
      const uint4 d4 = __ldg(reinterpret_cast<const uint4 *>(a.deg + v));
      p[0] = p4.x; p[1] = p4.y; p[2] = p4.z; p[3] = p4.w;
      d[0] = d4.x; d[1] = d4.y; d[2] = d4.z; d[3] = d4.w;
    }
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int64_t v = v0 + e * 32 + lane;
      if (v < a.n) {
        p[e] = __ldg(prow + v);
        d[e] = __ldg(a.deg + v);
      }
    }
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) enc[e] = key_enc(p[e], d[e]);
}

// Histogram of the keys of sampled chunks: block (row, part) takes chunks
// part * kSampleChunks and on, a warp at a time.
template <bool VEC>
__global__ void __launch_bounds__(kThreads) ncp_sample_kernel(NcpArgs a, int parts, int64_t chunks, int every) {
  __shared__ uint32_t h[kBins];
  const int warp = threadIdx.x >> 5;
  const int64_t row = blockIdx.x / parts, part = blockIdx.x % parts;
  const float *prow = a.p + row * a.n;
  for (int i = threadIdx.x; i < kBins; i += kThreads) h[i] = 0u;
  __syncthreads();
  for (int64_t c = part * kSampleChunks + warp; c < chunks && c < (part + 1) * kSampleChunks; c += kWarps) {
    uint32_t enc[4];
    sample_chunk<VEC>(a, prow, c, every, enc);
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (enc[e]) atomicAdd(&h[(enc[e] - 1u) >> kBinShift], 1u);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kBins; i += kThreads)
    if (h[i]) atomicAdd(a.hist + row * kBins + i, h[i]);
}

// The highest of kBins bins (count(bin) keys each, `base` more above all of them)
// with at least `want` keys in and above it; -1: none. Block-wide.
template <class Count>
__device__ int find_bin(uint32_t want, uint32_t base, uint32_t *w, int *s_bin, uint32_t *s_above, Count count) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kPer = kBins / kThreads;  // thread t: bins from the top, t * kPer and on
  uint32_t c[kPer], sum = 0;
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    c[i] = count(kBins - 1 - (tid * kPer + i));
    sum += c[i];
  }
  if (tid == 0) *s_bin = -1;
  const uint32_t incl = warp_prefix_incl(sum, lane);
  if (lane == 31) w[warp] = incl;
  __syncthreads();
  uint32_t above = base + incl - sum;
  for (int i = 0; i < warp; ++i) above += w[i];
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    if (above < want && above + c[i] >= want) {
      *s_bin = kBins - 1 - (tid * kPer + i);
      s_above[0] = above;         // above the bin
      s_above[1] = above + c[i];  // and with it
    }
    above += c[i];
  }
  __syncthreads();
  return *s_bin;
}

// Edge of each row: the highest bin edge with at least `want` sampled keys at
// or above it (encoded key; 1 = every key, when there are fewer). Where that
// would list more keys than there is room for, as in PPR rows, whose keys crowd
// in a few octaves, the row's sample is read again and the bin split by the next
// twelve bits (R-MAT 2^22, PPR rows of 419 seeds: 7.4 ms without, when most rows
// were streamed, 2.2 so). A row with too many keys even so (ties) is marked
// for the stream at once: the filter would read it for nothing.
template <bool VEC>
__global__ void __launch_bounds__(kThreads) ncp_edge_kernel(NcpArgs a, uint32_t want, int64_t chunks, int every,
                                                            ProfileBegin begin) {
  __shared__ uint32_t h[kBins], w[kWarps], s_above[2];
  __shared__ int s_bin;
  const int64_t row = blockIdx.x;
  if (begin != ProfileBegin::kNone && row == 0)
    for (int i = threadIdx.x; i < a.top; i += kThreads) profile_begin(a.ncp, i, begin == ProfileBegin::kAccumulate);
  const int bin = find_bin(want, 0u, w, &s_bin, s_above, [&](int b) { return __ldcg(a.hist + row * kBins + b); });
  if (bin < 0) {
    if (threadIdx.x == 0) a.edge[row] = 1u;
    return;
  }
  uint32_t edge = (uint32_t)bin << kBinShift;
  uint64_t keys = (uint64_t)s_above[1] * (uint64_t)every;
  if (keys > (uint64_t)kCap - kCap / 8) {
    const uint32_t above = s_above[0];
    for (int i = threadIdx.x; i < kBins; i += kThreads) h[i] = 0u;
    __syncthreads();
    const float *prow = a.p + row * a.n;
#pragma unroll 2
    for (int64_t c = threadIdx.x >> 5; c < chunks; c += kWarps) {
      uint32_t enc[4];
      sample_chunk<VEC>(a, prow, c, every, enc);
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (enc[e] && (int)((enc[e] - 1u) >> kBinShift) == bin)
          atomicAdd(&h[((enc[e] - 1u) >> (kBinShift - kBinsLog2)) & (uint32_t)(kBins - 1)], 1u);
    }
    __syncthreads();
    const int fine = find_bin(want, above, w, &s_bin, s_above, [&](int b) { return h[b]; });
    if (fine >= 0) {
      edge |= (uint32_t)fine << (kBinShift - kBinsLog2);
      keys = (uint64_t)s_above[1] * (uint64_t)every;
    }
  }
  if (threadIdx.x == 0) {
    a.edge[row] = edge + 1u;
    if (keys > (uint64_t)kCap + kCap / 4) a.listed[row] = (uint32_t)kCap + 1u;
  }
}

// ---- filter -----------------------------------------------------------------
constexpr int kFiltThreads = 256;
constexpr int kFiltVecs = 2;     // 16-byte loads of the row in flight a thread
constexpr int kFiltSteps = 8;    // such rounds a block
constexpr int kFiltElems = kFiltThreads * 4 * kFiltVecs * kFiltSteps;  // row elements of a block
constexpr int kFiltList = 3072;  // keys a block gathers; a row with more in one place is streamed instead

template <bool VEC>
__global__ void __launch_bounds__(kFiltThreads) ncp_filter_kernel(NcpArgs a, int segs) {
  __shared__ unsigned long long s_list[kFiltList];
  __shared__ uint32_t s_n, s_pos, s_base;
  __shared__ bool s_skip;
  const int64_t row = blockIdx.x / segs;
  const int64_t lo = (blockIdx.x % segs) * (int64_t)kFiltElems;
  const float *prow = a.p + row * a.n;
  if (threadIdx.x == 0) {
    s_n = 0u;
    s_pos = 0u;
    s_skip = __ldcg(a.listed + row) > (uint32_t)kCap;  // the row's list is not used any more
  }
  __syncthreads();
  if (s_skip) return;
  const uint32_t edge = a.edge[row];
  // A vertex is skipped without the IEEE division when p < (K (1 - 2^-20)) * d
  // in FP32, K = the edge's key (three roundings of at most 2^-24 each: the
  // conversion of d and the two products, so p / d < K (1 - 2^-21) and the
  // rounded key is below K); only while the products are normal and finite.
  const float Kc = __fmul_rn(__uint_as_float(edge - 1u), 0x1.ffffe0p-1f);
  const bool filt = Kc >= 1.17549435e-38f;  // FLT_MIN
  uint32_t pos = 0;
  for (int st = 0; st < kFiltSteps; ++st) {
    const int64_t base = lo + (int64_t)st * kFiltThreads * 4 * kFiltVecs;
    if (base >= a.n || *(volatile uint32_t *)&s_n > (uint32_t)kFiltList) break;
    float p[4 * kFiltVecs];
    uint32_t d[4 * kFiltVecs];
    auto index = [&](int i) {
      return VEC ? base + ((int64_t)(i >> 2) * kFiltThreads + threadIdx.x) * 4 + (i & 3)
                 : base + (int64_t)i * kFiltThreads + threadIdx.x;
    };
    if (VEC) {
#pragma unroll
      for (int k = 0; k < kFiltVecs; ++k) {
        const int64_t v = index(4 * k);
        float4 p4 = make_float4(0.f, 0.f, 0.f, 0.f);
        uint4 d4 = make_uint4(1u, 1u, 1u, 1u);
        if (v < a.n) {  // n is a multiple of 4: the whole vector is in the row
          p4 = __ldcs(reinterpret_cast<const float4 *>(prow + v));
          d4 = __ldg(reinterpret_cast<const uint4 *>(a.deg + v));
        }
        p[4 * k] = p4.x; p[4 * k + 1] = p4.y; p[4 * k + 2] = p4.z; p[4 * k + 3] = p4.w;
        d[4 * k] = d4.x; d[4 * k + 1] = d4.y; d[4 * k + 2] = d4.z; d[4 * k + 3] = d4.w;
      }
    } else {
#pragma unroll
      for (int i = 0; i < 4 * kFiltVecs; ++i) {
        const int64_t v = index(i);
        p[i] = v < a.n ? __ldcs(prow + v) : 0.f;
        d[i] = v < a.n ? __ldg(a.deg + v) : 1u;
      }
    }
#pragma unroll
    for (int i = 0; i < 4 * kFiltVecs; ++i) {
      if (!(p[i] > 0.f)) continue;
      ++pos;
      if (filt) {
        const float lim = __fmul_rn(Kc, __uint2float_rn(d[i] > 0u ? d[i] : 1u));
        if (lim <= 3.40282347e+38f && p[i] < lim) continue;
      }
      const uint32_t enc = key_enc(p[i], d[i]);
      if (enc < edge) continue;
      const unsigned long long key = sort_key(enc, (uint32_t)index(i));
      const uint32_t at = atomicAdd(&s_n, 1u);
      if (at < (uint32_t)kFiltList) s_list[at] = key;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) pos += __shfl_xor_sync(0xFFFFFFFFu, pos, o);
  if ((threadIdx.x & 31) == 0 && pos) atomicAdd(&s_pos, pos);
  __syncthreads();
  if (s_n > (uint32_t)kFiltList) {
    if (threadIdx.x == 0) atomicAdd(a.listed + row, (uint32_t)kCap + 1u);
    return;
  }
  const uint32_t n = s_n;
  if (threadIdx.x == 0) {
    if (s_pos) atomicAdd(a.positive + row, s_pos);
    s_base = n ? atomicAdd(a.listed + row, n) : 0u;
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < n; i += kFiltThreads)
    if (s_base + i < (uint32_t)kCap) a.list[row * kCap + s_base + i] = s_list[i];
}

// ---- order ------------------------------------------------------------------
// Place of the i-th key of a sorted buffer: sixteen consecutive keys lie in
// sixteen different banks' places, and so do the same ones of sixteen groups.
__device__ __forceinline__ uint32_t sort_place(uint32_t i) { return i ^ ((i >> 4) & 15u); }

// `kN` halving steps of a bitonic merge of runs of k keys, distances j, j / 2, ...:
// a thread takes the 2^kN keys that meet in them, so that shared memory and the
// barrier are passed once.
template <int kN>
__device__ __forceinline__ void merge_steps(unsigned long long *cand, uint32_t L2, uint32_t k, uint32_t j) {
  constexpr int kM = 1 << kN;
  const uint32_t step = j >> (kN - 1);
  for (uint32_t t = threadIdx.x; t < (L2 >> kN); t += kThreads) {
    const uint32_t base = ((t & ~(step - 1u)) << kN) | (t & (step - 1u));
    const bool up = (base & k) == 0u;  // (k is above every distance: the same for all of them)
    unsigned long long x[kM];
#pragma unroll
    for (int m = 0; m < kM; ++m) x[m] = cand[sort_place(base + (uint32_t)m * step)];
#pragma unroll
    for (int h = kM / 2; h > 0; h >>= 1) {
#pragma unroll
      for (int m = 0; m < kM; ++m) {
        if (m & h) continue;
        const unsigned long long a = x[m], b = x[m | h];
        const bool swap = (a > b) == up;
        x[m] = swap ? b : a;
        x[m | h] = swap ? a : b;
      }
    }
#pragma unroll
    for (int m = 0; m < kM; ++m) cand[sort_place(base + (uint32_t)m * step)] = x[m];
  }
  __syncthreads();
}

// Sorts the keys in cand[0, L) ascending (padded to a power of two of at least
// 16, at most kCap; block-wide): the i-th is then at cand[sort_place(i)].
__device__ void sort_keys(unsigned long long *cand, uint32_t L) {
  uint32_t L2 = 16;
  while (L2 < L) L2 <<= 1;
  for (uint32_t i = L + threadIdx.x; i < L2; i += kThreads) cand[i] = ~0ull;
  __syncthreads();
  for (uint32_t k = 2; k <= L2; k <<= 1) {
    uint32_t j = k >> 1;
    for (; j >= 8; j >>= 4) merge_steps<4>(cand, L2, k, j);
    if (j == 4) merge_steps<3>(cand, L2, k, j);
    if (j == 2) merge_steps<2>(cand, L2, k, j);
    if (j == 1) merge_steps<1>(cand, L2, k, j);
  }
}

// The first L sorted keys of a row: put(k, id, degree) in sweep order, then
// sum(k, arcs before k) for k in [0, L] (a graph has fewer than 2^32 arcs).
// Overwrites the keys; block-wide.
template <class Put, class Sum>
__device__ __forceinline__ void write_order(const NcpArgs &a, int64_t row, unsigned long long *cand, uint32_t L,
                                            uint32_t *s_w32, Put put, Sum sum_at) {
  int32_t *orow = a.order ? a.order + row * a.top : nullptr;
  const uint32_t per = (L + kThreads - 1) / kThreads;
  const uint32_t k0 = min(L, threadIdx.x * per), k1 = min(L, k0 + per);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t sum = 0;
  for (uint32_t k = k0; k < k1; ++k) {
    const uint32_t v = (uint32_t)cand[sort_place(k)], u = a.intl ? (uint32_t)__ldg(a.intl + v) : v;
    const uint32_t arc = __ldg(a.rp + u), deg = __ldg(a.rp + u + 1) - arc;
    if (orow) orow[k] = (int32_t)v;
    put(k, u, arc, deg);
    sum += deg;
    cand[sort_place(k)] = deg;  // (its key has been read)
  }
  const uint32_t incl = warp_prefix_incl(sum, lane);
  if (lane == 31) s_w32[warp] = incl;
  __syncthreads();
  uint32_t before = incl - sum;
  for (int w = 0; w < warp; ++w) before += s_w32[w];
  for (uint32_t k = k0; k < k1; ++k) {
    sum_at(k, before);
    before += (uint32_t)cand[sort_place(k)];
  }
  if (threadIdx.x == kThreads - 1) sum_at(L, before);  // its share is the last one, empty or not
}

// A row whose list cannot be used is streamed, the first kStreamSlots rows of a
// launch in parts, by up to kStreamParts blocks each.
constexpr int kStreamParts = 16;
constexpr int64_t kStreamSlots = 128;

__device__ __forceinline__ bool list_usable(const NcpArgs &a, int64_t row) {
  return a.list != nullptr && a.listed[row] <= (uint32_t)kCap && a.listed[row] >= min((uint32_t)a.top, a.positive[row]);
}

struct RowStream {
  uint32_t h[256], w32[kWarps], sel[2], n, m;
  unsigned long long thr;
  __device__ Stream on(unsigned char *smem) {
    return Stream{reinterpret_cast<unsigned long long *>(smem), reinterpret_cast<unsigned long long *>(smem + kBytesA),
                  h, w32, &n, &m, &thr, sel};
  }
};

__device__ __forceinline__ void stream_part(const NcpArgs &a, int64_t row, bool vec, const Stream &st, int part,
                                            int parts) {
  const int64_t ntiles = (a.n + kTile - 1) / kTile, lo = ntiles * part / parts, hi = ntiles * (part + 1) / parts;
  if (vec) stream_row<true>(a, a.p + row * a.n, st, (uint32_t)a.top, lo, hi);
  else stream_row<false>(a, a.p + row * a.n, st, (uint32_t)a.top, lo, hi);
}

__global__ void __launch_bounds__(kThreads, 2) ncp_stream_kernel(NcpArgs a, bool vec, int parts) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ RowStream rs;
  const int64_t row = blockIdx.x / parts;
  const int part = (int)(blockIdx.x % parts);
  if (list_usable(a, row)) return;
  const Stream st = rs.on(smem);
  stream_begin(st);
  stream_part(a, row, vec, st, part, parts);
  const uint32_t held = min(*st.n_buf, (uint32_t)a.top);
  unsigned long long *out = a.part + ((size_t)row * parts + part) * (size_t)a.top;
  for (uint32_t i = threadIdx.x; i < (uint32_t)a.top; i += kThreads) __stcg(out + i, i < held ? st.buf[i] : ~0ull);
}

__global__ void __launch_bounds__(kThreads, 2) ncp_order_kernel(NcpArgs a, bool vec, int parts) {
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned long long *cand = reinterpret_cast<unsigned long long *>(smem);
  __shared__ RowStream rs;
  uint32_t *s_w32 = rs.w32;
  const int64_t row = blockIdx.x;
  const uint32_t T = (uint32_t)a.top;
  uint32_t L;
  if (list_usable(a, row)) {
    L = a.listed[row];
    for (uint32_t i = threadIdx.x; i < L; i += kThreads) cand[i] = __ldcg(a.list + row * kCap + i);
    __syncthreads();
  } else {
    const Stream st = rs.on(smem);
    stream_begin(st);
    if (parts > 1 && row < kStreamSlots)
      stream_keys(a.part + (size_t)row * parts * (size_t)a.top, (int64_t)parts * a.top, st, T);
    else
      stream_part(a, row, vec, st, 0, 1);
    L = min(*st.n_buf, T);
  }
  sort_keys(cand, L);
  L = min(L, T);
  if (threadIdx.x == 0) a.kept[row] = L;
  write_order(
      a, row, cand, L, s_w32,
      [&](uint32_t k, uint32_t u, uint32_t, uint32_t deg) {
        a.ids[row * a.top + k] = u;
        a.gain[row * a.top + k] = (int32_t)deg;
      },
      [&](uint32_t k, uint32_t before) { a.first[row * ((int64_t)a.top + 1) + k] = before; });
}

// ---- inside -------------------------------------------------------------------
// The arcs of a row's kept vertices are one run, cut into pieces of kInsideArcs
// so that a hub's arcs are spread over blocks: block (row, part) takes pieces
// part, part + parts, ..., and leaves at once where there are fewer. An arc's
// owner is found by halving in the sums of the degrees, once for a thread's
// four arcs. Few of the neighbours are in the set, so two bits of a bitmap (32
// a member) are asked before the hash, whose probes for an absent vertex run to
// the next empty slot and keep the warp; a neighbour ranked before its vertex
// takes two from the vertex's gain.
constexpr int kInsideThreads = 1024;
constexpr uint32_t kInsideArcs = 1u << 15;
constexpr int kInsideParts = 16;
constexpr int kBitsLog2 = 17;
// hash keys and ranks, bitmap, first arc of each member in the run and in the graph
constexpr size_t kInsideSmem =
    (size_t)kHash * 6 + ((size_t)1 << kBitsLog2) / 8 + 2 * (size_t)kMaxTop * 4;
static_assert(kMaxTop <= 1 << 16, "ranks of 16 bits");

__device__ __forceinline__ uint32_t bit_a(uint32_t x, int shift) { return x >> shift; }
__device__ __forceinline__ uint32_t bit_b(uint32_t u, int shift) { return (u * 0x85EBCA6Bu) >> shift; }

// The kept vertices of a row in shared memory; the hash has at least twice as
// many slots as members, the bitmap sixteen bits a slot.
struct Members {
  uint32_t *hkey, *bits, *first, *arc;
  uint16_t *hval;
  uint32_t L, hmask;
  int hshift, bshift;

  __device__ Members(unsigned char *smem, uint32_t count) {
    hkey = reinterpret_cast<uint32_t *>(smem);
    bits = hkey + kHash;
    first = bits + (1 << kBitsLog2) / 32;
    arc = first + kMaxTop;
    hval = reinterpret_cast<uint16_t *>(arc + kMaxTop);
    L = count;
    int log2 = 8;
    while ((1u << log2) < 2u * L) ++log2;
    hmask = (1u << log2) - 1u;
    hshift = 32 - log2;
    bshift = hshift - (kBitsLog2 - kHashLog2);
  }
  __device__ void clear(int threads) {
    for (uint32_t i = threadIdx.x; i <= hmask; i += threads) hkey[i] = kEmpty;
    for (uint32_t i = threadIdx.x; i < (1u << (32 - bshift)) / 32u; i += threads) bits[i] = 0u;
    for (uint32_t i = L + threadIdx.x; i < (uint32_t)kMaxTop; i += threads) first[i] = 0xFFFFFFFFu;  // beyond every arc
  }
  __device__ void insert(uint32_t i, uint32_t u) {
    const uint32_t x = u * 0x9E3779B1u;
    atomicOr(&bits[bit_a(x, bshift) >> 5], 1u << (bit_a(x, bshift) & 31));
    atomicOr(&bits[bit_b(u, bshift) >> 5], 1u << (bit_b(u, bshift) & 31));
    uint32_t s = x >> hshift;
    for (uint32_t probe = 0; probe <= hmask; ++probe, s = (s + 1) & hmask) {
      if (atomicCAS(&hkey[s], kEmpty, u) == kEmpty) {
        hval[s] = (uint16_t)i;
        break;
      }
    }
  }
  // Arcs [begin, end) of the members' run, by a block of kT threads: four
  // consecutive ones a lane. A hub's arcs fill warps, whose lanes then add
  // their counts first (32 atomics on one word take their turns).
  template <int kT>
  __device__ void count(const uint32_t *adj, uint32_t begin, uint32_t end, int32_t *gain) const {
    constexpr int kU = 4;
    const int lane = threadIdx.x & 31;
    // (64 bits: begin + kT * kU may lie past 2^32)
    for (uint64_t base = begin + (uint64_t)(threadIdx.x & ~31u) * kU; base < end; base += kT * kU) {
      const uint64_t t0 = base + (uint64_t)lane * kU;
      uint32_t lo = 0;  // last member whose arcs start at or before t0 (those without arcs share a start)
      const uint32_t tc = (uint32_t)min(t0, (uint64_t)end - 1u);
#pragma unroll
      for (uint32_t half = kMaxTop / 2; half; half >>= 1)
        if (first[lo + half] <= tc) lo += half;
      uint32_t w[kU], own[kU];
#pragma unroll
      for (int i = 0; i < kU; ++i) {
        const uint64_t t = t0 + (uint64_t)i;
        w[i] = kEmpty;
        if (t < end) {
          while (lo + 1u < L && first[lo + 1u] <= (uint32_t)t) ++lo;
          w[i] = __ldg(adj + arc[lo] + ((uint32_t)t - first[lo]));
        }
        own[i] = lo;
      }
      uint32_t of = own[0];
      int32_t inside = 0;
#pragma unroll
      for (int i = 0; i < kU; ++i) {
        if (own[i] != of) {
          if (inside) atomicAdd(gain + of, -2 * inside);
          of = own[i];
          inside = 0;
        }
        const uint32_t x = w[i] * 0x9E3779B1u, ba = bit_a(x, bshift), bb = bit_b(w[i], bshift);
        const bool may = ((bits[ba >> 5] >> (ba & 31)) & (bits[bb >> 5] >> (bb & 31)) & 1u) != 0u;
        if (!may || w[i] == kEmpty) continue;
        uint32_t s = x >> hshift;
        for (uint32_t probe = 0; probe <= hmask; ++probe, s = (s + 1) & hmask) {
          const uint32_t hk = hkey[s];
          if (hk == w[i] && hval[s] < own[i]) ++inside;
          if (hk == w[i] || hk == kEmpty) break;
        }
      }
      __syncwarp();
      if (__all_sync(0xFFFFFFFFu, of == __shfl_sync(0xFFFFFFFFu, of, 0))) {
        inside = __reduce_add_sync(0xFFFFFFFFu, inside);
        if (lane == 0 && inside) atomicAdd(gain + of, -2 * inside);
      } else if (inside) {
        atomicAdd(gain + of, -2 * inside);
      }
    }
  }
};

__global__ void __launch_bounds__(kInsideThreads, 2) ncp_inside_kernel(NcpArgs a, int parts) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int64_t row = blockIdx.x / parts;
  const uint32_t L = a.kept[row], *first = a.first + row * ((int64_t)a.top + 1), tot = first[L];
  uint64_t at = (uint64_t)(blockIdx.x % parts) * kInsideArcs;
  if (at >= tot) return;
  Members m(smem, L);
  m.clear(kInsideThreads);
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < L; i += kInsideThreads) {
    const uint32_t u = a.ids[row * a.top + i];
    m.first[i] = first[i];
    m.arc[i] = __ldg(a.rp + u);
    m.insert(i, u);
  }
  __syncthreads();
  for (; at < tot; at += (uint64_t)parts * kInsideArcs)
    m.count<kInsideThreads>(a.adj, (uint32_t)at, (uint32_t)min(at + kInsideArcs, (uint64_t)tot), a.gain + row * a.top);
}

// ---- scan ---------------------------------------------------------------------
// kmax vertices kept; degree(k), gain(k) = degree(k) - 2 * inside(k).
template <class Degree>
__device__ __forceinline__ void scan_row(const NcpArgs &a, int64_t row, uint32_t kmax, const int32_t *gain,
                                         Degree degree) {
  __shared__ unsigned long long s_w64[2][kWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t T = (uint32_t)a.top;
  int32_t *orow = a.order ? a.order + row * a.top : nullptr;
  double *prow_phi = a.phi ? a.phi + row * a.top : nullptr;
  const uint32_t per = (kmax + kThreads - 1) / kThreads;
  const uint32_t k0 = min(kmax, (uint32_t)tid * per), k1 = min(kmax, k0 + per);
  long long cut_t = 0, vol_t = 0;
  for (uint32_t k = k0; k < k1; ++k) {
    cut_t += gain[k];
    vol_t += degree(k);
  }
  const long long cut_i = warp_prefix_incl(cut_t, lane), vol_i = warp_prefix_incl(vol_t, lane);
  if (lane == 31) {
    s_w64[0][warp] = (unsigned long long)cut_i;
    s_w64[1][warp] = (unsigned long long)vol_i;
  }
  __syncthreads();
  long long cut = cut_i - cut_t, vol = vol_i - vol_t;
  for (int w = 0; w < warp; ++w) {
    cut += (long long)s_w64[0][w];
    vol += (long long)s_w64[1][w];
  }
  const long long vol_all = (long long)a.m;
  for (uint32_t k = k0; k < k1; ++k) {
    cut += gain[k];
    vol += degree(k);
    const long long rest = vol_all - vol;
    const long long den = vol < rest ? vol : rest;
    const double phi = den > 0 ? (double)cut / (double)den : 1.0;
    if (prow_phi) prow_phi[k] = phi;
    if (a.ncp) atomicMin(a.ncp + k, dbl_enc(phi));
  }
  for (uint32_t k = kmax + tid; k < T; k += kThreads) {
    if (orow) orow[k] = -1;
    if (prow_phi) prow_phi[k] = __longlong_as_double(0x7FF8000000000000ll);  // NaN: no such prefix
  }
  if (tid == 0 && a.count) a.count[row] = (int32_t)kmax;
}

__global__ void __launch_bounds__(kThreads) ncp_scan_kernel(NcpArgs a) {
  const int64_t row = blockIdx.x;
  const uint32_t *first = a.first + row * ((int64_t)a.top + 1);
  scan_row(a, row, a.kept[row], a.gain + row * a.top, [&](uint32_t k) { return first[k + 1] - first[k]; });
}

// ---- rows of few vertices -------------------------------------------------------
// Everything for a row in one block and its shared memory, for rows of at most
// kSmallRow vertices, half as many more for a `top` of 512 and below: what the kernels above take there is mostly their launches.
// 9,000 vertices, 1 row, top 300: 44 us here and 72 through them; at the line the
// two meet (105 rows, top 4,096: 263 us here with 16,000 vertices, 255 through
// them with 17,000; 1 row, top 300: 57 and 70 with 17,000, top 512: 78 and 77 with 25,000).
// It takes rows of any length and no scratch, so longer rows come here too when
// there is no memory for the other kernels' scratch.
constexpr int64_t kSmallRow = 1 << 14;
// Little work and a small `top` are launches mostly, too: there the stream kernel's
// blocks leave a row's keys by parts and this kernel merges them, two launches for the
// six that find and filter a list. Calls back to back, top 16 / 64 / 256: 4 rows of 2^15
// vertices 33 / 36 / 51 us, and 50 / 52 / 60 by lists; 8 rows of 2^17 43 / 47 / 61 and 56 / 59 /
// 63; 2^18 56 / 59 / 76 and 60 / 62 / 68; 1 row of 2^20 85 / 94 / 113 and 60 / 58 / 64; top
// 512, 2^16 vertices 74 and 68.
constexpr int64_t kFewRow = 1 << 18;
constexpr int32_t kFewTop = 256;
constexpr int64_t kFewRowTop = 1 << 25;  // vertices of a row * top
constexpr int64_t kFewElems = 1 << 21;   // of the call
static_assert(kFewElems / kSmallRow <= kStreamSlots, "the stream kernel has room for every row of such a call");
constexpr size_t kSmallSmem = kInsideSmem + (size_t)kMaxTop * 4;  // and the gains
static_assert(kSmem <= kSmallSmem, "the row is streamed in the same memory");

// parts > 1: the row's keys come from the stream kernel's blocks
__global__ void __launch_bounds__(kThreads) ncp_small_kernel(NcpArgs a, bool vec, int parts) {
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned long long *cand = reinterpret_cast<unsigned long long *>(smem);
  __shared__ RowStream rs;
  __shared__ uint32_t s_tot;
  const int64_t row = blockIdx.x;
  const Stream st = rs.on(smem);
  stream_begin(st);
  if (parts > 1)
    stream_keys(a.part + (size_t)row * parts * (size_t)a.top, (int64_t)parts * a.top, st, (uint32_t)a.top);
  else
    stream_part(a, row, vec, st, 0, 1);
  const uint32_t L = min(*st.n_buf, (uint32_t)a.top);
  sort_keys(cand, L);
  // the sorted keys take the first kMaxTop * 8 bytes, hash keys later; the
  // vertices themselves wait in registers
  Members m(smem, L);
  int32_t *gain = reinterpret_cast<int32_t *>(smem + kInsideSmem);
  constexpr int kPer = kMaxTop / kThreads;
  uint32_t id[kPer];
  const uint32_t per = (L + kThreads - 1) / kThreads, k0 = min(L, threadIdx.x * per);
  write_order(
      a, row, cand, L, rs.w32,
      [&](uint32_t k, uint32_t u, uint32_t arc, uint32_t deg) {
#pragma unroll
        for (int i = 0; i < kPer; ++i)
          if (k - k0 == (uint32_t)i) id[i] = u;
        m.arc[k] = arc;
        gain[k] = (int32_t)deg;
      },
      [&](uint32_t k, uint32_t before) {
        if (k < L) m.first[k] = before;
        else s_tot = before;
      });
  __syncthreads();
  m.clear(kThreads);
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kPer; ++i)
    if ((uint32_t)i < per && k0 + (uint32_t)i < L) m.insert(k0 + (uint32_t)i, id[i]);
  __syncthreads();
  const uint32_t tot = s_tot;
  m.count<kThreads>(a.adj, 0u, tot, gain);
  __syncthreads();
  scan_row(a, row, L, gain, [&](uint32_t k) { return (k + 1u < L ? m.first[k + 1u] : tot) - m.first[k]; });
}

__global__ void ncp_profile_begin(unsigned long long *ncp, int32_t top, int accumulate) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < top) profile_begin(ncp, i, accumulate != 0);
}

__global__ void ncp_profile_end(unsigned long long *ncp, int32_t top) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < top) ncp[i] = (unsigned long long)__double_as_longlong(dbl_dec(ncp[i]));
}

// out-degree per original id: deg[orig[u]] = rp[u + 1] - rp[u]
__global__ void degree_table(const uint32_t *rp, const int32_t *orig, int64_t n, uint32_t *deg) {
  for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = orig ? orig[u] : u;
    deg[v] = rp[u + 1] - rp[u];
  }
}

bool aligned(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

}  // namespace
}  // namespace fg

using namespace fg;

extern "C" fg_status fg_ncp_sweep(fg_graph *g, const float *p, int32_t nq, int32_t top, int32_t *order_out,
                                  double *phi_out, int32_t *count_out, double *ncp_out, int32_t accumulate,
                                  void *stream_v) {
  if (!g) return fail(FG_ERR_INVALID_ARG, "graph is NULL");
  if (!p) return fail(FG_ERR_INVALID_ARG, "p is NULL");
  if (nq <= 0) return fail(FG_ERR_INVALID_ARG, "nq must be > 0 (got %d)", nq);
  if (top < 1 || top > FG_NCP_MAX_TOP)
    return fail(FG_ERR_INVALID_ARG, "top must be in [1, %d] (got %d)", FG_NCP_MAX_TOP, top);
  if (!order_out && !phi_out && !count_out && !ncp_out) return fail(FG_ERR_INVALID_ARG, "no output given");
  if (!aligned(p, 4) || !aligned(order_out, 4) || !aligned(count_out, 4) || !aligned(phi_out, 8) ||
      !aligned(ncp_out, 8))
    return fail(FG_ERR_INVALID_ARG, "misaligned pointer");
  int dev = -1;
  CUDA_TRY(cudaGetDevice(&dev));
  if (dev != g->device)
    return fail(FG_ERR_INVALID_ARG, "the graph lives on device %d but device %d is current", g->device, dev);
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_v);
  const int64_t n = g->n;

  {
    // degree table in original order, built once per graph (the only
    // synchronising step; later calls only read it)
    std::lock_guard<std::mutex> lk(g->mu);
    if (!g->deg.p) {
      static std::once_flag attr_once;
      static cudaError_t attr_err = cudaSuccess;
      std::call_once(attr_once, [] {
        attr_err = cudaFuncSetAttribute(ncp_order_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
        if (attr_err == cudaSuccess)
          attr_err = cudaFuncSetAttribute(ncp_stream_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
        if (attr_err == cudaSuccess)
          attr_err = cudaFuncSetAttribute(ncp_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)kSmallSmem);
        if (attr_err == cudaSuccess)
          attr_err = cudaFuncSetAttribute(ncp_inside_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)kInsideSmem);
      });
      CUDA_TRY(attr_err);
      DevBuf d;
      CUDA_TRY(d.reserve(sizeof(uint32_t) * (size_t)n));
      const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 16));
      degree_table<<<blocks, 256, 0, stream>>>(g->dg.rp, g->dg.orig, n, d.as<uint32_t>());
      cudaError_t e = cudaGetLastError();
      if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
      if (e != cudaSuccess) {
        d.release();
        return fail(FG_ERR_CUDA, "degree table: %s", cudaGetErrorString(e));
      }
      g->deg = d;
    }
  }

  NcpArgs a;
  a.p = p;
  a.deg = g->deg.as<uint32_t>();
  a.rp = g->dg.rp;
  a.adj = g->dg.adj;
  a.intl = g->dg.intl;
  a.n = n;
  a.m = g->dg.m;
  a.top = top;
  a.order = order_out;
  a.phi = phi_out;
  a.count = count_out;
  a.ncp = reinterpret_cast<unsigned long long *>(ncp_out);
  bool small = n <= kSmallRow || (n <= kSmallRow + kSmallRow / 2 && top <= 512);
  const bool vec = (n % 4 == 0) && aligned(p, 16);
  // Rows go through in launches of at most kRowsPerLaunch, which bounds the
  // scratch (about 80 KB + 12 * top bytes a row, from the stream-ordered
  // allocator).
  constexpr int64_t kRowsPerLaunch = 1024;
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  int64_t rows_max = std::min<int64_t>(nq, kRowsPerLaunch);
  bool few = !small && n <= kFewRow && top <= kFewTop && n * top <= kFewRowTop && n * nq <= kFewElems;
  size_t b_hist = 0, b_small = 0, b_list = 0, b_top = 0, b_part = 0;
  int stream_parts = 0;
  unsigned char *scratch = nullptr;
  for (; !small; rows_max = (rows_max + 1) / 2) {  // fewer rows a launch where memory is short
    b_hist = up((size_t)rows_max * kBins * 4);  // (few: only the parts)
    b_small = up((size_t)rows_max * 4);
    b_list = up((size_t)rows_max * kCap * 8);
    b_top = up((size_t)rows_max * ((size_t)top + 1) * 4);
    // two blocks an SM; one part (in the order kernel) for rows that one block streams in 50 us
    stream_parts = n <= kSampleAll && !few ? 1 : (int)std::max<int64_t>(1, std::min<int64_t>(kStreamParts, 304 / rows_max));
    b_part = stream_parts == 1 ? 0 : up((size_t)std::min(rows_max, kStreamSlots) * (size_t)stream_parts * (size_t)top * 8);
    if (few) b_hist = b_small = b_list = b_top = 0;
    const cudaError_t e0 = cudaMallocAsync(reinterpret_cast<void **>(&scratch),
                                           b_hist + 4 * b_small + b_list + 3 * b_top + b_part, stream);
    if (e0 == cudaSuccess) break;
    if (e0 != cudaErrorMemoryAllocation) CUDA_TRY(e0);
    (void)cudaGetLastError();
    scratch = nullptr;
    if (rows_max == 1) {  // none at all: one block a row, which streams a row of any length
      small = true;
      few = false;
      rows_max = std::min<int64_t>(nq, kRowsPerLaunch);
      break;
    }
  }
  if (a.ncp && (small || few)) {  // (else by the edge kernel)
    ncp_profile_begin<<<(top + 255) / 256, 256, 0, stream>>>(a.ncp, top, accumulate ? 1 : 0);
    CUDA_TRY(cudaGetLastError());
  }
  unsigned char *at = scratch;
  auto take = [&at](size_t b) {
    unsigned char *r = at;
    at += b;
    return r;
  };
  // (listed, positive and hist start at zero: one memset)
  a.listed = reinterpret_cast<uint32_t *>(take(b_small));
  a.positive = reinterpret_cast<uint32_t *>(take(b_small));
  a.hist = reinterpret_cast<uint32_t *>(take(b_hist));
  a.edge = reinterpret_cast<uint32_t *>(take(b_small));
  a.kept = reinterpret_cast<uint32_t *>(take(b_small));
  a.list = few ? nullptr : reinterpret_cast<unsigned long long *>(take(b_list));
  a.ids = reinterpret_cast<uint32_t *>(take(b_top));
  a.gain = reinterpret_cast<int32_t *>(take(b_top));
  a.first = reinterpret_cast<uint32_t *>(take(b_top));
  a.part = reinterpret_cast<unsigned long long *>(take(b_part));
  const int every = n > kSampleAll ? kSampleEvery : 1;
  const int64_t chunks = (n / every + kChunk - 1) / kChunk;  // (a sampled row's last chunks may lie past its end)
  const int sparts = (int)((chunks + kSampleChunks - 1) / kSampleChunks);
  // keys wanted above the edge among the sampled ones: with one in sixteen, the
  // share of `top` and six standard deviations of it, and a tenth of room
  const double share = (double)top / every;
  const uint32_t want = every == 1 ? (uint32_t)top : (uint32_t)(1.1 * share + 6.0 * std::sqrt(share) + 8.0);
  const int segs = (int)((n + kFiltElems - 1) / kFiltElems);
  cudaError_t e = cudaSuccess;
  for (int64_t r0 = 0; r0 < nq && e == cudaSuccess; r0 += rows_max) {
    const unsigned rows = (unsigned)std::min<int64_t>(rows_max, nq - r0);
    NcpArgs b = a;
    b.p = a.p + r0 * n;
    if (a.order) b.order = a.order + r0 * top;
    if (a.phi) b.phi = a.phi + r0 * top;
    if (a.count) b.count = a.count + r0;
    if (small || few) {
      if (few && stream_parts > 1)
        ncp_stream_kernel<<<rows * stream_parts, kThreads, kSmem, stream>>>(b, vec, stream_parts);
      ncp_small_kernel<<<rows, kThreads, kSmallSmem, stream>>>(b, vec, few ? stream_parts : 1);
      e = cudaGetLastError();
      continue;
    }
    e = cudaMemsetAsync(scratch, 0, 2 * b_small + b_hist, stream);
    if (vec) ncp_sample_kernel<true><<<rows * sparts, kThreads, 0, stream>>>(b, sparts, chunks, every);
    else ncp_sample_kernel<false><<<rows * sparts, kThreads, 0, stream>>>(b, sparts, chunks, every);
    const ProfileBegin begin = !a.ncp || r0 > 0 ? ProfileBegin::kNone
                               : accumulate     ? ProfileBegin::kAccumulate
                                                : ProfileBegin::kFresh;
    if (vec) ncp_edge_kernel<true><<<rows, kThreads, 0, stream>>>(b, want, chunks, every, begin);
    else ncp_edge_kernel<false><<<rows, kThreads, 0, stream>>>(b, want, chunks, every, begin);
    if (vec) ncp_filter_kernel<true><<<rows * segs, kFiltThreads, 0, stream>>>(b, segs);
    else ncp_filter_kernel<false><<<rows * segs, kFiltThreads, 0, stream>>>(b, segs);
    const unsigned streamed = (unsigned)std::min<int64_t>(rows, kStreamSlots);
    if (stream_parts > 1)
      ncp_stream_kernel<<<streamed * stream_parts, kThreads, kSmem, stream>>>(b, vec, stream_parts);
    ncp_order_kernel<<<rows, kThreads, kSmem, stream>>>(b, vec, stream_parts);
    ncp_inside_kernel<<<rows * kInsideParts, kInsideThreads, kInsideSmem, stream>>>(b, kInsideParts);
    ncp_scan_kernel<<<rows, kThreads, 0, stream>>>(b);
    if (e == cudaSuccess) e = cudaGetLastError();
  }
  if (scratch) cudaFreeAsync(scratch, stream);
  CUDA_TRY(e);
  if (a.ncp) {
    ncp_profile_end<<<(top + 255) / 256, 256, 0, stream>>>(a.ncp, top);
    CUDA_TRY(cudaGetLastError());
  }
  return FG_OK;
}
