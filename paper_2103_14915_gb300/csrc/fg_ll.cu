// Landmark labeling (LL) on top of a batch of SSSP / BFS queries (Sec. 1;
// Sec. 6.1 runs 1,024 SSSPs from randomly chosen landmark vertices). The
// batch's rows d(s_k, .) become per-vertex labels, and a pair (u, v) is
// answered from the two labels alone:
//     est(u, v) = min over k with d(s_k, u), d(s_k, v) finite of d(s_k, u) + d(s_k, v),
// an upper bound on d(u, v) on an undirected graph, exact when a landmark lies
// on a shortest u-v path.
//
// Both kernels move bytes and do almost no arithmetic, so HBM bandwidth bounds
// them:
//   label construction  [K][n] -> [n][K] transpose through 64 x 64 shared-memory
//                       tiles (each warp reads and writes 256 contiguous bytes
//                       per row; the padded tile keeps both phases free of bank
//                       conflicts), persistent blocks that load the next tile
//                       while writing the current one; 8 * K * n bytes;
//   query               few pairs: one warp per pair reads the two K-entry
//                       labels with 16-byte loads (K a multiple of 4) and
//                       reduces the minimum with shuffles; 8 * K + 16 bytes per
//                       pair. Many: the labels are taken in slices of columns,
//                       so that pairs meet in L2.
#include <algorithm>
#include <cstdint>

#include "fg_host.h"

namespace fg {
namespace {

constexpr int kT = 64;          // transpose tile
constexpr int kTRows = 8;       // thread rows per tile (block 32 x 8)
constexpr int kQThreads = 256;  // query block: 8 warps, one pair per warp at a time

// Persistent over tiles: block b takes tiles b, b + gridDim.x, ... (vertex
// tiles fastest, so neighbouring blocks read neighbouring row segments). Each
// thread holds its 16 elements of the next tile in registers, loaded while
// the current tile is written out of shared memory.
__global__ void __launch_bounds__(32 * kTRows) ll_transpose(const uint32_t *__restrict__ dist, int32_t K, int64_t n,
                                                            uint32_t *__restrict__ labels, int64_t ntv, int64_t ntiles) {
  __shared__ uint32_t tile[kT][kT + 1];
  const int tx = threadIdx.x, ty = threadIdx.y;
  constexpr int kPer = (kT / kTRows) * (kT / 32);  // elements per thread per tile
  uint32_t buf[kPer];
  auto load = [&](int64_t t) {
    const int64_t v0 = (t % ntv) * kT;
    const int64_t k0 = (t / ntv) * kT;
#pragma unroll
    for (int r = 0; r < kT / kTRows; ++r) {
      const int64_t k = k0 + ty + r * kTRows;
#pragma unroll
      for (int c = 0; c < kT / 32; ++c) {
        const int64_t v = v0 + tx + c * 32;
        buf[r * (kT / 32) + c] = (k < K && v < n) ? __ldcs(dist + (size_t)k * (size_t)n + (size_t)v) : 0u;
      }
    }
  };
  int64_t t = blockIdx.x;
  if (t < ntiles) load(t);
  for (; t < ntiles; t += gridDim.x) {
    __syncthreads();  // the previous tile has been written out of shared memory
#pragma unroll
    for (int r = 0; r < kT / kTRows; ++r)
#pragma unroll
      for (int c = 0; c < kT / 32; ++c) tile[ty + r * kTRows][tx + c * 32] = buf[r * (kT / 32) + c];
    __syncthreads();
    const int64_t v0 = (t % ntv) * kT;
    const int64_t k0 = (t / ntv) * kT;
    if (t + gridDim.x < ntiles) load(t + gridDim.x);  // in flight during the write-out below
#pragma unroll
    for (int r = 0; r < kT / kTRows; ++r) {
      const int64_t v = v0 + ty + r * kTRows;
#pragma unroll
      for (int c = 0; c < kT / 32; ++c) {
        const int64_t k = k0 + tx + c * 32;
        if (k < K && v < n) __stcs(labels + (size_t)v * (size_t)K + (size_t)k, tile[tx + c * 32][ty + r * kTRows]);
      }
    }
  }
}

__device__ __forceinline__ void take(uint32_t a, uint32_t b, unsigned long long &best) {
  if (a != 0xFFFFFFFFu && b != 0xFFFFFFFFu) {
    const unsigned long long d = (unsigned long long)a + (unsigned long long)b;
    best = d < best ? d : best;
  }
}

template <bool VEC>
__global__ void __launch_bounds__(kQThreads) ll_query_kernel(const uint32_t *__restrict__ labels, int64_t n, int32_t K,
                                                             const int32_t *__restrict__ pairs, int64_t Q,
                                                             unsigned long long *__restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (kQThreads / 32);
  for (int64_t i = ((int64_t)blockIdx.x * kQThreads + threadIdx.x) >> 5; i < Q; i += warps) {
    const int32_t u = __ldg(pairs + 2 * i), v = __ldg(pairs + 2 * i + 1);
    unsigned long long best = ~0ull;
    if (u >= 0 && (int64_t)u < n && v >= 0 && (int64_t)v < n) {
      const uint32_t *lu = labels + (size_t)u * (size_t)K, *lv = labels + (size_t)v * (size_t)K;
      if (VEC) {
        const uint4 *au = reinterpret_cast<const uint4 *>(lu), *av = reinterpret_cast<const uint4 *>(lv);
        for (int32_t j = lane; j < K / 4; j += 32) {
          const uint4 a = __ldg(au + j), b = __ldg(av + j);
          take(a.x, b.x, best);
          take(a.y, b.y, best);
          take(a.z, b.z, best);
          take(a.w, b.w, best);
        }
      } else {
        for (int32_t k = lane; k < K; k += 32) take(__ldg(lu + k), __ldg(lv + k), best);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long y = __shfl_xor_sync(0xFFFFFFFFu, best, o);
      best = y < best ? y : best;
    }
    if (lane == 0) out[i] = best;
  }
}

// Many pairs: a warp keeps up to kMine of them with their minima in shared memory
// and takes the labels in slices of kLanes * kC columns, kLanes lanes a pair, kC
// columns a lane, 32 words of a lane in flight. All blocks are resident and have
// the same number of pairs, so they stay on the same few slices, of which L2 holds
// about half: of the first line's 8.6 GB of labels 4.4 come from HBM, at 78 % of its
// peak, and a pair with few columns does not take a whole warp. Sums are taken in 32 bits while one of a pair's
// stays below 2^32 - 1 (it is then the least of all).
//   n = 2^18, K = 1,024, Q = 2^20  1.15 ms (7.4 TB/s) -> 0.75  (12 TB/s; each label once: 1.07 GB)
//   n = 2^15 (labels in L2)        0.67 -> 0.45
//   n = 2^18, K = 1,023            1.61 -> 1.12  (no 16-byte loads)
//   n = 2^18, K = 64 / 16          170 us -> 35 / 158 -> 17
// Slices of 128 columns (64 where K ends there): with 64 and 256 the first line is
// 0.81 and 0.92. Of more than 2^19 vertices L2 holds little of such a slice, and 64
// columns are the better ones: 2^20 vertices and K = 256 take 0.25 ms, not 0.28 (a
// warp per pair: 0.32); but not where 16-byte loads are out (K = 255: 0.40 and 0.36;
// 0.47). Below kSliceMinPairs a warp per pair is the faster one: Q = 4,000 of the first
// line 6.3 us and 25; 10,000 pairs of 9 columns 4.7 and 6.5; 32,768 pairs of 64 columns
// 19 and 16. Where L2 holds all labels (kL2Labels) slices win nothing by what they
// find there, and a warp streams a wide row without a vote and a shuffle tree every
// 128 columns: such rows of 16-byte loads, 2^12 vertices, take a warp per pair up to
// kSliceWidePairs pairs (512 columns: 2^15 pairs 24 us, 26 in slices; 2^16 35 and 36;
// 2^17 54 and 52), and beyond 2 * kWideRow columns for any number (1,024 columns: 2^16
// pairs 47 and 56, 2^20 522 and 562; 4,096 columns 134 and 174 for 2^16; without 16-byte
// loads, 767 columns, 2^20 552 and 474). The sizes do not tell of pairs that keep to a few vertices of a large
// graph: they are in L2 either way, and cost up to a third more in slices (64 of
// 2^18 vertices, 1,024 columns: 2^15 pairs 31 and 37 us, 2^20 518 and 537).
constexpr int kMine = 256;
constexpr int64_t kSliceMinPairs = 1 << 15;
constexpr int64_t kSliceBlocks = 152 * 4;
constexpr int32_t kWideRow = 256;
constexpr int64_t kSliceWidePairs = 1 << 16;
constexpr int64_t kL2Labels = 100ll << 20;  // (64 MB of labels are read at L2's rate, 134 MB are not)
constexpr int64_t kWideVertices = 1 << 19;  // 268 MB a slice of 128 columns

template <bool VEC, int kLanes, int kC>
__global__ void __launch_bounds__(kQThreads, 4) ll_slice_kernel(const uint32_t *__restrict__ labels, int64_t n, int32_t K,
                                                             const int32_t *__restrict__ pairs, int64_t Q, int per,
                                                             unsigned long long *__restrict__ out) {
  constexpr int kG = 32 / kLanes;             // pairs of a warp at a time
  constexpr int kU = kC >= 16 ? 1 : 16 / kC;  // such steps in flight
  constexpr uint32_t kInf = 0xFFFFFFFFu;
  __shared__ int2 s_pair[kQThreads / 32][kMine];
  __shared__ unsigned long long s_best[kQThreads / 32][kMine];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = lane % kLanes, grp = lane / kLanes;
  int2 *pr = s_pair[warp];
  unsigned long long *bs = s_best[warp];
  const int64_t w = (int64_t)blockIdx.x * (kQThreads / 32) + warp, warps = (int64_t)gridDim.x * (kQThreads / 32);
  auto load = [&](const uint32_t *row, int32_t k0, uint32_t (&x)[kC]) {
    if (VEC) {
#pragma unroll
      for (int c = 0; c < kC; c += 4) {
        const int32_t k = k0 + c * kLanes + 4 * sub;
        if (k >= K) break;
        const uint4 a = __ldg(reinterpret_cast<const uint4 *>(row + k));
        x[c] = a.x; x[c + 1] = a.y; x[c + 2] = a.z; x[c + 3] = a.w;
      }
    } else {
#pragma unroll
      for (int c = 0; c < kC; ++c) {
        const int32_t k = k0 + c * kLanes + sub;
        if (k < K) x[c] = __ldg(row + k);
      }
    }
  };
  for (int64_t i0 = w * per; i0 < Q; i0 += warps * per) {
    const int count = (int)min((int64_t)per, Q - i0);
    for (int i = lane; i < count; i += 32) {
      const int32_t u = __ldg(pairs + 2 * (i0 + i)), v = __ldg(pairs + 2 * (i0 + i) + 1);
      const bool ok = u >= 0 && (int64_t)u < n && v >= 0 && (int64_t)v < n;
      pr[i] = ok ? make_int2(u, v) : make_int2(-1, -1);
      bs[i] = ~0ull;
    }
    __syncwarp();
    for (int32_t k0 = 0; k0 < K; k0 += kLanes * kC) {
      for (int b = 0; b < count; b += kG * kU) {
        uint32_t x[kU][kC], y[kU][kC];
#pragma unroll
        for (int h = 0; h < kU; ++h) {
          const int i = b + h * kG + grp;
          const int2 p = i < count ? pr[i] : make_int2(-1, -1);
#pragma unroll
          for (int c = 0; c < kC; ++c) x[h][c] = y[h][c] = kInf;
          if (p.x >= 0) {
            load(labels + (size_t)p.x * (size_t)K, k0, x[h]);
            load(labels + (size_t)p.y * (size_t)K, k0, y[h]);
          }
        }
#pragma unroll
        for (int h = 0; h < kU; ++h) {
          const int i = b + h * kG + grp;
          uint32_t low = kInf;
#pragma unroll
          for (int c = 0; c < kC; ++c) {
            const uint32_t s = x[h][c] + y[h][c];
            low = min(low, s < x[h][c] ? kInf : s);
          }
#pragma unroll
          for (int o = kLanes / 2; o > 0; o >>= 1) low = min(low, __shfl_xor_sync(0xFFFFFFFFu, low, o));
          // No sum below 2^32 - 1: mostly a pair that no landmark of the slice
          // reaches (or no pair at all), with nothing to take. Only if a column
          // has two finite distances is their sum one of more than 32 bits.
          unsigned long long best = low == kInf ? ~0ull : low;
          if (__any_sync(0xFFFFFFFFu, low == kInf)) {
            uint32_t both = kInf;
#pragma unroll
            for (int c = 0; c < kC; ++c) both = min(both, max(x[h][c], y[h][c]));
            if (__any_sync(0xFFFFFFFFu, low == kInf && both != kInf)) {
              best = ~0ull;
#pragma unroll
              for (int c = 0; c < kC; ++c) take(x[h][c], y[h][c], best);
#pragma unroll
              for (int o = kLanes / 2; o > 0; o >>= 1) {
                const unsigned long long z = __shfl_xor_sync(0xFFFFFFFFu, best, o);
                best = z < best ? z : best;
              }
            }
          }
          if (sub == 0 && i < count && best < bs[i]) bs[i] = best;
        }
      }
    }
    __syncwarp();
    for (int i = lane; i < count; i += 32) out[i0 + i] = bs[i];
    __syncwarp();
  }
}

bool aligned(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

}  // namespace
}  // namespace fg

using namespace fg;

extern "C" fg_status fg_ll_build_labels(const uint32_t *dist, int32_t K, int64_t n, uint32_t *labels,
                                        void *stream_v) {
  if (!dist || !labels) return fail(FG_ERR_INVALID_ARG, "dist or labels is NULL");
  if (K < 1 || n < 1) return fail(FG_ERR_INVALID_ARG, "K and n must be >= 1 (got %d, %lld)", K, (long long)n);
  if (!aligned(dist, 4) || !aligned(labels, 4)) return fail(FG_ERR_INVALID_ARG, "misaligned pointer");
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_v);
  int dev = 0, sms = 0;
  CUDA_TRY(cudaGetDevice(&dev));
  CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int64_t ntv = (n + kT - 1) / kT, ntk = ((int64_t)K + kT - 1) / kT, ntiles = ntv * ntk;
  int per_sm = 0;
  CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ll_transpose, 32 * kTRows, 0));
  const int64_t blocks = std::min<int64_t>(ntiles, (int64_t)sms * std::max(per_sm, 1));  // all resident
  ll_transpose<<<(unsigned)blocks, dim3(32, kTRows), 0, stream>>>(dist, K, n, labels, ntv, ntiles);
  CUDA_TRY(cudaGetLastError());
  return FG_OK;
}

extern "C" fg_status fg_ll_query(const uint32_t *labels, int64_t n, int32_t K, const int32_t *pairs, int64_t Q,
                                 uint64_t *est_out, void *stream_v) {
  if (!labels || (Q > 0 && (!pairs || !est_out))) return fail(FG_ERR_INVALID_ARG, "NULL argument");
  if (K < 1 || n < 1 || Q < 0)
    return fail(FG_ERR_INVALID_ARG, "K, n must be >= 1 and Q >= 0 (got %d, %lld, %lld)", K, (long long)n,
                (long long)Q);
  if (!aligned(labels, 4) || !aligned(pairs, 4) || !aligned(est_out, 8))
    return fail(FG_ERR_INVALID_ARG, "misaligned pointer");
  if (Q == 0) return FG_OK;
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_v);
  const int64_t blocks = std::min<int64_t>((Q + kQThreads / 32 - 1) / (kQThreads / 32), 152ll * 64);
  unsigned long long *out = reinterpret_cast<unsigned long long *>(est_out);
  const bool vec = K % 4 == 0 && aligned(labels, 16);
  const bool wide_in_l2 = vec && K > kWideRow && n * (int64_t)K * 4 <= kL2Labels;
  const bool sliced = Q >= kSliceMinPairs && !(wide_in_l2 && (K > 2 * kWideRow || Q < kSliceWidePairs));
  if (sliced) {
    auto launch = [&](auto kernel) {
      const int64_t most = kSliceBlocks * (kQThreads / 32);  // warps
      const int64_t rounds = (Q + most * kMine - 1) / (most * kMine);
      const int per = (int)((Q + most * rounds - 1) / (most * rounds));
      kernel<<<(unsigned)kSliceBlocks, kQThreads, 0, stream>>>(labels, n, K, pairs, Q, per, out);
    };
    if (K <= 16) vec ? launch(ll_slice_kernel<true, 4, 4>) : launch(ll_slice_kernel<false, 4, 4>);
    else if (K <= 32) vec ? launch(ll_slice_kernel<true, 8, 4>) : launch(ll_slice_kernel<false, 8, 4>);
    else if (K <= 64 || (vec && n > kWideVertices)) vec ? launch(ll_slice_kernel<true, 8, 8>) : launch(ll_slice_kernel<false, 8, 8>);
    else vec ? launch(ll_slice_kernel<true, 16, 8>) : launch(ll_slice_kernel<false, 16, 8>);
  } else if (vec) {
    ll_query_kernel<true><<<(unsigned)blocks, kQThreads, 0, stream>>>(labels, n, K, pairs, Q, out);
  } else {
    ll_query_kernel<false><<<(unsigned)blocks, kQThreads, 0, stream>>>(labels, n, K, pairs, Q, out);
  }
  CUDA_TRY(cudaGetLastError());
  return FG_OK;
}
