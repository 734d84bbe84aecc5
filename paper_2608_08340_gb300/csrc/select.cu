// Floors of a search with buffered lists (k > 32) from its group pass: per
// query, the k-th largest of the maxima of disjoint groups of scores.  Each of
// the k groups holds a score that reaches it, so it bounds the query's k-th
// best score from below (partial selection, Sec. 4.4); with k well below the
// number of groups it lies close to that score, because the k best scores
// mostly fall into different groups.
#include "common.cuh"
#include "internal.h"

namespace oprag {

namespace {

constexpr int kSelThreads = 128;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kSelTop = 512;           // values ranked for the counted floors

// One CTA per query, up to kSelThreads * R group maxima in registers as
// order-preserving integers.  The k-th largest is found by a bisection between
// the smallest and the largest (a block-wide count a round); it stops at the
// first value that exactly k maxima reach, which is itself a valid floor
// between the k-th and the (k + 1)-th.  Bounded by its rounds, a barrier each,
// and with thousands of queries by their instructions.  The counted floors'
// ranks come from the values that reach the floor, ranked by counting.
// Measured on GB300, group pass and selection together, against a search bit by
// bit from the top: 300 queries of 50021 x 392, k = 100 39 (44) us, of 300000 x
// 128, k = 256 53 (61) us; 2048 queries of 300000 x 128, k = 100 49 (50) us.
template <int R>
__global__ void __launch_bounds__(kSelThreads)
group_select_kernel(const float* __restrict__ gmax, int64_t gld, int groups, int k,
                    float* __restrict__ kth, float* __restrict__ levels,
                    int* __restrict__ level_cnt) {
  __shared__ uint32_t ends[2][kSelWarps];
  __shared__ int part[2][kSelWarps];
  __shared__ __align__(16) uint32_t top[kSelTop];
  __shared__ int ntop;
  // Launched as a programmatic dependent of the group pass; the main pass may
  // start once every CTA of this grid has.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int qi = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const float* g = gmax + static_cast<int64_t>(qi) * gld;
  uint32_t v[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = r * kSelThreads + tid;
    // (NaN, the maximum of a group of NaN scores, holds no score)
    v[r] = i < groups ? score_order(fmaxf(__ldcs(g + i), -INFINITY)) : 0u;
  }
  const uint32_t none = score_order(-INFINITY);     // a group past the corpus's end
  uint32_t reached = none;
  if (k <= groups) {
    uint32_t lo = 0xffffffffu, hi = 0;
    int held = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (v[r] > none) {
        lo = min(lo, v[r]);
        ++held;
      }
      hi = max(hi, v[r]);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    held = __reduce_add_sync(0xffffffffu, held);
    if (lane == 0) {
      part[1][warp] = held;
      ends[0][warp] = lo;
      ends[1][warp] = hi;
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kSelWarps; ++w) {
      if (w != warp) held += part[1][w];
      lo = min(lo, ends[0][w]);
      hi = max(hi, ends[1][w]);
    }
    // With at least k values: at least k reach lo, fewer than k are above hi.
#pragma unroll 1
    for (int round = 0; held >= k && lo < hi; round ^= 1) {
      const uint32_t mid = lo + ((hi - lo) >> 1) + ((hi - lo) & 1u);
      int c = 0;
#pragma unroll
      for (int r = 0; r < R; ++r) c += v[r] >= mid ? 1 : 0;
      c = __reduce_add_sync(0xffffffffu, c);
      if (lane == 0) part[round][warp] = c;
      __syncthreads();
      c = 0;
#pragma unroll
      for (int w = 0; w < kSelWarps; ++w) c += part[round][w];
      if (c >= k) lo = mid;
      else hi = mid - 1;
      if (c == k) break;
    }
    if (held >= k) reached = lo;
  }
  // No floor when fewer than k groups hold a score.
  const float f = reached > none ? order_score(reached) : -INFINITY;
  if (tid == 0) kth[qi] = f;
  if (levels == nullptr) return;
  if (tid == 0) ntop = 0;
  __syncthreads();
  if (f > -INFINITY) {
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (v[r] >= reached) {
        const int at = atomicAdd(&ntop, 1);
        if (at < kSelTop) top[at] = v[r];
      }
  }
  __syncthreads();
  if (tid < kLevels) {
    levels[static_cast<int64_t>(qi) * kLevels + tid] = f;
    level_cnt[static_cast<int64_t>(qi) * kLevels + tid] = 0;
  }
  __syncthreads();
  const int n = min(ntop, kSelTop);
  for (int i = n + tid; i < (n + 3) / 4 * 4; i += kSelThreads) top[i] = 0u;
  __syncthreads();
  for (int i = tid; i < n; i += kSelThreads) {
    // The value's rank, equal values by position.
    const uint32_t x = top[i];
    int above = 0;
#pragma unroll 2
    for (int j = 0; j < n; j += 4) {
      const uint4 y = *reinterpret_cast<const uint4*>(top + j);
      above += y.x > x || (y.x == x && j < i) ? 1 : 0;
      above += y.y > x || (y.y == x && j + 1 < i) ? 1 : 0;
      above += y.z > x || (y.z == x && j + 2 < i) ? 1 : 0;
      above += y.w > x || (y.w == x && j + 3 < i) ? 1 : 0;
    }
#pragma unroll
    for (int l = 0; l < kLevels; ++l)
      if (above == level_rank(k, l) - 1)
        levels[static_cast<int64_t>(qi) * kLevels + l] = order_score(x);
  }
}

template <int R>
cudaError_t launch_r(const float* gmax, int64_t gld, int groups, int q, int k, float* kth,
                     float* levels, int* level_cnt, cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(q);
  cfg.blockDim = dim3(kSelThreads);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, group_select_kernel<R>, gmax, gld, groups, k, kth, levels,
                            level_cnt);
}

}  // namespace

cudaError_t launch_group_select(const float* gmax, int64_t gld, int groups, int q, int k,
                                float* kth, float* levels, int* level_cnt, cudaStream_t st) {
  if (q <= 0) return cudaSuccess;
  if (groups <= 4 * kSelThreads)
    return launch_r<4>(gmax, gld, groups, q, k, kth, levels, level_cnt, st);
  if (groups <= 8 * kSelThreads)
    return launch_r<8>(gmax, gld, groups, q, k, kth, levels, level_cnt, st);
  if (groups <= 16 * kSelThreads)
    return launch_r<16>(gmax, gld, groups, q, k, kth, levels, level_cnt, st);
  if (groups <= kSelectMaxGroups)
    return launch_r<kSelectMaxGroups / kSelThreads>(gmax, gld, groups, q, k, kth, levels,
                                                    level_cnt, st);
  return cudaErrorInvalidValue;
}

}  // namespace oprag
