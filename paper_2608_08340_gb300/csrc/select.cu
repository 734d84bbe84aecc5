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
// order-preserving integers.  The k-th largest is found bit by bit from the
// top (a block-wide count per bit, over all threads at once); the search stops
// at the first prefix that exactly k values reach, which is itself a valid
// floor between the k-th and the (k + 1)-th value.  Bounded by the latency of
// its rounds, a barrier each.  The counted floors' ranks come from the values that
// reach the floor, ranked by counting.
template <int R>
__global__ void __launch_bounds__(kSelThreads)
group_select_kernel(const float* __restrict__ gmax, int64_t gld, int groups, int k,
                    float* __restrict__ kth, float* __restrict__ levels,
                    int* __restrict__ level_cnt) {
  __shared__ int part[2][kSelWarps];
  __shared__ uint32_t top[kSelTop];
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
    v[r] = i < groups ? score_order(__ldcs(g + i)) : 0u;
  }
  uint32_t prefix = 0;
  if (k <= groups) {
#pragma unroll 1
    for (int bit = 31; bit >= 0; --bit) {
      const uint32_t cand = prefix | (1u << bit);
      int c = 0;
#pragma unroll
      for (int r = 0; r < R; ++r) c += v[r] >= cand ? 1 : 0;
      c = __reduce_add_sync(0xffffffffu, c);
      if (lane == 0) part[bit & 1][warp] = c;
      __syncthreads();
      c = 0;
#pragma unroll
      for (int w = 0; w < kSelWarps; ++w) c += part[bit & 1][w];
      if (c >= k) prefix = cand;
      if (c == k) break;
    }
  }
  // No floor when fewer than k groups hold a score.
  const float f = prefix > score_order(-INFINITY) ? order_score(prefix) : -INFINITY;
  if (tid == 0) kth[qi] = f;
  if (levels == nullptr) return;
  if (tid == 0) ntop = 0;
  __syncthreads();
  if (f > -INFINITY) {
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (v[r] >= prefix) {
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
  for (int i = tid; i < n; i += kSelThreads) {
    // The value's rank, equal values by position.
    const uint32_t x = top[i];
    int above = 0;
    for (int j = 0; j < n; ++j) above += top[j] > x || (top[j] == x && j < i) ? 1 : 0;
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
