// Global top-k reduction: merges the partial lists that the search kernels
// leave per (query tile, producer) into the final ranked top-k of each query.
// This is the step of Op_retrieve (Sec. 3.2; Sec. 4.1 Retrieval) that reduces
// local candidates to the global top-k, done inside one GPU: the producers
// are corpus slices instead of index shards.
//
// Three merges: for unsorted lists (buffered tensor-core lists, k > 32) a CTA
// per query over all their keys; for sorted lists head by head, one warp per
// query over at most 32 lists, one to four warps per query over up to 512.
#include "merge.cuh"
#include "oprag.h"

namespace oprag {

namespace {

// Few lists per query (at most 32): one warp per query merges the sorted
// lists directly.  Lane l holds the head of list l (with the next keys
// prefetched in registers); each round the warp takes the largest head
// (keys are unique, so exactly one lane wins) and that lane advances.
// CTAs of two warps under 64 registers a thread fit beside a running search
// CTA, so the early-launched merge waits in place.
constexpr int kHeads = 8;           // keys prefetched per list
constexpr int kWayWarps = 2;        // queries per CTA

__global__ void __launch_bounds__(kWayWarps * 32, 16)
merge_kway_kernel(ListSet ls, int q, int k, int64_t* __restrict__ out_ids,
                  float* __restrict__ out_scores) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int qi = blockIdx.x * kWayWarps + warp;
  if (qi >= q) return;
  const int tile = qi / ls.TH, row = qi % ls.TH;
  const int np = merge_list_count(ls, tile);
  const int kl = min(k, ls.klen);
  const uint64_t* list = ls.keys + ((static_cast<int64_t>(tile) * ls.P + lane) * ls.TH + row) *
                                       static_cast<int64_t>(ls.stride);
  const bool has_list = lane < np;
  uint64_t h[kHeads];
  int next = 0;       // keys of this list fetched so far
  auto refill = [&]() {
#pragma unroll
    for (int i = 0; i < kHeads; ++i) h[i] = next + i < kl ? list[next + i] : kEmptyKey;
    next += kHeads;
  };
  if (has_list) refill();
  else {
#pragma unroll
    for (int i = 0; i < kHeads; ++i) h[i] = kEmptyKey;
  }
  int avail = kHeads;
  uint64_t mine = kEmptyKey;      // the answer of rank (lane + 32 * m) for the current m
  for (int r = 0; r < k; ++r) {
    const uint64_t best = warp_max_key(h[0]);
    if (best != kEmptyKey && h[0] == best) {
#pragma unroll
      for (int i = 0; i + 1 < kHeads; ++i) h[i] = h[i + 1];
      h[kHeads - 1] = kEmptyKey;
      if (--avail == 0 && next < kl) {
        refill();
        avail = kHeads;
      }
    }
    if ((r & 31) == lane) mine = best;
    if ((r & 31) == 31 || r == k - 1) {
      const int i = (r & ~31) + lane;
      if (i <= r) {
        const int64_t o = static_cast<int64_t>(qi) * k + i;
        store_result(ls, out_ids, out_scores, o, mine);
      }
    }
  }
}

// More than 32 sorted lists, at most kSmallLists lists per lane: W warps per
// query (W = 1, 2 or 4 by list count; CTAs of four warps, 4 / W queries each).
// Launched early (programmatic dependent launch), a CTA waits in place and
// starts as soon as the search grid ends.  Lane l of warp w holds lists p =
// 32 w + l + 32 W u (u < kSmallLists): the first kSmallKeys keys of each,
// fetched with 16-byte loads all issued together.  Then the query's 32 W lanes
// take the k best head by head: each round the lanes' best heads go through a
// warp maximum (and, when W > 1, a maximum over the query's warps in shared
// memory); keys are unique, so one lane owns the winner and advances that list
// (fetching its next keys once the held ones are used up, which only k >
// kSmallKeys can need).  A round takes about 0.15 us, and few lists are drawn
// on beyond their first keys, so this holds up to k = 256: measured on GB300,
// 16 queries over 152 lists, against a CTA per query that filtered all P k keys
// through sorted buffers: k = 32 13 (56) us, k = 100 27 (76) us, k = 256 60
// (191) us; 1000 queries k = 32 11 (224) us.
constexpr int kSmallThreads = 128;
constexpr int kSmallLists = 4;
constexpr int kSmallKeys = 6;

template <int W>
__global__ void __launch_bounds__(kSmallThreads, 4)
merge_small_kernel(ListSet ls, int q, int k, int64_t* __restrict__ out_ids,
                   float* __restrict__ out_scores) {
  constexpr int kQPerCta = kSmallThreads / 32 / W;
  __shared__ uint64_t heads[2][kSmallThreads / 32];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int qs = warp / W, wq = warp % W;      // query slot in the CTA, warp of the query
  const int qi = blockIdx.x * kQPerCta + qs;
  if (qi >= q) return;                         // all W warps of the slot leave together
  const int tile = qi / ls.TH, row = qi % ls.TH;
  const int np = merge_list_count(ls, tile);
  const int kl = min(k, ls.klen);
  const uint64_t* base = ls.keys + (static_cast<int64_t>(tile) * ls.P * ls.TH + row) * ls.stride;
  const int64_t list_step = static_cast<int64_t>(ls.TH) * ls.stride;
  // Keys at or past kl of a list are not candidates; a missing list is empty.
  auto fetch = [&](int u, int from, uint64_t (&dst)[kSmallKeys]) {
    const int p = wq * 32 + lane + u * 32 * W;
    const uint64_t* l = base + p * list_step + from;
#pragma unroll
    for (int j = 0; j < kSmallKeys; j += 2) {
      ulonglong2 v = make_ulonglong2(kEmptyKey, kEmptyKey);
      if (p < np && from + j < kl) v = *reinterpret_cast<const ulonglong2*>(l + j);
      dst[j] = v.x;
      dst[j + 1] = from + j + 1 < kl ? v.y : kEmptyKey;
    }
  };
  uint64_t key[kSmallLists][kSmallKeys];
  int used[kSmallLists];
#pragma unroll
  for (int u = 0; u < kSmallLists; ++u) {
    fetch(u, 0, key[u]);
    used[u] = 0;
  }
  uint64_t mine = kEmptyKey;
  for (int r = 0; r < k; ++r) {
    uint64_t own = key[0][0];
#pragma unroll
    for (int u = 1; u < kSmallLists; ++u) own = umax64(own, key[u][0]);
    uint64_t best = warp_max_key(own);
    if constexpr (W > 1) {
      if (lane == 0) heads[r & 1][warp] = best;
      // The query's W warps (named barrier 1 + slot; constant ids, so
      // that the kernel reserves only the barriers it uses).
      if (qs == 0) asm volatile("bar.sync 1, %0;" ::"n"(32 * W) : "memory");
      else asm volatile("bar.sync 2, %0;" ::"n"(32 * W) : "memory");
#pragma unroll
      for (int j = 0; j < W; ++j) best = umax64(best, heads[r & 1][qs * W + j]);
    }
    if (best != kEmptyKey && own == best) {
      bool done = false;
#pragma unroll
      for (int u = 0; u < kSmallLists; ++u) {
        if (!done && key[u][0] == best) {
          done = true;
#pragma unroll
          for (int j = 0; j + 1 < kSmallKeys; ++j) key[u][j] = key[u][j + 1];
          key[u][kSmallKeys - 1] = kEmptyKey;
          if (++used[u] % kSmallKeys == 0 && used[u] < kl) fetch(u, used[u], key[u]);
        }
      }
    }
    if (wq != 0) continue;
    if ((r & 31) == lane) mine = best;
    if ((r & 31) == 31 || r == k - 1) {
      const int i = (r & ~31) + lane;
      if (i <= r) {
        const int64_t o = static_cast<int64_t>(qi) * k + i;
        store_result(ls, out_ids, out_scores, o, mine);
      }
    }
  }
}

// Unsorted lists (ListSet::counts), k > 32: W warps per query, a CTA of their
// own.  What bounds it is a chain of dependent steps on few keys, so each step
// is taken by all threads at once: the lists' counts are scanned into offsets
// in shared memory, every thread reads kUnsortedLoads of the concatenated keys
// (a binary search of the offsets finds a key's list), and the keys above the
// floor go to a buffer, which is cut down when the next round of keys might
// not fit and ranked at the end.  A good floor leaves little more than k keys.
// Measured on GB300 (event pairs of 2 us included), against a warp per query
// that sorts its buffer: 300 queries of 32768 x 256, k = 50 10 (14) us, of
// 300000 x 128 12 (20) us; 33 queries of 300000 x 128, k = 100 14 (33) us, 4000
// queries of 32768 x 256, k = 100 18 (29) us; 32768 rows in ascending order of
// their scores, 33 queries, k = 256 62 (381) us.
constexpr int kUnsortedLoads = 4;
constexpr int kRankMax = 256;       // keys that rank_buffer takes
static_assert(kRankMax >= OPRAG_K_MAX, "the k best can be ranked");
// Up to this many queries per SM, whose CTAs the SMs hold all at once, four warps
// a query; above, two.  Four against two warps,
// event-timed, k = 100: 300 queries of 300000 x 128 12 / 16 us, 1024 queries 16
// / 16 us, 4000 queries 35 / 31 us; 2048 queries of 1048576 x 768 27 / 23 us.
constexpr int kUnsortedWideQueries = 10;

template <int W>
struct Unsorted {
  static constexpr int kThreads = 32 * W;
  static constexpr int kRound = kThreads * kUnsortedLoads;   // keys read at a time
  static constexpr int kCap = 2 * kRound;                    // keys in the buffer
  static_assert(kCap - kRound >= kRankMax, "a cut buffer leaves room for a round");
};

// Drops the smallest of the buffer's c > limit keys (all different) until
// between k and limit are left, and returns how many; keys up to the new
// `floor` are not among the k best.  A bisection between the smallest and the
// largest key: a few rounds, where a sort takes some fifty.
template <int W>
__device__ __forceinline__ int cut_buffer(uint64_t* buf, int c, int k, int limit, uint64_t& floor) {
  constexpr int T = Unsorted<W>::kThreads, E = Unsorted<W>::kCap / T;
  __shared__ uint64_t ends[2][W];
  __shared__ int part[2][W];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint64_t v[E], lo = ~0ull, hi = 0;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const bool in = tid + e * T < c;
    v[e] = in ? buf[tid + e * T] : kEmptyKey;
    lo = umin64(lo, in ? v[e] : ~0ull);
    hi = umax64(hi, v[e]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = umin64(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = umax64(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (lane == 0) {
    ends[0][warp] = lo;
    ends[1][warp] = hi;
  }
  __syncthreads();          // also: every key of the buffer is in a register
#pragma unroll
  for (int w = 0; w < W; ++w) {
    lo = umin64(lo, ends[0][w]);
    hi = umax64(hi, ends[1][w]);
  }
  // c > limit keys are >= lo, and none is > hi; as no two are equal, some
  // value in (lo, hi] has exactly k keys at or above it.
  int kept = c, round = 0, before = 0;
  uint64_t mid = lo;
  while (lo < hi) {
    mid = lo + ((hi - lo) >> 1) + ((hi - lo) & 1);
    int mine = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) mine += v[e] >= mid ? 1 : 0;
    mine = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0) part[round][warp] = mine;
    __syncthreads();
    kept = before = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      if (w < warp) before += part[round][w];
      kept += part[round][w];
    }
    round ^= 1;             // written again only after the next barrier
    if (kept > limit) lo = mid;
    else if (kept < k) hi = mid - 1;
    else break;
  }
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const uint32_t bits = __ballot_sync(0xffffffffu, v[e] >= mid);
    const int at = before + __popc(bits & ((1u << lane) - 1u));
    if (v[e] >= mid && at < limit) buf[at] = v[e];
    before += __popc(bits);
  }
  floor = mid - 1;
  __syncthreads();
  return min(kept, limit);
}

// Sorts the buffer's c <= kRankMax keys, best first: every thread counts the
// keys above its own ones, with no barrier between.
template <int T, int E>
__device__ __forceinline__ void rank_buffer(uint64_t* buf, int c) {
  uint64_t v[E];
  int above[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int i = threadIdx.x + e * T;
    v[e] = i < c ? buf[i] : kEmptyKey;
    above[e] = 0;
  }
#pragma unroll 8
  for (int i = 0; i < c; ++i) {
    const uint64_t o = buf[i];
#pragma unroll
    for (int e = 0; e < E; ++e) above[e] += o > v[e] ? 1 : 0;
  }
  __syncthreads();
#pragma unroll
  for (int e = 0; e < E; ++e)
    if (static_cast<int>(threadIdx.x) + e * T < c) buf[above[e]] = v[e];
  __syncthreads();
}

template <int W>
__global__ void __launch_bounds__(Unsorted<W>::kThreads)
merge_unsorted_kernel(ListSet ls, int k, int64_t* __restrict__ out_ids,
                      float* __restrict__ out_scores) {
  constexpr int T = Unsorted<W>::kThreads, kRound = Unsorted<W>::kRound, kCap = Unsorted<W>::kCap;
  extern __shared__ int offs[];                     // P: keys of the lists before p
  __shared__ uint64_t buf[kCap];
  __shared__ int warp_sum[W];
  __shared__ int count;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int qi = blockIdx.x;
  const int tile = qi / ls.TH, row = qi % ls.TH;
  const int np = merge_list_count(ls, tile);
  const int* cnt = ls.counts + static_cast<int64_t>(tile) * ls.P * ls.TH + row;
  const uint64_t* base = ls.keys + (static_cast<int64_t>(tile) * ls.P * ls.TH + row) * ls.stride;
  const int64_t list_step = static_cast<int64_t>(ls.TH) * ls.stride;
  uint64_t worst = merge_floor_key(ls, qi, k);      // the same in every thread

  auto list_count = [&](int p) {
    return p < np ? max(0, min(cnt[static_cast<int64_t>(p) * ls.TH], ls.stride)) : 0;
  };
  if (tid == 0) count = 0;
  int total = 0, next = list_count(tid);
  for (int p0 = 0; p0 < np; p0 += T) {
    const int c = next;
    next = list_count(p0 + T + tid);
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    int before = total;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      if (w < warp) before += warp_sum[w];
      total += warp_sum[w];
    }
    if (p0 + tid < np) offs[p0 + tid] = before + incl - c;
    __syncthreads();        // warp_sum has been read; the offsets are written
  }

  for (int g = 0; g < total; g += kRound) {
    uint64_t key[kUnsortedLoads];
#pragma unroll
    for (int u = 0; u < kUnsortedLoads; ++u) {
      const int i = g + u * T + tid;
      key[u] = kEmptyKey;
      if (i < total) {
        int lo = 0, hi = np;                        // the last list with offs[p] <= i
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (offs[mid] <= i) lo = mid;
          else hi = mid;
        }
        key[u] = base[lo * list_step + (i - offs[lo])];
      }
    }
    uint32_t bits[kUnsortedLoads];
    int pass = 0;
#pragma unroll
    for (int u = 0; u < kUnsortedLoads; ++u) {
      bits[u] = __ballot_sync(0xffffffffu, key[u] > worst);
      pass += __popc(bits[u]);
    }
    if (pass != 0) {
      int slot = 0;
      if (lane == 0) slot = atomicAdd(&count, pass);
      slot = __shfl_sync(0xffffffffu, slot, 0);
#pragma unroll
      for (int u = 0; u < kUnsortedLoads; ++u) {
        if (key[u] > worst) buf[slot + __popc(bits[u] & ((1u << lane) - 1u))] = key[u];
        slot += __popc(bits[u]);
      }
    }
    __syncthreads();
    const int c = count;
    if (g + kRound < total && c > kCap - kRound) {
      const int kept = cut_buffer<W>(buf, c, k, kRankMax, worst);
      if (tid == 0) count = kept;
    }
    __syncthreads();
  }
  int c = count;
  const int limit = k <= 7 * kRankMax / 16 ? kRankMax / 2 : kRankMax;
  if (c > limit) c = cut_buffer<W>(buf, c, k, limit, worst);
  if (c <= kRankMax / 2) rank_buffer<T, kRankMax / 2 / T>(buf, c);
  else if (c <= 3 * kRankMax / 4) rank_buffer<T, (3 * kRankMax / 4 + T - 1) / T>(buf, c);
  else rank_buffer<T, kRankMax / T>(buf, c);
  for (int i = tid; i < k; i += T)
    store_result(ls, out_ids, out_scores, static_cast<int64_t>(qi) * k + i,
                 i < c ? buf[i] : kEmptyKey);
}

template <int W>
cudaError_t launch_unsorted(const ListSet& ls, int q, int k, int64_t* ids, float* scores, cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(q);
  cfg.blockDim = dim3(Unsorted<W>::kThreads);
  cfg.dynamicSmemBytes = static_cast<size_t>(ls.P) * sizeof(int);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, merge_unsorted_kernel<W>, ls, k, ids, scores);
}

template <typename Kern>
cudaError_t launch_warp_per_query(Kern kern, int warps, const ListSet& ls, int q, int k,
                                  int64_t* out_ids, float* out_scores, cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((q + warps - 1) / warps);
  cfg.blockDim = dim3(warps * 32);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, ls, q, k, out_ids, out_scores);
}

template <int W>
cudaError_t launch_small_w(const ListSet& ls, int q, int k, int64_t* out_ids, float* out_scores, cudaStream_t st) {
  constexpr int kQPerCta = kSmallThreads / 32 / W;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((q + kQPerCta - 1) / kQPerCta);
  cfg.blockDim = dim3(kSmallThreads);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, merge_small_kernel<W>, ls, q, k, out_ids, out_scores);
}

// Warps per query of merge_small_kernel: the fewest whose lanes hold all of
// a query's lists (kSmallLists each).  The lists' loads are issued together
// whatever W is, and with one warp per query the head-by-head rounds need no
// barrier.
cudaError_t launch_small(const ListSet& ls, int q, int k, int64_t* out_ids, float* out_scores, cudaStream_t st) {
  constexpr int kPerWarp = kSmallLists * 32;
  const int W = ls.P <= kPerWarp ? 1 : ls.P <= 2 * kPerWarp ? 2 : 4;
  // (at most three slices or two epilogue sets per SM: 456 lists on 152 SMs)
  if (ls.P > W * kPerWarp) return cudaErrorInvalidValue;
  if (W == 4) return launch_small_w<4>(ls, q, k, out_ids, out_scores, st);
  if (W == 2) return launch_small_w<2>(ls, q, k, out_ids, out_scores, st);
  return launch_small_w<1>(ls, q, k, out_ids, out_scores, st);
}

}  // namespace

namespace {

// One thread per query: a two-way merge of the queries' ranked lists.
__global__ void merge_two_kernel(int q, const int64_t* __restrict__ a_ids,
                                 const float* __restrict__ a_sc, int ka,
                                 const int64_t* __restrict__ b_ids,
                                 const float* __restrict__ b_sc, int kb, int k,
                                 int64_t* __restrict__ out_ids, int32_t* __restrict__ out_src,
                                 float* __restrict__ out_scores) {
  const int qi = blockIdx.x * blockDim.x + threadIdx.x;
  if (qi >= q) return;
  const int64_t* ai = a_ids + static_cast<int64_t>(qi) * ka;
  const float* as = a_sc + static_cast<int64_t>(qi) * ka;
  const int64_t* bi = b_ids + static_cast<int64_t>(qi) * kb;
  const float* bs = b_sc + static_cast<int64_t>(qi) * kb;
  int i = 0, j = 0;
  for (int r = 0; r < k; ++r) {
    const bool a_ok = i < ka && ai[i] >= 0;
    const bool b_ok = j < kb && bi[j] >= 0;
    // At equal scores list a (the knowledge index) comes first.
    const bool take_a = a_ok && (!b_ok || !(bs[j] > as[i]));
    const int64_t o = static_cast<int64_t>(qi) * k + r;
    if (take_a) {
      out_ids[o] = ai[i];
      out_scores[o] = as[i];
      out_src[o] = 0;
      ++i;
    } else if (b_ok) {
      out_ids[o] = bi[j];
      out_scores[o] = bs[j];
      out_src[o] = 1;
      ++j;
    } else {
      out_ids[o] = -1;
      out_scores[o] = -INFINITY;
      out_src[o] = -1;
    }
  }
}

}  // namespace

cudaError_t launch_merge_two(int q, const int64_t* a_ids, const float* a_sc, int ka,
                             const int64_t* b_ids, const float* b_sc, int kb, int k,
                             int64_t* out_ids, int32_t* out_src, float* out_scores,
                             cudaStream_t st) {
  if (q <= 0) return cudaSuccess;
  merge_two_kernel<<<(q + 127) / 128, 128, 0, st>>>(q, a_ids, a_sc, ka, b_ids, b_sc, kb, k,
                                                    out_ids, out_src, out_scores);
  return cudaGetLastError();
}

cudaError_t launch_merge(const ListSet& ls, int q, int k, int64_t* out_ids, float* out_scores,
                         int num_sms, cudaStream_t st) {
  if (q <= 0) return cudaSuccess;
  if (ls.counts != nullptr)
    return q <= kUnsortedWideQueries * num_sms
               ? launch_unsorted<4>(ls, q, k, out_ids, out_scores, st)
               : launch_unsorted<2>(ls, q, k, out_ids, out_scores, st);
  if (ls.P <= 32)
    return launch_warp_per_query(merge_kway_kernel, kWayWarps, ls, q, k, out_ids, out_scores, st);
  return launch_small(ls, q, k, out_ids, out_scores, st);
}

}  // namespace oprag
