// Tensor-core search of small query batches over a bf16 index: up to 32
// queries, k <= 16, dense scores (Sec. 4.4 dense scores and partial selection;
// Sec. 4.1 Retrieval).
//
// Such a search is one pass over the corpus, bound by HBM and by what happens
// before the first and after the last byte.  So the operands change places
// against search_tc.cuh: a tile of up to 128 corpus rows is the MMA's M side
// (one row per TMEM lane) and the queries, padded to N = 16 or 32, its N side.
// An epilogue thread then owns one row and the four epilogue warps share every
// tile, where with a query per lane one warp would filter the whole tile of a
// single query alone after the last copy has landed.
//
// Every CTA takes one slice of the corpus, all slices the same number of rows,
// cut into equal tiles (215.6 rows a CTA on 32768 become two tiles of 108
// rows instead of one or two of 128).  The first two tiles' keys go to fixed
// slots of each query's buffer in shared memory; a longer slice keeps the k
// best of them, whose last one is the floor of what later tiles push.  At the
// end the buffers' k best become one list per (query, CTA); for a few queries
// the last CTA to finish merges the lists itself, for more the merge kernel
// does (one launch less against one warp per query).
//
// Measured on GB300, cold L2, search and merge kernels (event pairs of 2 us
// included), against search_tc.cuh: 32768 x 768, k = 5: 1 query 25 (29) us, 8
// queries 27 (29) us, 16 queries 29 (31) us, 32 queries 31 (31) us; 16 queries
// and k = 16 33 (37) us; 1024 x 384, 1 query 15 (17) us.  (A bare TMA read of
// the 50 MB takes 16 us in the same setting.)  From 48 queries on the final
// selection of a CTA's queries by its six warps costs more than it saves: 64
// queries 37 against 31 us.
#include <algorithm>
#include <cfloat>

#include "merge.cuh"
#include "search_tc.cuh"
#include "tensor_map.h"

namespace oprag {

using namespace tc;

namespace {

constexpr int kSmallThreads = 192;           // producer, MMA issuer, four epilogue warps
constexpr int kSmallCap = 256;               // candidate keys per query: two tiles
constexpr int kSmallMaxStages = 10;
constexpr size_t kSmallSmem = 226 * 1024;
// Inline merge: one query per warp; a lane holds up to kInlineLists lists of 8.
constexpr int kInlineQueries = kSmallThreads / 32;
constexpr int kInlineLists = 5;

struct SmallParams {
  int64_t n;
  int q, k;
  int box;            // corpus rows per tile
  int64_t slice;      // corpus rows per CTA
  int kblocks;
  int stages;
  uint64_t* lists;    // [(query * grid + CTA) * stride]
  int stride;
  int* dev_err;
  long long wait_limit;
  unsigned int* done;   // CTAs finished (counts to grid - 1 and wraps); inline merge
  int64_t* out_ids;     // inline merge; nullptr: the lists are merged elsewhere
  float* out_scores;
};

__host__ __device__ constexpr uint32_t small_stage_bytes(int N) {
  return kAStageBytes + static_cast<uint32_t>(N) * 128;
}

// The warp puts the k <= 16 best of the c <= 256 keys of a buffer, best first,
// into dst (which may be the buffer); fewer keys end with empty ones.
__device__ __forceinline__ void small_best(const uint64_t* buf, int c, int k, uint64_t* dst) {
  const int lane = threadIdx.x & 31;
  uint64_t v[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) v[e] = lane + 32 * e < c ? buf[lane + 32 * e] : kEmptyKey;
  // Each lane's keys, best first (Batcher's network for eight).
  auto cx = [&](int a, int b) {
    const uint64_t hi = umax64(v[a], v[b]), lo = umin64(v[a], v[b]);
    v[a] = hi;
    v[b] = lo;
  };
  cx(0, 1); cx(2, 3); cx(4, 5); cx(6, 7);
  cx(0, 2); cx(1, 3); cx(4, 6); cx(5, 7);
  cx(1, 2); cx(5, 6);
  cx(0, 4); cx(1, 5); cx(2, 6); cx(3, 7);
  cx(2, 4); cx(3, 5);
  cx(1, 2); cx(3, 4); cx(5, 6);
  __syncwarp();
  uint64_t mine = kEmptyKey;
  for (int r = 0; r < k; ++r) {
    const uint64_t best = warp_max_key(v[0]);
    if (best != kEmptyKey && v[0] == best) {
#pragma unroll
      for (int e = 0; e < 7; ++e) v[e] = v[e + 1];
      v[7] = kEmptyKey;
    }
    if (r == lane) mine = best;
  }
  if (lane < k) dst[lane] = mine;
  __syncwarp();
}

// Merges one query's P <= 32 kInlineLists sorted lists of k <= 8 keys.
__device__ __forceinline__ void inline_merge(const SmallParams& p, int qi, int P) {
  const int lane = threadIdx.x & 31;
  uint64_t key[kInlineLists][8];
#pragma unroll
  for (int u = 0; u < kInlineLists; ++u) {
    const int l = lane + 32 * u;
    const uint64_t* src = p.lists + (static_cast<int64_t>(qi) * P + l) * p.stride;
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
      ulonglong2 x = make_ulonglong2(kEmptyKey, kEmptyKey);
      // (written by other CTAs of this launch: not through L1)
      if (l < P && j < p.k) x = __ldcg(reinterpret_cast<const ulonglong2*>(src + j));
      key[u][j] = x.x;
      key[u][j + 1] = j + 1 < p.k ? x.y : kEmptyKey;
    }
  }
  uint64_t mine = kEmptyKey;
  for (int r = 0; r < p.k; ++r) {
    uint64_t own = key[0][0];
#pragma unroll
    for (int u = 1; u < kInlineLists; ++u) own = umax64(own, key[u][0]);
    const uint64_t best = warp_max_key(own);
    if (best != kEmptyKey && own == best) {
#pragma unroll
      for (int u = 0; u < kInlineLists; ++u) {
        const bool won = key[u][0] == best;
#pragma unroll
        for (int j = 0; j < 7; ++j) key[u][j] = won ? key[u][j + 1] : key[u][j];
        key[u][7] = won ? kEmptyKey : key[u][7];
      }
    }
    if (r == lane) mine = best;
  }
  if (lane < p.k)
    store_result(ListSet{}, p.out_ids, p.out_scores, static_cast<int64_t>(qi) * p.k + lane, mine);
}

template <int N>
__global__ void __launch_bounds__(kSmallThreads, 1)
small_search_kernel(const __grid_constant__ CUtensorMap map_q,
                    const __grid_constant__ CUtensorMap map_e, const SmallParams p) {
  constexpr uint32_t kStage = small_stage_bytes(N);
  static_assert(N == 16 || N == 32, "an accumulator is read with one 32-column load");
  constexpr int kAccCols = 32;                          // TMEM columns per accumulator
  extern __shared__ __align__(1024) unsigned char smem_s[];
  unsigned char* ring = smem_s + ((1024 - (smem_addr(smem_s) & 1023)) & 1023);
  uint64_t* buf = reinterpret_cast<uint64_t*>(ring + p.stages * kStage);    // N x kSmallCap
  uint64_t* full = buf + N * kSmallCap;
  uint64_t* empty = full + kSmallMaxStages;
  uint64_t* tfull = empty + kSmallMaxStages;
  uint64_t* tempty = tfull + 2;
  uint64_t* mma_done = tempty + 2;
  int* cnt = reinterpret_cast<int*>(mma_done + 1);      // N
  float* flo = reinterpret_cast<float*>(cnt + N);       // N
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(flo + N);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* last_cta = reinterpret_cast<int*>(tmem_slot + 2);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t r_begin = p.slice * blockIdx.x;
  const int64_t r_end = min(p.n, r_begin + p.slice);
  const int tiles = static_cast<int>((r_end - r_begin + p.box - 1) / p.box);
  const uint32_t tx = static_cast<uint32_t>(p.box + N) * 128;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 4);
    }
    mbar_init(mma_done, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  auto load_stage = [&](int s, int kb, int tile) {
    unsigned char* sA = ring + s * kStage;
    mbar_arrive_expect_tx(&full[s], tx);
    tma_load_2d(sA, &map_e, &full[s], kb * kBlockK, static_cast<int>(r_begin) + tile * p.box);
    tma_load_2d(sA + kAStageBytes, &map_q, &full[s], kb * kBlockK, 0);
  };
  const int blocks = tiles * p.kblocks;
  int pre = 0;                 // blocks loaded before the setup barrier
  if (threadIdx.x == 0) {
    for (int tile = 0; tile < tiles && pre < p.stages; ++tile)
      for (int kb = 0; kb < p.kblocks && pre < p.stages; ++kb, ++pre) load_stage(pre, kb, tile);
  }
  if (warp == 1) tmem_alloc(tmem_slot, 2 * kAccCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == 0) {
    if (lane == 0) {
      // ------------------------------------------------ TMA producer
      uint32_t issued = 0, parity = 0;     // per stage: ever issued, parity of the last issue
      int s = 0, kb = 0, tile = 0;
      uint32_t ph = 0;
      for (int b = 0; b < blocks; ++b) {
        if (b >= pre) {
          if (!mbar_wait(&empty[s], ph ^ 1u, abort_flag, p.dev_err, p.wait_limit)) break;
          load_stage(s, kb, tile);
        }
        issued |= 1u << s;
        parity = (parity & ~(1u << s)) | (ph << s);
        if (++s == p.stages) {
          s = 0;
          ph ^= 1u;
        }
        if (++kb == p.kblocks) {
          kb = 0;
          ++tile;
        }
      }
      for (int i = 0; i < p.stages; ++i)
        if (issued & (1u << i)) mbar_drain(&full[i], (parity >> i) & 1u, p.dev_err);
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      // ------------------------------------------------ MMA issuer
      constexpr uint32_t idesc = idesc_bf16(kBlockM, N);
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int tile = 0; ok && tile < tiles; ++tile) {
        const int acc = tile & 1;
        const uint32_t acc_ph = static_cast<uint32_t>(tile >> 1) & 1u;
        if (!mbar_wait(&tempty[acc], acc_ph ^ 1u, abort_flag, p.dev_err, p.wait_limit)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(acc * kAccCols);
        for (int kb = 0; kb < p.kblocks; ++kb) {
          if (!mbar_wait(&full[s], ph, abort_flag, p.dev_err, p.wait_limit)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t a = sw128_desc(smem_addr(ring + s * kStage));
          const uint64_t b = sw128_desc(smem_addr(ring + s * kStage + kAStageBytes));
#pragma unroll
          for (int kk = 0; kk < kBlockK / kUmmaK; ++kk)
            mma_bf16(d_tmem, a + 2 * kk, b + 2 * kk, idesc, (kb | kk) != 0 ? 1u : 0u);
          mma_commit(&empty[s]);
          if (++s == p.stages) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (!ok) break;
        mma_commit(&tfull[acc]);
      }
      mma_commit(mma_done);
      mbar_drain(mma_done, 0, p.dev_err);
    }
    __syncwarp();
  } else {
    // ------------------------------------------------ epilogue
    const int eg = warp & 3;                  // TMEM lane group of this warp
    const int row = eg * 32 + lane;           // row within a tile
    bool ok = true;
    for (int tile = 0; tile < tiles; ++tile) {
      const int acc = tile & 1;
      const int64_t r = r_begin + static_cast<int64_t>(tile) * p.box + row;
      const bool valid = row < p.box && r < r_end;
      // (the warps meet at barriers below, so a wait that gives up does not
      // end one early: it goes on with what the accumulator holds)
      ok = mbar_wait(&tfull[acc], static_cast<uint32_t>(tile >> 1) & 1u, abort_flag, p.dev_err,
                     p.wait_limit) && ok;
      ok = __all_sync(0xffffffffu, ok);
      tc_fence_after();
      const uint32_t taddr = tmem_base + (static_cast<uint32_t>(eg * 32) << 16) +
                             static_cast<uint32_t>(acc * kAccCols);
      uint32_t v[32];
      tmem_ld32_async(taddr, v);
      tmem_wait_ld(v);
      // Hand the accumulator back.
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[acc]);
      if (tile < 2) {
        // Fixed slots of the first two tiles.  A score of -inf (one that
        // overflowed) is no result, as in the general kernel.
#pragma unroll
        for (int i = 0; i < N; ++i)
          if (i < p.q) {
            const float s = __uint_as_float(v[i]);
            buf[i * kSmallCap + tile * kBlockM + row] =
                valid && s > -INFINITY ? make_key(s, static_cast<uint32_t>(r)) : kEmptyKey;
          }
      } else {
#pragma unroll
        for (int i = 0; i < N; ++i) {
          if (i >= p.q) break;
          const float s = __uint_as_float(v[i]);
          if (valid && s >= flo[i])
            buf[i * kSmallCap + atomicAdd(cnt + i, 1)] = make_key(s, static_cast<uint32_t>(r));
        }
      }
      // Room for the next tile's 128 keys: keep the k best of a buffer that
      // may be too full, and raise its floor.
      if (tile >= 1 && tile + 1 < tiles) {
        asm volatile("bar.sync 1, 128;" ::: "memory");
        for (int c = warp - 2; c < p.q; c += 4) {
          const int have = tile == 1 ? 2 * kBlockM : cnt[c];
          if (have > kSmallCap - kBlockM) {
            uint64_t* b = buf + c * kSmallCap;
            small_best(b, have, p.k, b);
            if (lane == 0) {
              cnt[c] = p.k;
              flo[c] = fmaxf(key_floor(b[p.k - 1]), -FLT_MAX);
            }
          }
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem_base, 2 * kAccCols);
  for (int c = warp; c < p.q; c += kSmallThreads / 32) {
    const int have = tiles <= 2 ? tiles * kBlockM : cnt[c];
    small_best(buf + c * kSmallCap, have, p.k,
               p.lists + (static_cast<int64_t>(c) * gridDim.x + blockIdx.x) * p.stride);
  }
  if (p.out_ids == nullptr) return;
  // The last CTA to get here merges: its peers' lists are visible by then.
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) *last_cta = atomicInc(p.done, gridDim.x - 1) == gridDim.x - 1;
  __syncthreads();
  if (*last_cta == 0) return;
  __threadfence();
  if (warp < p.q) inline_merge(p, warp, static_cast<int>(gridDim.x));
}

template <int N>
cudaError_t launch_n(const CUtensorMap& mq, const CUtensorMap& me, const SmallParams& p, int grid,
                     size_t smem, cudaStream_t st) {
  static DeviceOnce once;
  const cudaError_t e = allow_smem(once, small_search_kernel<N>, kSmallSmem);
  if (e != cudaSuccess) return e;
  small_search_kernel<N><<<grid, kSmallThreads, smem, st>>>(mq, me, p);
  return cudaGetLastError();
}

}  // namespace

bool small_applies(const SearchShape& s) {
  return s.q <= kSmallMaxQueries && s.k <= 16 && s.n_second == 0 && !s.fused_lex && !s.lex_block &&
         s.group == 0;
}

// One slice of equal tiles per SM; at least 32 rows a slice.
SmallPlan small_plan(const SearchShape& s, int num_sms) {
  SmallPlan pl{};
  const int64_t per = std::max<int64_t>(32, (s.n + num_sms - 1) / num_sms);
  const int64_t tiles = (per + kBlockM - 1) / kBlockM;
  pl.box = static_cast<int>((per + tiles - 1) / tiles);
  pl.slice = pl.box * tiles;
  pl.grid = static_cast<int>((s.n + pl.slice - 1) / pl.slice);
  pl.inline_merge = s.q <= kInlineQueries && s.k <= 8 && pl.grid <= 32 * kInlineLists;
  return pl;
}

size_t small_scratch_bytes(const SearchShape& s, const SmallPlan& pl) {
  return static_cast<size_t>(s.q) * pl.grid * list_len_for(s.k) * sizeof(uint64_t);
}

cudaError_t launch_small_search(const void* E, const void* Q, const SearchShape& s,
                                const SmallPlan& pl, void* scratch, int* dev_err,
                                unsigned int* done, long long wait_limit, int64_t* out_ids,
                                float* out_scores, ListSet* lists, cudaStream_t st) {
  const int N = s.q <= 16 ? 16 : 32;
  CUtensorMap mq, me;
  if (!encode_rows_map(&mq, Q, s.q, s.d, N, kBF16) ||
      !encode_rows_map(&me, E, s.n, s.d, pl.box, kBF16))
    return cudaErrorInvalidValue;
  SmallParams p{};
  p.n = s.n;
  p.q = s.q;
  p.k = s.k;
  p.box = pl.box;
  p.slice = pl.slice;
  p.kblocks = (s.d + kBlockK - 1) / kBlockK;
  p.lists = static_cast<uint64_t*>(scratch);
  p.stride = list_len_for(s.k);
  p.dev_err = dev_err;
  p.wait_limit = wait_limit > 0 ? wait_limit : kWaitLimitCycles;
  if (pl.inline_merge) {
    p.done = done;
    p.out_ids = out_ids;
    p.out_scores = out_scores;
  }
  const size_t fixed = static_cast<size_t>(N) * kSmallCap * sizeof(uint64_t) +
                       (2 * kSmallMaxStages + 5) * sizeof(uint64_t) + N * 8 + 32 + 1024;
  p.stages = static_cast<int>(
      std::min<size_t>(kSmallMaxStages, (kSmallSmem - fixed) / small_stage_bytes(N)));
  const size_t smem = fixed + p.stages * small_stage_bytes(N);
  lists->keys = p.lists;
  lists->P = pl.grid;
  lists->TH = 1;
  lists->stride = p.stride;
  lists->klen = p.stride;
  if (N == 16) return launch_n<16>(mq, me, p, pl.grid, smem, st);
  return launch_n<32>(mq, me, p, pl.grid, smem, st);
}

}  // namespace oprag
