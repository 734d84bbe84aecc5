// Search of fp32 indices: the query x chunk inner products of Sec. 4.4 as a
// register-tiled fp32 product on the CUDA cores (the scores must be fp32 sums
// of fp32 products, which the tensor cores do not give), with the partial
// top-k selection (Sec. 4.4, Sec. 7) fused behind it.
//
// A CTA of 256 threads takes one query tile of TY * TM queries and one
// contiguous slice of the corpus, in tiles of 4 * TX rows (TX = 256 / TY).
// Thread (ty, tx) holds the scores of queries ty + TY i (i < TM) and rows
// tx + TX j (j < 4); a warp covers 4 ty and 8 tx, so that each of its 16-byte
// shared-memory reads touches at most 128 different bytes (measured: 2.1
// cycles of the SM each; 4.2 for 16 rows or more).  K blocks of 32 floats of
// both operands come through a TMA ring (128-byte swizzle: eight rows' reads
// of one k group touch all banks once) that the warps feed in turn, every eighth
// block each: a ninth warp would cap every thread at 168 registers.
//
// Sums: chains of eight products, four of them added up per K block, and the
// blocks' sums added with compensation (Kahan), so that the error does not grow
// with d.  Up to d = kFineDim the streaming kernel, whose lanes then held one
// chain of four products each, was closer to 64 bits than that; there the
// chains have four products and four of them (two up to d = 32) are added up
// before each compensated addition.  Relative error against 64 bits (root mean
// square, 1e-8, over the 10 best of 100 queries), in brackets the streaming
// kernel's: d = 16 4.3 (4.2; 40 queries 4.2 and 4.3), 32 4.0 (4.4), 64 3.9 (4.3),
// 128 4.0 (4.7), 136 4.2 (4.5), 768 3.3 (5.1), 1280 3.5 (5.9).  With chains of
// eight throughout 4.7, 4.8, 4.6 and 4.5 up to d = 128, and 263 instead of 285 us
// (100000 x 64, 256 queries), 66 instead of 73 us (32768 x 64, 100 queries).
// One chain of 64 products per two blocks, added to two plain sums in turn, gave
// 6.8 at d = 768 and 177 instead of 195 us at 100 queries of 32768 x 768.
//
// What bounds it: from about 16 queries on the FMA pipes and, next to them,
// the shared-memory reads that feed them (a warp step of four k: 112 FMA issue
// slots and 11 reads with TM = 7), below that HBM.  The tile shape follows the
// batch (config_for): TY = 4 (256 corpus rows) up to 32 queries, TY = 8 up to
// 64, TY = 16 above.  Measured on GB300, 32768 x 768 and k = 10, search kernel,
// against the streaming kernel this one replaced (each chunk of eight queries
// streamed the corpus again, five shuffles per score): 1 query 27 (41) us, 16
// queries 43 (92) us, 32 queries 68 (172) us, 100 queries 195 (529) us or 25.8
// TFLOP/s, 256 queries 393 (1297) us; 86132 x 1192 and 8 queries 96 (111) us.
//
// Selection.  Each query of the tile has a buffer of candidate keys in shared
// memory.  A score enters it when it reaches the query's floor: the k-th
// largest of a warp's group maxima in the first tile (k distinct scores reach
// it), then what compactions prove and what the other slices of the search
// publish (qfloor).  A buffer that could overflow within the next tile is
// sorted by one warp and cut to its k best; at the end the buffers are sorted
// into one list per (query, slice) for the merge kernel.
#pragma once
#include <cfloat>

#include "common.cuh"
#include "internal.h"

namespace oprag {
namespace f32 {

constexpr int kThreads = 256;
constexpr int kBK = 32;                    // floats per K block: one 128-byte swizzle row
constexpr int kRowBytes = kBK * 4;
constexpr int kRowsPerThread = 4;
constexpr int kFineDim = 128;              // dimensions of the finer sums
constexpr int kMaxCap = 512;               // candidate keys per query
constexpr int kMaxStages = 16;
constexpr size_t kSmemMax = 226 * 1024;

struct Params {
  const float* E;       // n x d
  const float* Q;       // q x d
  int64_t n;
  int d;
  int q;
  int k;
  Fusion fu;
  uint64_t* lists;      // [(tile * G + slice) * TH + query] * stride
  int stride;
  int cap;
  int stages;
  int stage;            // bytes of a ring stage: b_bytes of corpus rows, then the queries
  int b_bytes;
  uint64_t* qfloor;     // optional: shared k-th bounds, tagged gen
  uint32_t gen;
  int* dev_err;
  long long wait_limit;
};

// Launch shape of one search (host side, also its scratch size).
struct Config {
  int TY, TM;
  int th;        // queries per tile, TY * TM
  int qt;        // query tiles
  int G;         // corpus slices
  int cap, stages, stage, b_bytes;
  size_t smem;
};

// Adds sums to the scores with their rounding errors carried (Kahan).
template <int TM, int TN>
__device__ __forceinline__ void add_sums(const float (&s)[TM][kRowsPerThread],
                                         float (&tot)[TM][kRowsPerThread],
                                         float (&lost)[TM][kRowsPerThread]) {
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const float add = s[i][j] - lost[i][j], sum = tot[i][j] + add;
      lost[i][j] = (sum - tot[i][j]) - add;
      tot[i][j] = sum;
    }
}

// One K block: eight groups of four k (zeros past d), TN of the thread's four
// rows.  mid: the block's sums, of four chains of eight products, 0 for the
// other rows.  kFine: chains of four, four of them added up in mid (two when
// `finest`) and then to the scores.  a0 / b0: the thread's first query / corpus
// row of the stage.
template <int TY, int TM, int TN, bool kFine>
__device__ __forceinline__ void mul_block(const unsigned char* a0, const unsigned char* b0, int ty,
                                          int tx, float (&mid)[TM][kRowsPerThread],
                                          float (&tot)[TM][kRowsPerThread],
                                          float (&lost)[TM][kRowsPerThread], bool finest) {
  constexpr int TX = kThreads / TY;
  constexpr int kChain = kFine ? 4 : 8;
  constexpr int kSum = 4 * kChain / 4;              // steps of a second-level sum
  float acc[TM][TN];
#pragma unroll
  for (int s = 0; s < kBK / 4; ++s) {
    const bool first = s % (kChain / 4) == 0, last = (s + 1) % (kChain / 4) == 0;
    const int ob = (s ^ (tx & 7)) << 4;
    float4 b[TN];
#pragma unroll
    for (int j = 0; j < TN; ++j)
      b[j] = *reinterpret_cast<const float4*>(b0 + j * TX * kRowBytes + ob);
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      // row ty + TY i of the tile; its swizzle phase alternates when TY = 4
      const int oa = (s ^ ((ty + TY * i) & 7)) << 4;
      const float4 a = *reinterpret_cast<const float4*>(a0 + i * TY * kRowBytes + oa);
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[i][j] = first ? a.x * b[j].x : fmaf(a.x, b[j].x, acc[i][j]);
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a.y, b[j].y, acc[i][j]);
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a.z, b[j].z, acc[i][j]);
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a.w, b[j].w, acc[i][j]);
      if (last)
#pragma unroll
        for (int j = 0; j < TN; ++j)
          mid[i][j] = s % kSum < kChain / 4 ? acc[i][j] : mid[i][j] + acc[i][j];
    }
    if (kFine && (s + 1) % kSum == 0) add_sums<TM, TN>(mid, tot, lost);
    if (kFine && (s + 1) % kSum == kSum / 2 && finest) {
      add_sums<TM, TN>(mid, tot, lost);
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) mid[i][j] = 0.f;
    }
  }
  if (!kFine)
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = TN; j < kRowsPerThread; ++j) mid[i][j] = 0.f;
}

// The fused score of query qg and row r (Sec. 4.4), the dense one without a block.
__device__ __forceinline__ float fuse(const Fusion& fu, float s, int qg, int64_t r) {
  if (fu.bm25 == nullptr) return s;
  const float m = fu.bm25_max[qg], inv_max = m > 0.f ? 1.f / m : 0.f;
  return fmaf(fu.alpha, s, (1.f - fu.alpha) * (fu.bm25[qg * fu.ld + r] * inv_max));
}

// max(m, |a|, |b|), NaN when one of them is.
__device__ __forceinline__ float max_abs_nan(float m, float a, float b) {
  asm("max.NaN.f32 %0, %0, %1, %2;" : "+f"(m) : "f"(fabsf(a)), "f"(fabsf(b)));
  return m;
}

// Scores that passed the fp32 range: the carried errors of the sums turn an
// infinite sum into NaN, so those scores are formed again as plain sums in the
// order of the dimensions, where an overflowed sum of finite products keeps its
// infinity.  They are looked for once per tile, behind the pushes of the other
// scores.  Measured against no such care, 32768 x 768: 100 queries 194 (194) us, 60
// 118 (114), 32 77 (73), 20 51 (49), and 414 (418) us at 256 queries of 65536 x 384;
// with a check in each K block, to drop the carried errors there, 100 queries took
// 6 us more, and with the scores formed before the selection 2 us (32 queries 80).
// Returns bit 4 i + j for each.
template <int TM>
__device__ __forceinline__ uint32_t find_overflowed(const float (&score)[TM][kRowsPerThread]) {
  float any = 0.f;
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < kRowsPerThread; j += 2)
      any = max_abs_nan(any, score[i][j], score[i][j + 1]);
  uint32_t redo = 0;
  if (any != any) {
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < kRowsPerThread; ++j)
        if (score[i][j] != score[i][j]) redo |= 1u << (kRowsPerThread * i + j);
  }
  return redo;
}

// Forms the scores of `redo` (all of rows and queries that exist) and pushes those
// that reach their query's floor.  r0, ql0: the thread's first corpus row, and its
// first query of the tile at q0.
template <int TY>
static __device__ __noinline__ void push_overflowed(const Params& p, uint32_t redo, int64_t r0,
                                                    int q0, int ql0, uint64_t* buf, int* cnt,
                                                    const uint32_t* flo) {
  constexpr int TX = kThreads / TY;
#pragma unroll 1
  for (; redo != 0; redo &= redo - 1) {
    const int at = __ffs(redo) - 1;
    const int64_t r = r0 + TX * (at % kRowsPerThread);
    const int ql = ql0 + TY * (at / kRowsPerThread), qg = q0 + ql;
    const float4* e = reinterpret_cast<const float4*>(p.E + r * p.d);
    const float4* q = reinterpret_cast<const float4*>(p.Q + static_cast<int64_t>(qg) * p.d);
    float s = 0.f;
#pragma unroll 2
    for (int t = 0; t < p.d / 4; ++t) {
      const float4 x = __ldg(e + t), y = __ldg(q + t);
      s = fmaf(x.w, y.w, fmaf(x.z, y.z, fmaf(x.y, y.y, fmaf(x.x, y.x, s))));
    }
    s = fuse(p.fu, s, qg, r);
    if (s >= order_score(flo[ql]))
      buf[ql * p.cap + atomicAdd(cnt + ql, 1)] = make_key(s, static_cast<uint32_t>(r));
  }
}

// keep_best for c <= 32 E keys: a bitonic sort.
template <int E>
__device__ __noinline__ void sort_best(uint64_t* buf, int c, int k, uint64_t* dst) {
  const int lane = threadIdx.x & 31;
  uint64_t v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) v[e] = lane * E + e < c ? buf[lane * E + e] : kEmptyKey;
  warp_sort_desc<E>(v);
  __syncwarp();
#pragma unroll
  for (int e = 0; e < E; ++e)
    if (lane * E + e < min(c, k)) dst[lane * E + e] = v[e];
  __syncwarp();
}

// keep_best for c <= 32 E keys, by counting.
template <int E>
__device__ __forceinline__ void rank_best(const uint64_t* buf, int c, int k, uint64_t* dst) {
  const int lane = threadIdx.x & 31;
  uint64_t v[E];
  int above[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    v[e] = lane + 32 * e < c ? buf[lane + 32 * e] : kEmptyKey;
    above[e] = 0;
  }
#pragma unroll 4
  for (int i = 0; i < c; ++i) {
    const uint64_t o = buf[i];
#pragma unroll
    for (int e = 0; e < E; ++e) above[e] += o > v[e] ? 1 : 0;
  }
  __syncwarp();
#pragma unroll
  for (int e = 0; e < E; ++e)
    if (lane + 32 * e < c && above[e] < k) dst[above[e]] = v[e];
  __syncwarp();
}

// The warp puts the min(c, k) best of the c keys of a buffer, best first, into
// dst (which may be the buffer).  Up to 64 keys -- the usual case, a good
// floor leaves few more than k -- every lane counts the keys above its own
// ones: no chain of dependent exchanges (14 queries a warp at the end of a
// search: 1 us instead of 10 us of bitonic sorts).  More keys are sorted.
__device__ __forceinline__ void keep_best(uint64_t* buf, int c, int k, uint64_t* dst) {
  if (c <= 32) rank_best<1>(buf, c, k, dst);
  else if (c <= 64) rank_best<2>(buf, c, k, dst);
  else if (c <= 128) sort_best<4>(buf, c, k, dst);
  else if (c <= 256) sort_best<8>(buf, c, k, dst);
  else sort_best<16>(buf, c, k, dst);
}

// The newest block copied into a stage (-1: none), where warp w has issued the
// blocks w, w + 8, ... up to newest[w] (-1: none).  Only that copy can still be
// in flight: a block is issued after the one before it in its stage has landed.
// (Its phase is the one to wait for; an older block's phase has the parity of a
// copy that nobody will issue.)
__host__ __device__ inline int newest_block(const int* newest, int stages, int stage) {
  int best = -1;
  for (int w = 0; w < kThreads / 32; ++w) {
    int m = newest[w];
    // the warp's blocks come back to a stage after at most `stages` steps
    for (int i = 0; i < stages && m > best; ++i, m -= kThreads / 32)
      if (m % stages == stage) best = m;
  }
  return best;
}

// The value of rank r (0-based, descending) among the 8 E values of each group
// of eight lanes: a bitonic sort, element l E + e in lane l of the group.
template <int E>
__device__ __forceinline__ float rank_of_8(float (&v)[E], int r) {
  const int l = threadIdx.x & 7;
#pragma unroll
  for (int size = 2; size <= 8 * E; size <<= 1) {
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      if (stride < E) {
#pragma unroll
        for (int e = 0; e < E; ++e)
          if ((e & stride) == 0) {
            const bool desc = ((l * E + e) & size) == 0;
            const float hi = fmaxf(v[e], v[e | stride]), lo = fminf(v[e], v[e | stride]);
            v[e] = desc ? hi : lo;
            v[e | stride] = desc ? lo : hi;
          }
      } else {
        const int lm = stride / E;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const bool desc = ((l * E + e) & size) == 0;
          const float o = __shfl_xor_sync(0xffffffffu, v[e], lm);
          v[e] = (((l & lm) == 0) == desc) ? fmaxf(v[e], o) : fminf(v[e], o);
        }
      }
    }
  }
  float m = v[0];
#pragma unroll
  for (int e = 1; e < E; ++e)
    if (e == (r & (E - 1))) m = v[e];
  return __shfl_sync(0xffffffffu, m, r / E, 8);
}

template <int TY, int TM, bool kFine>
__global__ void __launch_bounds__(kThreads, 1)
f32_search_kernel(const __grid_constant__ CUtensorMap map_q,
                  const __grid_constant__ CUtensorMap map_e, const __grid_constant__ Params p) {
  constexpr int TX = kThreads / TY;
  constexpr int BM = TY * TM, BN = TX * kRowsPerThread;
  constexpr int WY = TY / 4;                          // warps along the queries
  extern __shared__ __align__(1024) unsigned char smem_f[];
  // (an offset, not a rounded pointer: the compiler then still knows that the
  // ring is shared memory)
  unsigned char* ring = smem_f + ((1024 - (smem_addr(smem_f) & 1023)) & 1023);
  uint64_t* buf = reinterpret_cast<uint64_t*>(ring + p.stages * p.stage);
  uint64_t* full = buf + static_cast<size_t>(BM) * p.cap;
  uint64_t* empty = full + kMaxStages;
  int* cnt = reinterpret_cast<int*>(empty + kMaxStages);
  uint32_t* flo = reinterpret_cast<uint32_t*>(cnt + BM);    // score_order of each floor
  volatile int* abort_flag = reinterpret_cast<volatile int*>(flo + BM);

  // Let the merge kernel get scheduled; it waits for this grid to finish.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int q0 = blockIdx.y * BM;
  const int64_t r_begin = p.n * blockIdx.x / gridDim.x;
  const int64_t r_end = p.n * (blockIdx.x + 1) / gridDim.x;
  const int tiles = static_cast<int>((r_end - r_begin + BN - 1) / BN);
  const int nkb = (p.d + kBK - 1) / kBK;
  const bool finest = nkb == 1;

  if (tid == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], kThreads / 32);
    }
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_map(&map_q);
    prefetch_map(&map_e);
  }
  if (tid < BM) {
    cnt[tid] = 0;
    // (up to 32 results a score of -inf, one that overflowed, is none)
    flo[tid] = score_order(p.k <= 32 ? -FLT_MAX : -INFINITY);
  }
  __syncthreads();

  // Groups of TX rows (1 .. 4) that the tile at row r0 needs.
  auto groups_of = [&](int64_t r0) {
    const int64_t left = r_end - r0;
    return left >= BN ? kRowsPerThread : static_cast<int>((left + TX - 1) / TX);
  };

  // Loads.  Block m = 8 i + w is issued by lane 0 of warp w, at the start of
  // the warps' own block m + lag - stages, into the stage that block m - stages
  // used; with lag 2 its wait for the other warps to leave that stage is
  // almost never one.  The warps take turns because issuing a block's copies
  // takes a thread about as long as one of its math steps.
  const int blocks = tiles * nkb;
  const int lag = p.stages >= 4 ? 2 : 1;
  int ld_m = warp, ld_s = warp % p.stages, ld_kb = warp % nkb;
  uint32_t ld_ph = (warp / p.stages) & 1;
  int ld_last = -1;            // the warp's newest block
  int64_t ld_r0 = r_begin + static_cast<int64_t>(warp / nkb) * BN;
  auto load_next = [&]() {
    if (lane == 0 && !*abort_flag &&
        mbar_wait(&empty[ld_s], ld_ph ^ 1u, abort_flag, p.dev_err, p.wait_limit)) {
      unsigned char* sB = ring + ld_s * p.stage;
      const int tn = groups_of(ld_r0);
      mbar_arrive_expect_tx(&full[ld_s], static_cast<uint32_t>((tn * TX + BM) * kRowBytes));
      for (int j = 0; j < tn; ++j)
        tma_load_2d(sB + j * TX * kRowBytes, &map_e, &full[ld_s], ld_kb * kBK,
                    static_cast<int>(ld_r0) + j * TX);
      tma_load_2d(sB + p.b_bytes, &map_q, &full[ld_s], ld_kb * kBK, q0);
      ld_last = ld_m;
    }
    __syncwarp();
    ld_m += kThreads / 32;
    for (ld_s += kThreads / 32; ld_s >= p.stages; ld_s -= p.stages) ld_ph ^= 1u;
    for (ld_kb += kThreads / 32; ld_kb >= nkb; ld_kb -= nkb) ld_r0 += BN;
  };
  while (ld_m < p.stages - lag && ld_m < blocks) load_next();

  // A wait that gives up does not end a warp early (the warps meet at
  // barriers): it goes on with whatever the stage holds, and every later wait
  // returns at once because the abort word is set.
  const int ty = (warp % WY) * 4 + (lane >> 3);
  const int tx = (warp / WY) * 8 + (lane & 7);
  float acc[TM][kRowsPerThread], tot[TM][kRowsPerThread], lost[TM][kRowsPerThread];
  int st = 0, blk = 0;
  uint32_t ph = 0;
#pragma unroll 1
  for (int tile = 0; tile < tiles; ++tile) {
    const int64_t r0 = r_begin + static_cast<int64_t>(tile) * BN;
    const int tn = groups_of(r0);
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < kRowsPerThread; ++j) tot[i][j] = lost[i][j] = 0.f;
    // What the other slices have published about this tile's queries.
    if (p.qfloor != nullptr && tile > 0 && tid < BM && q0 + tid < p.q) {
      const unsigned long long v =
          __ldcg(reinterpret_cast<const unsigned long long*>(p.qfloor + q0 + tid));
      if (static_cast<uint32_t>(v >> 32) == p.gen)
        atomicMax(flo + tid, static_cast<uint32_t>(v));
    }
#pragma unroll 1
    for (int kb = 0; kb < nkb; ++kb, ++blk) {
      if (ld_m == blk + p.stages - lag && ld_m < blocks) load_next();
      mbar_wait(&full[st], ph, abort_flag, p.dev_err, p.wait_limit);
      __syncwarp();
      const unsigned char* sB = ring + st * p.stage + tx * kRowBytes;
      const unsigned char* sA = ring + st * p.stage + p.b_bytes + ty * kRowBytes;
      if (tn == 4) mul_block<TY, TM, 4, kFine>(sA, sB, ty, tx, acc, tot, lost, finest);
      else if (tn == 3) mul_block<TY, TM, 3, kFine>(sA, sB, ty, tx, acc, tot, lost, finest);
      else if (tn == 2) mul_block<TY, TM, 2, kFine>(sA, sB, ty, tx, acc, tot, lost, finest);
      else mul_block<TY, TM, 1, kFine>(sA, sB, ty, tx, acc, tot, lost, finest);
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[st]);
      if (++st == p.stages) {
        st = 0;
        ph ^= 1u;
      }
      if (!kFine) add_sums<TM, kRowsPerThread>(acc, tot, lost);
    }

    // ---- selection
    // The scores (in the accumulators' place), -inf where there is none.
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int qg = q0 + ty + TY * i;
      float inv_max = 0.f;
      const float* brow = nullptr;
      if (p.fu.bm25 != nullptr && qg < p.q) {
        const float m = p.fu.bm25_max[qg];
        inv_max = m > 0.f ? 1.f / m : 0.f;
        brow = p.fu.bm25 + static_cast<int64_t>(qg) * p.fu.ld;
      }
#pragma unroll
      for (int j = 0; j < kRowsPerThread; ++j) {
        const int64_t r = r0 + tx + TX * j;
        float v = tot[i][j];
        if (brow != nullptr && r < r_end)
          v = fmaf(p.fu.alpha, v, (1.f - p.fu.alpha) * (brow[r] * inv_max));
        acc[i][j] = r < r_end && qg < p.q ? v : -INFINITY;
      }
    }
    if (tile == 0 && p.k <= 32 && r_end - r_begin > 64) {
      // First floors: the k-th largest of the maxima of 8, 16 or 32 groups of
      // the warp's 32 scores of a query (k distinct scores reach it), then
      // the best such bound of the CTA and of the slices that are as far.  (A
      // slice of up to 64 rows takes them all: ranking 64 keys is cheaper.)
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const int ql = ty + TY * i;
        // NaN counts for nothing (fmaxf with -inf): the sorts' minima and maxima
        // would put a second copy of another score in its place.
        const float none = -INFINITY;
        float b;
        if (p.k <= 8) {
          float m[1] = {fmaxf(fmaxf(fmaxf(acc[i][0], acc[i][1]), fmaxf(acc[i][2], acc[i][3])), none)};
          b = rank_of_8<1>(m, p.k - 1);
        } else if (p.k <= 16) {
          float m[2] = {fmaxf(fmaxf(acc[i][0], acc[i][1]), none),
                        fmaxf(fmaxf(acc[i][2], acc[i][3]), none)};
          b = rank_of_8<2>(m, p.k - 1);
        } else {
          float m[4] = {fmaxf(acc[i][0], none), fmaxf(acc[i][1], none), fmaxf(acc[i][2], none),
                        fmaxf(acc[i][3], none)};
          b = rank_of_8<4>(m, p.k - 1);
        }
        if ((lane & 7) == 0 && b > -INFINITY) atomicMax(flo + ql, score_order(b));
      }
      __syncthreads();
      if (p.qfloor != nullptr && tid < BM && q0 + tid < p.q) {
        const unsigned long long mine =
            (static_cast<unsigned long long>(p.gen) << 32) | flo[tid];
        const unsigned long long old =
            atomicMax(reinterpret_cast<unsigned long long*>(p.qfloor + q0 + tid), mine);
        if (old > mine && static_cast<uint32_t>(old >> 32) == p.gen)
          flo[tid] = static_cast<uint32_t>(old);
      }
    }
    // The previous tile's compactions and the floors are done.
    __syncthreads();
    // One slot reservation per thread and query, all of them in flight before
    // the first key is stored (a returning atomic per score took 5 us more of
    // 100 queries' search).
    int at[TM];
    uint32_t take = 0;                 // bit 4 i + j: the score enters
    static_assert(TM * kRowsPerThread <= 32, "one mask bit per score");
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int ql = ty + TY * i;
      const float fl = order_score(flo[ql]);
      uint32_t m = 0;
#pragma unroll
      for (int j = 0; j < kRowsPerThread; ++j)
        if (acc[i][j] >= fl && r0 + tx + TX * j < r_end) m |= 1u << j;
      if (q0 + ql >= p.q) m = 0;
      at[i] = m != 0 ? atomicAdd(cnt + ql, __popc(m)) : 0;
      take |= m << (kRowsPerThread * i);
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      uint64_t* b = buf + (ty + TY * i) * p.cap + at[i];
#pragma unroll
      for (int j = 0; j < kRowsPerThread; ++j)
        if ((take >> (kRowsPerThread * i + j)) & 1u)
          *b++ = make_key(acc[i][j], static_cast<uint32_t>(r0 + tx + TX * j));
    }
    const uint32_t redo = find_overflowed<TM>(acc);
    if (redo != 0) push_overflowed<TY>(p, redo, r0 + tx, q0, ty, buf, cnt, flo);
    __syncthreads();
    // Buffers without room for another tile, or of the last tile: keep the k
    // best.
    const bool last = tile + 1 == tiles;
    for (int ql = warp; ql < BM; ql += kThreads / 32) {
      if (q0 + ql >= p.q) break;
      const int c = cnt[ql];
      uint64_t* b = buf + ql * p.cap;
      if (last) {
        uint64_t* dst = p.lists + ((static_cast<int64_t>(blockIdx.y) * gridDim.x + blockIdx.x) * BM +
                                   ql) * p.stride;
        keep_best(b, c, p.k, dst);
        for (int i = c + lane; i < p.k; i += 32) dst[i] = kEmptyKey;
      } else if (c > p.cap - BN) {
        keep_best(b, c, p.k, b);
        if (lane == 0) {
          cnt[ql] = min(c, p.k);
          if (c >= p.k) {
            const uint32_t o = static_cast<uint32_t>(b[p.k - 1] >> 32);
            atomicMax(flo + ql, o);
            if (p.qfloor != nullptr)
              atomicMax(reinterpret_cast<unsigned long long*>(p.qfloor + q0 + ql),
                        (static_cast<unsigned long long>(p.gen) << 32) | o);
          }
        }
      }
    }
  }
  // After a wait gave up, copies may still fly: the CTA outlives them.  Every
  // wait lies before the last tile's barriers, so all warps read the same here.
  if (*abort_flag) {
    int* newest = reinterpret_cast<int*>(buf);
    __syncthreads();           // the buffers have been read
    if (lane == 0) newest[warp] = ld_last;
    __syncthreads();
    if (tid < p.stages) {
      const int m = newest_block(newest, p.stages, tid);
      if (m >= 0) mbar_drain(&full[tid], (m / p.stages) & 1, p.dev_err);
    }
  }
}

template <int TY, int TM, bool kFine>
cudaError_t launch_tm(const Config& c, const CUtensorMap& mq, const CUtensorMap& me,
                      const Params& p, cudaStream_t st) {
  static DeviceOnce once;
  const cudaError_t e = allow_smem(once, f32_search_kernel<TY, TM, kFine>, kSmemMax);
  if (e != cudaSuccess) return e;
  f32_search_kernel<TY, TM, kFine><<<dim3(c.G, c.qt), kThreads, c.smem, st>>>(mq, me, p);
  return cudaGetLastError();
}

// Query tiles of up to 8 TY queries.  Instantiated in translation units of
// their own (parallel builds).
template <int TY, bool kFine>
cudaError_t launch_ty(const Config& c, const CUtensorMap& mq, const CUtensorMap& me,
                      const Params& p, cudaStream_t st) {
  if constexpr (TY == 4) {
    if (c.TM == 1) return launch_tm<TY, 1, kFine>(c, mq, me, p, st);
    if (c.TM == 2) return launch_tm<TY, 2, kFine>(c, mq, me, p, st);
    if (c.TM == 3) return launch_tm<TY, 3, kFine>(c, mq, me, p, st);
    if (c.TM == 4) return launch_tm<TY, 4, kFine>(c, mq, me, p, st);
  }
  switch (c.TM) {
    case 5: return launch_tm<TY, 5, kFine>(c, mq, me, p, st);
    case 6: return launch_tm<TY, 6, kFine>(c, mq, me, p, st);
    case 7: return launch_tm<TY, 7, kFine>(c, mq, me, p, st);
    default: return launch_tm<TY, 8, kFine>(c, mq, me, p, st);
  }
}

}  // namespace f32
}  // namespace oprag
