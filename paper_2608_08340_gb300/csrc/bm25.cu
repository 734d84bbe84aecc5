// Lexical half of the hybrid search (Sec. 4.4): BM25 of every (query, chunk)
// pair through inverted postings, touching only the chunks that hold a query
// term and giving the same scores as a scan of the whole corpus.
//
// The per-posting weight idf(t) * tf (k1 + 1) / (tf + k1 (1 - b + b |d| / avgdl))
// does not depend on the query, so it is computed once on the device when the
// sparse side is attached; a query's BM25 for chunk d is then the sum of the
// weights of its terms' postings at d (a repeated term counts again).
//
// Work items are (tile of 1024 chunks, query), tile-major, in one contiguous
// share per CTA; a warp takes one item.  Its lanes hold the tile's sums in
// registers while the query's dense terms (held by more than half of the
// chunks, stored as rows of weights with zeros where absent) are added, then
// the sums go to the warp's row in shared memory, where the sparse terms
// scatter their postings (each chunk at most once per term, so one term's adds
// never collide); a table built with the postings gives where each sparse
// term's postings enter the tile.  The order -- dense terms in the query's
// order, then sparse terms in the query's order -- is the order of the rerank
// too, so both give the same sums.  Adding a zero weight leaves an fp32 sum
// unchanged.  The warp writes the tile's row of the q x n BM25 matrix and
// folds the tile maximum into the per-query maximum that normalises the
// lexical score.
//
// A query holds about four of the thirty or so dense terms, so with many queries
// (kFewQueries) a CTA looks the terms of a tile's queries up together and copies
// that tile of all dense rows to shared
// memory once and the items read them there: 1024 queries on 32768 chunks read
// 19 MB of dense rows from L2 instead of 530 MB.  What is left is the write of
// the block (134 MB) and the shared-memory passes (about 30 KB per item).
// Measured on GB300 (8 Zipf terms a query): 64 us instead of 88 us for one CTA
// per query and tile of 8192 chunks with its sums in shared memory.
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace oprag {

namespace {

constexpr int kDocTile = kBm25DocTile;
constexpr int kBm25Warps = 20;
constexpr int kBm25Threads = kBm25Warps * 32;
constexpr int kVec = kDocTile / 4 / 32;      // float4 groups of a tile per lane
constexpr int kPostBatch = 4;                // postings per lane and chunk
constexpr int kChunks = 4;                   // chunks loaded before their adds
// Dense rows kept in shared memory (4 KB each), beside the warps' rows: the
// commonest terms of a Zipf corpus; others are read from L2.
constexpr int kBm25MaxRows = 29;
// Queries of a tile in one CTA from which its dense rows are copied: a query
// reads about four of them, so below that direct reads move fewer bytes.
constexpr int kStageMinQueries = 8;
// Queries up to which a warp takes its item's terms and dense rows by itself, so
// that no barrier and no tile boundary holds the other warps up.  Measured, 500000
// / 32768 chunks: 4 queries 15 / 12 us against 31 / 12 us, 16 queries 31 / 12
// against 54 / 16, 64 queries 79 / 14 against 98 / 19, 128 queries 142 / 19
// against 157 / 22; from 192 on 500000 chunks take the same (204, 204 us), and with
// a thousand queries the copies of the dense rows tell (see above).
constexpr int kFewQueries = 160;
// Queries and terms of one batch whose lookups are done together.
constexpr int kBatchQueries = 120;
constexpr int kBatchTerms = 2048;

// One lane's term of a query: its dense row (-1: postings [lo, hi) of the
// tile's cell, -2: none).
struct TermSlot {
  int slot, lo, hi;
};

__device__ __forceinline__ TermSlot load_term(const SparseIndex& sp,
                                              const int32_t* __restrict__ q_terms, int ti, int t1,
                                              int tile) {
  TermSlot t{-2, 0, 0};
  const int32_t term = ti < t1 ? q_terms[ti] : -1;
  if (term >= 0 && term < sp.vocab) {
    const int64_t row = sp.row_of(term);
    t.slot = sp.dense_slot[term];
    const int32_t* tp = tile_cell(sp.tile_ptr, row, tile);
    t.lo = tp[0];
    t.hi = tp[1];
  }
  return t;
}

template <bool kFew>
__global__ void __launch_bounds__(kBm25Threads, 1)
bm25_matrix_kernel(SparseIndex sp, int64_t n, const int32_t* __restrict__ q_indptr,
                   const int32_t* __restrict__ q_terms, int q, float* __restrict__ out, int64_t ld,
                   float* __restrict__ out_max, int rows) {
  extern __shared__ __align__(16) float smem_b[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* row = smem_b + warp * kDocTile;
  float4* row4 = reinterpret_cast<float4*>(row);
  // Term lookups of the batch, by raw term position, and its query offsets.
  int* t_slot = reinterpret_cast<int*>(smem_b + kBm25Warps * kDocTile);
  int* t_lo = t_slot + kBatchTerms;
  int* t_hi = t_lo + kBatchTerms;
  int* q_ptr = t_hi + kBatchTerms;
  float4* dense4 = reinterpret_cast<float4*>(q_ptr + kBatchQueries + 8);
  const int64_t total = static_cast<int64_t>(sp.ntiles) * q;
  const int64_t w1 = total * (blockIdx.x + 1) / gridDim.x;
  int loaded = -1;             // tile whose dense rows are in shared memory
  for (int64_t w = total * blockIdx.x / gridDim.x; w < w1;) {
    // A batch: queries of one tile, or with few queries the share's next items,
    // a warp each.
    const int64_t wa = w;
    const int tile_a = static_cast<int>(w / q);
    const int qa = static_cast<int>(w - static_cast<int64_t>(tile_a) * q);
    const int q_tile = static_cast<int>(min(static_cast<int64_t>(q), qa + (w1 - w)));
    const int items = kFew ? static_cast<int>(min(w1 - w, static_cast<int64_t>(kBm25Warps)))
                           : min(q_tile - qa, kBatchQueries);
    w += items;
    int staged = 0, tb = 0;
    bool listed = false;       // else the terms are looked up per item
    if constexpr (!kFew) {
      const int64_t d0 = static_cast<int64_t>(tile_a) * kDocTile;
      const int nv = static_cast<int>((min(n - d0, static_cast<int64_t>(kDocTile)) + 3) / 4);
      __syncthreads();         // the previous batch has been computed
      for (int i = threadIdx.x; i <= items; i += kBm25Threads) q_ptr[i] = q_indptr[qa + i];
      if (loaded != tile_a && q_tile - qa >= kStageMinQueries) {
        for (int i = threadIdx.x; i < rows * (kDocTile / 4); i += kBm25Threads) {
          const int r = i / (kDocTile / 4), v = i % (kDocTile / 4);
          if (v < nv)
            dense4[i] = __ldg(reinterpret_cast<const float4*>(sp.dense_w + r * sp.dense_ld + d0) + v);
        }
        loaded = tile_a;
      }
      staged = loaded == tile_a ? rows : 0;
      __syncthreads();
      tb = q_ptr[0];
      listed = q_ptr[items] - tb <= kBatchTerms;
      if (listed) {
        for (int i = threadIdx.x; i < q_ptr[items] - tb; i += kBm25Threads) {
          const TermSlot t = load_term(sp, q_terms, tb + i, tb + i + 1, tile_a);
          t_slot[i] = t.slot;
          t_lo[i] = t.lo;
          t_hi[i] = t.hi;
        }
        __syncthreads();
      }
    }
    for (int item = warp; item < items; item += kBm25Warps) {
      const int tile = kFew ? static_cast<int>((wa + item) / q) : tile_a;
      const int qi = kFew ? static_cast<int>((wa + item) % q) : qa + item;
      const int64_t d0 = static_cast<int64_t>(tile) * kDocTile;
      const int first_doc = static_cast<int>(d0);
      const int nv = static_cast<int>((min(n - d0, static_cast<int64_t>(kDocTile)) + 3) / 4);
      const int b0 = kFew ? q_indptr[qi] : q_ptr[item];
      const int b1 = kFew ? q_indptr[qi + 1] : q_ptr[item + 1];
      auto term = [&](int ti, int t1) {
        if (!listed) return load_term(sp, q_terms, ti, t1, tile);
        return ti < t1 ? TermSlot{t_slot[ti - tb], t_lo[ti - tb], t_hi[ti - tb]} : TermSlot{-2, 0, 0};
      };
      float4 acc[kVec];
#pragma unroll
      for (int u = 0; u < kVec; ++u) acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      // Dense terms, 32 of the query's terms at a time.
      for (int base = b0; base < b1; base += 32) {
        const int slot = term(base + lane, b1).slot;
        for (uint32_t m = __ballot_sync(0xffffffffu, slot >= 0); m != 0; m &= m - 1) {
          const int s = __shfl_sync(0xffffffffu, slot, __ffs(m) - 1);
          float4 x[kVec];
          if (s < staged) {
#pragma unroll
            for (int u = 0; u < kVec; ++u) x[u] = dense4[s * (kDocTile / 4) + lane + 32 * u];
          } else {
            const float4* src = reinterpret_cast<const float4*>(sp.dense_w + s * sp.dense_ld + d0);
#pragma unroll
            for (int u = 0; u < kVec; ++u)
              x[u] = lane + 32 * u < nv ? __ldg(src + lane + 32 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
          }
#pragma unroll
          for (int u = 0; u < kVec; ++u) {
            acc[u].x += x[u].x;
            acc[u].y += x[u].y;
            acc[u].z += x[u].z;
            acc[u].w += x[u].w;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kVec; ++u) row4[lane + 32 * u] = acc[u];
      __syncwarp();
      // Sparse terms: the postings go in chunks of 32 kPostBatch of one term;
      // kChunks chunks (of one or several terms) are loaded together, then
      // added one after the other.
      for (int base = b0; base < b1; base += 32) {
        const TermSlot t = term(base + lane, b1);
        uint32_t m = __ballot_sync(0xffffffffu, t.slot == -1 && t.lo < t.hi);
        int p = 0, hi = 0;       // the current term's postings still to load
        while (p < hi || m != 0) {
          int2 e[kChunks][kPostBatch];
#pragma unroll
          for (int h = 0; h < kChunks; ++h) {
            if (p >= hi && m != 0) {
              const int src = __ffs(m) - 1;
              p = __shfl_sync(0xffffffffu, t.lo, src);
              hi = __shfl_sync(0xffffffffu, t.hi, src);
              m &= m - 1;
            }
#pragma unroll
            for (int u = 0; u < kPostBatch; ++u) {
              const int i = p + lane + 32 * u;
              e[h][u] = i < hi ? __ldg(sp.post + i) : make_int2(-1, 0);
            }
            p += 32 * kPostBatch;
          }
#pragma unroll
          for (int h = 0; h < kChunks; ++h) {
            // (one term's chunks are distinct: all reads before the writes;
            // chunk -1 and a wider cell's other tiles are outside the row)
            float v[kPostBatch];
#pragma unroll
            for (int u = 0; u < kPostBatch; ++u) {
              const uint32_t at = static_cast<uint32_t>(e[h][u].x) - static_cast<uint32_t>(first_doc);
              if (at < kDocTile) v[u] = row[at];
            }
#pragma unroll
            for (int u = 0; u < kPostBatch; ++u) {
              const uint32_t at = static_cast<uint32_t>(e[h][u].x) - static_cast<uint32_t>(first_doc);
              if (at < kDocTile) row[at] = v[u] + __int_as_float(e[h][u].y);
            }
            __syncwarp();
          }
        }
      }
      float top = 0.f;
      float4* orow = out != nullptr
                         ? reinterpret_cast<float4*>(out + static_cast<int64_t>(qi) * ld + d0)
                         : nullptr;
#pragma unroll
      for (int u = 0; u < kVec; ++u) {
        if (lane + 32 * u < nv) {
          const float4 v = row4[lane + 32 * u];
          if (orow != nullptr) orow[lane + 32 * u] = v;
          top = fmaxf(fmaxf(top, fmaxf(v.x, v.y)), fmaxf(v.z, v.w));
        }
      }
      // BM25 is never negative, so the float order equals the int order.
      const int bits = __reduce_max_sync(0xffffffffu, __float_as_int(top));
      if (lane == 0 && bits > 0) atomicMax(reinterpret_cast<int*>(out_max + qi), bits);
      __syncwarp();            // the row is read before the next item overwrites it
    }
  }
}

// One thread per query, by the classes of its terms: the head terms' counts
// (as bf16, twice: against the high and the low half of the split weights),
// its first kLexMidReg distinct mid rows and first kLexRegTerms distinct tail
// terms that have postings, each with its multiplicity, in first-occurrence
// order, and the raw term index where a further distinct one first occurs
// (the end of the query's terms if none does).
__global__ void lex_prep_kernel(const int32_t* __restrict__ lex_class,
                                const int64_t* __restrict__ post_ptr, int vocab,
                                const int32_t* __restrict__ q_indptr,
                                const int32_t* __restrict__ q_terms, int q, LexPrep out) {
  const int qi = blockIdx.x * blockDim.x + threadIdx.x;
  if (qi >= q) return;
  float cnt[kLexHeadTerms];
#pragma unroll
  for (int i = 0; i < kLexHeadTerms; ++i) cnt[i] = 0.f;
  const int t0 = q_indptr[qi], t1 = q_indptr[qi + 1];
  int4* tails = out.terms + static_cast<int64_t>(qi) * kLexRegTerms;
  int2* mids = out.mid + static_cast<int64_t>(qi) * kLexMidReg;
  int nt = 0, nm = 0, first_ovf = t1;
  for (int i = t0; i < t1; ++i) {
    const int32_t term = q_terms[i];
    if (term < 0 || term >= vocab) continue;
    const int c = lex_class[term];
    if (c >= 0) {
#pragma unroll
      for (int s = 0; s < kLexHeadTerms; ++s) cnt[s] += s == c ? 1.f : 0.f;
    } else if (c <= -2) {
      const int row = -2 - c;
      int j = 0;
      while (j < nm && mids[j].x != row) ++j;
      if (j < nm) mids[j].y = __float_as_int(__int_as_float(mids[j].y) + 1.f);
      else if (nm < kLexMidReg) mids[nm++] = make_int2(row, __float_as_int(1.f));
      else if (first_ovf == t1) first_ovf = i;
    } else {
      const int64_t a = post_ptr[term], b = post_ptr[term + 1];
      if (a >= b) continue;
      int j = 0;
      while (j < nt && tails[j].w != term) ++j;
      if (j < nt)
        tails[j].z = __float_as_int(__int_as_float(tails[j].z) + 1.f);
      else if (nt < kLexRegTerms)
        tails[nt++] = make_int4(static_cast<int>(a), static_cast<int>(b), __float_as_int(1.f), term);
      else if (first_ovf == t1)
        first_ovf = i;
    }
  }
  out.term_cnt[qi] = nt;
  out.mid_cnt[qi] = nm;
  out.ovf[qi] = first_ovf;
  __nv_bfloat16* row = static_cast<__nv_bfloat16*>(out.qcount) + static_cast<int64_t>(qi) * kLexK;
#pragma unroll
  for (int s = 0; s < kLexHeadTerms; ++s) {
    row[s] = __float2bfloat16_rn(cnt[s]);
    row[kLexHeadTerms + s] = __float2bfloat16_rn(cnt[s]);
  }
}

}  // namespace

cudaError_t launch_lex_prep(const int32_t* lex_class, const int64_t* post_ptr, int vocab,
                            const int32_t* q_indptr, const int32_t* q_terms, int q,
                            const LexPrep& out, cudaStream_t st) {
  if (q <= 0) return cudaSuccess;
  lex_prep_kernel<<<(q + 127) / 128, 128, 0, st>>>(lex_class, post_ptr, vocab, q_indptr, q_terms,
                                                   q, out);
  return cudaGetLastError();
}

cudaError_t launch_bm25_matrix(const SparseIndex& sp, int64_t n, const int32_t* q_indptr,
                               const int32_t* q_terms, int q, float* out, int64_t ld,
                               float* out_max, int num_sms, cudaStream_t st) {
  if (q <= 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(out_max, 0, sizeof(float) * q, st);
  if (e != cudaSuccess) return e;
  const int rows = std::min(sp.dense_rows, kBm25MaxRows);
  constexpr size_t kRow = kDocTile * sizeof(float);
  constexpr size_t kFixed = kBm25Warps * kRow +
                            (3 * kBatchTerms + kBatchQueries + 8) * sizeof(int);
  // One CTA per SM (its shared memory), fewer when there are fewer items.
  const int64_t items = static_cast<int64_t>(sp.ntiles) * q;
  const int grid = static_cast<int>(std::min<int64_t>(items, num_sms));
  if (q <= kFewQueries) {
    static DeviceOnce once;
    e = allow_smem(once, bm25_matrix_kernel<true>, kFixed);
    if (e != cudaSuccess) return e;
    bm25_matrix_kernel<true><<<grid, kBm25Threads, kFixed, st>>>(sp, n, q_indptr, q_terms, q, out,
                                                                 ld, out_max, 0);
    return cudaGetLastError();
  }
  static DeviceOnce once;
  e = allow_smem(once, bm25_matrix_kernel<false>, kFixed + kBm25MaxRows * kRow);
  if (e != cudaSuccess) return e;
  bm25_matrix_kernel<false><<<grid, kBm25Threads, kFixed + rows * kRow, st>>>(
      sp, n, q_indptr, q_terms, q, out, ld, out_max, rows);
  return cudaGetLastError();
}

}  // namespace oprag
