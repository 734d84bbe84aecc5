// Lexical rerank of a dense top-N: the dense-first hybrid policy (Sec. 4.1
// Retrieval; Sec. 5.5).  Per query: BM25 of each candidate chunk through the
// sparse index, the BM25 maximum over the candidates, the weighted fusion of
// Sec. 4.4 and the ranked top-k of the fused scores.
//
// One CTA of four warps per query; a thread holds one or two candidates.  A
// candidate's BM25 is the sum of its query terms' weights: a dense term's
// weight is read from its row, a sparse term's is found by a binary search of
// the term's postings around the candidate's 1024-chunk tile (the table of the
// BM25 pass gives their range).  The searches' scattered reads of L2 bound the
// kernel, and their latency, so a thread searches kTermBatch terms at once.
// The sums and the fused score are formed exactly as in the BM25 pass and the
// fused search epilogue, so with every chunk a candidate the result equals the
// full hybrid search bit for bit.  A candidate's rank is counted against the
// other keys in shared memory (no chain of exchanges).  Measured on GB300,
// 32768 chunks, 1024 queries of 8 terms, 128 candidates: 21.7 us; a term's
// whole list searched instead, 24 us; one warp per query and one term at a
// time, 58 us.
#include "common.cuh"
#include "internal.h"

namespace oprag {

namespace {

constexpr int kRerankThreads = 128;
constexpr int kTermBatch = 8;

template <int E>
__global__ void __launch_bounds__(kRerankThreads)
rerank_kernel(SparseIndex sp, int ncand, const int64_t* __restrict__ cand_ids,
              const float* __restrict__ cand_scores, const int32_t* __restrict__ q_indptr,
              const int32_t* __restrict__ q_terms, float alpha, int k,
              int64_t* __restrict__ out_ids, float* __restrict__ out_scores) {
  __shared__ int term_slot[kTermBatch];            // dense row, -1: postings, -2: no term
  __shared__ int64_t term_row[kTermBatch];         // the term's tile_row
  __shared__ uint64_t keys[kRerankThreads * E];
  __shared__ float warp_max[kRerankThreads / 32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int qi = blockIdx.x;
  int32_t doc[E];
  float dense[E], lex[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int c = tid + e * kRerankThreads;
    const int64_t id = c < ncand ? cand_ids[static_cast<int64_t>(qi) * ncand + c] : -1;
    doc[e] = static_cast<int32_t>(id);
    dense[e] = c < ncand ? cand_scores[static_cast<int64_t>(qi) * ncand + c] : 0.f;
    lex[e] = 0.f;
  }
  const int t0 = q_indptr[qi], t1 = q_indptr[qi + 1];
  // Adds the dense and / or the sparse terms of one batch, dense terms first.
  auto add_batch = [&](int base, bool with_dense, bool with_sparse) {
    __syncthreads();        // the previous batch's term table has been read
    if (tid < kTermBatch) {
      int slot = -2;
      int64_t row = 0;
      const int32_t term = base + tid < t1 ? q_terms[base + tid] : -1;
      if (term >= 0 && term < sp.vocab) {
        slot = sp.dense_slot[term];
        row = sp.row_of(term);
      }
      term_slot[tid] = slot >= 0 ? (with_dense ? slot : -2) : (with_sparse ? slot : -2);
      term_row[tid] = row;
    }
    __syncthreads();
    // Dense weights, and each candidate's part of the sparse terms' postings:
    // those of the cell of the candidate's tile of chunks.
    float w[kTermBatch][E];
    int lo[kTermBatch][E], hi[kTermBatch][E], end[kTermBatch][E];
#pragma unroll
    for (int b = 0; b < kTermBatch; ++b) {
      const int slot = term_slot[b];
#pragma unroll
      for (int e = 0; e < E; ++e) {
        w[b][e] = 0.f;
        lo[b][e] = hi[b][e] = 0;
        if (doc[e] < 0) continue;
        if (slot >= 0) w[b][e] = __ldg(sp.dense_w + slot * sp.dense_ld + doc[e]);
        if (slot == -1) {
          const int32_t* tp = tile_cell(sp.tile_ptr, term_row[b], doc[e] / kBm25DocTile);
          lo[b][e] = __ldg(tp);
          hi[b][e] = __ldg(tp + 1);
        }
      }
    }
#pragma unroll
    for (int b = 0; b < kTermBatch; ++b)
#pragma unroll
      for (int e = 0; e < E; ++e) end[b][e] = hi[b][e];
    // Lower bound of each candidate in each range (chunks ascending).
    bool more = true;
    while (more) {
      more = false;
#pragma unroll
      for (int b = 0; b < kTermBatch; ++b) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
          if (lo[b][e] < hi[b][e]) {
            const int mid = lo[b][e] + ((hi[b][e] - lo[b][e]) >> 1);
            if (__ldg(&sp.post[mid].x) < doc[e]) lo[b][e] = mid + 1;
            else hi[b][e] = mid;
            more |= lo[b][e] < hi[b][e];
          }
        }
      }
    }
#pragma unroll
    for (int b = 0; b < kTermBatch; ++b)
#pragma unroll
      for (int e = 0; e < E; ++e) lex[e] += w[b][e];
#pragma unroll
    for (int b = 0; b < kTermBatch; ++b) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        w[b][e] = 0.f;
        if (lo[b][e] < end[b][e]) {
          const int2 pe = __ldg(sp.post + lo[b][e]);
          if (pe.x == doc[e]) w[b][e] = __int_as_float(pe.y);
        }
      }
    }
#pragma unroll
    for (int b = 0; b < kTermBatch; ++b)
#pragma unroll
      for (int e = 0; e < E; ++e) lex[e] += w[b][e];
  };
  // The BM25 pass's order: all dense terms, then all sparse terms.
  if (t1 - t0 <= kTermBatch) {
    add_batch(t0, true, true);
  } else {
    for (int base = t0; base < t1; base += kTermBatch) add_batch(base, true, false);
    for (int base = t0; base < t1; base += kTermBatch) add_batch(base, false, true);
  }
  // BM25 maximum over the candidates (BM25 is never negative).
  float m = 0.f;
#pragma unroll
  for (int e = 0; e < E; ++e)
    if (doc[e] >= 0) m = fmaxf(m, lex[e]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) warp_max[warp] = m;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kRerankThreads / 32; ++i) m = fmaxf(m, warp_max[i]);
  const float inv_max = m > 0.f ? 1.f / m : 0.f;
  const float a = alpha, b1 = 1.f - alpha;
  uint64_t key[E];
  int above[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    key[e] = doc[e] >= 0 ? make_key(fmaf(a, dense[e], b1 * (lex[e] * inv_max)),
                                    static_cast<uint32_t>(doc[e]))
                         : kEmptyKey;
    keys[tid + e * kRerankThreads] = key[e];
    above[e] = 0;
  }
  __syncthreads();
#pragma unroll 8
  for (int i = 0; i < ncand; ++i) {
    const uint64_t o = keys[i];
    // equal keys (only empty ones) rank by position
#pragma unroll
    for (int e = 0; e < E; ++e)
      above[e] += o > key[e] || (o == key[e] && i < tid + e * kRerankThreads) ? 1 : 0;
  }
#pragma unroll
  for (int e = 0; e < E; ++e)
    if (tid + e * kRerankThreads < ncand && above[e] < k) {
      const int64_t o = static_cast<int64_t>(qi) * k + above[e];
      out_ids[o] = key[e] == kEmptyKey ? -1 : static_cast<int64_t>(key_id(key[e]));
      out_scores[o] = key[e] == kEmptyKey ? -INFINITY : key_score(key[e]);
    }
}

}  // namespace

cudaError_t launch_rerank(const SparseIndex& sp, int q, int ncand, const int64_t* cand_ids,
                          const float* cand_scores, const int32_t* q_indptr,
                          const int32_t* q_terms, float alpha, int k, int64_t* out_ids,
                          float* out_scores, cudaStream_t st) {
  if (q <= 0) return cudaSuccess;
  if (ncand < 1 || ncand > kRerankMaxCand || k > ncand) return cudaErrorInvalidValue;
  if (ncand <= kRerankThreads)
    rerank_kernel<1><<<q, kRerankThreads, 0, st>>>(sp, ncand, cand_ids, cand_scores, q_indptr,
                                                   q_terms, alpha, k, out_ids, out_scores);
  else
    rerank_kernel<2><<<q, kRerankThreads, 0, st>>>(sp, ncand, cand_ids, cand_scores, q_indptr,
                                                   q_terms, alpha, k, out_ids, out_scores);
  return cudaGetLastError();
}

}  // namespace oprag
