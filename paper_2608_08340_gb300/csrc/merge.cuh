// Pieces of the merges of a query's partial lists (the global top-k reduction
// of Op_retrieve, Sec. 3.2 / Sec. 4.1 Retrieval).
#pragma once
#include "common.cuh"
#include "internal.h"

namespace oprag {

// Writes result o of the merge: a key's id (split into the corpus and the id
// within it for a search over two stacked corpora) and score, or the empty
// result (-1, -inf).
__device__ __forceinline__ void store_result(const ListSet& ls, int64_t* out_ids, float* out_scores,
                                             int64_t o, uint64_t key) {
  if (key == kEmptyKey) {
    out_ids[o] = -1;
    out_scores[o] = -INFINITY;
    if (ls.out_src != nullptr) ls.out_src[o] = -1;
    return;
  }
  int64_t id = static_cast<int64_t>(key_id(key));
  if (ls.out_src != nullptr) {
    const bool second = id >= ls.split;
    ls.out_src[o] = second ? 1 : 0;
    if (second) id -= ls.split;
  }
  out_ids[o] = id;
  out_scores[o] = key_score(key);
}

// Lists that exist for the query tile `tile` (see ListSet).
__device__ __forceinline__ int merge_list_count(const ListSet& ls, int tile) {
  int np = ls.P;
  if (ls.C > 0) {
    int c0 = static_cast<int>(static_cast<int64_t>(tile / ls.pair) * ls.C / ls.qt) - 1;
    c0 = c0 < 0 ? 0 : c0;
    np = min(ls.P, (ls.C - c0) * ls.sets);
  }
  return np;
}

// The smallest key that can still be among the query's k best: a counted
// floor f whose band counts up to it sum to k or more proves k real scores
// >= f, so every key of the top k has a score >= f (the key of score f with
// the largest id ranks below all of them).  kEmptyKey (admit all) without
// counted floors.
__device__ __forceinline__ uint64_t merge_floor_key(const ListSet& ls, int qi, int k) {
  if (ls.levels == nullptr || ls.level_cnt == nullptr) return kEmptyKey;
  int cnt[kLevels];
  float floors[kLevels];
#pragma unroll
  for (int i = 0; i < kLevels; ++i) {       // all loads before the first use
    const int64_t o = static_cast<int64_t>(qi) * kLevels + i;
    cnt[i] = ls.level_cnt[o];
    floors[i] = ls.levels[o];
  }
  int sum = 0;
#pragma unroll
  for (int i = 0; i < kLevels; ++i) {
    sum += cnt[i];
    if (sum >= k) return floors[i] > -INFINITY ? make_key(floors[i], kNoId) : kEmptyKey;
  }
  return kEmptyKey;
}

}  // namespace oprag
