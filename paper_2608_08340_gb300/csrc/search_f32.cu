// Host side of the fp32 search of search_f32.cuh: tile shape, corpus slices and
// scratch size.
#include <algorithm>

#include "search_f32.cuh"
#include "tensor_map.h"

namespace oprag {

using namespace f32;

namespace f32 {

extern template cudaError_t launch_ty<4, false>(const Config&, const CUtensorMap&,
                                                const CUtensorMap&, const Params&, cudaStream_t);
extern template cudaError_t launch_ty<4, true>(const Config&, const CUtensorMap&,
                                               const CUtensorMap&, const Params&, cudaStream_t);
extern template cudaError_t launch_ty<8, false>(const Config&, const CUtensorMap&,
                                                const CUtensorMap&, const Params&, cudaStream_t);
extern template cudaError_t launch_ty<8, true>(const Config&, const CUtensorMap&,
                                               const CUtensorMap&, const Params&, cudaStream_t);
extern template cudaError_t launch_ty<16, false>(const Config&, const CUtensorMap&,
                                                 const CUtensorMap&, const Params&, cudaStream_t);
extern template cudaError_t launch_ty<16, true>(const Config&, const CUtensorMap&,
                                                const CUtensorMap&, const Params&, cudaStream_t);

}  // namespace f32

namespace {

// Tile shape for q queries and k results, then (G > 0) everything else for G
// corpus slices.  The smallest TY that holds the batch in one tile: a warp
// covers four ty, so that a small TY reads each corpus row from shared memory
// fewer times and pads the batch less.  k > 32 keeps TY = 4, since candidate
// buffers of k + BN keys fit only 32 queries.  The queries are split evenly
// over the tiles.
Config config_for(const SearchShape& s, int G) {
  Config c{};
  c.TY = s.q <= 32 || s.k > 32 ? 4 : s.q <= 64 ? 8 : 16;
  c.qt = (s.q + 8 * c.TY - 1) / (8 * c.TY);
  const int per_tile = (s.q + c.qt - 1) / c.qt;
  c.TM = (per_tile + c.TY - 1) / c.TY;
  if (c.TY > 4) c.TM = std::max(c.TM, 5);     // smaller ones take the next smaller TY
  c.th = c.TY * c.TM;
  c.qt = (s.q + c.th - 1) / c.th;
  c.G = G;
  const int bn = kThreads / c.TY * kRowsPerThread;
  c.cap = std::min(kMaxCap, (s.k + bn + 31) / 32 * 32);
  // buffers, counts and floors, barriers and the abort word, ring alignment
  const size_t fixed = static_cast<size_t>(c.th) * (c.cap * sizeof(uint64_t) + 8) +
                       2 * kMaxStages * sizeof(uint64_t) + 16 + 1024;
  // A stage holds the corpus rows of the widest tile of a slice (short slices
  // then have more K blocks in flight) and the queries, in whole swizzle atoms.
  const int tx = kThreads / c.TY;
  const int64_t rows = (s.n + G - 1) / G;
  const int groups = static_cast<int>(std::min<int64_t>(kRowsPerThread, (rows + tx - 1) / tx));
  c.b_bytes = groups * tx * kRowBytes;
  c.stage = (c.b_bytes + c.th * kRowBytes + 1023) / 1024 * 1024;
  c.stages = static_cast<int>(std::min<size_t>(kMaxStages, (kSmemMax - fixed) / c.stage));
  c.smem = fixed + c.stages * static_cast<size_t>(c.stage);
  return c;
}

}  // namespace

// Corpus slices per query tile: one CTA per SM in as few full waves as
// possible (a second or third wave only when it fills the SMs better), at
// least 16 rows a slice.
int f32_slices(const SearchShape& s, int num_sms) {
  const Config c = config_for(s, 1);
  const int64_t most = std::max<int64_t>(1, (s.n + 15) / 16);
  int best = 1;
  double best_fill = 0.0;
  for (int w = 1; w <= 3; ++w) {
    const int64_t g = std::max<int64_t>(1, static_cast<int64_t>(w) * num_sms / c.qt);
    const int64_t ctas = g * c.qt, waves = (ctas + num_sms - 1) / num_sms;
    const double fill = static_cast<double>(ctas) / static_cast<double>(waves * num_sms);
    if (fill > best_fill + 0.05) {
      best_fill = fill;
      best = static_cast<int>(g);
    }
  }
  return static_cast<int>(std::min<int64_t>(best, most));
}

size_t f32_scratch_bytes(const SearchShape& s, int slices) {
  const Config c = config_for(s, slices);
  return sizeof(uint64_t) * static_cast<size_t>(c.qt) * slices * c.th * list_len_for(s.k);
}

cudaError_t launch_f32_search(const void* E, const void* Q, const SearchShape& s, const Fusion& fu,
                              void* scratch, int slices, ListSet* lists, cudaStream_t st,
                              uint64_t* qfloor, uint32_t gen, int* dev_err,
                              long long wait_limit) {
  const Config c = config_for(s, slices);
  CUtensorMap mq, me;
  if (!encode_rows_map(&mq, Q, s.q, s.d, c.th, kF32) ||
      !encode_rows_map(&me, E, s.n, s.d, kThreads / c.TY, kF32))
    return cudaErrorInvalidValue;
  Params p{};
  p.E = static_cast<const float*>(E);
  p.Q = static_cast<const float*>(Q);
  p.n = s.n;
  p.d = s.d;
  p.q = s.q;
  p.k = s.k;
  p.fu = fu;
  p.lists = static_cast<uint64_t*>(scratch);
  p.stride = list_len_for(s.k);
  p.cap = c.cap;
  p.stages = c.stages;
  p.stage = c.stage;
  p.b_bytes = c.b_bytes;
  p.qfloor = qfloor;
  p.gen = gen;
  p.dev_err = dev_err;
  p.wait_limit = wait_limit > 0 ? wait_limit : kWaitLimitCycles;
  lists->keys = p.lists;
  lists->P = slices;
  lists->TH = c.th;
  lists->stride = p.stride;
  lists->klen = p.stride;
  const bool fine = s.d <= kFineDim;
  if (c.TY == 4)
    return fine ? launch_ty<4, true>(c, mq, me, p, st) : launch_ty<4, false>(c, mq, me, p, st);
  if (c.TY == 8)
    return fine ? launch_ty<8, true>(c, mq, me, p, st) : launch_ty<8, false>(c, mq, me, p, st);
  return fine ? launch_ty<16, true>(c, mq, me, p, st) : launch_ty<16, false>(c, mq, me, p, st);
}

}  // namespace oprag
