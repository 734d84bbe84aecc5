// Tail of Op_embed (Sec. 4.3): the hidden states of each chunk or query of a
// padded batch are mean-pooled over its unmasked tokens and L2-normalised,
// and the vector is written in the index's dtype, ready for oprag_search.
//
// A row's result does not depend on the batch it comes in, nor on its padding:
// tokens belong to eight lanes by their position (sixteen consecutive tokens to a
// lane), each lane is summed in order, the lanes are added in order, and the
// squared norm is summed over the elements in a fixed order, however many CTAs
// share the row.
//
// One CTA of 256 threads per row when the rows fill the SMs twice: thread i
// accumulates, in fp32, the 16-byte groups i and i + 256 of the row's elements,
// lane by lane, the loads of eight or sixteen tokens in flight at once; a block
// reduction of the squared mean gives the norm.  HBM-bound: the unmasked hidden
// states are read once.
//
// Wide rows need more threads and smaller batches leave SMs without loads in
// flight: then a cluster of SD x ST CTAs shares a row, an SD-th of its elements
// and an ST-th of its lanes each (a padded row's real tokens, which come first,
// are spread evenly).  With ST > 1 a CTA leaves its lanes' sums in shared memory
// and finishes an ST-th of its elements: it adds the eight lanes through
// distributed shared memory.  Every CTA then forms the whole norm from the squared
// norms of the groups of all.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include "common.cuh"
#include "internal.h"

namespace oprag {

namespace {

constexpr int kPoolThreads = 256;
constexpr int kLanes = 8;               // partial sums of a row
// Consecutive tokens of a lane (with eight, rows that one CTA reads alone are read
// with more jumps: 256 x 512 x 4096 without padding 178 instead of 174 us).
constexpr int kTokenBlock = 16;
constexpr int kMaxShare = 2 * kPoolThreads;      // 16-byte groups of a token per CTA

template <typename TIn>
struct Group;                                   // one 16-byte group of inputs
template <>
struct Group<uint16_t> {
  static constexpr int kN = 8;
  __device__ static void add(const uint4& v, float (&a)[8]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      a[2 * i] += __uint_as_float(w[i] << 16);
      a[2 * i + 1] += __uint_as_float(w[i] & 0xFFFF0000u);
    }
  }
};
template <>
struct Group<float> {
  static constexpr int kN = 4;
  __device__ static void add(const uint4& v, float (&a)[4]) {
    a[0] += __uint_as_float(v.x);
    a[1] += __uint_as_float(v.y);
    a[2] += __uint_as_float(v.z);
    a[3] += __uint_as_float(v.w);
  }
};

template <int N>
__device__ __forceinline__ void store_floats(float* dst, const float (&a)[N]) {
#pragma unroll
  for (int i = 0; i < N; i += 4)
    *reinterpret_cast<float4*>(dst + i) = make_float4(a[i], a[i + 1], a[i + 2], a[i + 3]);
}

// R 16-byte groups per thread and token.  kSplit: a cluster of SD * ST CTAs per
// row, rank = dim part * ST + lane part.
template <typename TIn, int R, bool kSplit>
__global__ void __launch_bounds__(kPoolThreads, 2)
embed_pool_kernel(const TIn* __restrict__ hidden, int tokens, int dim,
                  const uint8_t* __restrict__ mask, void* __restrict__ out, int out_bf16, int SD,
                  int ST) {
  namespace cg = cooperative_groups;
  constexpr int N = Group<TIn>::kN;
  constexpr int kStep = 16 / R;                   // tokens loaded together
  static_assert(kTokenBlock % kStep == 0, "a step lies in one block");
  extern __shared__ __align__(16) float sums[];   // lanes' sums, then squares
  __shared__ float red[kPoolThreads / 32];
  __shared__ int part_count;
  cg::cluster_group cluster = cg::this_cluster();
  const int S = kSplit ? SD * ST : 1;
  const int rank = kSplit ? static_cast<int>(cluster.block_rank()) : 0;
  const int dpart = kSplit ? rank / ST : 0, tpart = kSplit ? rank % ST : 0;
  const int lane_step = kSplit ? ST : 1;
  const int b = blockIdx.x / S, wl = threadIdx.x & 31;
  const int groups = dim / N;
  const int share = kSplit ? (groups + SD - 1) / SD : groups;    // groups of a dim part
  const int first = dpart * share;
  const int mine = min(share, groups - first);    // (none when <= 0)
  const uint4* row = reinterpret_cast<const uint4*>(hidden + static_cast<int64_t>(b) * tokens * dim) +
                     first;
  const uint8_t* mrow = mask + static_cast<int64_t>(b) * tokens;
  float tot[R][N], acc[R][N];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int i = 0; i < N; ++i) tot[r][i] = 0.f;
  // The steps of this CTA's lanes, one after the other.  The mask of a step's
  // tokens, a byte per thread of the warp, is read a step ahead.
  const int lanes = min(kLanes, (tokens + kTokenBlock - 1) / kTokenBlock);   // that hold tokens
  auto read_mask = [&](int l, int t) -> uint32_t {
    return l < lanes && wl < kStep && t + wl < tokens ? mrow[t + wl] : 0u;
  };
  int count = 0;
  int l = tpart, t = l * kTokenBlock;
  uint32_t byte = read_mask(l, t);
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int i = 0; i < N; ++i) acc[r][i] = 0.f;
#pragma unroll 1
  while (l < lanes) {
    const uint32_t m = __ballot_sync(0xffffffffu, byte != 0);
    const int at = t, lane = l;
    t += kStep;
    if (t % kTokenBlock == 0) t += (kLanes - 1) * kTokenBlock;
    if (t >= tokens) {
      l += lane_step;
      t = l * kTokenBlock;
    }
    byte = read_mask(l, t);
    if (m != 0) {                                 // (no padding)
      count += __popc(m);
      uint4 v[kStep][R];
#pragma unroll
      for (int u = 0; u < kStep; ++u)
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int g = threadIdx.x + r * kPoolThreads;
          v[u][r] = ((m >> u) & 1u) && g < mine ? __ldg(row + static_cast<int64_t>(at + u) * groups + g)
                                                : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
      for (int u = 0; u < kStep; ++u)
#pragma unroll
        for (int r = 0; r < R; ++r)
          if ((m >> u) & 1u) Group<TIn>::add(v[u][r], acc[r]);
    }
    if (l == lane) continue;
    // The lane is complete.
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int g = threadIdx.x + r * kPoolThreads;
      if (kSplit && ST > 1) {
        if (g < mine) store_floats(sums + (lane / ST * share + g) * N, acc[r]);
      }
#pragma unroll
      for (int i = 0; i < N; ++i) {
        if (!kSplit || ST == 1) tot[r][i] += acc[r][i];
        acc[r][i] = 0.f;
      }
    }
  }
  // The groups that this CTA finishes: [g0, g1) of its dim part.
  int g0 = 0, g1 = mine;
  const int finish = kSplit ? (share + ST - 1) / ST : share;
  if constexpr (kSplit) {
    if (ST > 1) {
      if (threadIdx.x == 0) part_count = count;
      cluster.sync();
      g0 = tpart * finish;
      g1 = min(mine, g0 + finish);
      count = 0;
      for (int p = 0; p < ST; ++p) count += *cluster.map_shared_rank(&part_count, dpart * ST + p);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int g = g0 + threadIdx.x + r * kPoolThreads;
        if (g >= g1) continue;
        float4 x[kLanes][N / 4];
#pragma unroll
        for (int l = 0; l < kLanes; ++l) {
          const float4* p = reinterpret_cast<const float4*>(
              cluster.map_shared_rank(sums, dpart * ST + l % ST) + (l / ST * share + g) * N);
#pragma unroll
          for (int i = 0; i < N / 4; ++i)
            x[l][i] = l < lanes ? p[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int l = 0; l < kLanes; ++l)
#pragma unroll
          for (int i = 0; i < N; i += 4) {
            tot[r][i] += x[l][i / 4].x;
            tot[r][i + 1] += x[l][i / 4].y;
            tot[r][i + 2] += x[l][i / 4].z;
            tot[r][i + 3] += x[l][i / 4].w;
          }
      }
    }
  }
  const float inv_c = count > 0 ? 1.f / static_cast<float>(count) : 0.f;
  // The squared norm: each group's squares in order, thread i adds the row's
  // groups i, i + 256, ..., then warps and the CTA are added up.
  float ss = 0.f;
  float* squares = sums + (kSplit && ST > 1 ? kLanes / ST * share * N : 0);   // a float per group
#pragma unroll
  for (int r = 0; r < R; ++r) {
    float sq = 0.f;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      tot[r][i] *= inv_c;
      sq = fmaf(tot[r][i], tot[r][i], sq);
    }
    if constexpr (kSplit) {
      const int g = g0 + threadIdx.x + r * kPoolThreads;
      if (g < g1) squares[g - g0] = sq;
    } else {
      ss += sq;
    }
  }
  if constexpr (kSplit) {
    cluster.sync();
#pragma unroll 4
    for (int g = threadIdx.x; g < groups; g += kPoolThreads) {
      const int d = g / share, q = (g - d * share) / finish;
      ss += cluster.map_shared_rank(squares, d * ST + q)[g - d * share - q * finish];
    }
    cluster.barrier_arrive();             // this CTA reads no more
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if (wl == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  float total = 0.f;
#pragma unroll
  for (int w = 0; w < kPoolThreads / 32; ++w) total += red[w];
  const float norm = sqrtf(total);
  const float scale = count > 0 && norm > 0.f ? 1.f / norm : 0.f;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int g = g0 + threadIdx.x + r * kPoolThreads;
    if (g >= g1) continue;
    const int64_t o0 = static_cast<int64_t>(b) * dim + static_cast<int64_t>(first + g) * N;
    if (out_bf16) {
      __nv_bfloat16* o = static_cast<__nv_bfloat16*>(out) + o0;
#pragma unroll
      for (int i = 0; i < N; i += 2)
        *reinterpret_cast<__nv_bfloat162*>(o + i) =
            __floats2bfloat162_rn(tot[r][i] * scale, tot[r][i + 1] * scale);
    } else {
#pragma unroll
      for (int i = 0; i < N; ++i) tot[r][i] *= scale;
      store_floats(static_cast<float*>(out) + o0, tot[r]);
    }
  }
  if constexpr (kSplit) cluster.barrier_wait();   // nor do the peers read from it
}

// Parts of a row's elements, so that a CTA takes two groups a thread at most, and
// of its lanes: as many as keep the batch within two CTAs per SM, with eight
// CTAs (the portable cluster size) and one per 8 tokens at most.
// Measured on GB300 with events (a pair takes 6 us of it), in brackets one CTA
// per row and one chain of tokens, bf16: 1 x 512 x 4096 21 (85) us, 64 x 512 x 4096
// with padding 48 (92) us, 152 x 512 x 4096 121 (116) us, with padding 90 (101) us,
// 1 x 64 x 768 10 (13) us, 128 x 256 x 768 23 (37) us, 512 x 1024 x 512 158 (205)
// us, 20 x 512 x 8192 38 (148) us, 4 x 300 x 16384 38 (132) us; 256 x 512 x 4096
// stays at one CTA (133, 135 us).
struct Split {
  int dim, lanes;
};

Split split_for(int batch, int tokens, int groups, int num_sms) {
  Split s{1, 1};
  while (s.dim < 8 && groups > s.dim * kMaxShare) s.dim *= 2;
  while (s.dim * s.lanes < 8 && static_cast<int64_t>(batch) * 2 * s.dim * s.lanes <= 2 * num_sms &&
         16 * s.lanes <= tokens)
    s.lanes *= 2;
  return s;
}

template <typename TIn, int R>
cudaError_t launch_r(const TIn* hidden, int batch, int tokens, int dim, const uint8_t* mask,
                     void* out, int out_bf16, Split s, cudaStream_t st) {
  if (s.dim * s.lanes == 1) {
    embed_pool_kernel<TIn, R, false><<<batch, kPoolThreads, 0, st>>>(hidden, tokens, dim, mask, out,
                                                                     out_bf16, 1, 1);
    return cudaGetLastError();
  }
  // the lanes' sums of a part, and a float per group
  constexpr int kGroupBytes = Group<TIn>::kN * sizeof(float);
  const int lanes_bytes = s.lanes > 1 ? kLanes / s.lanes * kGroupBytes : 0;
  static DeviceOnce once;
  const cudaError_t e = allow_smem(once, embed_pool_kernel<TIn, R, true>,
                                   R * kPoolThreads * (kLanes / 2 * kGroupBytes + sizeof(float)));
  if (e != cudaSuccess) return e;
  const size_t share = (dim / Group<TIn>::kN + s.dim - 1) / s.dim;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(batch) * s.dim * s.lanes);
  cfg.blockDim = dim3(kPoolThreads);
  cfg.dynamicSmemBytes = share * (lanes_bytes + sizeof(float));
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = s.dim * s.lanes;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, embed_pool_kernel<TIn, R, true>, hidden, tokens, dim, mask, out,
                            out_bf16, s.dim, s.lanes);
}

template <typename TIn>
cudaError_t launch_typed(const void* hidden, int batch, int tokens, int dim, const uint8_t* mask,
                         void* out, int out_bf16, int num_sms, cudaStream_t st) {
  const int groups = dim / Group<TIn>::kN;
  const Split s = split_for(batch, tokens, groups, num_sms);
  const int share = (groups + s.dim - 1) / s.dim;
  if (share > kMaxShare) return cudaErrorInvalidValue;
  const TIn* h = static_cast<const TIn*>(hidden);
  if (share <= kPoolThreads)
    return launch_r<TIn, 1>(h, batch, tokens, dim, mask, out, out_bf16, s, st);
  return launch_r<TIn, 2>(h, batch, tokens, dim, mask, out, out_bf16, s, st);
}

}  // namespace

cudaError_t launch_embed_pool(int hidden_dtype, const void* hidden, int batch, int tokens, int dim,
                              const uint8_t* mask, int out_dtype, void* out, cudaStream_t st) {
  if (batch <= 0) return cudaSuccess;
  const int out_bf16 = out_dtype == kBF16 ? 1 : 0;
  int dev = 0, sms = 1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  return hidden_dtype == kBF16
             ? launch_typed<uint16_t>(hidden, batch, tokens, dim, mask, out, out_bf16, sms, st)
             : launch_typed<float>(hidden, batch, tokens, dim, mask, out, out_bf16, sms, st);
}

}  // namespace oprag
