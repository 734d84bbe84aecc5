// Tail of Op_embed (Sec. 4.3): the hidden states of each chunk or query of a
// padded batch are mean-pooled over its unmasked tokens and L2-normalised,
// and the vector is written in the index's dtype, ready for oprag_search.
//
// One CTA of 256 threads per batch row when the rows fill the SMs twice: thread
// i accumulates, in fp32, the 16-byte groups i, i + 256, ... of the row's dim
// elements over the tokens, the loads of kTokenBatch tokens in flight at once;
// a block reduction of the squared mean gives the norm.  HBM-bound: the
// unmasked hidden states are read once.
//
// Smaller batches leave SMs without loads in flight, so a cluster of S CTAs
// shares a row: CTA r takes the token blocks r, r + S, ... (a padded row's real
// tokens, which come first, are spread evenly), leaves its partial sums in
// shared memory and finishes one S-th of the row: it adds the S partial sums,
// in CTA order, through distributed shared memory, and the squared norms of
// the parts are exchanged the same way.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include "common.cuh"
#include "internal.h"

namespace oprag {

namespace {

constexpr int kPoolThreads = 256;
constexpr int kTokenBatch = 8;

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

template <typename TIn, int R, bool kSplit>
__global__ void __launch_bounds__(kPoolThreads)
embed_pool_kernel(const TIn* __restrict__ hidden, int tokens, int dim,
                  const uint8_t* __restrict__ mask, void* __restrict__ out, int out_bf16) {
  namespace cg = cooperative_groups;
  constexpr int N = Group<TIn>::kN;
  extern __shared__ __align__(16) float part[];   // this CTA's partial sums (dim)
  __shared__ float red[kPoolThreads / 32];
  __shared__ float part_ss;                       // squared norm of this CTA's part
  __shared__ int part_count;
  cg::cluster_group cluster = cg::this_cluster();
  const int S = kSplit ? static_cast<int>(cluster.num_blocks()) : 1;
  const int rank = kSplit ? static_cast<int>(cluster.block_rank()) : 0;
  const int b = blockIdx.x / S;
  const int groups = dim / N;
  const uint4* row0 = reinterpret_cast<const uint4*>(hidden + static_cast<int64_t>(b) * tokens * dim);
  const uint8_t* mrow = mask + static_cast<int64_t>(b) * tokens;
  float acc[R][N];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int i = 0; i < N; ++i) acc[r][i] = 0.f;
  // Tokens are added in increasing order (a fixed summation order for a given S).
  constexpr int TB = R <= 2 ? kTokenBatch : kTokenBatch / 2;   // register budget
  int count = 0;
  for (int t = rank * TB; t < tokens; t += S * TB) {
    bool m[TB];
#pragma unroll
    for (int u = 0; u < TB; ++u) {
      m[u] = t + u < tokens && mrow[t + u] != 0;
      count += static_cast<int>(m[u]);
    }
    uint4 v[TB][R];
#pragma unroll
    for (int u = 0; u < TB; ++u)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int g = threadIdx.x + r * kPoolThreads;
        v[u][r] = m[u] && g < groups ? __ldg(row0 + static_cast<int64_t>(t + u) * groups + g)
                                     : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
    for (int u = 0; u < TB; ++u)
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (m[u]) Group<TIn>::add(v[u][r], acc[r]);
  }
  // This CTA's part of the row: groups [g0, g1), its mean and squared norm.
  int g0 = 0, g1 = groups;
  if constexpr (kSplit) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int g = threadIdx.x + r * kPoolThreads;
      if (g < groups) {
#pragma unroll
        for (int i = 0; i < N; i += 4)
          *reinterpret_cast<float4*>(part + g * N + i) =
              make_float4(acc[r][i], acc[r][i + 1], acc[r][i + 2], acc[r][i + 3]);
      }
    }
    if (threadIdx.x == 0) part_count = count;
    cluster.sync();
    g0 = groups * rank / S;
    g1 = groups * (rank + 1) / S;
    count = 0;
    for (int s = 0; s < S; ++s) count += *cluster.map_shared_rank(&part_count, s);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int g = g0 + threadIdx.x + r * kPoolThreads;
#pragma unroll
      for (int i = 0; i < N; ++i) acc[r][i] = 0.f;
      if (g < g1) {
        for (int s = 0; s < S; ++s) {
          const float* p = cluster.map_shared_rank(part, s) + g * N;
#pragma unroll
          for (int i = 0; i < N; i += 4) {
            const float4 v = *reinterpret_cast<const float4*>(p + i);
            acc[r][i] += v.x;
            acc[r][i + 1] += v.y;
            acc[r][i + 2] += v.z;
            acc[r][i + 3] += v.w;
          }
        }
      }
    }
  }
  const float inv_c = count > 0 ? 1.f / static_cast<float>(count) : 0.f;
  float ss = 0.f;
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int i = 0; i < N; ++i) {
      acc[r][i] *= inv_c;
      ss = fmaf(acc[r][i], acc[r][i], ss);
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int w = 0; w < kPoolThreads / 32; ++w) t += red[w];
    part_ss = t;
  }
  float total = 0.f;
  if constexpr (kSplit) {
    cluster.sync();
    for (int s = 0; s < S; ++s) total += *cluster.map_shared_rank(&part_ss, s);
  } else {
    __syncthreads();
    total = part_ss;
  }
  const float norm = sqrtf(total);
  const float scale = count > 0 && norm > 0.f ? 1.f / norm : 0.f;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int g = g0 + threadIdx.x + r * kPoolThreads;
    if (g >= g1) continue;
    const int64_t e0 = static_cast<int64_t>(b) * dim + static_cast<int64_t>(g) * N;
    if (out_bf16) {
      __nv_bfloat16* o = static_cast<__nv_bfloat16*>(out) + e0;
#pragma unroll
      for (int i = 0; i < N; i += 2)
        *reinterpret_cast<__nv_bfloat162*>(o + i) =
            __floats2bfloat162_rn(acc[r][i] * scale, acc[r][i + 1] * scale);
    } else {
      float* o = static_cast<float*>(out) + e0;
#pragma unroll
      for (int i = 0; i < N; i += 4)
        *reinterpret_cast<float4*>(o + i) = make_float4(acc[r][i] * scale, acc[r][i + 1] * scale,
                                                        acc[r][i + 2] * scale, acc[r][i + 3] * scale);
    }
  }
  if constexpr (kSplit) cluster.sync();   // the peers have read this CTA's shared memory
}

// CTAs per row: as many as keep the batch within two CTAs per SM, at most
// eight (the portable cluster size) and one per block of tokens.  Measured on
// GB300 against one CTA per row, bf16: 1 x 512 x 4096 11.8 (41.0) us, 8 x 512 x
// 4096 13.1 (55.0) us, 64 x 512 x 4096 37.1 (82.0) us, 152 x 512 x 4096 72.5
// (88.5) us, 1 x 64 x 768 4.3 (5.7) us; 256 x 512 x 4096 stays at one (118 us;
// split in two 121 us).
int split_for(int batch, int tokens, int num_sms) {
  int s = 1;
  while (s < 8 && static_cast<int64_t>(batch) * 2 * s <= 2 * num_sms &&
         2 * s * kTokenBatch <= tokens)
    s *= 2;
  return s;
}

template <typename TIn, int R>
cudaError_t launch_r(const TIn* hidden, int batch, int tokens, int dim, const uint8_t* mask,
                     void* out, int out_bf16, int split, cudaStream_t st) {
  if (split == 1) {
    embed_pool_kernel<TIn, R, false><<<batch, kPoolThreads, 0, st>>>(hidden, tokens, dim, mask, out,
                                                                     out_bf16);
    return cudaGetLastError();
  }
  const size_t smem = static_cast<size_t>(dim) * sizeof(float);
  // (for every dim: with the static shared memory, 48 KB of sums are too many
  // for a kernel without the opt-in)
  static DeviceOnce once;
  const cudaError_t e =
      allow_smem(once, embed_pool_kernel<TIn, R, true>, R * kPoolThreads * 16 / sizeof(TIn) * sizeof(float));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(batch) * split);
  cfg.blockDim = dim3(kPoolThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = split;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, embed_pool_kernel<TIn, R, true>, hidden, tokens, dim, mask, out,
                            out_bf16);
}

template <typename TIn>
cudaError_t launch_typed(const void* hidden, int batch, int tokens, int dim, const uint8_t* mask,
                         void* out, int out_bf16, int split, cudaStream_t st) {
  const int groups = dim / Group<TIn>::kN;
  const int r = (groups + kPoolThreads - 1) / kPoolThreads;
  const TIn* h = static_cast<const TIn*>(hidden);
  if (r <= 1) return launch_r<TIn, 1>(h, batch, tokens, dim, mask, out, out_bf16, split, st);
  if (r <= 2) return launch_r<TIn, 2>(h, batch, tokens, dim, mask, out, out_bf16, split, st);
  if (r <= 4) return launch_r<TIn, 4>(h, batch, tokens, dim, mask, out, out_bf16, split, st);
  if (r <= 8) return launch_r<TIn, 8>(h, batch, tokens, dim, mask, out, out_bf16, split, st);
  return cudaErrorInvalidValue;
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
  const int split = split_for(batch, tokens, sms);
  return hidden_dtype == kBF16
             ? launch_typed<uint16_t>(hidden, batch, tokens, dim, mask, out, out_bf16, split, st)
             : launch_typed<float>(hidden, batch, tokens, dim, mask, out, out_bf16, split, st);
}

}  // namespace oprag
