// k_post.cu - covariance post-step of Sec. 3.2: the sketch of Q~, the
// product with its diagonal set to zero, from the sketch of the product.
// Entry (i, i) of AB enters the sketch of repetition t at bucket
// (h1_t(i) + h2_t(i)) mod b with sign s1_t(i) s2_t(i) (the decomposed
// splitting and sign functions of Sec. 2.2), so removing it is one
// subtraction per (i, t).  (AB)_ii = sum_k A_ik B_ki: a cluster of up to 8
// blocks owns 32 consecutive i and its warps take the inner indices in turn (A
// read down its columns, A_ik at A[k lda + i], and B along its rows, B_ki at
// B[k ldb + i]: 32 consecutive i per warp load), then the partial sums of each
// i are added in FP64 in warp and block order.  1500 positions of 3000 inner
// indices in FP32 took 85 us with one block per 32 positions (47 of the 152
// SMs) and FP64 terms (2 a clock and SM, and as slow to convert): 22 us.
#include <algorithm>
#include <cooperative_groups.h>

#include "cms_internal.h"
#include "sketch_generic.cuh"

namespace cms {
namespace {

__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ double to_f64(T v) { return static_cast<double>(v); }
template <> __device__ __forceinline__ double to_f64<__nv_bfloat16>(__nv_bfloat16 v) {
  return static_cast<double>(__bfloat162float(v));
}

// The sum of A_ik B_ki over k = k0, k0 + step, ...: FP64 storage in FP64, FP32
// and BF16 storage as the sum and its error in FP32 (products split by a fused
// multiply-add, additions by Knuth's two-sum; 48 bits, of which the sketch
// keeps 24), in FP64 where a value leaves FP32's range on the way: an infinity,
// or a sum so small that products may have underflowed (each loses at most 2^-149
// then, 2^31 of them 2^-118).
template <typename T>
__device__ __forceinline__ double diag_part(const T* A, int64_t lda, const T* B, int64_t ldb, int64_t k0, int64_t n2,
                                            int64_t step) {
  if constexpr (sizeof(T) < 8) {
    float s = 0.f, e = 0.f;
#pragma unroll 8
    for (int64_t k = k0; k < n2; k += step) {
      const float x = to_f32(A[k * lda]), y = to_f32(B[k * ldb]);
      const float p = x * y, pe = fmaf(x, y, -p);
      const float t = s + p, v = t - s;
      e += ((s - (t - v)) + (p - v)) + pe;
      s = t;
    }
    if (fabsf(s) >= 0x1p-70f && isfinite(s) && isfinite(e)) return static_cast<double>(s) + static_cast<double>(e);
    if (s == 0.f && e == 0.f) {   // nothing to add, or all of it underflowed
      bool any = false;
#pragma unroll 8
      for (int64_t k = k0; k < n2; k += step) any |= to_f32(A[k * lda]) != 0.f && to_f32(B[k * ldb]) != 0.f;
      if (!any) return 0.0;
    }
  }
  double s = 0.0;
#pragma unroll 4
  for (int64_t k = k0; k < n2; k += step) s = fma(to_f64(A[k * lda]), to_f64(B[k * ldb]), s);
  return s;
}

template <typename T>
__global__ void __launch_bounds__(1024)
k_remove_diagonal(const T* __restrict__ A, int64_t lda, const T* __restrict__ B, int64_t ldb, int64_t m,
                  int64_t n2, const uint32_t* __restrict__ hs, int64_t n, int d, int64_t b,
                  float* __restrict__ c) {
  __shared__ double part[32][33];
  __shared__ double sum[32];
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int rank = static_cast<int>(cluster.block_rank()), ranks = static_cast<int>(cluster.num_blocks());
  const int64_t i = static_cast<int64_t>(blockIdx.y) * 32 + lane;
  part[w][lane] = i < m ? diag_part(A + i, lda, B + i, ldb, rank * 32 + w, n2, 32 * ranks) : 0.0;
  __syncthreads();
  if (w == 0) {
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < 32; ++q) s += part[q][lane];
    sum[lane] = s;
  }
  cluster.sync();
  if (rank == 0 && w == 0 && i < m) {
    double diag = sum[lane];
    for (int q = 1; q < ranks; ++q) diag += cluster.map_shared_rank(sum, q)[lane];
    for (int t = 0; t < d; ++t) {
      const uint32_t w1 = hs[(static_cast<size_t>(t) * 2 + 0) * n + i];
      const uint32_t w2 = hs[(static_cast<size_t>(t) * 2 + 1) * n + i];
      uint64_t z = static_cast<uint64_t>(w1 & kBucketMask) + (w2 & kBucketMask);
      if (z >= static_cast<uint64_t>(b)) z -= static_cast<uint64_t>(b);
      const double sv = ((w1 ^ w2) >> 31) ? -diag : diag;
      atomicAdd(&c[static_cast<size_t>(t) * b + z], static_cast<float>(-sv));
    }
  }
  cluster.sync();   // the other blocks' sums are read
}

template <typename T>
cudaError_t launch_diagonal(const void* A, int64_t lda, const void* B, int64_t ldb, int64_t m, int64_t n2,
                            const cms_hashes* h, float* c, cudaStream_t s) {
  const int64_t cols = (m + 31) / 32;
  int ranks = 1;
  while (ranks < 8 && cols * ranks * 2 <= 2 * 152 && n2 >= 256 * ranks) ranks *= 2;
  cudaLaunchConfig_t cfg{};
  cfg.blockDim = dim3(1024);
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = ranks;
  at.val.clusterDim.y = 1;
  at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  // (65535 rows of blocks a launch: 2^21 positions)
  const T* a = static_cast<const T*>(A);
  const T* bp = static_cast<const T*>(B);
  for (int64_t i0 = 0; i0 < m; i0 += 65535 * 32) {
    cfg.gridDim = dim3(ranks, static_cast<unsigned>(std::min<int64_t>((m - i0 + 31) / 32, 65535)));
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_remove_diagonal<T>, a + i0, lda, bp + i0, ldb, m - i0, n2,
                                             static_cast<const uint32_t*>(h->d_hs + i0), h->n, h->d, h->b, c);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_remove_diagonal(const void* A, int64_t lda, const void* B, int64_t ldb, int64_t n1, int64_t n2,
                                   int64_t n3, int dt, const cms_hashes* h, float* c, cudaStream_t s) {
  const int64_t m = std::min(n1, n3);
  if (m == 0) return cudaSuccess;
  ProfScope prof_scope("k_remove_diagonal", s);
  switch (dt) {
    case CMS_F32: return launch_diagonal<float>(A, lda, B, ldb, m, n2, h, c, s);
    case CMS_BF16: return launch_diagonal<__nv_bfloat16>(A, lda, B, ldb, m, n2, h, c, s);
    default: return launch_diagonal<double>(A, lda, B, ldb, m, n2, h, c, s);
  }
}

}  // namespace cms
