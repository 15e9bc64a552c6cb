// k_direct.cu - the sketch from the product's entries, for sketches that are
// long beside n1 n3: tensor-core tiles of AB whose entries are added to the
// buckets (h1(i) + h2(j)) mod b of every repetition as they leave the
// accumulators, or from a buffer of entries: all of them up to 16.8 M, bands of
// rows for FINDSIGNIFICANTENTRIES.
//
// Sec. 2.2 forms c from the spectra of the columns of A and rows of B, d n2
// transforms of length b.  By the same identity c_t[z] is the signed sum of
// the entries of AB whose key is z, which takes n1 n2 n3 multiply-adds on the
// tensor cores and d n1 n3 additions into c.  Where b is not much smaller
// than n1 n3 this is by far the cheaper side of the identity.
//
//  * k_direct_pack lays A (B) out once per call as K-major tiles of 128 rows
//    in the 128-byte swizzle that tcgen05.mma reads, so that a stage of the
//    product is one contiguous 16 KB bulk copy per operand, whatever the
//    caller's leading dimension and alignment.  FP32 values (and FP64 values
//    rounded to FP32) are split in two FP16 terms, v = hi + lo to 2^-23 of v
//    or 2^-40 of the largest value of the 128 x 128 block, after a scaling of
//    the block by a power of two; BF16 values are exact.
//    Its last block bounds every bucket (Cauchy-Schwarz) and fixes the grid
//    of the integer sums.
//  * k_direct_tile (k_direct_tile.cu) multiplies tiles of AB on the tensor
//    cores.  Entries are scaled to 64-bit integers and added to the buckets
//    with integer reductions: the order of the additions does not matter, so
//    the sketch is the same in every run.  Its scatter warps add them while the
//    next tile is multiplied, or the entries are stored (at most 16.8 M of a
//    product) and
//    k_direct_grid or k_direct_window adds them with the whole chip: a tile's
//    additions take an SM 12 us a repetition, so that a last wave of few tiles
//    would wait for them (2265 x 2265 x 503, d = 7: 318 us fused, 24 + 197 us
//    in two).
//  * k_direct_finish converts the sums to FP32.
//
// Measured on one GB300 (whole calls, transform route -> this one): X^T X of
// 4096 x 2048 FP32, b = 2^16, d = 5 with its hash draw and dense decode 2.93
// -> 0.31 ms; 8192 x 4096 BF16, b = 2^16, d = 3 7.54 -> 0.35 ms; 16384 x
// 32768 BF16, b = 2^20, d = 7 834 -> 50.6 ms; 64 uneven products of n = 512 ..
// 8192, b = 16 n, d = 3 416 -> 25.2 ms.  What bounds it: the additions into
// the buckets (random 64-bit reductions run at 205 G/s on the whole chip, one
// 32-byte sector each: 36.7 of the large product's 51 ms), then shared memory,
// which the operands' copies and the tensor cores' reads of them share (about 110
// bytes per clock and SM).
#include <algorithm>
#include <climits>
#include <cmath>
#include <cuda_fp16.h>

#include "direct_tile.cuh"
#include "warp_fft.cuh"

namespace cms {
namespace {

using namespace wfft;
using namespace dtile;

constexpr double kFixedSeconds = 36e-6;   // launches of a single product
constexpr double kMargin = 4e-6;
constexpr double kInL2 = 110e6;           // bytes of packed operands that stay in L2
// Bytes of stored entries.  Products of one sketch stay below it; the masked
// sums of FINDSIGNIFICANTENTRIES, which have no fused form, take AB in bands of
// tile rows one after the other above it.
constexpr size_t kMaxStored = size_t{256} << 20;
constexpr int kWindow = 28672;             // buckets in shared memory (224 KB)
constexpr int kBadExp = 0x4000;         // block with an infinity or a NaN
constexpr int kMinExp = -126;           // smallest normal values: scales stay representable


__device__ __forceinline__ float load_val(const float* p) { return __ldg(p); }
__device__ __forceinline__ float load_val(const __nv_bfloat16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ float load_val(const double* p) { return static_cast<float>(__ldg(p)); }

// 2^e for |e| <= 126
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }

// The product whose blocks start[q] .. start[q + 1] - 1 hold block `x`.
__device__ __forceinline__ int find_instance(const int* __restrict__ start, int count, int x) {
  int lo = 0, hi = count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(start + mid) <= x) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

struct PackSide {
  const void* X;       // rows of ld elements, inner index k
  int64_t ld;
  int64_t n;           // columns used
  const int8_t* bal;   // [k]: power of two that multiplies row k (A's; B's is the inverse), NULL: none
  int tiles;           // 0: the side is the other one's bytes
  uint8_t* out;        // [tile][stage] images
  int2* blocks;        // [tile][superblock]: exponent, sum of squares of the scaled values
};

struct PackArgs {
  PackSide side[2];
  int64_t K;
  int nsb;
  int dt;
  int64_t n1, n3;
  uint32_t* ticket;    // blocks done; left at 0
  DirectScale* scale;
};

__device__ __forceinline__ float block_sum256(float v, float* sh) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) r += sh[w];
  return r;
}

__device__ __forceinline__ int block_max256(int v, int* sh) {
  v = __reduce_max_sync(0xFFFFFFFFu, v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  int r = sh[0];
#pragma unroll
  for (int w = 1; w < 8; ++w) r = max(r, sh[w]);
  return r;
}

// The grid of the integer sums, by the last block of a product's packing.
// A bucket is a sum of at most n1 n3 entries, so |c_z| <= sqrt(n1 n3) |AB|_F
// <= sqrt(n1 n3) |A|_F |B|_F: the largest shift that keeps this below 2^62.
__device__ void direct_scale(const PackArgs& p, float* fsh, int* ish) {
  float q[2];
  int em[2];
  for (int sd = 0; sd < 2; ++sd) {
    const PackSide& s = p.side[sd];
    const int64_t count = static_cast<int64_t>(s.tiles) * p.nsb;
    int m = kMinExp;
    for (int64_t x = threadIdx.x; x < count; x += 256) m = max(m, __ldcg(&s.blocks[x].x));
    em[sd] = block_max256(m, ish);
    float acc = 0.f;
    for (int64_t x = threadIdx.x; x < count; x += 256) {
      const int2 v = __ldcg(&s.blocks[x]);
      const int de = 2 * (v.x - em[sd]);
      acc += de < -120 ? 0.f : __int_as_float(v.y) * pow2f(de);
    }
    q[sd] = block_sum256(acc, fsh);
  }
  if (threadIdx.x != 0) return;
  if (p.side[1].tiles == 0) { q[1] = q[0]; em[1] = em[0]; }
  DirectScale r;
  r.emax[0] = em[0];
  r.emax[1] = em[1];
  r.bad = em[0] >= kBadExp || em[1] >= kBadExp;
  // squares of values below 2^15: at most 2^30 K n each, inside FP32's range
  const float bound = 1.01f * sqrtf(static_cast<float>(p.n1) * static_cast<float>(p.n3)) * sqrtf(q[0]) * sqrtf(q[1]);
  r.shift = 0;
  if (bound > 0.f) r.shift = min(61 - ((__float_as_int(bound) >> 23) - 127), 126);
  *p.scale = r;
  *p.ticket = 0;
}

// ---- inner indices brought to one magnitude ----
// Blocks of 128 inner indices share an exponent, and all of AB one grid of the
// integer sums.  Both are fine for a_k b_k of any size, but not for a large a_k
// with a small b_k beside a small a_k with a large b_k: columns of A scaled by
// 2^-20 .. 2^20 and rows of B by the inverse were off by 0.36 in relative L2
// (2.6e-7 through the spectra).  So the larger of the two lends half of the
// difference of their exponents to the smaller: a_k 2^g and b_k 2^-g, exact.
// X^T X needs none (a_k and b_k are the same).  The kernel also zeroes the
// call's sums, so that it takes the place of a memset, not one more launch: a
// few warps per inner index, bound by reading the operands once more; the packing
// reads them at the same time and waits before it uses the balance (1777 x 1003,
// 1203 inner indices, FP32: 68 us a call without, 72 with it, 79 one after the
// other; 256 x 256 x 256 in FP64 31 us either way).
struct BalanceSide {
  const void* X;
  int64_t ld;
  int64_t n;
};
struct BalanceArgs {
  BalanceSide side[2];
  int64_t K;
  int dt;
  int warps;           // per inner index: 1, 2, 4 or 8
  int8_t* bal;
  uint4* zero;         // words of 16 bytes to set to zero
  int64_t words;
};

// Largest magnitude of values x, x + step, ... of a row, as FP32 bits.
template <typename T>
__device__ __forceinline__ uint32_t row_max(const BalanceSide& s, int64_t k, int x, int step) {
  const T* row = static_cast<const T*>(s.X) + k * s.ld;
  uint32_t m = 0;
#pragma unroll 8
  for (int64_t i = x; i < s.n; i += step) m = max(m, __float_as_uint(load_val(row + i)) & 0x7FFFFFFFu);
  return m;
}

// `warps` of the block's 8 take an inner index (the same count of turns in
// every warp of the block: they meet at barriers).
template <typename T>
__device__ __forceinline__ void balance_rows(const BalanceArgs& p, int64_t block, int64_t blocks) {
  __shared__ uint32_t part[2][8];
  const int warp = threadIdx.x >> 5, per = 8 / p.warps, row = warp / p.warps;
  const int x = threadIdx.x - row * p.warps * 32, step = 32 * p.warps;
  for (int64_t k0 = block * per; k0 < p.K; k0 += blocks * per) {
    const int64_t k = k0 + row;
    uint32_t m[2] = {0, 0};
    if (k < p.K) {
      m[0] = row_max<T>(p.side[0], k, x, step);
      m[1] = row_max<T>(p.side[1], k, x, step);
    }
    m[0] = __reduce_max_sync(0xFFFFFFFFu, m[0]);
    m[1] = __reduce_max_sync(0xFFFFFFFFu, m[1]);
    if (p.warps > 1) {
      __syncthreads();
      if ((threadIdx.x & 31) == 0) { part[0][warp] = m[0]; part[1][warp] = m[1]; }
      __syncthreads();
      if (x == 0)
        for (int w = 1; w < p.warps; ++w) { m[0] = max(m[0], part[0][warp + w]); m[1] = max(m[1], part[1][warp + w]); }
    }
    if (x == 0 && k < p.K) {
      // none for a row of zeros, or with an infinity or a NaN; rounded to zero:
      // a difference of one is left alone
      const bool none = m[0] == 0 || m[1] == 0 || max(m[0], m[1]) >= 0x7F800000u;
      const int half = (static_cast<int>(m[1] >> 23) - static_cast<int>(m[0] >> 23)) / 2;
      p.bal[k] = static_cast<int8_t>(none ? 0 : min(max(half, -126), 126));
    }
  }
}
__device__ __forceinline__ void balance_task(const BalanceArgs& p, int64_t block, int64_t blocks) {
  if (p.dt == CMS_BF16) balance_rows<__nv_bfloat16>(p, block, blocks);
  else if (p.dt == CMS_F64) balance_rows<double>(p, block, blocks);
  else balance_rows<float>(p, block, blocks);
}

__global__ void __launch_bounds__(256) k_direct_balance(const BalanceArgs p) {
  next_kernel_may_start();
  for (int64_t q = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x; q < p.words;
       q += static_cast<int64_t>(gridDim.x) * 256)
    p.zero[q] = make_uint4(0, 0, 0, 0);
  balance_task(p, blockIdx.x, gridDim.x);
}

__global__ void __launch_bounds__(256) k_direct_balance_batched(const BalanceArgs* __restrict__ args) {
  const BalanceArgs p = args[blockIdx.y];
  balance_task(p, blockIdx.x, gridDim.x);
}

// Multiplies the values of inner index k by their power of two (side 0: A).
__device__ __forceinline__ float balanced(float v, int g, int side) { return v * pow2f(side ? -g : g); }

template <typename T, bool SPLIT>
__device__ __forceinline__ void pack_block(const PackArgs& p, int sb, int tile, int sd, uint8_t* img, float* fsh,
                                           int* ish) {
  constexpr int kImages = SPLIT ? 4 : 2;   // stages of a superblock
  constexpr int kPerStage = kSuper / kImages;
  const PackSide& s = p.side[sd];
  const int64_t K = p.K;
  const int r = threadIdx.x & (kTile - 1), half = threadIdx.x >> 7;
  const int64_t i = static_cast<int64_t>(tile) * kTile + r;
  const int64_t k0 = static_cast<int64_t>(sb) * kSuper + half * 64;
  const T* X = static_cast<const T*>(s.X) + i;
  float x[64];
  const int kn = i < s.n ? static_cast<int>(min(max(K - k0, static_cast<int64_t>(0)), static_cast<int64_t>(64))) : 0;
  if (kn == 64) {
#pragma unroll
    for (int q = 0; q < 64; ++q) x[q] = load_val(X + (k0 + q) * s.ld);
  } else {
#pragma unroll
    for (int q = 0; q < 64; ++q) x[q] = q < kn ? load_val(X + (k0 + q) * s.ld) : 0.f;
  }
  // (the operands are read while the kernel before, which finds the balance
  // and zeroes the sums, still runs)
  wait_for_kernel_before();
  if (s.bal != nullptr) {
    // (64 bytes of the same 64 inner indices for every row)
    if (kn == 64) {
      uint32_t w[16];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint4 v = __ldcg(reinterpret_cast<const uint4*>(s.bal + k0) + q);
        w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
      }
#pragma unroll
      for (int q = 0; q < 64; ++q) x[q] = balanced(x[q], static_cast<int8_t>(w[q / 4] >> (q % 4 * 8)), sd);
    } else {
#pragma unroll
      for (int q = 0; q < 64; ++q)
        if (q < kn) x[q] = balanced(x[q], s.bal[k0 + q], sd);
    }
  }
  uint32_t m = 0;
#pragma unroll
  for (int q = 0; q < 64; ++q) m = max(m, __float_as_uint(x[q]) & 0x7FFFFFFFu);
  m = static_cast<uint32_t>(block_max256(static_cast<int>(m), ish));
  const bool bad = m >= 0x7F800000u;
  const int e = bad ? 0 : max(static_cast<int>(m >> 23) - 127, kMinExp);
  // two factors: 2^(14 - e) alone may leave FP32's range
  const int sh = direct_scale_log2(SPLIT) - e;
  const float f1 = pow2f(sh / 2), f2 = pow2f(sh - sh / 2);
  float nn = 0.f;
#pragma unroll
  for (int q = 0; q < 64; ++q) {
    x[q] = x[q] * f1 * f2;
    nn = fmaf(x[q], x[q], nn);
  }
  nn = block_sum256(nn, fsh);
  const uint32_t rowoff = (r >> 3) * 1024 + (r & 7) * 128;
  // chunk c: 8 of this thread's 64 inner indices, in the image's 16-byte
  // column c (swizzled by the row)
  auto put = [&](int image, int c, const uint32_t (&w)[4]) {
    *reinterpret_cast<uint4*>(img + image * kStageBytes + rowoff + ((c ^ (r & 7)) << 4)) =
        make_uint4(w[0], w[1], w[2], w[3]);
  };
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float a = x[8 * c + 2 * q], b = x[8 * c + 2 * q + 1];
      if constexpr (SPLIT) {
        const __half ha = __float2half_rn(a), hb = __float2half_rn(b);
        const __half2 h2 = __halves2half2(ha, hb);
        const __half2 l2 = __floats2half2_rn(a - __half2float(ha), b - __half2float(hb));
        hi[q] = *reinterpret_cast<const uint32_t*>(&h2);
        lo[q] = *reinterpret_cast<const uint32_t*>(&l2);
      } else {
        const __nv_bfloat162 h2 = __floats2bfloat162_rn(a, b);
        hi[q] = *reinterpret_cast<const uint32_t*>(&h2);
      }
    }
    if constexpr (SPLIT) {
      put(half * 2 + c / 4, c & 3, hi);
      put(half * 2 + c / 4, 4 + (c & 3), lo);
    } else {
      put(half, c, hi);
    }
  }
  fence_proxy_async();
  __syncthreads();
  if (threadIdx.x == 0) {
    s.blocks[static_cast<size_t>(tile) * p.nsb + sb] = make_int2(bad ? kBadExp : e, __float_as_int(nn));
    const int64_t left = min(K - static_cast<int64_t>(sb) * kSuper, static_cast<int64_t>(kSuper));
    const uint32_t bytes = static_cast<uint32_t>((left + kPerStage - 1) / kPerStage) * kStageBytes;
    const int64_t per_tile = (K + kPerStage - 1) / kPerStage;   // images of a tile
    uint8_t* dst = s.out + (static_cast<size_t>(tile) * per_tile + static_cast<size_t>(sb) * kImages) * kStageBytes;
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(img)),
                 "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
  }
}

// Block `idx` of a product's packing: superblocks fastest, then the tiles of
// A, then those of B.
__device__ __forceinline__ void pack_task(const PackArgs& p, uint32_t idx) {
  extern __shared__ __align__(1024) uint8_t img[];
  __shared__ float fsh[8];
  __shared__ int ish[8];
  __shared__ bool last;
  const uint32_t nsb = static_cast<uint32_t>(p.nsb);
  const uint32_t total = nsb * static_cast<uint32_t>(p.side[0].tiles + p.side[1].tiles);
  int tile = static_cast<int>(idx / nsb);
  const int sb = static_cast<int>(idx - tile * nsb);
  const int sd = tile >= p.side[0].tiles;
  if (sd) tile -= p.side[0].tiles;
  if (p.dt == CMS_BF16) pack_block<__nv_bfloat16, false>(p, sb, tile, sd, img, fsh, ish);
  else if (p.dt == CMS_F64) pack_block<double, true>(p, sb, tile, sd, img, fsh, ish);
  else pack_block<float, true>(p, sb, tile, sd, img, fsh, ish);
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(p.ticket, 1u) == total - 1;
  }
  __syncthreads();
  if (last) {
    __threadfence();
    direct_scale(p, fsh, ish);
  }
  if (threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

__global__ void __launch_bounds__(256) k_direct_pack(const PackArgs p) {
  next_kernel_may_start();
  pack_task(p, blockIdx.x);
}

// ---- pre-sketched operands: b well below n ----
// By Fig. 1 c_t is the cyclic convolution of the count sketches of a_k and
// b_k, summed over k: with A'_t = S1 A (b x n2) and B'_t = B S2 (n2 x b) it is
// the sum over the entries of A'_t B'_t whose two positions add up to z mod b,
// the direct route's problem with b in the place of n1 and n3.
//
//  * k_pre_transpose: the operand as slabs [superblock][i][128] of FP32, so
//    that an entry of a column is 512 contiguous bytes over its inner indices
//    and a slab (n x 512 bytes) stays in L2 while every repetition and side
//    reads it;
//  * k_pre_lists: the entries of every bucket, from the bucket lists by h mod
//    C: bucket z = C z1 + z2 has the row u = z2 R + z1 of A'_t;
//  * k_pre_pack: 128 buckets x 128 inner indices per block, a warp 16 buckets:
//    the sums of its entries' rows in registers, then scaled, split and
//    stored as k_direct_pack does.
// X^T X of 2048 x 16384 FP32, b = 2048, d = 5: 7.2 ms through the
// shared-memory transform kernel (every entry gathered for each of its rows,
// with its twiddle), 6.9 ms through the tiles of n1 x n3 (1.3e9 additions),
// 0.62 ms this way (transpose 74 us, lists 6, sums and packing 200, tiles
// 306).  What bounds it: the tiles (b^2 n2 d multiply-adds), and the 1.3 GB of
// rows read by the sums.  It is the cheapest way from b of about n / 4 down;
// over 130 calls of n = 64 .. 16384, b = n / 8 .. 32 n, 64 to 8192 inner
// indices it won 22 times, by up to 6.7 over the transform route.
struct PreArgs {
  const void* X[2];
  int64_t ld[2];
  int64_t n[2];
  const int8_t* bal;      // powers of two of the inner indices, NULL: none
  int alias;
  int64_t K;
  int nsb, d;
  int hn;                 // hash domain
  int R, C, classes, tiles;   // classes of R buckets per tile of 128 rows
  float* slab[2];         // [superblock][n][128]
  const uint32_t* hs;     // [t][side][hn]
  const uint32_t* perm;
  const uint32_t* off;    // [t][side][C + 1]
  uint32_t* ent;          // [t][side][hn]: x | sign << 31, by row
  uint32_t* start;        // [t][side][tiles 128 + 1]
  uint32_t* vhs;          // [2][tiles 128]: bucket of each row
  PackArgs pack;          // repetition 0
  size_t rep_images;
  int rep_blocks;
};

template <typename T>
__global__ void __launch_bounds__(256) k_pre_transpose(const PreArgs p) {
  __shared__ float sh[kSuper][33];
  const int side = blockIdx.z;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t i = static_cast<int64_t>(blockIdx.x) * 32 + lane;
  const int64_t k0 = static_cast<int64_t>(blockIdx.y) * kSuper;
  wait_for_kernel_before();
  if (static_cast<int64_t>(blockIdx.x) * 32 >= p.n[side]) return;
  const T* X = static_cast<const T*>(p.X[side]);
#pragma unroll
  for (int q = 0; q < kSuper / 8; ++q) {
    const int k = q * 8 + warp;
    float v = i < p.n[side] && k0 + k < p.K ? load_val(X + (k0 + k) * p.ld[side] + i) : 0.f;
    if (p.bal != nullptr && k0 + k < p.K) v = balanced(v, p.bal[k0 + k], side);
    sh[k][lane] = v;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int x = q * 8 + warp;
    const int64_t xi = static_cast<int64_t>(blockIdx.x) * 32 + x;
    if (xi >= p.n[side]) continue;
    float* dst = p.slab[side] + (static_cast<size_t>(blockIdx.y) * p.n[side] + xi) * kSuper;
#pragma unroll
    for (int g = 0; g < 4; ++g) dst[g * 32 + lane] = sh[g * 32 + lane][x];
  }
}

// A warp per class z2 of one (t, side): its entries by z1, in their order.
__global__ void __launch_bounds__(256) k_pre_lists(const PreArgs p) {
  const int lane = threadIdx.x & 31;
  const int z2 = static_cast<int>(blockIdx.x) * 8 + (threadIdx.x >> 5);
  const size_t ts = blockIdx.y;
  const int rows = p.tiles * kTile;
  if (z2 >= p.C) return;
  const uint32_t* off = p.off + ts * (p.C + 1);
  const uint32_t e0 = off[z2], e1 = off[z2 + 1];
  uint32_t* ent = p.ent + ts * p.hn;
  uint32_t* start = p.start + ts * (rows + 1);
  const int row0 = z2 / p.classes * kTile + z2 % p.classes * p.R;   // of bucket (z1 = 0, z2)
  uint32_t at = e0;
  for (int z1 = 0; z1 < p.R; ++z1) {
    if (lane == 0) {
      start[row0 + z1] = at;
      if (ts < 2) p.vhs[ts * rows + row0 + z1] = static_cast<uint32_t>(z1 * p.C + z2);
    }
    for (uint32_t e = e0; e < e1; e += 32) {
      uint32_t w = 0, x = 0;
      bool mine = false;
      if (e + lane < e1) {
        x = p.perm[ts * p.hn + e + lane];
        w = p.hs[ts * p.hn + x];
        mine = static_cast<int>((w & kBucketMask) / static_cast<uint32_t>(p.C)) == z1;
      }
      const unsigned m = __ballot_sync(0xFFFFFFFFu, mine);
      if (mine) ent[at + __popc(m & ((1u << lane) - 1u))] = x | (w & 0x80000000u);
      at += __popc(m);
    }
  }
  // rows of the tile that hold no bucket (128 is no multiple of R, or the last tile)
  const bool last_of_tile = z2 % p.classes == p.classes - 1 || z2 == p.C - 1;
  const int pad_end = z2 == p.C - 1 ? rows + 1 : (z2 / p.classes + 1) * kTile;
  if (last_of_tile)
    for (int r = row0 + p.R + lane; r < pad_end; r += 32) {
      start[r] = e1;
      if (ts < 2 && r < rows) p.vhs[ts * rows + r] = 0;
    }
}

__global__ void __launch_bounds__(256) k_pre_pack(const PreArgs p) {
  extern __shared__ __align__(1024) uint8_t img[];
  __shared__ float fsh[8];
  __shared__ int ish[8];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // superblocks slowest: their slab stays in L2
  const int per_sb = p.tiles * 2 * p.d;
  const int sb = static_cast<int>(blockIdx.x) / per_sb;
  int rest = static_cast<int>(blockIdx.x) - sb * per_sb;
  const int ts = rest / p.tiles, tile = rest - ts * p.tiles;
  const int t = ts >> 1, side = ts & 1;
  const int64_t n = p.n[side];
  const float* slab = p.slab[p.alias ? 0 : side] + static_cast<size_t>(sb) * n * kSuper + lane * 4;
  const uint32_t* ent = p.ent + static_cast<size_t>(ts) * p.hn;
  const uint32_t* start = p.start + static_cast<size_t>(ts) * (p.tiles * kTile + 1) + tile * kTile + warp * 16;
  const uint32_t bound = lane <= 16 ? start[lane] : 0;
  float v[16][4];
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    const uint32_t e0 = __shfl_sync(0xFFFFFFFFu, bound, r), e1 = __shfl_sync(0xFFFFFFFFu, bound, r + 1);
    float a[4] = {0.f, 0.f, 0.f, 0.f};
    for (uint32_t e = e0; e < e1; e += 32) {
      const uint32_t mine = e + lane < e1 ? ent[e + lane] : 0x7FFFFFFFu;
      const int cnt = static_cast<int>(min(e1 - e, 32u));
      float s[4] = {0.f, 0.f, 0.f, 0.f};
      for (int q = 0; q < cnt; q += 4) {
        float4 x[4];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          const uint32_t w = __shfl_sync(0xFFFFFFFFu, mine, min(q + g, 31));
          const uint32_t xi = w & kBucketMask;
          x[g] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (q + g < cnt && static_cast<int64_t>(xi) < n)
            x[g] = __ldg(reinterpret_cast<const float4*>(slab + static_cast<size_t>(xi) * kSuper));
          if (w >> 31) x[g] = make_float4(-x[g].x, -x[g].y, -x[g].z, -x[g].w);
        }
        s[0] += (x[0].x + x[1].x) + (x[2].x + x[3].x);
        s[1] += (x[0].y + x[1].y) + (x[2].y + x[3].y);
        s[2] += (x[0].z + x[1].z) + (x[2].z + x[3].z);
        s[3] += (x[0].w + x[1].w) + (x[2].w + x[3].w);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) a[q] += s[q];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) v[r][q] = a[q];
  }
  uint32_t m = 0;
#pragma unroll
  for (int r = 0; r < 16; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) m = max(m, __float_as_uint(v[r][q]) & 0x7FFFFFFFu);
  m = static_cast<uint32_t>(block_max256(static_cast<int>(m), ish));
  const bool bad = m >= 0x7F800000u;
  const int e = bad ? 0 : max(static_cast<int>(m >> 23) - 127, kMinExp);
  const int sh = direct_scale_log2(true) - e;
  const float f1 = pow2f(sh / 2), f2 = pow2f(sh - sh / 2);
  float nn = 0.f;
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    uint32_t hi[2], lo[2];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      v[r][q] = v[r][q] * f1 * f2;
      nn = fmaf(v[r][q], v[r][q], nn);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const __half ha = __float2half_rn(v[r][2 * q]), hb = __float2half_rn(v[r][2 * q + 1]);
      const __half2 h2 = __halves2half2(ha, hb);
      const __half2 l2 = __floats2half2_rn(v[r][2 * q] - __half2float(ha), v[r][2 * q + 1] - __half2float(hb));
      hi[q] = *reinterpret_cast<const uint32_t*>(&h2);
      lo[q] = *reinterpret_cast<const uint32_t*>(&l2);
    }
    // inner indices 4 lane .. 4 lane + 3: image lane / 8 (32 of them), 8-byte
    // half of 16-byte column (lane / 2) mod 4 (hi) and 4 beyond (lo)
    const int row = warp * 16 + r;
    uint8_t* base = img + (lane >> 3) * kStageBytes + (row >> 3) * 1024 + (row & 7) * 128 + (lane & 1) * 8;
    const int c = (lane >> 1) & 3;
    *reinterpret_cast<uint2*>(base + ((c ^ (row & 7)) << 4)) = make_uint2(hi[0], hi[1]);
    *reinterpret_cast<uint2*>(base + (((c + 4) ^ (row & 7)) << 4)) = make_uint2(lo[0], lo[1]);
  }
  nn = block_sum256(nn, fsh);
  fence_proxy_async();
  __syncthreads();
  PackArgs pk = p.pack;
#pragma unroll
  for (int sd = 0; sd < 2; ++sd) {
    pk.side[sd].out += t * p.rep_images;
    pk.side[sd].blocks += static_cast<size_t>(t) * p.rep_blocks;
  }
  pk.ticket += t;
  pk.scale += t;
  if (threadIdx.x == 0) {
    pk.side[side].blocks[static_cast<size_t>(tile) * p.nsb + sb] = make_int2(bad ? kBadExp : e, __float_as_int(nn));
    const int64_t left = min(p.K - static_cast<int64_t>(sb) * kSuper, static_cast<int64_t>(kSuper));
    const int64_t per_tile = (p.K + 31) / 32;
    uint8_t* dst = pk.side[side].out + (static_cast<size_t>(tile) * per_tile + static_cast<size_t>(sb) * 4) * kStageBytes;
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(img)),
                 "r"(static_cast<uint32_t>((left + 31) / 32) * kStageBytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    __threadfence();
    last = atomicAdd(pk.ticket, 1u) == static_cast<uint32_t>(2 * p.tiles * p.nsb) - 1;
  }
  __syncthreads();
  if (last) {
    __threadfence();
    direct_scale(pk, fsh, ish);
  }
  if (threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// A value added to its bucket's sum, to the sums of the bits set in the
// position i of its row, and to those of the bits set in j.
__device__ __forceinline__ void bucket_add_masked(unsigned long long* c, size_t set, int bits, uint32_t i, uint32_t j,
                                                  uint32_t ha, uint32_t hb, uint32_t b, long long v) {
  uint32_t z = (ha & kBucketMask) + (hb & kBucketMask);
  if (z >= b) z -= b;
  const long long iv = ((ha ^ hb) >> 31) ? -v : v;
  c += z;
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(c), "l"(iv) : "memory");
  for (int m = 0; m < bits; ++m) {
    c += set;
    if ((i >> m) & 1u) asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(c), "l"(iv) : "memory");
  }
  for (int m = 0; m < bits; ++m) {
    c += set;
    if ((j >> m) & 1u) asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(c), "l"(iv) : "memory");
  }
}

__global__ void __launch_bounds__(256)
k_direct_pack_batched(const PackArgs* __restrict__ args, const int* __restrict__ start, int count) {
  __shared__ PackArgs sp;
  const int q = find_instance(start, count, static_cast<int>(blockIdx.x));
  for (int w = threadIdx.x; w < static_cast<int>(sizeof(PackArgs) / 4); w += 256)
    reinterpret_cast<uint32_t*>(&sp)[w] = reinterpret_cast<const uint32_t*>(args + q)[w];
  __syncthreads();
  pack_task(sp, blockIdx.x - static_cast<uint32_t>(__ldg(start + q)));
}

struct GridArgs {
  const float* grid;           // [part][tile row - row0][tile column][128 columns][128 rows]
  size_t part;                 // entries from one part to the next
  int row0;
  int parts;
  int tiles1, tiles3, sym;
  const uint32_t* hs;          // [t][side][n]
  const DirectScale* scale;
  unsigned long long* acc;     // [copy][t][b], or [1 + 2 bits][t][b]
  int copies, bits;
  int n, n1, n3, b, d;
};

// The entries of the grid, and the mirror images of a symmetric product's,
// added to the buckets: a block takes 16 columns of a tile, a warp two, a lane
// four rows of each, and the repetitions from blockIdx.z on.  The parts of an
// entry are added as integers.
constexpr int kGridCols = 2;
template <bool MASKED>
__global__ void __launch_bounds__(256) k_direct_grid(const GridArgs p) {
  next_kernel_may_start();
  wait_for_kernel_before();
  if (p.scale->bad) return;
  const int tile = static_cast<int>(blockIdx.x), tr = tile / p.tiles3, ti = p.row0 + tr, tj = tile - tr * p.tiles3;
  if (p.sym && ti > tj) return;
  const bool mirror = p.sym && ti < tj;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int q0 = (static_cast<int>(blockIdx.y) * 8 + warp) * kGridCols;   // columns of the tile
  const int i0 = ti * kTile + lane, j0 = tj * kTile + q0;                 // rows i0 + 32 r
  const int cols = min(kGridCols, p.n3 - j0);
  if (cols <= 0) return;
  const float* src = p.grid + static_cast<size_t>(tile) * kTile * kTile + q0 * kTile + lane;
  long long v[kGridCols][4];
#pragma unroll
  for (int q = 0; q < kGridCols; ++q)
#pragma unroll
    for (int r = 0; r < 4; ++r) v[q][r] = __float2ll_rn(__ldcg(src + q * kTile + r * 32));
#pragma unroll 4
  for (int s = 1; s < p.parts; ++s) {
    src += p.part;
#pragma unroll
    for (int q = 0; q < kGridCols; ++q)
#pragma unroll
      for (int r = 0; r < 4; ++r) v[q][r] += __float2ll_rn(__ldcg(src + q * kTile + r * 32));
  }
  const uint32_t b = static_cast<uint32_t>(p.b);
  const size_t set = static_cast<size_t>(p.d) * p.b;
  unsigned long long* sums = p.acc + (p.copies > 1 ? static_cast<size_t>(blockIdx.x + blockIdx.y) % p.copies * set : 0);
  auto add = [&](unsigned long long* c, uint32_t i, uint32_t j, uint32_t ha, uint32_t hb, long long iv) {
    if constexpr (MASKED) bucket_add_masked(c, set, p.bits, i, j, ha, hb, b, iv);
    else {
      uint32_t z = (ha & kBucketMask) + (hb & kBucketMask);
      if (z >= b) z -= b;
      const long long w = ((ha ^ hb) >> 31) ? -iv : iv;
      asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(c + z), "l"(w) : "memory");
    }
  };
  for (int t = blockIdx.z; t < p.d; t += gridDim.z) {
    const uint32_t* h1 = p.hs + static_cast<size_t>(2 * t) * p.n;
    const uint32_t* h2 = h1 + p.n;
    unsigned long long* c = sums + static_cast<size_t>(t) * p.b;
    uint32_t hr[4], hm[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const bool in = i0 + 32 * r < p.n1;
      hr[r] = in ? __ldg(h1 + i0 + 32 * r) : 0;
      hm[r] = mirror && in ? __ldg(h2 + i0 + 32 * r) : 0;
    }
#pragma unroll
    for (int q = 0; q < kGridCols; ++q) {
      if (q >= cols) break;
      const uint32_t hc = __ldg(h2 + j0 + q), hx = mirror ? __ldg(h1 + j0 + q) : 0;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int i = i0 + 32 * r;
        if (i >= p.n1) continue;
        add(c, i, j0 + q, hr[r], hc, v[q][r]);
        if (mirror) add(c, j0 + q, i, hx, hm[r], v[q][r]);
      }
    }
  }
}

// __float2ll_rn for |v| < 2^63 without the 64-bit conversion (2 a clock and SM)
__device__ __forceinline__ long long to_units(float v) {
  const uint32_t bits = __float_as_uint(v);
  const int shift = static_cast<int>((bits >> 23) & 0xFFu) - 150;
  const long long big = static_cast<long long>(static_cast<unsigned long long>((bits & 0x7FFFFFu) | 0x800000u) << (shift & 63));
  const long long small = __float2int_rn(v);
  return shift < 0 ? small : (static_cast<int>(bits) < 0 ? -big : big);
}

// Byte of a window's bucket (z4: four times the bucket).  The hashes are linear
// in the position mod a prime, so that a warp's 32 rows are mostly an even
// progression of buckets: one step in 16 words would put them in two banks.
__device__ __forceinline__ uint32_t window_byte(uint32_t z4) { return z4 ^ ((z4 >> 5) & 0x7Cu); }

// The entries of the grid added to the buckets with the first kWindow buckets
// of a repetition in a block's shared memory (two words each) and the others'
// additions in L2: a block adds its share of the tiles for one repetition.
// 64 bits are added in two halves, the low half's carry taken from the value
// that its addition returns (64-bit additions in shared memory are a loop of
// compare and swap, a quarter as fast).  Beside k_direct_grid, bound by 1.35 G
// reductions a second and SM: 4096 x 4096 entries, d = 3, b = 2^16 (44% of the
// buckets in the window) 228 -> 175 us; 1500 x 1500, d = 5, b = 30000 (all but
// 4%) 78 -> 45 us, 30 clocks for a warp's 32 additions, most of them latency.
// Three windows a repetition, every entry read for each, took 279 us where one
// takes 175.
__global__ void __launch_bounds__(1024, 1) k_direct_window(const GridArgs p, int shares) {
  extern __shared__ uint32_t words[];        // low halves, then high halves
  next_kernel_may_start();
  const int t = static_cast<int>(blockIdx.x) / shares, share = static_cast<int>(blockIdx.x) - t * shares;
  const uint32_t b = static_cast<uint32_t>(p.b), mine = min(b, static_cast<uint32_t>(kWindow));
  const uint32_t b4 = 4 * b, mine4 = 4 * mine;
  const uint32_t used = (mine + 31) & ~31u;
  for (uint32_t q = threadIdx.x; q < used; q += 1024) words[q] = words[kWindow + q] = 0;
  __syncthreads();
  wait_for_kernel_before();
  if (p.scale->bad) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t* h1 = p.hs + static_cast<size_t>(2 * t) * p.n;
  const uint32_t* h2 = h1 + p.n;
  unsigned long long* out = p.acc + static_cast<size_t>(t) * b;
  const uint32_t base = smem_u32(words);
  // four rows: their low halves are on their way together
  auto add4 = [&](const uint32_t (&row4)[4], const int (&rowneg)[4], uint32_t col4, int colneg, const long long (&v)[4]) {
    uint32_t z4[4], l[4], h[4], old[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const uint32_t z = row4[r] + col4;
      z4[r] = min(z, z - b4);              // (row4 + col4) mod b4
      const int m = (rowneg[r] ^ colneg) >> 31;
      const unsigned long long iv = static_cast<unsigned long long>((v[r] ^ m) - m);
      l[r] = static_cast<uint32_t>(iv);
      h[r] = static_cast<uint32_t>(iv >> 32);
      asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %3, %4;\n\tmov.u32 %0, 0;\n\t"
                   "@p atom.shared.add.u32 %0, [%1], %2;\n\t}"
                   : "=&r"(old[r])
                   : "r"(base + window_byte(z4[r])), "r"(l[r]), "r"(z4[r]), "r"(mine4)
                   : "memory");
      if (z4[r] >= mine4)
        asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(out + z4[r] / 4), "l"(iv) : "memory");
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 x, y;\n\tsetp.lt.u32 p, %0, %1;\n\t"
                   "add.cc.u32 x, %4, %5;\n\taddc.u32 y, %6, 0;\n\t"
                   "@p red.shared.add.u32 [%2+%3], y;\n\t}" ::"r"(z4[r]), "r"(mine4), "r"(base + window_byte(z4[r])),
                   "n"(4 * kWindow), "r"(old[r]), "r"(l[r]), "r"(h[r])
                   : "memory");
    }
  };
  // half tiles: two columns a warp, four rows of each a lane
  const int tiles = p.sym ? p.tiles3 * (p.tiles3 + 1) / 2 : p.tiles1 * p.tiles3;
  for (int u = share; u < 2 * tiles; u += shares) {
    int ti, tj;
    const int q = u >> 1;
    if (p.sym) {
      tj = static_cast<int>((sqrtf(8.f * static_cast<float>(q) + 1.f) - 1.f) * 0.5f);
      while (tj * (tj + 1) / 2 > q) --tj;
      while ((tj + 1) * (tj + 2) / 2 <= q) ++tj;
      ti = q - tj * (tj + 1) / 2;
    } else {
      ti = q / p.tiles3;
      tj = q - ti * p.tiles3;
    }
    const bool mirror = p.sym && ti != tj;
    const int i0 = ti * kTile + lane, q0 = (u & 1) * 64 + warp * 2, j0 = tj * kTile + q0;
    if (j0 >= p.n3) continue;
    const float* src = p.grid + (static_cast<size_t>(ti) * p.tiles3 + tj) * kTile * kTile + q0 * kTile + lane;
    long long v[2][4];
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int r = 0; r < 4; ++r) v[c][r] = to_units(__ldcg(src + c * kTile + r * 32));
#pragma unroll 2
    for (int x = 1; x < p.parts; ++x) {
      src += p.part;
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int r = 0; r < 4; ++r) v[c][r] += to_units(__ldcg(src + c * kTile + r * 32));
    }
    uint32_t row4[4];
    int rowneg[4];
    auto rows = [&](const uint32_t* hh) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {   // (entries past the last row are zero)
        const uint32_t w = i0 + 32 * r < p.n1 ? __ldg(hh + i0 + 32 * r) : 0;
        rowneg[r] = static_cast<int>(w);
        row4[r] = 4 * (w & kBucketMask);
      }
    };
    const int cols = min(2, p.n3 - j0);
    rows(h1);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (c >= cols) break;
      const uint32_t w = __ldg(h2 + j0 + c);
      add4(row4, rowneg, 4 * (w & kBucketMask), static_cast<int>(w), v[c]);
    }
    if (mirror) {
      rows(h2);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        if (c >= cols) break;
        const uint32_t w = __ldg(h1 + j0 + c);
        add4(row4, rowneg, 4 * (w & kBucketMask), static_cast<int>(w), v[c]);
      }
    }
  }
  __syncthreads();
  for (uint32_t q = threadIdx.x; q < mine; q += 1024) {
    const uint32_t w = window_byte(4 * q) / 4;
    const unsigned long long sum = static_cast<unsigned long long>(words[kWindow + w]) << 32 | words[w];
    if (sum) asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(out + q), "l"(sum) : "memory");
  }
}

// `per` buckets share a scale.  COPIES: 32 buckets per block, the copies
// dealt to its 8 warps.
template <bool COPIES>
__global__ void __launch_bounds__(256) k_direct_finish(const unsigned long long* acc, int copies, float* c, int64_t len,
                                                       int64_t per, const DirectScale* scale, int log2s) {
  wait_for_kernel_before();
  if constexpr (COPIES) {
    __shared__ unsigned long long part[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t q = static_cast<int64_t>(blockIdx.x) * 32 + lane;
    unsigned long long v = 0;
    if (q < len) {
#pragma unroll 4
      for (int r = warp; r < copies; r += 8) v += __ldcg(acc + r * len + q);
    }
    part[warp][lane] = v;
    __syncthreads();
    if (warp == 0 && q < len) {
#pragma unroll
      for (int w = 1; w < 8; ++w) v += part[w][lane];
      c[q] = direct_value(v, scale[q / per], log2s);
    }
  } else {
    for (int64_t q = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x; q < len;
         q += static_cast<int64_t>(gridDim.x) * 256)
      c[q] = direct_value(acc[q], scale[q / per], log2s);
  }
}

// The bits |sum| > half of each (repetition, bucket) and side, decoded into a
// position (0: none).  The rho copies of a bit of E are the same mask, so
// their sketches are the same sums, and a complement's sums are the total's
// less the bit's: a bit is 1 when its sum alone is above, 0 when its
// complement's alone is, and no bit (a tie of the votes) otherwise.
__global__ void __launch_bounds__(256)
k_direct_sig_decode(const unsigned long long* __restrict__ acc, int bits, int64_t len, int64_t n1, int64_t n3,
                    float half, const DirectScale* __restrict__ scale, int log2s, uint64_t* __restrict__ keys) {
  const DirectScale sc = *scale;
  const int64_t q = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x;
  if (q >= len) return;
  const unsigned long long total = acc[q];
  int64_t pos[2];
  for (int sd = 0; sd < 2; ++sd) {
    int64_t x = 0;
    const unsigned long long* a = acc + static_cast<size_t>(1 + sd * bits) * len + q;
    for (int m = 0; m < bits; ++m) {
      const unsigned long long s1 = a[static_cast<size_t>(m) * len];
      const bool one = fabsf(direct_value(s1, sc, log2s)) > half;
      const bool zero = fabsf(direct_value(total - s1, sc, log2s)) > half;
      if (one == zero) { x = -1; break; }
      x |= static_cast<int64_t>(one) << m;
    }
    pos[sd] = x;
    if (x < 0) break;
  }
  uint64_t key = 0;
  if (pos[0] >= 0 && pos[0] < n1 && pos[1] >= 0 && pos[1] < n3)
    key = static_cast<uint64_t>(pos[0]) * static_cast<uint64_t>(n3) + static_cast<uint64_t>(pos[1]) + 1u;
  keys[q] = key;
}

}  // namespace

uint32_t read_clear_error_direct() { return dtile::read_clear_error_tile(); }

namespace {

// How the tiles are cut and where their entries go.
//  wide   units of two tiles side by side (an operand tile of A serves both:
//         96 KB from L2 for 2 x 128 x 128 x 128 BF16 products instead of 128),
//         or one tile with its inner indices dealt to the block's halves
//         (twice the units, where tiles are few);
//  splits of the inner dimension while SMs have no unit;
//  grid   entries stored for a launch of its own (additions from every SM,
//         about 6 us more; at most 16.8 M, 64 MB of scratch: above that it would
//         still pay where most buckets are in the window, 4500 x 4500, K = 4000,
//         b = 30000, d = 5 FP32 560 us against 785, and not elsewhere, 8192 x 8192,
//         b = 2^17 2186 against 2008), or added by the tile kernel while it multiplies on.
// Times: a chunk of 64 (FP16 terms) or 128 (BF16) inner indices of a tile
// 0.40 us (BF16 alone on its operands 0.53: the copies from L2 bound it), and
// more where the packed operands (`packed` bytes) do not stay in L2: 2.0 times as
// much in units of two tiles and 2.45 in units of one (BF16 1.7 and 2.2; fitted,
// as the line at 110 MB of the 129, to 320 calls of n = 32 .. 17000 and 64 to 2 M
// inner indices by either route; 5022 x 19702 FP32, b = 3125, d = 1: 0.96 ms
// estimated without it, 1.76 ms taken, 1.01 by the spectra).  The shape of the
// units is chosen without it.
void choose_tiles(DirectPlan& p, bool sym, int reps, double entries, double adds, double full_rate, double sm_rate,
                  double window, double packed, bool may_grid, bool may_fuse, bool shared, int sms) {
  // stored entries added: in L2, or with a share of the buckets in shared memory
  // (2.7 us less per million of its additions, 4 us more)
  p.window = entries * adds * window >= 3e6;
  const double added = entries * reps * adds / full_rate * (p.window ? 1.0 - 0.65 * window : 1.0) + (p.window ? 4e-6 : 0.0);
  double best = 1e30, best_mma = 0.0;
  for (int wide = 0; wide < 2; ++wide) {
    if (!wide && shared) continue;
    const int units = tile_units(p.tiles1, p.tiles3, wide != 0, sym);
    for (int s = 1; s <= std::min(p.nsb, 64); ++s) {
      const int per = (p.nsb + s - 1) / s, real = (p.nsb + per - 1) / per;
      if (s > 1 && static_cast<int64_t>(units) * s * reps > 2 * sms) break;   // every SM has work
      if (real != s && s > 1) continue;
      const double blocks = static_cast<double>(units) * real * reps;
      const double chunk = wide ? 0.85e-6 : (p.split ? 0.43e-6 : 0.55e-6);
      const double unit = per * (p.split ? 2.0 : 1.0) * chunk + 3e-6;
      // (a batch's products share the last wave)
      const double waves = shared ? std::max(1.0, blocks / sms) : std::ceil(blocks / sms);
      const double mma = waves * unit;
      for (int grid = 0; grid < 2; ++grid) {
        if (grid ? !may_grid : !may_fuse) continue;
        const double parts = real * (wide || per * (p.split ? 2 : 1) == 1 ? 1.0 : 2.0);
        const double t =
            grid ? mma + 3e-6 + added + entries * reps * (sym ? 4.0 : 8.0) * parts / 4e12 + parts * 0.1e-6
                 : mma + std::max(entries * reps * adds * real / full_rate,
                                  waves * entries * adds / units / sm_rate);
        if (t < best) {
          best = t;
          best_mma = mma;
          p.wide = wide != 0;
          p.grid = grid != 0;
          p.sb_per_split = per;
          p.splits = real;
        }
      }
    }
  }
  p.units = tile_units(p.tiles1, p.tiles3, p.wide, sym);
  const double beyond = p.split ? (p.wide ? 2.0 : 2.45) : (p.wide ? 1.7 : 2.2);
  p.beyond_l2 = packed > kInL2;
  p.seconds = best + kFixedSeconds + (p.beyond_l2 ? (beyond - 1.0) * best_mma : 0.0);
  p.blocks = static_cast<int>(std::min<int64_t>(static_cast<int64_t>(p.units) * p.splits * reps, sms));
  const int chunks = p.sb_per_split * (p.split ? 2 : 1);
  p.need_fold = (p.wide ? chunks : (chunks + 1) / 2) > 64;
  p.need_hand = !p.grid;
  p.need_merge = !p.wide && !p.grid && chunks > 1;
  p.parts = p.splits * (!p.wide && chunks > 1 ? 2 : 1);
}

size_t al1k(size_t x) { return (x + 1023) & ~static_cast<size_t>(1023); }

// Copies of `words` sums.  Reductions to few words queue up (23 G/s on 2^10
// words, 100 on 2^14, 165 on 2^16, 200 from 2^18 on), so tiles share several
// copies of a short sketch's sums, which the conversion adds up.
int sum_copies(int64_t words, int64_t units) {
  return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>({256, (int64_t{1} << 18) / words, units})));
}

}  // namespace

DirectPlan make_direct_plan(const cms_hashes* h, int64_t n1, int64_t n2, int64_t n3, int dt, bool alias, int sms,
                            int sets, bool batch) {
  DirectPlan p;
  p.split = dt != CMS_BF16;
  p.alias = alias;
  p.tiles1 = static_cast<int>((n1 + kTile - 1) / kTile);
  p.tiles3 = static_cast<int>((n3 + kTile - 1) / kTile);
  p.nsb = static_cast<int>((n2 + kSuper - 1) / kSuper);
  const int per = p.split ? 32 : 64;
  const int64_t images = (n2 + per - 1) / per;
  const double entries = static_cast<double>(n1) * static_cast<double>(n3);
  const double packed = static_cast<double>(p.tiles1 + (alias ? 0 : p.tiles3)) * static_cast<double>(images) * kStageBytes;
  const int64_t words = static_cast<int64_t>(h->d) * h->b;
  auto choose = [&](DirectPlan& q, double rate) {
    choose_tiles(q, alias, 1, entries, 0.5 * h->d * (sets + 1), rate, 1.35e9,
                 sets == 1 ? std::min(1.0, static_cast<double>(kWindow) / static_cast<double>(h->b)) : 0.0, packed,
                 !batch && (sets > 1 || entries <= 16.8e6), sets == 1, batch, sms);
  };
  choose(p, 2.05e11);
  // reductions to few words queue up (see sum_copies), where each split of the
  // inner dimension adds its own share: few splits there.  A batch has at most four
  // copies: 242 x 6456 BF16, b = 64, d = 1 took 89 us an instance with the splits for
  // the full rate, 42 by the spectra, 12 so.  The estimate stays the full rate's,
  // which the choice of route was fitted with.
  const double spread = (batch ? 4.0 : sets > 1 ? 1e9 : 256.0) * static_cast<double>(words) / 1024.0;
  const double rate = 2.3e10 * std::pow(spread, 0.53);
  if (rate < 2.05e11) {
    const double seconds = p.seconds;
    choose(p, rate);
    p.seconds = seconds;
  }
  // large operands: read (twice where their inner indices are balanced) and
  // packed at 5 TB/s; small ones are in the fixed part
  if (p.beyond_l2) {
    const double values = static_cast<double>(alias ? n1 : n1 + n3) * static_cast<double>(n2);
    p.seconds += (values * (dt == CMS_F64 ? 8.0 : dt == CMS_BF16 ? 2.0 : 4.0) * (alias ? 1.0 : 2.0) + packed) / 5e12;
  }
  // (a batch's products queue up less: others' additions are under way too)
  p.copies = sets > 1 ? 1 : sum_copies(words, static_cast<int64_t>(p.units) * p.splits);
  if (batch) p.copies = std::min(p.copies, 4);
  p.sets = sets;
  size_t o = 0;
  const int t3 = alias ? 0 : p.tiles3;
  // sums and the ticket (zero before a run)
  p.acc_bytes = static_cast<size_t>(p.copies) * sets * words * 8;
  p.off_acc = o;    o = al1k(o + p.acc_bytes + 256);
  p.zero_bytes = o;
  p.off_grid = o;
  if (p.grid) {
    // (whole bands of the order of units)
    const size_t row = static_cast<size_t>(p.parts) * p.tiles3 * kTile * kTile * sizeof(float);
    p.band = p.tiles1;
    if (row * p.tiles1 > kMaxStored) p.band = std::max(kBand, static_cast<int>(kMaxStored / row) / kBand * kBand);
    o = al1k(o + row * p.band);
  }
  p.off_work = o;   o = al1k(o + (batch ? 0 : tile_work_bytes(p.blocks, p.need_fold, p.need_hand, p.need_merge)));
  p.off_scale = o;  o = al1k(o + sizeof(DirectScale));
  p.off_blocks = o; o = al1k(o + static_cast<size_t>(p.tiles1 + t3) * p.nsb * sizeof(int2));
  p.off_bal = o;
  if (!alias) o = al1k(o + static_cast<size_t>(n2));
  p.off_pa = o;     o = al1k(o + static_cast<size_t>(p.tiles1) * images * kStageBytes);
  p.off_pb = alias ? p.off_pa : o;
  if (!alias) o = al1k(o + static_cast<size_t>(p.tiles3) * images * kStageBytes);
  p.ws_bytes = o;
  return p;
}

// Estimated time of the transform route (make_sketch_plan): launches, the
// conventional 5 b log2 b + 4 b flops per repetition and inner index, and the
// gathers of its front end (every entry of a_k and b_k for each computed row),
// at rates fitted per kernel family to 160 calls of n = 64 .. 16384, b = n / 8
// .. 32 n, 64 to 8192 inner indices.  Of 1330 calls of n = 8 .. 17000, b = 2 .. 400 n,
// 64 to 2 M inner indices, every storage type, 7 are slower by the chosen route than
// by the spectra by more than 8%, at most by 1.37 (4667 x 14591 x 4018 FP32, b = 600, d
// = 1: 0.76 and 0.56 ms) (n = 454, K = 142, b = 810, d = 4 BF16:
// 96 us by the spectra, 44 us this way; n = 6746, K = 184, b = 1620, d = 4 the
// other way round: 160 and 1136 us).
static double transform_seconds(const SketchPlan& p, int64_t n1, int64_t n2, int64_t n3, bool batch) {
  const double b = static_cast<double>(p.b);
  const double dk = static_cast<double>(p.d) * static_cast<double>(n2);
  const double gflop = dk * (5.0 * b * std::log2(std::max(b, 2.0)) + 4.0 * b) * 1e-9;
  const int rows = p.fast ? (p.nrows + 1) / 2 * 2 : p.nrows;   // the register kernels take two at a time
  const double mgather = dk * rows * static_cast<double>(n1 + n3) * 1e-6;
  double fixed, work;
  if (p.wide) fixed = 60.0, work = 66.0 * gflop;
  else if (p.ws) fixed = 50.0, work = 25.0 * gflop;
  else if (!p.fast) fixed = 34.0, work = 208.0 * gflop + 4.0 * mgather;
  else if (p.tmem_rec) fixed = 95.0, work = 30.0 * gflop + 1.6 * mgather;
  else fixed = 50.0, work = 52.0 * gflop + 1.6 * mgather;
  // a row's block adds up the partial spectra of the inner dimension's chunks,
  // 256 points at a time: latency where the rows are few, shared in a batch
  const double inverse = (p.fast ? 0.13 : 0.09) * p.nkc * static_cast<double>(p.C) / 256.0;
  return 1e-6 * (batch ? work + 12.0 : fixed + work + inverse);
}

// Pre-sketched operands: the direct route's tiles over b x b x n2 for each
// repetition.
PrePlan make_pre_plan(const cms_hashes* h, int64_t n1, int64_t n2, int64_t n3, bool alias, int sms) {
  PrePlan q;
  if (h->C <= 0 || h->R > kTile || h->d_perm == nullptr) return q;
  q.R = static_cast<int>(h->R);
  q.C = static_cast<int>(h->C);
  q.classes = kTile / q.R;
  q.tiles = (q.C + q.classes - 1) / q.classes;
  if (q.tiles > 128) return q;    // b above about 16384 is never cheap
  if (h->b < 64) return q;        // nor is a tile with few rows (5120 x 415, b = 27, d = 3: 325 us, 175 by the spectra)
  const int64_t rows = static_cast<int64_t>(q.tiles) * kTile;
  DirectPlan& p = q.direct;
  p.split = true;
  p.tiles1 = p.tiles3 = q.tiles;
  p.nsb = static_cast<int>((n2 + kSuper - 1) / kSuper);
  const double packed = 2.0 * static_cast<double>(rows) * static_cast<double>(n2) * 4.0 * h->d;
  choose_tiles(p, false, h->d, static_cast<double>(rows) * rows, 1.0, 5.0e11, 4e9, 0.0, packed, false, true, false, sms);
  const double n = static_cast<double>(alias ? n1 : n1 + n3), k = static_cast<double>(p.nsb) * kSuper;
  // sums of rows: 5 TB/s together, 24 GB/s a block of which 304 run at a time
  // (10847 x 947 x 5263 BF16, b = 128, d = 1: 16 blocks, 0.33 ms, 0.18 by the spectra)
  const double blocks = 2.0 * p.nsb * q.tiles * h->d;
  const double sums = std::max(static_cast<double>(n1 + n3) * k * h->d * 4.0 / 5e12,
                               static_cast<double>(std::max(n1, n3)) * 512.0 / q.tiles * std::max(1.0, blocks / 304.0) / 2.4e10);
  p.seconds += 14e-6 + n * k * 8.0 / 4e12 + sums +
              2.0 * static_cast<double>(rows) * k * h->d * 4.0 / 3e12;
  // (beyond L2 the measured times were 1.0 to 1.5 of the rest)
  if (p.beyond_l2) p.seconds = 1.1 * (p.seconds + (alias ? 0.0 : n * k * 4.0 / 5e12));
  const int64_t words = static_cast<int64_t>(h->d) * h->b;
  p.copies = sum_copies(words, static_cast<int64_t>(p.units) * p.splits);
  const int64_t images = (n2 + 31) / 32;
  size_t o = 0;
  p.acc_bytes = static_cast<size_t>(p.copies) * words * 8;
  // sums and a ticket per repetition: zero before a run
  p.off_acc = o;    o = al1k(o + p.acc_bytes + 256);
  p.zero_bytes = o;
  p.off_work = o;   o = al1k(o + tile_work_bytes(p.blocks, p.need_fold, p.need_hand, p.need_merge));
  p.off_scale = o;  o = al1k(o + sizeof(DirectScale) * h->d);
  q.rep_blocks = 2 * q.tiles * p.nsb;
  p.off_blocks = o; o = al1k(o + static_cast<size_t>(q.rep_blocks) * h->d * sizeof(int2));
  const size_t side = static_cast<size_t>(q.tiles) * images * kStageBytes;
  q.rep_images = 2 * side;
  p.off_pa = o;
  p.off_pb = o + side;
  o = al1k(o + q.rep_images * h->d);
  q.off_ent = o;    o = al1k(o + static_cast<size_t>(2 * h->d) * h->n * 4);
  q.off_start = o;  o = al1k(o + static_cast<size_t>(2 * h->d) * (rows + 1) * 4);
  q.off_vhs = o;    o = al1k(o + static_cast<size_t>(2) * rows * 4);
  p.off_bal = o;
  if (!alias) o = al1k(o + static_cast<size_t>(n2));
  q.off_slab = o;   o = al1k(o + static_cast<size_t>(p.nsb) * (alias ? n1 : n1 + n3) * kSuper * 4);
  p.ws_bytes = o;
  q.usable = true;
  return q;
}

bool choose_direct(const cms_hashes* h, const SketchPlan& plan, int64_t n1, int64_t n2, int64_t n3, int dt, bool alias,
                   int sms, DirectPlan* out, bool batch) {
  // under 64 inner indices the packing and the padding to a superblock show;
  // the launches of a batch are shared by its instances
  if (n2 < 64 || n1 < 1 || n3 < 1 || h->n > 65535 || !tile_kernel_usable()) return false;
  // (no plan for calls that the launches alone decide: planning is host time)
  const double transform = transform_seconds(plan, n1, n2, n3, batch);
  if (!batch && transform <= kFixedSeconds + kMargin + 3e-6) return false;
  *out = make_direct_plan(h, n1, n2, n3, dt, alias, sms, 1, batch);
  double best = out->ws_bytes <= kDirectMaxWorkspace ? out->seconds - (batch ? kFixedSeconds : 0.0) : 1e30;
  if (!batch) {
    const PrePlan pre = make_pre_plan(h, n1, n2, n3, alias, sms);
    if (pre.usable && pre.direct.seconds < best && pre.direct.ws_bytes <= kDirectMaxWorkspace) {
      *out = pre.direct;
      out->pre = true;
      out->alias_operands = alias;
      out->sms = sms;
      best = pre.direct.seconds;
    }
  }
  // a margin for the estimates' error: where both are mostly launches, and a
  // tenth beyond L2.  In a batch the other way round there with several
  // repetitions: its transform body takes up to 2.6 times as long as the single
  // call's (6827 x 58270 FP32, b = 2592, d = 3: 10.9 ms an instance, 8.1 by the tiles),
  // with one as long (5022 x 19702, b = 3125, d = 1: 1.03 and 1.69).
  const double beyond = !out->beyond_l2 ? 1.0 : !batch ? 1.1 : h->d > 1 ? 1.0 / 1.2 : 1.0;
  return best * beyond + (batch ? 0.0 : kMargin) < transform;
}

// The masked sums of FINDSIGNIFICANTENTRIES in one pass: an entry is added to
// its bucket's total and, in the mean, to half of the 2 `bits` masked sums,
// against 2 ell products.
bool choose_direct_significant(const cms_hashes* h, const SketchPlan& plan, int64_t n1, int64_t n2, int64_t n3, int dt,
                               bool alias, int sms, int bits, int ell, DirectPlan* out) {
  if (n2 < 64 || n1 < 1 || n3 < 1 || h->n > 65535 || !tile_kernel_usable()) return false;
  *out = make_direct_plan(h, n1, n2, n3, dt, alias, sms, 1 + 2 * bits, false);
  if (out->ws_bytes > kDirectMaxWorkspace) return false;
  return out->seconds + static_cast<double>(out->acc_bytes) / 3e12 < 2.0 * ell * transform_seconds(plan, n1, n2, n3, false);
}

namespace {

PackArgs pack_args(const DirectPlan& p, const void* A, int64_t lda, const void* B, int64_t ldb,
                   int64_t n1, int64_t n2, int64_t n3, int dt, char* ws) {
  int2* blocks = reinterpret_cast<int2*>(ws + p.off_blocks);
  PackArgs a{};
  const int8_t* bal = p.alias ? nullptr : reinterpret_cast<const int8_t*>(ws + p.off_bal);
  a.side[0] = PackSide{A, lda, n1, bal, p.tiles1, reinterpret_cast<uint8_t*>(ws + p.off_pa), blocks};
  a.side[1] = PackSide{B, ldb, n3, bal, p.alias ? 0 : p.tiles3, reinterpret_cast<uint8_t*>(ws + p.off_pb),
                       blocks + static_cast<size_t>(p.tiles1) * p.nsb};
  a.K = n2;
  a.nsb = p.nsb;
  a.dt = dt;
  a.n1 = n1;
  a.n3 = n3;
  a.ticket = reinterpret_cast<uint32_t*>(ws + p.off_acc + p.acc_bytes);
  a.scale = reinterpret_cast<DirectScale*>(ws + p.off_scale);
  return a;
}

TileArgs tile_args(const DirectPlan& p, const cms_hashes* h, int64_t n1, int64_t n2, int64_t n3, char* ws) {
  TileArgs a{};
  a.pa = reinterpret_cast<uint8_t*>(ws + p.off_pa);
  a.pb = reinterpret_cast<uint8_t*>(ws + p.off_pb);
  a.ea = reinterpret_cast<int2*>(ws + p.off_blocks);
  a.eb = p.alias ? a.ea : a.ea + static_cast<size_t>(p.tiles1) * p.nsb;
  a.reps = 1;
  a.scale = reinterpret_cast<DirectScale*>(ws + p.off_scale);
  a.hs = h->d_hs;
  a.acc = reinterpret_cast<unsigned long long*>(ws + p.off_acc);
  a.K = n2;
  a.n = static_cast<int>(h->n);
  a.n1 = static_cast<int>(n1);
  a.n3 = static_cast<int>(n3);
  a.b = static_cast<int>(h->b);
  a.d = h->d;
  a.tiles1 = p.tiles1;
  a.tiles3 = p.tiles3;
  a.nsb = p.nsb;
  a.sb_per_split = p.sb_per_split;
  a.splits = p.splits;
  a.units = p.units;
  a.copies = p.copies;
  a.grid = reinterpret_cast<float*>(ws + p.off_grid);
  a.row0 = a.unit0 = 0;
  a.rows = p.tiles1;
  a.parts = p.parts;
  a.split = p.split ? 1 : 0;
  a.sym = p.alias ? 1 : 0;
  return a;
}

BalanceArgs balance_args(const DirectPlan& p, const void* A, int64_t lda, const void* B, int64_t ldb, int64_t n1,
                         int64_t n2, int64_t n3, int dt, char* ws) {
  BalanceArgs a{};
  a.side[0] = BalanceSide{A, lda, n1};
  a.side[1] = BalanceSide{B, ldb, n3};
  a.K = n2;
  a.dt = dt;
  // warps on every SM, and at least four loads a lane
  a.warps = 1;
  while (a.warps < 8 && n2 * a.warps < 152 * 32 && std::max(n1, n3) >= 256 * a.warps) a.warps *= 2;
  a.bal = reinterpret_cast<int8_t*>(ws + p.off_bal);
  return a;
}

// Zeroed sums and tickets, and the inner indices' powers of two where A and B differ.
cudaError_t launch_start(const DirectPlan& p, bool alias, const void* A, int64_t lda, const void* B, int64_t ldb,
                         int64_t n1, int64_t n2, int64_t n3, int dt, char* ws, cudaStream_t s) {
  if (alias) return cudaMemsetAsync(ws + p.off_acc, 0, p.zero_bytes, s);
  BalanceArgs a = balance_args(p, A, lda, B, ldb, n1, n2, n3, dt, ws);
  a.zero = reinterpret_cast<uint4*>(ws + p.off_acc);
  a.words = static_cast<int64_t>(p.zero_bytes / 16);
  ProfScope prof_scope("k_direct_balance", s);
  const int64_t work = std::max((n2 * a.warps + 7) / 8, (a.words + 1023) / 1024);
  k_direct_balance<<<static_cast<unsigned>(std::min<int64_t>(work, 152 * 8)), 256, 0, s>>>(a);
  return cudaGetLastError();
}

int pack_blocks(const DirectPlan& p) { return p.nsb * (p.tiles1 + (p.alias ? 0 : p.tiles3)); }

template <typename F>
cudaError_t with_smem(F kern, uint32_t bytes) {
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
}

}  // namespace

size_t direct_batch_bytes(int count, int sms) {
  auto al = [](size_t x) { return (x + 255) & ~static_cast<size_t>(255); };
  // arguments, then the tile kernel's words (folds and tiles handed over)
  return al(count * sizeof(PackArgs)) + al(count * sizeof(TileArgs)) + 2 * al((count + 1) * sizeof(int)) +
         al(count * sizeof(BalanceArgs)) + tile_work_bytes(sms, true, true, false);
}

cudaError_t build_direct_batch(const std::vector<DirectSpec>& specs, int sms, void* d_buf, DirectBatch* out,
                               cudaStream_t s) {
  auto al = [](size_t x) { return (x + 255) & ~static_cast<size_t>(255); };
  const int count = static_cast<int>(specs.size());
  std::vector<unsigned char> host(direct_batch_bytes(count, 0));
  out->buf = d_buf;
  out->count = count;
  out->o_tile = al(count * sizeof(PackArgs));
  out->o_ps = out->o_tile + al(count * sizeof(TileArgs));
  out->o_ts = out->o_ps + al((count + 1) * sizeof(int));
  out->o_bal = out->o_ts + al((count + 1) * sizeof(int));
  out->o_work = out->o_bal + al(count * sizeof(BalanceArgs));
  out->balanced = 0;
  int* ps = reinterpret_cast<int*>(host.data() + out->o_ps);
  int* ts = reinterpret_cast<int*>(host.data() + out->o_ts);
  int np = 0, nt = 0;
  out->pack_smem = 0;
  for (int q = 0; q < count; ++q) {
    const DirectSpec& d = specs[q];
    reinterpret_cast<PackArgs*>(host.data())[q] =
        pack_args(d.plan, d.A, d.lda, d.B, d.ldb, d.n1, d.n2, d.n3, d.dt, d.ws);
    reinterpret_cast<TileArgs*>(host.data() + out->o_tile)[q] = tile_args(d.plan, d.h, d.n1, d.n2, d.n3, d.ws);
    if (!d.plan.alias)
      reinterpret_cast<BalanceArgs*>(host.data() + out->o_bal)[out->balanced++] =
          balance_args(d.plan, d.A, d.lda, d.B, d.ldb, d.n1, d.n2, d.n3, d.dt, d.ws);
    ps[q] = np;
    ts[q] = nt;
    np += pack_blocks(d.plan);
    nt += d.plan.units * d.plan.splits;
    out->need_fold |= d.plan.need_fold;
    out->pack_smem = std::max<uint32_t>(out->pack_smem, (d.plan.split ? 4 : 2) * kStageBytes);
  }
  ps[count] = np;
  ts[count] = nt;
  out->pack_blocks = np;
  out->units = nt;
  out->tile_blocks = std::min(nt, sms);
  cudaError_t e = cudaSuccess;
  for (int q = 0; q < count && e == cudaSuccess; ++q)
    e = cudaMemsetAsync(specs[q].ws + specs[q].plan.off_acc, 0, specs[q].plan.zero_bytes, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_buf, host.data(), host.size(), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);   // the host copy goes out of scope
  return e;
}

cudaError_t launch_direct_batched(const DirectBatch& d, cudaStream_t s) {
  if (d.count == 0) return cudaSuccess;
  const char* base = static_cast<const char*>(d.buf);
  cudaError_t e;
  for (int q = 0; q < d.balanced; q += 65535) {
    ProfScope prof_scope("k_direct_balance_batched", s);
    const int blocks = std::min(std::max(152 * 8 / d.balanced, 8), 152 * 2);   // of a product
    k_direct_balance_batched<<<dim3(blocks, std::min(d.balanced - q, 65535)), 256, 0, s>>>(
        reinterpret_cast<const BalanceArgs*>(base + d.o_bal) + q);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  {
    ProfScope prof_scope("k_direct_pack_batched", s);
    if ((e = with_smem(k_direct_pack_batched, d.pack_smem)) != cudaSuccess) return e;
    k_direct_pack_batched<<<d.pack_blocks, 256, d.pack_smem, s>>>(reinterpret_cast<const PackArgs*>(base),
                                                                  reinterpret_cast<const int*>(base + d.o_ps), d.count);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  ProfScope prof_scope("k_direct_tile_batched", s);
  TileLaunch l{};
  l.args = reinterpret_cast<const TileArgs*>(base + d.o_tile);
  l.start = reinterpret_cast<const int*>(base + d.o_ts);
  l.count = d.count;
  l.total = d.units;
  l.need_fold = d.need_fold ? 1 : 0;
  l.need_hand = 1;
  l.work = reinterpret_cast<float*>(const_cast<char*>(base) + d.o_work);
  return launch_tiles(TileArgs{}, l, true, false, d.tile_blocks, s);
}

namespace {

cudaError_t launch_product_tiles(const DirectPlan& p, const TileArgs& a, char* ws, cudaStream_t s) {
  ProfScope prof_scope("k_direct_tile", s);
  TileLaunch l{};
  l.total = a.units * p.splits * a.reps;
  l.need_fold = p.need_fold ? 1 : 0;
  l.need_hand = p.need_hand ? 1 : 0;
  l.need_merge = p.need_merge ? 1 : 0;
  l.work = reinterpret_cast<float*>(ws + p.off_work);
  return launch_tiles(a, l, p.wide, p.grid, std::min(p.blocks, l.total), s);
}

// Stored entries into the sums.
cudaError_t launch_stored(const DirectPlan& p, const cms_hashes* h, const TileArgs& a, cudaStream_t s) {
  cudaError_t e;
  GridArgs g{};
  g.grid = a.grid;
  g.part = static_cast<size_t>(a.rows) * p.tiles3 * kTile * kTile;
  g.row0 = a.row0;
  g.parts = p.parts;
  g.tiles1 = p.tiles1;
  g.tiles3 = p.tiles3;
  g.sym = p.alias ? 1 : 0;
  g.hs = h->d_hs;
  g.scale = a.scale;
  g.acc = a.acc;
  g.copies = p.copies;
  g.bits = (p.sets - 1) / 2;
  g.n = a.n; g.n1 = a.n1; g.n3 = a.n3; g.b = a.b; g.d = a.d;
  // an SM adds 1.35 G/s: few tiles are shared by the repetitions' blocks
  if (p.window) {
    ProfScope window_scope("k_direct_window", s);
    if ((e = with_smem(k_direct_window, 8 * kWindow)) != cudaSuccess) return e;
    const int shares = std::max(1, 152 / h->d);
    return launch_after(k_direct_window, dim3(h->d * shares), 1024, 8 * kWindow, s, g, shares);
  }
  const int tiles = a.rows * p.tiles3, per_tile = kTile / (8 * kGridCols);
  ProfScope grid_scope("k_direct_grid", s);
  const dim3 gg(tiles, per_tile, std::min(h->d, std::max(1, 152 * 2 / (tiles * per_tile))));
  return launch_after(p.sets > 1 ? k_direct_grid<true> : k_direct_grid<false>, gg, 256, 0, s, g);
}

// Zeroed sums, packing, tiles.
cudaError_t launch_sums(const DirectPlan& p, const cms_hashes* h, const void* A, int64_t lda, const void* B,
                        int64_t ldb, int64_t n1, int64_t n2, int64_t n3, int dt, char* ws, cudaStream_t s) {
  cudaError_t e = launch_start(p, p.alias, A, lda, B, ldb, n1, n2, n3, dt, ws, s);
  if (e != cudaSuccess) return e;
  {
    ProfScope prof_scope("k_direct_pack", s);
    const uint32_t smem = (p.split ? 4 : 2) * kStageBytes;
    if ((e = with_smem(k_direct_pack, smem)) != cudaSuccess) return e;
    const PackArgs a = pack_args(p, A, lda, B, ldb, n1, n2, n3, dt, ws);
    if (p.alias) {
      k_direct_pack<<<pack_blocks(p), 256, smem, s>>>(a);
      e = cudaGetLastError();
    } else {
      e = launch_after(k_direct_pack, dim3(pack_blocks(p)), 256, smem, s, a);
    }
    if (e != cudaSuccess) return e;
  }
  TileArgs a = tile_args(p, h, n1, n2, n3, ws);
  if (!p.grid) return launch_product_tiles(p, a, ws, s);
  for (int row = 0; row < p.tiles1 && e == cudaSuccess; row += p.band) {
    // the bands' units follow each other (tile_unit); one band: all of them
    a.row0 = row;
    a.rows = std::min(p.band, p.tiles1 - row);
    a.unit0 = tile_units(row, p.tiles3, p.wide, p.alias);
    a.units = tile_units(row + a.rows, p.tiles3, p.wide, p.alias) - a.unit0;
    e = launch_product_tiles(p, a, ws, s);
    if (e == cudaSuccess) e = launch_stored(p, h, a, s);
  }
  return e;
}

// `per` buckets share a scale.
cudaError_t launch_finish(const DirectPlan& p, const cms_hashes* h, float* c, int64_t per, char* ws, cudaStream_t s) {
  const int64_t len = static_cast<int64_t>(h->d) * h->b;
  const unsigned long long* acc = reinterpret_cast<const unsigned long long*>(ws + p.off_acc);
  const DirectScale* scale = reinterpret_cast<const DirectScale*>(ws + p.off_scale);
  ProfScope prof_scope("k_direct_finish", s);
  if (p.copies > 1)
    return launch_after(k_direct_finish<true>, dim3(static_cast<unsigned>((len + 31) / 32)), 256, 0, s, acc, p.copies, c,
                        len, per, scale, direct_scale_log2(p.split));
  return launch_after(k_direct_finish<false>, dim3(static_cast<unsigned>(std::min<int64_t>((len + 255) / 256, 152 * 8))),
                      256, 0, s, acc, 1, c, len, per, scale, direct_scale_log2(p.split));
}

}  // namespace

namespace {

cudaError_t launch_pre(const DirectPlan& chosen, const cms_hashes* h, const void* A, int64_t lda, const void* B,
                       int64_t ldb, int64_t n1, int64_t n2, int64_t n3, int dt, float* c, char* ws, cudaStream_t s) {
  const bool alias = chosen.alias_operands;
  const PrePlan q = make_pre_plan(h, n1, n2, n3, alias, chosen.sms);
  const DirectPlan& p = q.direct;
  const int rows = q.tiles * kTile;
  PreArgs a{};
  a.X[0] = A; a.X[1] = B;
  a.ld[0] = lda; a.ld[1] = ldb;
  a.n[0] = n1; a.n[1] = n3;
  a.bal = alias ? nullptr : reinterpret_cast<const int8_t*>(ws + p.off_bal);
  a.alias = alias ? 1 : 0;
  a.K = n2;
  a.nsb = p.nsb;
  a.d = h->d;
  a.hn = static_cast<int>(h->n);
  a.R = q.R; a.C = q.C; a.classes = q.classes; a.tiles = q.tiles;
  a.slab[0] = reinterpret_cast<float*>(ws + q.off_slab);
  a.slab[1] = alias ? a.slab[0] : a.slab[0] + static_cast<size_t>(p.nsb) * n1 * kSuper;
  a.hs = h->d_hs;
  a.perm = h->d_perm;
  a.off = h->d_off;
  a.ent = reinterpret_cast<uint32_t*>(ws + q.off_ent);
  a.start = reinterpret_cast<uint32_t*>(ws + q.off_start);
  a.vhs = reinterpret_cast<uint32_t*>(ws + q.off_vhs);
  a.pack = pack_args(p, nullptr, 0, nullptr, 0, rows, n2, rows, CMS_F32, ws);
  a.rep_images = q.rep_images;
  a.rep_blocks = q.rep_blocks;
  cudaError_t e = launch_start(p, alias, A, lda, B, ldb, n1, n2, n3, dt, ws, s);
  if (e != cudaSuccess) return e;
  {
    ProfScope prof_scope("k_pre_transpose", s);
    void (*const kern)(const PreArgs) = dt == CMS_BF16  ? k_pre_transpose<__nv_bfloat16>
                                        : dt == CMS_F64 ? k_pre_transpose<double>
                                                        : k_pre_transpose<float>;
    // 65535 superblocks a launch, the limit of y (8388480 inner indices)
    const int64_t esz = dt == CMS_BF16 ? 2 : dt == CMS_F64 ? 8 : 4;
    for (int first = 0; first < p.nsb; first += 65535) {
      PreArgs part = a;
      const int64_t k0 = static_cast<int64_t>(first) * kSuper;
      for (int side = 0; side < 2; ++side) {
        part.X[side] = static_cast<const char*>(a.X[side]) + k0 * a.ld[side] * esz;
        part.slab[side] = a.slab[side] + k0 * a.n[side];
      }
      if (a.bal != nullptr) part.bal = a.bal + k0;
      part.K = n2 - k0;
      const dim3 grid(static_cast<unsigned>((std::max(n1, n3) + 31) / 32), std::min(p.nsb - first, 65535), alias ? 1 : 2);
      if (alias) {
        kern<<<grid, 256, 0, s>>>(part);
        e = cudaGetLastError();
      } else {
        e = launch_after(kern, grid, 256, 0, s, part);
      }
      if (e != cudaSuccess) return e;
    }
  }
  {
    ProfScope prof_scope("k_pre_lists", s);
    k_pre_lists<<<dim3((q.C + 7) / 8, 2 * h->d), 256, 0, s>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  {
    ProfScope prof_scope("k_pre_pack", s);
    if ((e = with_smem(k_pre_pack, 4 * kStageBytes)) != cudaSuccess) return e;
    k_pre_pack<<<p.nsb * q.tiles * 2 * h->d, 256, 4 * kStageBytes, s>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  TileArgs ta = tile_args(p, h, rows, n2, rows, ws);
  ta.hs = a.vhs;
  ta.n = rows;
  ta.d = 1;
  ta.reps = h->d;
  ta.rep_images = q.rep_images;
  ta.rep_blocks = q.rep_blocks;
  if ((e = launch_product_tiles(p, ta, ws, s)) != cudaSuccess) return e;
  return launch_finish(p, h, c, h->b, ws, s);
}

}  // namespace

cudaError_t launch_direct(const DirectPlan& p, const cms_hashes* h, const void* A, int64_t lda, const void* B,
                          int64_t ldb, int64_t n1, int64_t n2, int64_t n3, int dt, float* c, char* ws,
                          cudaStream_t s) {
  if (p.pre) return launch_pre(p, h, A, lda, B, ldb, n1, n2, n3, dt, c, ws, s);
  cudaError_t e = launch_sums(p, h, A, lda, B, ldb, n1, n2, n3, dt, ws, s);
  if (e != cudaSuccess) return e;
  return launch_finish(p, h, c, static_cast<int64_t>(h->d) * h->b, ws, s);
}

cudaError_t launch_direct_significant(const DirectPlan& p, const cms_hashes* h, const void* A, int64_t lda,
                                      const void* B, int64_t ldb, int64_t n1, int64_t n2, int64_t n3, int dt,
                                      float delta, uint64_t* keys, char* ws, cudaStream_t s) {
  cudaError_t e = launch_sums(p, h, A, lda, B, ldb, n1, n2, n3, dt, ws, s);
  if (e != cudaSuccess) return e;
  const int64_t len = static_cast<int64_t>(h->d) * h->b;
  ProfScope prof_scope("k_direct_sig_decode", s);
  k_direct_sig_decode<<<static_cast<unsigned>((len + 255) / 256), 256, 0, s>>>(
      reinterpret_cast<const unsigned long long*>(ws + p.off_acc), (p.sets - 1) / 2, len, n1, n3, 0.5f * delta,
      reinterpret_cast<const DirectScale*>(ws + p.off_scale), direct_scale_log2(p.split), keys);
  return cudaGetLastError();
}

}  // namespace cms
