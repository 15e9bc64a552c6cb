// k_sketch_sparse.cu - COMPRESSEDPRODUCT for sparse inputs (Sec. 2.2, "A and
// B sparse ... nonzeros of a column (row) retrieved in linear time";
// Theorem 5's setting): A given by columns (CSC: colptr, rowidx, val), B by
// rows (CSR: rowptr, colidx, val).  Only inner indices k with a nonzero
// column a_k AND a nonzero row b_k contribute; they are compacted first, in
// increasing k, by a deterministic scan.
//
// The per-k work is the same four-step split as the dense kernels
// (b = R * 1024, a block owns one row f1 for one repetition and a range of
// nonempty k): the pruned first stage scatters the few nonzeros of a_k / b_k
// into Y[f1][z2] = sum s(x) v_x w_b^{f1 h(x)}, one warp per (side, k), in a
// fixed order (lanes with distinct buckets add in parallel, colliding lanes
// in lane order), then the radix-32 x radix-32 warp FFT, the spectral
// product (split across the two sides' warps) and Kahan-compensated
// accumulation, exactly as in k_sketch_fast.cu.
#include <algorithm>
#include <cstdlib>
#include <type_traits>

#include "cms_internal.h"
#include "direct_tile.cuh"
#include "warp_fft.cuh"

namespace cms {
namespace {

using namespace wfft;

constexpr int kC = kFeC;       // 1024
constexpr int kG = 4;          // nonempty inner indices per group
constexpr int kThreads = 256;  // 8 warps = 2 sides x kG
constexpr int kFlush = 16;     // groups between Kahan folds (64 products)
constexpr int kPitch = 33;
constexpr int kRegion = 32 * kPitch;
constexpr int kSplitBlocks = 1024;   // chunks of the inner-index split

struct SparseArgs {
  const int64_t* ptr0;         // colptr of A (side 0)
  const int64_t* ptr1;         // rowptr of B (side 1)
  const int32_t* idx0;         // row indices of A
  const int32_t* idx1;         // column indices of B
  const void* val0;
  const void* val1;
  int nside0, nside1;          // n1, n3
  int n;
  int64_t b;
  int nrows;
  int nkc;                     // k-chunks per (repetition, row): fixed by the launch
  const int32_t* klist;
  const int32_t* kcount;       // device: length of klist (written by the split kernels)
  int ntask;
  int d;
  int skip_empty;              // 1: a block returns at once when the list is empty
  int sepy;                    // 1: scatter into per-warp Y buffers kept zero between groups
  const uint32_t* hs;
  int tw_shift, nhi;
  float2* partial;
};

template <typename T> __device__ __forceinline__ float ld_val(const void* p, int64_t e);
template <> __device__ __forceinline__ float ld_val<float>(const void* p, int64_t e) {
  return __ldg(static_cast<const float*>(p) + e);
}
template <> __device__ __forceinline__ float ld_val<double>(const void* p, int64_t e) {
  return static_cast<float>(__ldg(static_cast<const double*>(p) + e));
}
template <> __device__ __forceinline__ float ld_val<__nv_bfloat16>(const void* p, int64_t e) {
  return __bfloat162float(static_cast<const __nv_bfloat16*>(p)[e]);
}

size_t sparse_smem_bytes(int tw_shift, int nhi, bool sepy) {
  return static_cast<size_t>(2 * kG) * kRegion * 8 + static_cast<size_t>(kC) * 16 +
         (static_cast<size_t>(1) << tw_shift) * 8 + static_cast<size_t>(nhi) * 8 +
         (sepy ? static_cast<size_t>(2 * kG) * kC * 8 : 0);
}

// One (repetition, row, chunk of the list).
template <typename T>
__device__ __forceinline__ void sparse_task(const SparseArgs& p, int task) {
  extern __shared__ __align__(128) unsigned char sm[];
  float2* work = reinterpret_cast<float2*>(sm);
  float4* acc = reinterpret_cast<float4*>(sm + static_cast<size_t>(2 * kG) * kRegion * 8);
  float2* tlo = reinterpret_cast<float2*>(acc + kC);
  float2* thi = tlo + (1 << p.tw_shift);
  // per warp: the scatter target Y (kept zero between groups: each lane
  // clears what it wrote once the FFT has read it)
  float2* ysc = thi + p.nhi;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // chunks slowest: a short list leaves the last ones empty, and the blocks,
  // which take every gridDim-th task, all get their share of the others (with the
  // chunks fastest, one inner index of 640 x 640, b = 2^20, d = 7: 2.33 ms, 1.96 so)
  const int row = task % p.nrows;
  const int t = task / p.nrows % p.d;
  const int kc = task / (p.nrows * p.d);
  const uint32_t f1 = static_cast<uint32_t>(row);
  const int S = 1 << p.tw_shift;
  const ModB modb = make_modb(p.b);
  // the chunking follows the list length found on the device: nkc chunks of
  // a whole number of groups; trailing chunks may be empty (zero partials)
  const int K = *p.kcount;
  const int kchunk = max(kG, ((K + p.nkc - 1) / p.nkc + kG - 1) / kG * kG);
  const int l_begin = min(K, kc * kchunk);
  const int l_end = min(K, l_begin + kchunk);

  for (int i = tid; i < S; i += kThreads) {
    float s, c;
    sincospif(2.0f * static_cast<float>(i) / static_cast<float>(p.b), &s, &c);
    tlo[i] = make_float2(c, -s);
  }
  for (int i = tid; i < p.nhi; i += kThreads) {
    const double a = 2.0 * static_cast<double>(static_cast<int64_t>(i) * S) / static_cast<double>(p.b);
    double s, c;
    sincospi(a, &s, &c);
    thi[i] = make_float2(static_cast<float>(c), static_cast<float>(-s));
  }
  for (int i = tid; i < kC; i += kThreads) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (p.sepy)
    for (int i = tid; i < 2 * kG * kC; i += kThreads) ysc[i] = make_float2(0.f, 0.f);
  float2 anchor[4];
  float2 step;
  {
    float s, c;
    sincospif(2.0f * static_cast<float>(lane) / static_cast<float>(kC), &s, &c);
    step = make_float2(c, -s);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      sincospif(2.0f * static_cast<float>((lane * 8 * q) & (kC - 1)) / static_cast<float>(kC), &s, &c);
      anchor[q] = make_float2(c, -s);
    }
  }
  __syncthreads();

  const int side_w = warp / kG;
  const int g_w = warp % kG;
  float2* region = work + warp * kRegion;
  float2* ybuf = p.sepy ? ysc + warp * kC : region;
  const float2* partner = work + (warp ^ kG) * kRegion;   // same k slot, other side
  const uint32_t* tab = p.hs + (static_cast<size_t>(t) * 2 + side_w) * p.n;
  const int64_t* ptr = side_w ? p.ptr1 : p.ptr0;
  const int32_t* idx = side_w ? p.idx1 : p.idx0;
  const void* val = side_w ? p.val1 : p.val0;
  const int nside = side_w ? p.nside1 : p.nside0;

  float2 part[16];
#pragma unroll
  for (int m = 0; m < 16; ++m) part[m] = make_float2(0.f, 0.f);
  // the only per-group exchange is between the two warps of a k slot (its
  // two sides): they meet at a 64-thread barrier of their own (1 + k slot)
  auto pair_sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(1 + g_w) : "memory"); };

  // one nonzero of the warp's (side, k): its bucket and contribution
  // s(x) v w_b^{f1 h(x)} (a lane without one gets a unique sentinel bucket)
  auto contribution = [&](bool valid, int32_t x, float v, uint32_t w, uint32_t& z2, float2& c) {
    z2 = 0x80000000u | static_cast<uint32_t>(lane);
    c = make_float2(0.f, 0.f);
    if (valid && x >= 0 && x < nside) {
      const uint32_t h = w & kBucketMask;
      float2 tw = wb(tlo, thi, mulmod(h, f1, modb), p.tw_shift);
      if (w >> 31) { tw.x = -tw.x; tw.y = -tw.y; }
      c = make_float2(v * tw.x, v * tw.y);
      z2 = h & (kC - 1);
    }
  };
  // added to Y[z2]: lanes with distinct buckets in parallel, lanes sharing
  // a bucket in lane order (round q takes each bucket's q-th lane, so the
  // rounds are as many as the largest multiplicity)
  auto scatter = [&](uint32_t z2, float2 contrib) {
    const uint32_t same = __match_any_sync(0xFFFFFFFFu, z2);
    const uint32_t rank = __popc(same & ((1u << lane) - 1u));
    const uint32_t nrank = __reduce_max_sync(0xFFFFFFFFu, rank);
    for (uint32_t q = 0; q <= nrank; ++q) {
      if (rank == q && !(z2 >> 31)) {
        float2 y = ybuf[z2];
        y.x += contrib.x;
        y.y += contrib.y;
        ybuf[z2] = y;
      }
      __syncwarp();
    }
  };
  // The first 32 nonzeros of each group's (side, k) are fetched during the
  // two previous groups' FFTs, one dependent level per FFT stage (inner
  // index and column bounds two groups ahead, row index and value and hash
  // one group ahead), and their buckets and contributions formed at the end
  // of the previous group, so the scatter finds them in registers; further
  // nonzeros of a long column are loaded when scattered.
  int64_t pe0 = 0, pe1 = 0;     // this group's column bounds
  int64_t ne0 = 0, ne1 = 0;     // the next group's
  uint32_t pz2;
  float2 pc;
  {
    int32_t px = -1;
    float pv = 0.f;
    uint32_t pw = 0;
    if (l_begin + g_w < l_end) {
      const int k = p.klist[l_begin + g_w];
      pe0 = ptr[k];
      pe1 = ptr[k + 1];
      if (pe0 + lane < pe1) {
        px = idx[pe0 + lane];
        pv = ld_val<T>(val, pe0 + lane);
        if (px >= 0 && px < nside) pw = __ldg(tab + px);
      }
    }
    contribution(pe0 + lane < pe1, px, pv, pw, pz2, pc);
    if (l_begin + kG + g_w < l_end) {
      const int k1 = p.klist[l_begin + kG + g_w];
      ne0 = ptr[k1];
      ne1 = ptr[k1 + 1];
    }
  }

  int group = 0;
  for (int l0 = l_begin; l0 < l_end; l0 += kG, ++group) {
    const int gcnt = min(kG, l_end - l0);
    // ---- scatter the nonzeros of this warp's (side, k) into its zero Y ---
    // (without separate buffers the FFT region is zeroed first)
    if (!p.sepy) {
      pair_sync();   // the partner has read this region's published half
      float4* r4 = reinterpret_cast<float4*>(region);
#pragma unroll
      for (int i = 0; i < kC / 2 / 32; ++i) r4[lane + 32 * i] = make_float4(0.f, 0.f, 0.f, 0.f);
      __syncwarp();
    }
    if (g_w < gcnt) {
      scatter(pz2, pc);
      for (int64_t base = pe0 + 32; base < pe1; base += 32) {
        const int64_t e = base + lane;
        const bool valid = e < pe1;
        int32_t x = -1;
        float v = 0.f;
        uint32_t w = 0;
        if (valid) {
          x = idx[e];
          v = ld_val<T>(val, e);
          if (x >= 0 && x < nside) w = __ldg(tab + x);
        }
        uint32_t z2;
        float2 c;
        contribution(valid, x, v, w, z2, c);
        scatter(z2, c);
      }
    }
    __syncwarp();
    // first prefetch level, two groups ahead: the inner index
    const int ln2 = l0 + 2 * kG + g_w;
    const int nk2 = ln2 < l_end ? p.klist[ln2] : -1;
    // ---- FFT of length 1024 ----------------------------------------------
    float2 x[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) x[j] = ybuf[lane + 32 * j];
    __syncwarp();
    // leave Y zero for the next group: each lane clears the bucket of its
    // nonzero (a column of more than 32 nonzeros clears the whole buffer)
    if (p.sepy && g_w < gcnt) {
      if (pe1 - pe0 > 32) {
        float4* y4 = reinterpret_cast<float4*>(ybuf);
#pragma unroll
        for (int i = 0; i < kC / 2 / 32; ++i) y4[lane + 32 * i] = make_float4(0.f, 0.f, 0.f, 0.f);
      } else if (!(pz2 >> 31)) {
        ybuf[pz2] = make_float2(0.f, 0.f);
      }
    }
    dft32<false>(x);
    // third level, next group: the lane's nonzero (row index and value)
    int32_t nx = -1;
    float nv = 0.f;
    if (ne0 + lane < ne1) {
      nx = idx[ne0 + lane];
      nv = ld_val<T>(val, ne0 + lane);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float2 w = anchor[q];
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        if (q + r > 0) x[8 * q + r] = cmul(x[8 * q + r], w);
        w = cmul(w, step);
      }
    }
    if (p.sepy) pair_sync();   // the partner has read this region's published half
    else __syncwarp();
#pragma unroll
    for (int f = 0; f < 32; ++f) region[f * kPitch + lane] = x[f];
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 32; ++j) x[j] = region[lane * kPitch + j];
    // fourth level, next group: its hash
    const uint32_t nw = (nx >= 0 && nx < nside) ? __ldg(tab + nx) : 0u;
    // second level, two groups ahead: the column bounds
    int64_t qe0 = 0, qe1 = 0;
    if (nk2 >= 0) {
      qe0 = ptr[nk2];
      qe1 = ptr[nk2 + 1];
    }
    dft32<false>(x);
    __syncwarp();
    if (side_w == 0) {
#pragma unroll
      for (int m = 16; m < 32; ++m) region[lane + 32 * m] = x[m];
    } else {
#pragma unroll
      for (int m = 0; m < 16; ++m) region[lane + 32 * m] = x[m];
    }
    pair_sync();   // the partner's half is published
    if (g_w < gcnt) {
      if (side_w == 0) {
#pragma unroll
        for (int m = 0; m < 16; ++m) {
          const float2 q = partner[lane + 32 * m];
          part[m].x = fmaf(x[m].x, q.x, part[m].x);
          part[m].x = fmaf(-x[m].y, q.y, part[m].x);
          part[m].y = fmaf(x[m].x, q.y, part[m].y);
          part[m].y = fmaf(x[m].y, q.x, part[m].y);
        }
      } else {
#pragma unroll
        for (int m = 0; m < 16; ++m) {
          const float2 q = partner[lane + 32 * (16 + m)];
          part[m].x = fmaf(x[16 + m].x, q.x, part[m].x);
          part[m].x = fmaf(-x[16 + m].y, q.y, part[m].x);
          part[m].y = fmaf(x[16 + m].x, q.y, part[m].y);
          part[m].y = fmaf(x[16 + m].y, q.x, part[m].y);
        }
      }
    }
    pe0 = ne0;
    pe1 = ne1;
    contribution(pe0 + lane < pe1, nx, nv, nw, pz2, pc);
    ne0 = qe0;
    ne1 = qe1;
    const bool last = l0 + kG >= l_end;
    if ((group % kFlush) == kFlush - 1 || last) {
      __syncthreads();
      const int own = side_w * 16;
#pragma unroll
      for (int m = 0; m < 16; ++m) {
        region[lane + 32 * (own + m)] = part[m];
        part[m] = make_float2(0.f, 0.f);
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < kC / kThreads; ++u) {
        const int f = tid + kThreads * u;
        const int sd = f >> 9;          // bins f < 512 live with side a
        float2 s = work[(sd * kG + 0) * kRegion + f];
#pragma unroll
        for (int g = 1; g < kG; ++g) {
          const float2 v = work[(sd * kG + g) * kRegion + f];
          s.x += v.x;
          s.y += v.y;
        }
        float4 a = acc[f];
        kahan_add(a.x, a.z, s.x);
        kahan_add(a.y, a.w, s.y);
        acc[f] = a;
      }
      __syncthreads();   // every region read before any warp writes its own again
    }
  }
  __syncthreads();
  float2* out = p.partial + ((static_cast<size_t>(t) * p.nrows + f1) * p.nkc + kc) * kC;
  for (int f = tid; f < kC; f += kThreads) {
    const float4 a = acc[f];
    out[f] = make_float2(a.x - a.z, a.y - a.w);
  }
}

// A few blocks per SM over all tasks: with a block per task the launch took
// 33 us when the list was empty (6156 blocks of the exact sparse workload,
// each alone on its SM, only to return), now 5 us.
template <typename T>
__global__ void __launch_bounds__(kThreads, 1) k_sketch_sparse(const SparseArgs p) {
  if (p.skip_empty && *p.kcount == 0) return;
  for (int task = blockIdx.x; task < p.ntask; task += gridDim.x) {
    sparse_task<T>(p, task);
    __syncthreads();   // the next task initialises the shared memory that this one read
  }
}

// Sparse-k hybrid: the nonempty inner indices split, in increasing k, into
// those whose outer product a_k b_k has at most `limit` terms (sketched
// directly, Sec. 2.2 "sketching a matrix product naively") and the rest
// (the FFT route); limit < 0 sends every nonempty index to the FFT route.
// Two passes over contiguous chunks of k (one block each): counts per
// chunk, and an ordered write of every chunk behind the chunks before it
// (each block adds up their counts; a scan kernel of its own between the two
// cost 6 us of the call).  counts[0] = FFT list length, counts[1] = direct
// list length.
//  The direct list fills dlist from its front; inner indices of more than
// kHeavyTerms terms fill it from its back (DirectTerms::heavy of them, in any
// order): all blocks share each of those.
constexpr int64_t kHeavyTerms = 16384;
__device__ __forceinline__ void classify_k(const int64_t* __restrict__ a_ptr, const int64_t* __restrict__ b_ptr,
                                           int64_t n2, int64_t limit, int64_t k, bool* fft, bool* direct, bool* heavy) {
  int64_t na = 0, nb = 0;
  if (k < n2) {
    na = a_ptr[k + 1] - a_ptr[k];
    nb = b_ptr[k + 1] - b_ptr[k];
  }
  const bool live = na > 0 && nb > 0;
  *direct = live && limit >= 0 && na * nb <= limit;
  *heavy = *direct && na * nb > kHeavyTerms;
  *fft = live && !*direct;
}

// Largest magnitude of n values as the bits of an FP32 number (rounded up;
// infinities and NaN stay above every finite value); the whole warp.
__device__ __forceinline__ uint32_t abs_bits(float v) { return __float_as_uint(v) & 0x7FFFFFFFu; }
__device__ __forceinline__ uint32_t abs_bits(__nv_bfloat16 v) { return abs_bits(__bfloat162float(v)); }
__device__ __forceinline__ uint32_t abs_bits(double v) { return abs_bits(__double2float_ru(fabs(v))); }

template <typename T>
__device__ __forceinline__ uint32_t warp_max_abs(const T* __restrict__ v, const int32_t* __restrict__ idx, int64_t n,
                                                 int nside) {
  uint32_t m = 0;
  for (int64_t q = threadIdx.x & 31; q < n; q += 32)
    if (idx[q] >= 0 && idx[q] < nside) m = max(m, abs_bits(v[q]));
  return __reduce_max_sync(0xFFFFFFFFu, m);
}

// What the integer sums of the direct part need: the largest product of a
// direct inner index, and the number of terms.
struct DirectTerms {
  unsigned long long terms;
  uint32_t max_bits;       // of an FP32 number
  uint32_t heavy;          // length of the list at dlist's back
};

// Power of two by which a term is scaled before it is rounded to an integer:
// the sum of all terms stays below 2^62 (terms < 2^bits, each < 2^(e + 1)).
__device__ __forceinline__ int term_shift(const DirectTerms& m) {
  if (m.max_bits == 0) return 0;
  const int bits = 64 - __clzll(static_cast<long long>(m.terms));
  const int e = max(static_cast<int>(m.max_bits >> 23), 1) - 127;
  return 62 - bits - (e + 1);
}

template <typename T>
__global__ void __launch_bounds__(1024)
k_split_count(const int64_t* __restrict__ a_ptr, const int64_t* __restrict__ b_ptr, int64_t n2, int64_t limit,
              int64_t chunk, int32_t* __restrict__ part, const int32_t* __restrict__ a_idx,
              const T* __restrict__ a_val, const int32_t* __restrict__ b_idx, const T* __restrict__ b_val, int n1,
              int n3, DirectTerms* __restrict__ terms) {
  __shared__ int32_t tot[2];
  if (threadIdx.x < 2) tot[threadIdx.x] = 0;
  __syncthreads();
  const int64_t k0 = static_cast<int64_t>(blockIdx.x) * chunk;
  const int64_t k1 = min(n2, k0 + chunk);
  int cf = 0, cd = 0;
  unsigned long long nterm = 0;
  uint32_t mx = 0;
  for (int64_t base = k0; base < k1; base += blockDim.x) {
    const int64_t k = base + threadIdx.x;
    bool f = false, dr = false, hv = false;
    if (k < k1) classify_k(a_ptr, b_ptr, n2, limit, k, &f, &dr, &hv);
    cf += f;
    cd += dr && !hv;
    if (terms == nullptr) continue;
    // the warp measures its direct inner indices one after the other
    for (unsigned todo = __ballot_sync(0xFFFFFFFFu, dr); todo; todo &= todo - 1) {
      const int64_t kk = base + (threadIdx.x & ~31u) + __ffs(todo) - 1;
      const int64_t a0 = a_ptr[kk], na = a_ptr[kk + 1] - a0, b0 = b_ptr[kk], nb = b_ptr[kk + 1] - b0;
      const uint32_t ma = warp_max_abs(a_val + a0, a_idx + a0, na, n1);
      const uint32_t mb = warp_max_abs(b_val + b0, b_idx + b0, nb, n3);
      nterm += static_cast<unsigned long long>(na * nb);
      const uint32_t inf = 0x7F800000u;
      mx = max(mx, ma >= inf || mb >= inf ? 0x7FC00000u
                                          : __float_as_uint(__fmul_ru(__uint_as_float(ma), __uint_as_float(mb))));
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    cf += __shfl_down_sync(0xFFFFFFFFu, cf, o);
    cd += __shfl_down_sync(0xFFFFFFFFu, cd, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&tot[0], cf);
    atomicAdd(&tot[1], cd);
    if (nterm > 0) {
      atomicAdd(&terms->terms, nterm);
      atomicMax(&terms->max_bits, mx);
    }
  }
  __syncthreads();
  if (threadIdx.x < 2) part[2 * blockIdx.x + threadIdx.x] = tot[threadIdx.x];
}

__global__ void __launch_bounds__(1024)
k_split_write(const int64_t* __restrict__ a_ptr, const int64_t* __restrict__ b_ptr, int64_t n2, int64_t limit,
              int64_t chunk, const int32_t* __restrict__ part, int32_t* __restrict__ flist,
              int32_t* __restrict__ dlist, int32_t* __restrict__ counts, DirectTerms* __restrict__ terms) {
  __shared__ int32_t warp_tot[2][32];
  __shared__ int32_t running[2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // lengths of the lists before this chunk (at most 1024 chunks)
  if (tid < 2) running[tid] = 0;
  __syncthreads();
  for (int side = 0; side < 2; ++side) {
    int32_t v = tid < static_cast<int>(blockIdx.x) ? part[2 * tid + side] : 0;
    v = __reduce_add_sync(0xFFFFFFFFu, v);
    if (lane == 0 && v > 0) atomicAdd(&running[side], v);
  }
  __syncthreads();
  if (blockIdx.x == gridDim.x - 1 && tid < 2) counts[tid] = running[tid] + part[2 * blockIdx.x + tid];
  const int64_t k0 = static_cast<int64_t>(blockIdx.x) * chunk;
  const int64_t k1 = min(n2, k0 + chunk);
  for (int64_t base = k0; base < k1; base += 1024) {
    const int64_t k = base + tid;
    bool f = false, dr = false, hv = false;
    if (k < k1) classify_k(a_ptr, b_ptr, n2, limit, k, &f, &dr, &hv);
    if (hv) dlist[n2 - 1 - static_cast<int64_t>(atomicAdd(&terms->heavy, 1u))] = static_cast<int32_t>(k);
    dr = dr && !hv;
    const unsigned bf = __ballot_sync(0xFFFFFFFFu, f);
    const unsigned bd = __ballot_sync(0xFFFFFFFFu, dr);
    const unsigned lt = (1u << lane) - 1u;
    if (lane == 0) { warp_tot[0][warp] = __popc(bf); warp_tot[1][warp] = __popc(bd); }
    __syncthreads();
    int before_f = 0, before_d = 0;
    for (int w = 0; w < warp; ++w) { before_f += warp_tot[0][w]; before_d += warp_tot[1][w]; }
    if (f) flist[running[0] + before_f + __popc(bf & lt)] = static_cast<int32_t>(k);
    if (dr) dlist[running[1] + before_d + __popc(bd & lt)] = static_cast<int32_t>(k);
    __syncthreads();
    if (tid < 2) {
      int tot = 0;
      for (int w = 0; w < 32; ++w) tot += warp_tot[tid][w];
      running[tid] += tot;
    }
    __syncthreads();
  }
}

template <typename T> __device__ __forceinline__ double val_f64(const T* v, int64_t i);
template <> __device__ __forceinline__ double val_f64<float>(const float* v, int64_t i) { return v[i]; }
template <> __device__ __forceinline__ double val_f64<double>(const double* v, int64_t i) { return v[i]; }
template <> __device__ __forceinline__ double val_f64<__nv_bfloat16>(const __nv_bfloat16* v, int64_t i) {
  return static_cast<double>(__bfloat162float(v[i]));
}

// Direct sketch of the outer products of the listed inner indices: for every
// nonzero pair (A_ik, B_kj) and repetition t, s1(i) s2(j) A_ik B_kj goes to
// bucket (h1(i) + h2(j)) mod b.  A block takes an inner index of the list at a
// time, in pieces of up to 4096 terms from up to kDirN nonzeros, whose values
// and hashes sit in shared memory, so that a term costs its addition alone (6.3
// M random 64-bit reductions of the exact sparse workload: 31 us at the chip's
// 205 G/s; with the hashes read per term and a 64-bit division per pair 42 us).
// A piece is 32 x 128 where both sides have that many, and longer along one
// side where the other is short (a column of 100000 nonzeros against one
// element: 32 x 128 at most took 4.5 ms, 32 threads at work; 0.08 so).  The
// pieces of heavy inner indices are dealt to all blocks, one adding 1.35 G/s (one
// product of 640 x 640, b = 2^20, d = 7: 1.73 ms by one block, 0.12 so).
//  INT: terms rounded to integers at a common scale (term_shift) and added
//       as 64-bit integers: the same sums in any order.
//  else: FP64 (products of two FP32 or BF16 values are exact), added
//       atomically: their order varies, at FP64 rounding.
constexpr int kDirN = 512, kDirTerms = 4096, kDirT = 8;

// Nonzeros of A and of B in a piece of an na x nb outer product.
struct Piece {
  int a, b;
};
__device__ __forceinline__ Piece piece_of(int64_t na, int64_t nb) {
  Piece q;
  if (na <= 32 && nb <= 128) {   // one piece, without the divisions
    q.a = static_cast<int>(na);
    q.b = static_cast<int>(nb);
    return q;
  }
  q.a = static_cast<int>(min(na, static_cast<int64_t>(32)));
  q.b = static_cast<int>(min(nb, static_cast<int64_t>(min(kDirTerms / q.a, kDirN - q.a))));
  q.a = static_cast<int>(min(na, static_cast<int64_t>(min(kDirTerms / q.b, kDirN - q.b))));
  return q;
}

struct ScatterArgs {
  const int64_t* a_ptr;
  const int32_t* a_idx;
  const void* a_val;
  const int64_t* b_ptr;
  const int32_t* b_idx;
  const void* b_val;
  int n1, n3;
  int64_t n, n2;
  const int32_t* dlist;
  const int32_t* counts;
  const uint32_t* hs;
  int d;
  int64_t b;
  double* cd;
  const DirectTerms* terms;
};

template <typename T, bool INT, bool HEAVY>
__device__ __forceinline__ void scatter(const ScatterArgs& p) {
  const int64_t* __restrict__ a_ptr = p.a_ptr;
  const int64_t* __restrict__ b_ptr = p.b_ptr;
  const int32_t* __restrict__ a_idx = p.a_idx;
  const int32_t* __restrict__ b_idx = p.b_idx;
  const T* __restrict__ a_val = static_cast<const T*>(p.a_val);
  const T* __restrict__ b_val = static_cast<const T*>(p.b_val);
  const int32_t* __restrict__ dlist = p.dlist;
  const uint32_t* __restrict__ hs = p.hs;
  const DirectTerms* __restrict__ terms = p.terms;
  double* __restrict__ cd = p.cd;
  const int n1 = p.n1, n3 = p.n3, d = p.d;
  const int64_t n = p.n, n2 = p.n2, b = p.b;
  __shared__ double val[kDirN];            // A's nonzeros, then B's
  __shared__ int pos[kDirN];
  __shared__ uint32_t hash[kDirT][kDirN];
  const int count = HEAVY ? static_cast<int>(terms->heavy) : p.counts[1];
  const int tid = threadIdx.x;
  double up = 1.0;
  if (INT) {
    if (count == 0 || terms->max_bits >= 0x7F800000u) return;   // the conversion writes NaN
    up = ldexp(1.0, term_shift(*terms));
  }
  int q = blockIdx.x;                      // place in the list
  int64_t ca = 0, cb = 0;                  // nonzeros of the piece's corner
  __shared__ long long last[HEAVY ? 256 : 1], part[8];   // of 256 heavy ones: pieces up to each
  int h0 = -256;
  long long c = 0, total = 0, turn = 0;    // this block's next piece, pieces of these 256, and before them
  for (;;) {
    int64_t k;
    if constexpr (!HEAVY) {
      if (q >= count) return;
      k = dlist[q];
    } else {
      while (c >= total) {
        turn += total;
        h0 += 256;
        if (h0 >= count) return;
        long long pieces = 0;
        if (h0 + tid < count) {
          const int64_t kk = dlist[n2 - 1 - (h0 + tid)];
          const int64_t na = a_ptr[kk + 1] - a_ptr[kk], nb = b_ptr[kk + 1] - b_ptr[kk];
          const Piece pc = piece_of(na, nb);
          pieces = (na + pc.a - 1) / pc.a * ((nb + pc.b - 1) / pc.b);
        }
        const int lane = tid & 31, warp = tid >> 5;
        for (int o = 1; o < 32; o <<= 1) {
          const long long y = __shfl_up_sync(0xFFFFFFFFu, pieces, o);
          if (lane >= o) pieces += y;
        }
        __syncthreads();
        if (lane == 31) part[warp] = pieces;
        __syncthreads();
        for (int w = 0; w < warp; ++w) pieces += part[w];
        last[tid] = pieces;
        __syncthreads();
        total = last[255];
        c = (static_cast<long long>(blockIdx.x) + gridDim.x - turn % gridDim.x) % gridDim.x;
      }
      int lo = 0, hi = 255;                // the first with last > c
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (last[mid] > c) hi = mid;
        else lo = mid + 1;
      }
      k = dlist[n2 - 1 - (h0 + lo)];
      ca = c - (lo > 0 ? last[lo - 1] : 0);   // the piece's number, for now
    }
    const int64_t a0 = a_ptr[k], na = a_ptr[k + 1] - a0;
    const int64_t b0 = b_ptr[k], nb = b_ptr[k + 1] - b0;
    const Piece pc = piece_of(na, nb);
    if constexpr (HEAVY) {
      const int64_t per = (nb + pc.b - 1) / pc.b, x = ca;
      ca = x / per * pc.a;
      cb = x % per * pc.b;
    }
    const int la = static_cast<int>(min(na - ca, static_cast<int64_t>(pc.a)));
    const int lb = static_cast<int>(min(nb - cb, static_cast<int64_t>(pc.b)));
    __syncthreads();
    for (int e = tid; e < la + lb; e += 256) {
      // an index outside the matrix marks its entry as none (-1)
      if (e < la) {
        const int i = a_idx[a0 + ca + e];
        pos[e] = i >= 0 && i < n1 ? i : -1;
        val[e] = val_f64<T>(a_val, a0 + ca + e) * up;
      } else {
        const int j = b_idx[b0 + cb + e - la];
        pos[e] = j >= 0 && j < n3 ? j : -1;
        val[e] = val_f64<T>(b_val, b0 + cb + e - la);
      }
    }
    __syncthreads();
    for (int t0 = 0; t0 < d; t0 += kDirT) {
      const int lt = min(kDirT, d - t0);
      if (t0 > 0) __syncthreads();
      for (int e = tid; e < lt * (la + lb); e += 256) {
        const int t = e / (la + lb), x = e - t * (la + lb);
        const uint32_t* row = hs + (static_cast<size_t>(t0 + t) * 2 + (x < la ? 0 : 1)) * n;
        hash[t][x] = pos[x] >= 0 ? row[pos[x]] : 0;
      }
      __syncthreads();
      for (int e = tid; e < la * lb; e += 256) {
        const int i = e / lb, j = la + e - i * lb;
        if (pos[i] < 0 || pos[j] < 0) continue;
        // once per pair: FP64 arithmetic is slow beside the additions
        const double v = val[i] * val[j];
        const long long iv = INT ? __double2ll_rn(v) : 0;
        for (int t = 0; t < lt; ++t) {
          const uint32_t w1 = hash[t][i], w2 = hash[t][j];
          uint32_t z = (w1 & kBucketMask) + (w2 & kBucketMask);
          if (z >= static_cast<uint32_t>(b)) z -= static_cast<uint32_t>(b);
          const bool neg = ((w1 ^ w2) >> 31) != 0;
          double* dst = cd + static_cast<size_t>(t0 + t) * b + z;
          if (INT) atomicAdd(reinterpret_cast<unsigned long long*>(dst), static_cast<unsigned long long>(neg ? -iv : iv));
          else atomicAdd(dst, neg ? -v : v);
        }
      }
    }
    if constexpr (HEAVY) {
      c += gridDim.x;
    } else if ((cb += pc.b) >= nb) {
      cb = 0;
      if ((ca += pc.a) >= na) {
        ca = 0;
        q += gridDim.x;
      }
    }
  }
}

// The list, and beside it (a programmatic launch, where inner indices may be that
// long) the heavy ones: in one kernel their code cost the list's 2 to 3 us of 37.
template <typename T, bool INT>
__global__ void __launch_bounds__(256) k_direct_scatter(const ScatterArgs p) {
  dtile::next_kernel_may_start();
  scatter<T, INT, false>(p);
}
template <typename T, bool INT>
__global__ void __launch_bounds__(256) k_direct_scatter_heavy(const ScatterArgs p) {
  scatter<T, INT, true>(p);
  dtile::wait_for_kernel_before();   // this kernel's end implies the list's
}

// c = FFT-route c + direct part (rounded once to FP32), or the direct part
// alone when no inner index took the FFT route.
template <bool INT>
__global__ void k_add_direct(float* __restrict__ c, const double* __restrict__ cd, int64_t len,
                             const int32_t* __restrict__ counts, const DirectTerms* __restrict__ terms) {
  const bool fft = counts[0] > 0;
  int shift = 0;
  bool bad = false;
  if (INT) {
    if (terms->terms == 0 && fft) return;
    bad = terms->max_bits >= 0x7F800000u;
    shift = term_shift(*terms);
  }
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < len;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const double v = cd[i];
    if (INT && !fft) {   // without FP64 arithmetic (FP64 took 41 us for 3 x 2^20 buckets)
      c[i] = bad ? __int_as_float(0x7FC00000) : scale_pow2(__ll2float_rn(__double_as_longlong(v)), -shift);
    } else if (INT) {
      const double w = ldexp(static_cast<double>(__double_as_longlong(v)), -shift);
      c[i] = bad ? __int_as_float(0x7FC00000) : static_cast<float>(static_cast<double>(c[i]) + w);
    } else {
      c[i] = static_cast<float>(fft ? static_cast<double>(c[i]) + v : v);
    }
  }
}

}  // namespace

int make_sparse_plan(const cms_hashes* h, int64_t n2, int64_t K, int num_sms, size_t smem_optin,
                     SketchPlan* plan, size_t* off_klist, std::string* why) {
  SketchPlan p;
  p.b = h->b;
  p.d = h->d;
  if (h->C != kFeC) {
    *why = "the sparse path needs b to be a multiple of 1024 (b = R * 1024)";
    return CMS_ERR_UNSUPPORTED;
  }
  p.R = h->R;
  p.C = h->C;
  p.nrows = static_cast<int>(p.R / 2 + 1);
  p.nradC = factor_radices(p.C, p.radC, 16);
  int sh = 0;
  while ((static_cast<int64_t>(1) << (2 * sh)) < p.b) ++sh;
  p.tw_shift = sh;
  p.nhi = static_cast<int>((p.b + (static_cast<int64_t>(1) << sh) - 1) >> sh);
  // separate, zero-kept scatter buffers when they fit beside the rest (a
  // debug switch in the environment keeps the in-place form, the path of
  // sketches too long for them)
  p.sparse_sepy = sparse_smem_bytes(p.tw_shift, p.nhi, true) <= smem_optin &&
                  std::getenv("CMS_SPARSE_INPLACE_Y") == nullptr;
  p.smem = sparse_smem_bytes(p.tw_shift, p.nhi, p.sparse_sepy);
  p.G = kG;
  p.threads = kThreads;
  const int64_t units = static_cast<int64_t>(p.d) * p.nrows;
  const int64_t slots = num_sms;
  const int64_t lo = std::max<int64_t>(1, (2 * slots + units - 1) / units);
  const int64_t hi = std::max<int64_t>(lo, 4 * lo);
  // chunks over the list of nonempty k; the workspace covers the largest count
  int64_t nkc;
  if (K < 0) {
    nkc = hi;
  } else {
    nkc = 1;
    double best = -1.0;
    const int64_t maxc = std::max<int64_t>(1, (K + kG - 1) / kG);
    for (int64_t c2 = std::min(lo, maxc); c2 <= std::min(hi, maxc); ++c2) {
      const int64_t tasks = units * c2;
      const int64_t waves = (tasks + slots - 1) / slots;
      const double eff = static_cast<double>(tasks) / static_cast<double>(waves * slots);
      if (eff > best + 1e-9) { best = eff; nkc = c2; }
    }
  }
  const int64_t KK = K < 0 ? n2 : K;
  int64_t kchunk = KK > 0 ? (KK + nkc - 1) / nkc : kG;
  kchunk = ((kchunk + kG - 1) / kG) * kG;
  if (K >= 0) nkc = KK > 0 ? (KK + kchunk - 1) / kchunk : 1;
  p.kchunk = kchunk;
  p.nkc = static_cast<int>(nkc);
  auto align256 = [](size_t x) { return (x + 255) & ~static_cast<size_t>(255); };
  size_t off = 0;
  p.off_partial = off; off = align256(off + static_cast<size_t>(units) * hi * p.C * 8);
  p.off_V = off;       off = align256(off + static_cast<size_t>(units) * p.C * 8);
  p.off_twC = off;     off = align256(off + static_cast<size_t>(p.C) * 8);
  p.off_twR = off;     off = align256(off + static_cast<size_t>(p.R) * 8);
  *off_klist = off;    off = align256(off + static_cast<size_t>(std::max<int64_t>(n2, 1) + 1) * 4);
  // sparse-k hybrid: the direct list, the list counts, the FP64 direct sketch
  p.off_dlist = off;   off = align256(off + (static_cast<size_t>(std::max<int64_t>(n2, 1)) + 2 + 2 * kSplitBlocks) * 4);
  p.off_cd = off;      off = align256(off + static_cast<size_t>(p.d) * p.b * 8 + sizeof(DirectTerms));
  p.ws_bytes = off;
  (void)why;
  *plan = p;
  return CMS_OK;
}

namespace {
DirectTerms* direct_terms(const cms_hashes* h, double* cd) {
  return reinterpret_cast<DirectTerms*>(cd + static_cast<size_t>(h->d) * h->b);
}
}  // namespace

cudaError_t launch_nonempty_split(const cms_hashes* h, const SparseArgsHost& in, int dt, int64_t n2, int64_t limit,
                                  int integer, int32_t* flist, int32_t* dlist, int32_t* counts, int32_t* scratch,
                                  double* cd, cudaStream_t s) {
  // the direct part's sums and its measure start at zero
  cudaError_t e = cudaMemsetAsync(cd, 0, static_cast<size_t>(h->d) * h->b * sizeof(double) + sizeof(DirectTerms), s);
  if (e != cudaSuccess) return e;
  if (n2 <= 0) return cudaMemsetAsync(counts, 0, 2 * sizeof(int32_t), s);
  const int64_t nblk = std::min<int64_t>(kSplitBlocks, (n2 + 1023) / 1024);
  const int64_t chunk = ((n2 + nblk - 1) / nblk + 1023) / 1024 * 1024;
  const unsigned g = static_cast<unsigned>((n2 + chunk - 1) / chunk);
  ProfScope prof_scope("k_nonempty_split", s);
  auto count = [&](auto* tag) {
    using T = std::remove_pointer_t<decltype(tag)>;
    k_split_count<T><<<g, 1024, 0, s>>>(in.a_ptr, in.b_ptr, n2, limit, chunk, scratch, in.a_idx,
                                        static_cast<const T*>(in.a_val), in.b_idx, static_cast<const T*>(in.b_val),
                                        in.n1, in.n3, integer ? direct_terms(h, cd) : nullptr);
  };
  if (dt == CMS_F32) count(static_cast<float*>(nullptr));
  else if (dt == CMS_BF16) count(static_cast<__nv_bfloat16*>(nullptr));
  else count(static_cast<double*>(nullptr));
  k_split_write<<<g, 1024, 0, s>>>(in.a_ptr, in.b_ptr, n2, limit, chunk, scratch, flist, dlist, counts,
                                   direct_terms(h, cd));
  return cudaGetLastError();
}

cudaError_t launch_direct_scatter(const cms_hashes* h, const SparseArgsHost& in, int dt, int integer, int64_t limit,
                                  const int32_t* dlist, const int32_t* counts, int64_t n2, double* cd, cudaStream_t s) {
  if (n2 <= 0) return cudaSuccess;
  // the lists' lengths are on the device: blocks stride over them, and return
  // at once when they are empty (two waves of blocks: with one, those with two
  // inner indices end last, 40.8 us for 2048 of them and 36.7 with two)
  const ScatterArgs a{in.a_ptr, in.a_idx, in.a_val, in.b_ptr, in.b_idx, in.b_val, in.n1, in.n3, h->n, n2, dlist,
                      counts, h->d_hs, h->d, h->b, cd, direct_terms(h, cd)};
  cudaError_t e = cudaSuccess;
  auto go = [&](auto* tag, auto integer_tag) {
    using T = std::remove_pointer_t<decltype(tag)>;
    constexpr bool kInt = decltype(integer_tag)::value;
    {
      ProfScope prof_scope("k_direct_scatter", s);
      k_direct_scatter<T, kInt><<<static_cast<unsigned>(std::min<int64_t>(n2, 152 * 16)), 256, 0, s>>>(a);
      e = cudaGetLastError();
    }
    if (e != cudaSuccess || limit <= kHeavyTerms) return;
    ProfScope prof_scope("k_direct_scatter_heavy", s);
    e = dtile::launch_after(k_direct_scatter_heavy<T, kInt>, dim3(152 * 4), 256, 0, s, a);
  };
  auto both = [&](auto* tag) {
    if (integer) go(tag, std::true_type{});
    else go(tag, std::false_type{});
  };
  if (dt == CMS_F32) both(static_cast<float*>(nullptr));
  else if (dt == CMS_BF16) both(static_cast<__nv_bfloat16*>(nullptr));
  else both(static_cast<double*>(nullptr));
  return e;
}

cudaError_t launch_add_direct(const cms_hashes* h, float* c, double* cd, int integer, const int32_t* counts,
                              cudaStream_t s) {
  const int64_t len = static_cast<int64_t>(h->d) * h->b;
  const unsigned grid = static_cast<unsigned>(std::min<int64_t>((len + 255) / 256, 4096));
  ProfScope prof_scope("k_add_direct", s);
  if (integer) k_add_direct<true><<<grid, 256, 0, s>>>(c, cd, len, counts, direct_terms(h, cd));
  else k_add_direct<false><<<grid, 256, 0, s>>>(c, cd, len, counts, nullptr);
  return cudaGetLastError();
}

cudaError_t launch_sketch_sparse(const SketchPlan& plan, const cms_hashes* h, const SparseArgsHost& in,
                                 int dt, const int32_t* klist, const int32_t* kcount, int skip_empty,
                                 float2* partial, cudaStream_t s) {
  SparseArgs a{};
  a.ptr0 = in.a_ptr; a.ptr1 = in.b_ptr;
  a.idx0 = in.a_idx; a.idx1 = in.b_idx;
  a.val0 = in.a_val; a.val1 = in.b_val;
  a.n = static_cast<int>(h->n);
  a.nside0 = in.n1; a.nside1 = in.n3;
  a.b = plan.b;
  a.nrows = plan.nrows;
  a.nkc = plan.nkc;
  a.klist = klist;
  a.kcount = kcount;
  a.skip_empty = skip_empty;
  a.sepy = plan.sparse_sepy ? 1 : 0;
  a.hs = h->d_hs;
  a.tw_shift = plan.tw_shift;
  a.nhi = plan.nhi;
  a.partial = partial;
  const int smem = static_cast<int>(plan.smem);
  a.ntask = static_cast<int>(static_cast<int64_t>(plan.d) * plan.nrows * plan.nkc);
  a.d = plan.d;
  const unsigned grid = static_cast<unsigned>(std::min(a.ntask, 4 * 152));
  cudaError_t e = cudaSuccess;
  switch (dt) {
    case CMS_F32:
      e = cudaFuncSetAttribute(k_sketch_sparse<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (e == cudaSuccess) { ProfScope ps("k_sketch_sparse", s); k_sketch_sparse<float><<<grid, kThreads, smem, s>>>(a); }
      break;
    case CMS_BF16:
      e = cudaFuncSetAttribute(k_sketch_sparse<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (e == cudaSuccess) { ProfScope ps("k_sketch_sparse", s); k_sketch_sparse<__nv_bfloat16><<<grid, kThreads, smem, s>>>(a); }
      break;
    default:
      e = cudaFuncSetAttribute(k_sketch_sparse<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (e == cudaSuccess) { ProfScope ps("k_sketch_sparse", s); k_sketch_sparse<double><<<grid, kThreads, smem, s>>>(a); }
      break;
  }
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace cms
