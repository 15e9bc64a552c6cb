// k_direct_tile.cu - the tensor-core tiles of the direct route (k_direct.cu).
//
// One block per SM, 640 threads, over units of work in a fixed order:
//  * warp 1 copies stages (16 KB per operand tile: 32 inner indices as two
//    FP16 terms, or 64 in BF16) with bulk copies, as far ahead as shared
//    memory holds (192 KB);
//  * warp 0 issues the products (tcgen05.mma, 128 x 128 tiles, FP32 sums in
//    tensor memory) for two halves in turn: the two tiles of a 128 x 256 unit
//    (wide), or one tile with its inner indices dealt to the halves;
//  * warps 4-7 and 8-11, one group per half, drain the tensor cores' sums
//    every 64 (FP16 terms) or 128 (BF16) inner indices into FP32 registers, so
//    that the tensor cores work on one half while the other is drained;
//  * warps 12-19 add finished tiles to the buckets (GRID off), handed over
//    through L2, while the next unit is multiplied: the additions (205 G/s on
//    the chip) and the products overlap.
//
// Why 64 or 128 inner indices: the tensor cores cut the products and the sum
// they join to a common exponent; relative to 64 bits the drained sums of
// FP16 terms are off by 4.1e-7 after 128 and 2.1e-7 after 64 inner indices, of
// BF16 (8-bit factors) by 1.6e-7 after 128.  The cross terms hi lo go to a
// second accumulator: in the first, each would be cut to the large sum's
// precision (6.1e-7).  From 64 drains on the registers are folded into words
// of the block's own in L2 every 32 drains: a longer chain of FP32 additions
// to one large sum would lose half a bit per doubling.
//
// What bounds it: shared memory.  A 128 x 128 x 16 product takes 70 clocks on
// resident operands and about 110 beside the copies of the next ones, and the
// scatter warps' reductions pass through the same unit.  Two blocks of 128
// threads a SM that drained their own tiles took 57.3 ms for X^T X of 16384 x
// 32768 BF16 (b = 2^20, d = 7) and 205 us for 4096 x 2048 FP32 (b = 2^16, d =
// 5); this layout takes 50.6 ms and, entries stored, 61 + 106 us.  Two groups
// of 192 threads (each with its own issuer) took 76 ms; keeping the buckets
// in L2 by an evict-last hint on the reductions gave 8% of the 50.6.
//
// Registers: 96 x 640 at launch >= 40 x 128 + 168 x 256 + 48 x 256 after
// setmaxnreg.
#include <algorithm>
#include <atomic>

#include "direct_tile.cuh"
#include "warp_fft.cuh"

namespace cms {
namespace dtile {
namespace {

using namespace wfft;

constexpr int kThreads = 640;
constexpr int kRegsCtl = 40, kRegsEpi = 168, kRegsAdd = 48;
constexpr int kAddWarps = 8;
constexpr int kFold = 32;               // drains between folds
constexpr int kFoldFrom = 64;           // drains above which they are folded
constexpr int kTileFloats = kTile * kTile;
constexpr int kBarMergeFull = 1, kBarMergeFree = 2;   // both groups of drains

__device__ uint32_t g_tile_error = 0;   // 1: a wait gave up

template <bool WIDE> struct Ring {
  static constexpr int kSlots = WIDE ? 4 : 6;
  static constexpr int kBytes = (WIDE ? 3 : 2) * kStageBytes;
};
constexpr uint32_t tile_smem_bytes() { return 1024 + 12 * kStageBytes; }

// 2^e for |e| <= 126
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }

// Shared-memory matrix descriptors of K-major operands in the 128-byte
// swizzle (8-row groups 1024 bytes apart): the low word holds the address, the
// high word is the same for all.
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr) { return ((addr >> 4) & 0x3FFFu) | (1u << 16); }
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);

// The issuing thread's instructions count: at 64 clocks a product they are
// what the tensor cores wait for (a 64-bit descriptor built per product and
// run-time loops around it took 160 clocks each).
template <bool ACC>
__device__ __forceinline__ void mma_f16(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "mov.b64 da, {%1, %4};\n\tmov.b64 db, {%2, %4};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t}" ::"r"(d),
      "r"(a), "r"(b), "r"(idesc), "r"(kDescHi), "n"(ACC ? 1 : 0)
      : "memory");
}
__device__ __forceinline__ void mma_f16(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc, bool acc) {
  if (acc) mma_f16<true>(d, a, b, idesc);
  else mma_f16<false>(d, a, b, idesc);
}

// The products of one stage: 16 inner indices are 32 bytes (2 units of 16)
// along the rows.  The sums start over with the first stage of a drain (first)
// and of the cross terms (cross_first).
__device__ __forceinline__ void stage_split(uint32_t main, uint32_t cross, uint32_t a, uint32_t b, uint32_t idesc,
                                            bool first, bool cross_first) {
  mma_f16(main, a, b, idesc, !first);
  mma_f16(cross, a, b + 4, idesc, !cross_first);
  mma_f16<true>(main, a + 2, b + 2, idesc);
  mma_f16<true>(cross, a + 2, b + 6, idesc);
  mma_f16<true>(cross, a + 4, b, idesc);
  mma_f16<true>(cross, a + 6, b + 2, idesc);
}
__device__ __forceinline__ void stage_bf16(uint32_t main, uint32_t a, uint32_t b, uint32_t idesc, bool first) {
  mma_f16(main, a, b, idesc, !first);
  mma_f16<true>(main, a + 2, b + 2, idesc);
  mma_f16<true>(main, a + 4, b + 4, idesc);
  mma_f16<true>(main, a + 6, b + 6, idesc);
}

// The barrier's phase completes when the tensor-core work issued so far has.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void named_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ void tmem_wait_ld8x2(uint32_t (&a)[8], uint32_t (&b)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
                 "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]), "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7])
               :
               : "memory");
}

__device__ __forceinline__ bool elect_one() {
  uint32_t v;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(v));
  return v != 0;
}

__device__ __forceinline__ int uniform(int v) { return __shfl_sync(0xFFFFFFFFu, v, 0); }

struct Unit {
  const TileArgs* p;
  int q;            // unit within its product's tiles
  int split, rep;
  int ti, tc;       // tile row; column of units
  int st0, nst;     // stages
  int sb0;
  int chunks;       // of two stages
};

// Unit `idx` of the launch.
template <bool WIDE>
__device__ __forceinline__ void get_unit(const TileArgs& one, const TileLaunch& l, int idx, Unit& u) {
  u.p = &one;
  if (l.count > 0) {
    // a batch's units are in falling order of their inner dimension: a block
    // takes one from the front and one from the back in turn, so that the
    // additions of a short product overlap the multiplications of a long one
    const int g = gridDim.x, k = idx / g, r = (k >> 1) * g + idx - k * g;
    idx = k & 1 ? l.total - 1 - r : r;
    int lo = 0, hi = l.count - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (__ldg(l.start + mid) <= idx) lo = mid;
      else hi = mid - 1;
    }
    u.p = l.args + lo;
    idx -= __ldg(l.start + lo);
  }
  const TileArgs& p = *u.p;
  u.q = p.unit0 + idx % p.units;
  idx /= p.units;
  u.split = idx % p.splits;
  u.rep = idx / p.splits;
  tile_unit(u.q, p.tiles1, p.tiles3, WIDE, p.sym != 0, &u.ti, &u.tc);
  const int images = p.split ? 4 : 2, per = kSuper / images;
  u.sb0 = u.split * p.sb_per_split;
  const int per_tile = static_cast<int>((p.K + per - 1) / per);
  u.st0 = u.sb0 * images;
  u.nst = min(per_tile, min(p.nsb, u.sb0 + p.sb_per_split) * images) - u.st0;
  u.chunks = (u.nst + 1) / 2;
}

// Column tile of a half, or -1 when it has none.
template <bool WIDE>
__device__ __forceinline__ int half_col(const Unit& u, int half) {
  if (!WIDE) return u.tc;
  const int tj = 2 * u.tc + half;
  return tj < u.p->tiles3 && (!u.p->sym || tj >= u.ti) ? tj : -1;
}

// (h1 + h2) mod b, with the sign s1 s2 in bit 31.
__device__ __forceinline__ uint32_t bucket_of(uint32_t ha, uint32_t hb, uint32_t b) {
  uint32_t z = (ha & kBucketMask) + (hb & kBucketMask);
  if (z >= b) z -= b;
  return z | ((ha ^ hb) & 0x80000000u);
}

// L2 keeps the sums (59 MB at b = 2^20, d = 7) over the operands' stages.
__device__ __forceinline__ uint64_t policy_keep() {
  uint64_t v;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(v));
  return v;
}
__device__ __forceinline__ void bucket_add(unsigned long long* c, uint32_t z, float v, uint64_t keep) {
  const float w = __uint_as_float(__float_as_uint(v) ^ (z & 0x80000000u));
  asm volatile("red.relaxed.gpu.global.add.L2::cache_hint.u64 [%0], %1, %2;" ::"l"(c + (z & kBucketMask)),
               "l"(__float2ll_rn(w)), "l"(keep)
               : "memory");
}

// A thread's row of a tile: columns one after the other, so that a warp's
// rows make whole lines (rows stored by their threads took 32 sectors an
// instruction; added to 64-bit sums by the splits, 20 us of a small product's
// 60).
__device__ __forceinline__ void store_grid(const TileArgs& p, const float (&acc)[kTile], int part, int ti, int tj,
                                           int row) {
  float* g = p.grid + ((static_cast<size_t>(part) * p.rows + ti - p.row0) * p.tiles3 + tj) * kTileFloats + row;
#pragma unroll
  for (int q = 0; q < kTile; ++q) __stcg(g + q * kTile, acc[q]);
}

// Tensor-memory sums of 128 columns into the registers.
template <bool CROSS>
__device__ __forceinline__ void drain(uint32_t col, uint32_t cross, float f, float (&acc)[kTile]) {
  if constexpr (CROSS) {
#pragma unroll
    for (int g = 0; g < kTile / 8; ++g) {
      uint32_t v[8], w[8];
      tmem_ld8_nowait(col + g * 8, v);
      tmem_ld8_nowait(cross + g * 8, w);
      tmem_wait_ld8x2(v, w);
#pragma unroll
      for (int q = 0; q < 8; ++q)
        acc[g * 8 + q] = fmaf(__uint_as_float(v[q]) + __uint_as_float(w[q]), f, acc[g * 8 + q]);
    }
  } else {
#pragma unroll
    for (int g = 0; g < kTile / 16; ++g) {
      uint32_t v[8], w[8];
      tmem_ld8_nowait(col + g * 16, v);
      tmem_ld8_nowait(col + g * 16 + 8, w);
      tmem_wait_ld8x2(v, w);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        acc[g * 16 + q] = fmaf(__uint_as_float(v[q]), f, acc[g * 16 + q]);
        acc[g * 16 + 8 + q] = fmaf(__uint_as_float(w[q]), f, acc[g * 16 + 8 + q]);
      }
    }
  }
}

template <bool WIDE, bool GRID>
__global__ void __launch_bounds__(kThreads, 1) k_direct_tile(const __grid_constant__ TileArgs one, const TileLaunch l) {
  constexpr int kSlots = Ring<WIDE>::kSlots, kBytes = Ring<WIDE>::kBytes;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[kSlots], freed[kSlots], ready[4], drained[4], stored[2], scattered[2];
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_err;
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31;
  if constexpr (GRID) next_kernel_may_start();
  constexpr int kStoring = WIDE ? 256 : 128;
  if (tid == 0) {
    for (int q = 0; q < kSlots; ++q) { mbar_init(&full[q], 1); mbar_init(&freed[q], 1); }
    for (int q = 0; q < 4; ++q) { mbar_init(&ready[q], 1); mbar_init(&drained[q], WIDE ? 256 : 128); }
    for (int q = 0; q < 2; ++q) { mbar_init(&stored[q], kStoring); mbar_init(&scattered[q], 32 * kAddWarps); }
    s_err = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    tmem_alloc(&s_tmem, 512);
    tmem_relinquish();
  }
  tmem_fence_before_sync();
  __syncthreads();
  tmem_fence_after_sync();
  wait_for_kernel_before();
  const uint32_t tmem = static_cast<uint32_t>(uniform(static_cast<int>(s_tmem)));
  const size_t per_block = static_cast<size_t>((l.need_fold ? 2 : 0) + (l.need_hand ? 4 : 0) + (l.need_merge ? 1 : 0)) * kTileFloats;
  float* work = l.work + blockIdx.x * per_block;
  float* hand = work + (l.need_fold ? 2 : 0) * kTileFloats;
  float* merge = hand + (l.need_hand ? 4 : 0) * kTileFloats;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsCtl));
    if (warp == 1 && lane == 0) {
      // ---- copies ----
      bool ok = true;
      int slot = 0, phase = 0, issued = 0;
      for (int idx = blockIdx.x; idx < l.total && ok; idx += gridDim.x) {
        Unit u;
        get_unit<WIDE>(one, l, idx, u);
        const TileArgs& p = *u.p;
        const int per_tile = static_cast<int>((p.K + (p.split ? 31 : 63)) / (p.split ? 32 : 64));
        const int c0 = half_col<WIDE>(u, 0), c1 = WIDE ? half_col<WIDE>(u, 1) : -1;
        const uint8_t* ga = p.pa + u.rep * p.rep_images + (static_cast<size_t>(u.ti) * per_tile + u.st0) * kStageBytes;
        const uint8_t* gb = p.pb + u.rep * p.rep_images;
        const uint8_t* gb0 = gb + (static_cast<size_t>(max(c0, 0)) * per_tile + u.st0) * kStageBytes;
        const uint8_t* gb1 = gb + (static_cast<size_t>(max(c1, 0)) * per_tile + u.st0) * kStageBytes;
        const uint32_t bytes = (1 + (c0 >= 0) + (c1 >= 0)) * kStageBytes;
        for (int st = 0; st < u.nst; ++st) {
          if (issued >= kSlots) ok = !s_err && mbar_wait_bounded(&freed[slot], phase ^ 1);
          if (!ok) break;
          uint8_t* dst = ring + slot * kBytes;
          const size_t off = static_cast<size_t>(st) * kStageBytes;
          mbar_arrive_expect_tx(&full[slot], bytes);
          bulk_g2s(dst, ga + off, kStageBytes, &full[slot]);
          if (c0 >= 0) bulk_g2s(dst + kStageBytes, gb0 + off, kStageBytes, &full[slot]);
          if (c1 >= 0) bulk_g2s(dst + 2 * kStageBytes, gb1 + off, kStageBytes, &full[slot]);
          ++issued;
          if (++slot == kSlots) { slot = 0; phase ^= 1; }
        }
      }
      if (!ok) s_err = 1;
      // every copy has landed before the block may leave
      for (int q = max(0, issued - kSlots); q < issued; ++q)
        (void)mbar_wait_bounded(&full[q % kSlots], (q / kSlots) & 1);
    } else if (warp == 0) {
      // ---- products: the whole warp, so that slots, descriptors and addresses
      // stay in uniform registers; one lane issues ----
      bool ok = true;
      uint32_t slot = 0, phase = 0;
      int uses[4] = {0, 0, 0, 0};   // of each accumulator (narrow: half * 2 + buffer; wide: buffer)
      const uint32_t ring0 = smem_u32(ring);
      for (int idx = blockIdx.x; idx < l.total && ok; idx += gridDim.x) {
        Unit u;
        get_unit<WIDE>(one, l, idx, u);
        const bool split = uniform(u.p->split) != 0;
        const bool act0 = uniform(half_col<WIDE>(u, 0)) >= 0, act1 = WIDE && uniform(half_col<WIDE>(u, 1)) >= 0;
        const int nst = uniform(u.nst), chunks = uniform(u.chunks);
        // wide: both tiles as one product of 256 columns where both are there
        const int n_cols = act0 && act1 ? 2 * kTile : kTile;
        const uint32_t skip = WIDE && !act0 ? 1 : 0;     // the second tile alone
        // D: FP32; A, B: FP16 (0) or BF16 (1), K-major; N / 8, M / 16
        const uint32_t idesc = (1u << 4) | ((split ? 0u : 1u) << 7) | ((split ? 0u : 1u) << 10) |
                               (static_cast<uint32_t>(n_cols / 8) << 17) | (static_cast<uint32_t>(kTile / 16) << 24);
        for (int ch = 0; ch < chunks; ++ch) {
          const int ns = min(2, nst - 2 * ch);
          // narrow: chunks alternate between the halves' accumulators
          const int buf = WIDE ? (split ? 0 : ch & 1) : (split ? 0 : (ch >> 1) & 1);
          const int a = WIDE ? buf : (ch & 1) * 2 + buf;
          const int used = a == 0 ? uses[0] : a == 1 ? uses[1] : a == 2 ? uses[2] : uses[3];
          if (used > 0) ok = !s_err && mbar_wait_bounded(&drained[a], (used - 1) & 1);
          // (the cross terms of a product of a batch lie where a BF16 product
          // before it had its second buffer)
          if (ok && WIDE && split && ch == 0 && uses[1] > 0) ok = mbar_wait_bounded(&drained[1], (uses[1] - 1) & 1);
          ok = __all_sync(0xFFFFFFFFu, ok);
          if (!ok) break;
          tmem_fence_after_sync();
          const uint32_t main = tmem + (WIDE ? buf * 256 + skip * kTile : (ch & 1) * 256 + buf * kTile);
          const uint32_t cross = WIDE ? tmem + 256 + skip * kTile : main + kTile;
          const bool cross_first = !WIDE || (ch & 1) == 0;      // the cross terms start over
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            if (q >= ns) break;
            ok = __all_sync(0xFFFFFFFFu, mbar_wait_bounded(&full[slot], phase));
            if (!ok) break;
            tmem_fence_after_sync();
            const uint32_t da = desc_lo(ring0 + slot * kBytes);
            const uint32_t db = da + ((1 + skip) * kStageBytes >> 4);
            if (elect_one()) {
              if (split) stage_split(main, cross, da, db, idesc, q == 0, q == 0 && cross_first);
              else stage_bf16(main, da, db, idesc, q == 0);
              mma_commit(&freed[slot]);
              if (q == ns - 1) mma_commit(&ready[a]);
            }
            __syncwarp();
            if (++slot == kSlots) { slot = 0; phase ^= 1; }
          }
          if (!ok) break;
          if (a == 0) ++uses[0]; else if (a == 1) ++uses[1]; else if (a == 2) ++uses[2]; else ++uses[3];
        }
      }
      if (!ok && lane == 0) s_err = 1;
      // the products' arrivals have come before the block may leave
      for (int a = 0; a < 4; ++a) {
        const int used = a == 0 ? uses[0] : a == 1 ? uses[1] : a == 2 ? uses[2] : uses[3];
        if (used > 0) (void)mbar_wait_bounded(&ready[a], (used - 1) & 1);
      }
    }
    __syncwarp();
  } else if (warp >= 12) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsAdd));
    if constexpr (!GRID) {
      // ---- additions into the buckets ----
      bool ok = true;
      int k = 0;   // tiles handed over
      const uint64_t keep = policy_keep();
      for (int idx = blockIdx.x; idx < l.total && ok; idx += gridDim.x, ++k) {
        Unit u;
        get_unit<WIDE>(one, l, idx, u);
        const TileArgs& p = *u.p;
        const int s = k & 1;
        ok = !s_err && mbar_wait_bounded_sleep(&stored[s], (k >> 1) & 1);
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (!ok) break;
        if (!p.scale[u.rep].bad) {
          const size_t set = static_cast<size_t>(p.d) * (p.reps > 1 ? p.reps : 1) * p.b;
          unsigned long long* sums = p.acc + static_cast<size_t>(u.rep) * p.b +
          (p.copies > 1 ? static_cast<size_t>(u.q + u.split) % p.copies * set : 0);
          const uint32_t b = static_cast<uint32_t>(p.b);
          for (int half = 0; half < (WIDE ? 2 : 1); ++half) {
            const int tj = half_col<WIDE>(u, half);
            if (tj < 0) continue;
            const bool mirror = p.sym && u.ti != tj;
            const float* src = hand + (s * 2 + half) * kTileFloats;
            const int j0 = tj * kTile, cols = min(kTile, p.n3 - j0);
            // blocks of 32 rows x 8 columns, taken by the warps in turn; the
            // hashes of the next repetition are on their way while this
            // one's additions leave
            for (int blk = warp - 12; blk < 64; blk += kAddWarps) {
              const int i = u.ti * kTile + (blk & 3) * 32 + lane, q0 = (blk >> 2) * 8;
              if (q0 >= cols) break;
              float v[8];
#pragma unroll
              for (int q = 0; q < 8; ++q) v[q] = __ldcg(src + (q0 + q) * kTile + (blk & 3) * 32 + lane);
              const bool row = i < p.n1;
              const int here = min(8, cols - q0);
              const uint32_t* h1 = p.hs;
              uint32_t hr, hm = 0, hc[8], hx[8];
              auto fetch = [&](const uint32_t* a, const uint32_t* c) {
                hr = row ? __ldg(a + i) : 0;
                if (mirror) hm = row ? __ldg(c + i) : 0;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                  hc[q] = q < here ? __ldg(c + j0 + q0 + q) : 0;
                  if (mirror) hx[q] = q < here ? __ldg(a + j0 + q0 + q) : 0;
                }
              };
              fetch(h1, h1 + p.n);
              for (int t = 0; t < p.d; ++t) {
                unsigned long long* c = sums + static_cast<size_t>(t) * p.b;
                uint32_t zr[8], zm[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                  zr[q] = bucket_of(hr, hc[q], b);
                  zm[q] = mirror ? bucket_of(hx[q], hm, b) : 0;
                }
                h1 += 2 * static_cast<size_t>(p.n);
                if (t + 1 < p.d) fetch(h1, h1 + p.n);
                if (row) {
#pragma unroll
                  for (int q = 0; q < 8; ++q)
                  if (q < here) bucket_add(c, zr[q], v[q], keep);
                  if (mirror) {
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                    if (q < here) bucket_add(c, zm[q], v[q], keep);
                  }
                }
              }
            }
          }
        }
        mbar_arrive(&scattered[s]);
      }
      if (!ok) s_err = 1;
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpi));
    // ---- one group per half: drain, fold, finish ----
    const int half = (warp - 4) >> 2;
    const int row = tid & 127;
    // this group's columns: narrow its half's two buffers (the sum and the cross
    // terms), wide its tile's part of two 256-column buffers
    const uint32_t tm = tmem + (static_cast<uint32_t>(warp & 3) << 21) + half * (WIDE ? kTile : 256);
    constexpr uint32_t kNext = WIDE ? 256 : kTile;    // the other buffer
    float* fold = work + half * kTileFloats + row;
    bool ok = true;
    int used0 = 0, used1 = 0, k = 0;
    bool merged = false;
    // (after a wait that gave up the units go on without waiting: the two
    // groups meet at their barriers the same number of times)
    for (int idx = blockIdx.x; idx < l.total; idx += gridDim.x, ++k) {
      Unit u;
      get_unit<WIDE>(one, l, idx, u);
      const TileArgs& p = *u.p;
      const int tj = half_col<WIDE>(u, half);
      const bool split = p.split != 0;
      const int mine = WIDE ? u.chunks : (u.chunks + 1 - half) / 2;     // drains of this half
      const bool folds = l.need_fold && mine > kFoldFrom;
      const DirectScale sc = p.scale[u.rep];
      float acc[kTile];
#pragma unroll
      for (int q = 0; q < kTile; ++q) acc[q] = 0.f;
      {
        // (plain loads: a programmatic launch may run while the packing still
        // writes the exponents, which the read-only path does not allow)
        const size_t rb = static_cast<size_t>(u.rep) * p.rep_blocks + u.sb0;
        const int2* ea = p.ea + rb + static_cast<size_t>(u.ti) * p.nsb;
        const int2* eb = p.eb + rb + static_cast<size_t>(max(tj, 0)) * p.nsb;
        for (int lc = 0; lc < mine; ++lc) {
          const int ch = WIDE ? lc : 2 * lc + half;
          const int sb = split ? ch >> 1 : ch;
          const int de = ea[sb].x - sc.emax[0] + eb[sb].x - sc.emax[1];
          const float f = de < -126 ? 0.f : pow2f(min(de, 0));
          const int buf = split ? 0 : lc & 1;
          const int a = WIDE ? buf : half * 2 + buf;
          uint64_t* rd = &ready[a];
          const int used = buf ? used1 : used0;
          if (ok) ok = mbar_wait_bounded(rd, used & 1);
          ok = __all_sync(0xFFFFFFFFu, ok);
          if (!ok) break;
          if (buf) ++used1; else ++used0;
          tmem_fence_after_sync();
          if (tj >= 0) {
            if (split && (!WIDE || (ch & 1) || ch == u.chunks - 1)) drain<true>(tm, tm + kNext, f, acc);
            else drain<false>(tm + buf * kNext, 0, f, acc);
          }
          tmem_fence_before_sync();
          mbar_arrive(&drained[a]);
          if (folds && tj >= 0 && (lc + 1) % kFold == 0 && lc + 1 < mine) {
            // one thread adds to each word, in order: the same sum in every run
            const bool first = lc + 1 == kFold;
#pragma unroll
            for (int q = 0; q < kTile; ++q) {
              if (first) __stcg(fold + q * kTile, acc[q]);
              else asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(fold + q * kTile), "f"(acc[q]) : "memory");
              acc[q] = 0.f;
            }
          }
        }
        if (folds && ok && tj >= 0) {
#pragma unroll
          for (int g = 0; g < kTile / 16; ++g) {
            float v[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) v[q] = __ldcg(fold + (g * 16 + q) * kTile);
#pragma unroll
            for (int q = 0; q < 16; ++q) acc[g * 16 + q] += v[q];
          }
        }
      }
      if (!WIDE && !GRID && u.chunks > 1) {
        // the second half's sums join the first's
        if (half == 1) {
          if (merged) named_sync(kBarMergeFree, 256);
#pragma unroll
          for (int q = 0; q < kTile; ++q) __stcg(merge + q * kTile + row, acc[q]);
          named_arrive(kBarMergeFull, 256);
        } else {
          if (merged) named_arrive(kBarMergeFree, 256);
          named_sync(kBarMergeFull, 256);
#pragma unroll
          for (int g = 0; g < kTile / 16; ++g) {
            float v[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) v[q] = __ldcg(merge + (g * 16 + q) * kTile + row);
#pragma unroll
            for (int q = 0; q < 16; ++q) acc[g * 16 + q] += v[q];
          }
        }
        merged = true;
      }
      if (!WIDE && half == 1 && !(GRID && p.parts > p.splits)) continue;
      const float up = pow2f(sc.shift / 2), up2 = pow2f(sc.shift - sc.shift / 2);
#pragma unroll
      for (int q = 0; q < kTile; ++q) acc[q] = acc[q] * up * up2;
      if constexpr (GRID) {
        if (ok && tj >= 0 && !sc.bad) store_grid(p, acc, WIDE ? u.split : u.split * (p.parts / p.splits) + half, u.ti, tj, row);
      } else {
        const int s = k & 1;
        if (k >= 2 && ok) ok = !s_err && mbar_wait_bounded_sleep(&scattered[s], ((k >> 1) - 1) & 1);
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (ok && tj >= 0) {
          float* dst = hand + (s * 2 + half) * kTileFloats + row;
#pragma unroll
          for (int q = 0; q < kTile; ++q) __stcg(dst + q * kTile, acc[q]);
        }
        mbar_arrive(&stored[s]);
      }
    }
    if (!ok) s_err = 1;
  }
  tmem_fence_before_sync();
  __syncthreads();
  if (tid == 0 && s_err) atomicOr(&g_tile_error, 1u);
  if (warp == 0) tmem_dealloc(tmem, 512);
  if (tid == 0) {
    for (int q = 0; q < kSlots; ++q) { mbar_inval(&full[q]); mbar_inval(&freed[q]); }
    for (int q = 0; q < 4; ++q) { mbar_inval(&ready[q]); mbar_inval(&drained[q]); }
    for (int q = 0; q < 2; ++q) { mbar_inval(&stored[q]); mbar_inval(&scattered[q]); }
  }
}

}  // namespace

uint32_t read_clear_error_tile() {
  uint32_t v = 0, zero = 0;
  if (cudaMemcpyFromSymbol(&v, g_tile_error, sizeof(v)) != cudaSuccess) return 0xFFFFFFFFu;
  if (v) cudaMemcpyToSymbol(g_tile_error, &zero, sizeof(zero));
  return v;
}

namespace {
using Kernel = void (*)(const TileArgs, const TileLaunch);
Kernel kernel_of(bool wide, bool grid) {
  return wide ? (grid ? k_direct_tile<true, true> : k_direct_tile<true, false>)
              : (grid ? k_direct_tile<false, true> : k_direct_tile<false, false>);
}
}  // namespace

// The register split needs the launch's registers to add up, or the request
// for more would never be granted; checked once against the compiled kernels.
bool tile_kernel_usable() {
  static std::atomic<int> ok{-1};   // concurrent first calls store the same value
  int v = ok.load(std::memory_order_relaxed);
  if (v < 0) {
    v = 1;
    for (int q = 0; q < 4; ++q) {
      cudaFuncAttributes fa{};
      if (cudaFuncGetAttributes(&fa, kernel_of((q & 1) != 0, (q & 2) != 0)) != cudaSuccess ||
          fa.maxThreadsPerBlock < kThreads || fa.numRegs * kThreads < 128 * kRegsCtl + 256 * kRegsEpi + 32 * kAddWarps * kRegsAdd)
        v = 0;
    }
    ok.store(v, std::memory_order_relaxed);
  }
  return v == 1;
}

cudaError_t launch_tiles(const TileArgs& one, const TileLaunch& l, bool wide, bool grid, int blocks, cudaStream_t s) {
  if (!tile_kernel_usable()) return cudaErrorInvalidConfiguration;
  const Kernel k = kernel_of(wide, grid);
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(tile_smem_bytes()));
  if (e != cudaSuccess) return e;
  // stored entries: small products, set up while the packing ends.  Fused: blocks
  // placed one by one as the packing leaves the SMs cost more than that saves
  // (16384 x 32768 BF16: 51.0 -> 56.3 ms).
  if (grid) return launch_after(k, dim3(blocks), kThreads, tile_smem_bytes(), s, one, l);
  k<<<blocks, kThreads, tile_smem_bytes(), s>>>(one, l);
  return cudaGetLastError();
}

}  // namespace dtile
}  // namespace cms
