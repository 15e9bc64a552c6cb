// direct_tile.cuh - the tiles of the direct route: arguments, order and
// launch (k_direct_tile.cu), shared with the packing and planning side
// (k_direct.cu).
#pragma once

#include "cms_internal.h"

namespace cms {
namespace dtile {

constexpr int kTile = 128;              // rows and columns of a tile
constexpr int kSuper = 128;             // inner indices with one scale
constexpr int kStageBytes = kTile * 128;   // one operand's share of a stage
constexpr int kBand = 12;               // rows of tiles that blocks work through together

struct TileArgs {
  const uint8_t* pa;
  const uint8_t* pb;
  const int2* ea;              // (exponent, -) per superblock
  const int2* eb;
  const DirectScale* scale;
  const uint32_t* hs;          // [t][side][n]
  unsigned long long* acc;     // [copy][t][b]
  int copies;                  // tiles add to copy (tile mod copies)
  // more than one pair of operands (repetitions of pre-sketched operands):
  // bytes and superblocks from one pair's to the next; one scale and b
  // buckets each
  size_t rep_images;
  int rep_blocks;
  int reps;
  // entries in units of the integer sums: [part][tile row - row0][tile
  // column][128 columns][128 rows], a part per split of the inner dimension, or
  // two where a unit's halves hold a share of it each; rows tile rows from row0
  // on, whose units follow unit0
  float* grid;
  int row0, rows, unit0;
  int64_t K;
  int n, n1, n3, b, d;
  int tiles1, tiles3;
  int nsb, sb_per_split, splits;
  int parts;                   // of the grid: splits, or twice as many
  int units;                   // of work per split and repetition (tile_units; of the rows)
  int split;                   // two FP16 terms per value
  int sym;                     // A = X^T, B = X: tiles on and above the diagonal
};

// One launch: a product (count = 0), or the products of a batch, `total`
// units of work in all.  work: per block, folds (two tiles), the tiles handed
// to the scatter warps (four) and the partial tile of the second half (one;
// entries that are stored leave the halves as two parts), as far as the
// launch needs them.
struct TileLaunch {
  const TileArgs* args;        // of a batch, device
  const int* start;            // first unit of each
  int count;
  int total;
  int need_fold, need_hand, need_merge;
  float* work;
};

// Columns of a unit's work: two tiles side by side, or one (its inner indices
// dealt to the block's two halves).
__host__ __device__ inline int unit_cols(int tiles3, bool wide) { return wide ? (tiles3 + 1) / 2 : tiles3; }

// Rows that column c of units has in the band from row r0 on (tiles on and
// above the diagonal when sym).
__host__ __device__ inline int band_rows(int r0, int rows, int c, bool wide, bool sym) {
  if (!sym) return rows;
  const int lim = (wide ? 2 * c + 1 : c) - r0 + 1;
  return lim < 0 ? 0 : (lim < rows ? lim : rows);
}

__host__ __device__ inline int tile_units(int tiles1, int tiles3, bool wide, bool sym) {
  const int cols = unit_cols(tiles3, wide);
  int total = 0;
  for (int r0 = 0; r0 < tiles1; r0 += kBand) {
    const int rows = tiles1 - r0 < kBand ? tiles1 - r0 : kBand;
    const int c0 = sym ? (wide ? r0 / 2 : r0) : 0;
    int c = c0;
    for (; c < cols && sym && c < c0 + kBand; ++c) total += band_rows(r0, rows, c, wide, sym);
    if (c < cols) total += (cols - c) * rows;
  }
  return total;
}

// Tile row and column of units for unit q.
__host__ __device__ inline void tile_unit(int q, int tiles1, int tiles3, bool wide, bool sym, int* row, int* col) {
  const int cols = unit_cols(tiles3, wide);
  for (int r0 = 0; r0 < tiles1; r0 += kBand) {
    const int rows = tiles1 - r0 < kBand ? tiles1 - r0 : kBand;
    const int c0 = sym ? (wide ? r0 / 2 : r0) : 0;
    int c = c0;
    for (; c < cols && sym && c < c0 + kBand; ++c) {
      const int r = band_rows(r0, rows, c, wide, sym);
      if (q < r) { *row = r0 + q; *col = c; return; }
      q -= r;
    }
    if (c >= cols) continue;
    const int full = (cols - c) * rows;
    if (q < full) { *row = r0 + q % rows; *col = c + q / rows; return; }
    q -= full;
  }
  *row = 0;
  *col = 0;
}

// Bytes of `work` for a launch of `blocks` blocks.
inline size_t tile_work_bytes(int blocks, bool fold, bool hand, bool merge) {
  return static_cast<size_t>(blocks) * ((fold ? 2 : 0) + (hand ? 4 : 0) + (merge ? 1 : 0)) * kTile * kTile * sizeof(float);
}

// The kernels of a call follow each other by programmatic launches: the next
// one is set up (its blocks' barriers, tensor memory, zeroed words) while the
// last blocks of the one before finish, and waits for all of its results (256 x
// 256 x 256 in FP64, b = 1024: 37.9 -> 32.3 us a call).  Every block waits, so
// that a kernel's end implies the end of those before it.  What the kernels
// before wrote is read by plain or L2 loads: the read-only path (__ldg) is for
// the hash tables, which are complete before the first of them starts.
__device__ __forceinline__ void next_kernel_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_kernel_before() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... A>
cudaError_t launch_after(void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

bool tile_kernel_usable();
uint32_t read_clear_error_tile();
// one: the product when l.count = 0.  wide: units of two tiles; grid: entries
// stored in TileArgs::grid, else added to the buckets.
cudaError_t launch_tiles(const TileArgs& one, const TileLaunch& l, bool wide, bool grid, int blocks, cudaStream_t s);

}  // namespace dtile
}  // namespace cms
