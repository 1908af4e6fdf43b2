// Adafactor on the compact gradient R (Sec. "GaLore with memory-efficient optimizers": Adafactor with
// first-order statistics; the update itself is Shazeer and Stern's, the paper prints none): declarations.
#pragma once

#include "common.cuh"
#include "planes.cuh"

namespace galore {

constexpr double kAdafactorDecay = 0.8;     // beta2_t = 1 - t^-0.8
constexpr float kAdafactorEps1 = 1e-30f;    // added to R^2
constexpr float kAdafactorClip = 1.0f;      // the update is divided by max(1, rms / clip)
constexpr int kAfTileCols = 128;            // tile of the statistics pass: 128 columns x
// 64 rows; 32 or 16 (four per warp, all in flight at once) where such tiles would leave SMs idle; more where a column
// would have more than 64 partial sums to add up
inline int af_tile_rows(int64_t rows, int64_t cols) {
  const int64_t tiles = ((rows + 63) / 64) * ((cols + kAfTileCols - 1) / kAfTileCols);
  const int base = tiles < 64 ? 16 : tiles < 128 ? 32 : 64, least = 16 * (int)((rows + 16 * 64 - 1) / (16 * 64));
  return base > least ? base : least;
}
constexpr int kAfSumBlocks = 592;           // parts of the rms pass's sum: fixed, so its total is reproducible

// One layer's Adafactor step.  R partials, N and M are row-major with their own row pitches.
struct AdafactorItem {
  float* Rpart;            // split-K partials of R; slice 0 receives their sum
  int splits;
  int64_t split_stride;
  int rows, cols;          // shape of R and M
  int64_t r_ld, n_ld, s_ld;
  float* M;                // first moment (fp32)
  float *v_row, *v_col;    // running means of R^2 + eps_1 along rows (rows entries) and columns (cols entries)
  __nv_bfloat16* Nout;     // the new first moment once more, as the operand of the back-projection: bf16, or three
  int64_t n_plane;         // bf16 planes `n_plane` elements apart
  PlaneSplit split;        // a matrix (the projector) to be split into planes beside the update
  float beta1;
  double t;                // completed steps + 1
  float* scratch;          // adafactor_scratch_bytes(rows, cols) bytes
  bool squares_ready;      // the projection has left the sums of R^2 where adafactor_squares() says
  int tile_rows, tiles_r;  // rows of a tile of the sums of R^2, tiles of them: adafactor_group_add() fills them in
};
// Where a projection may leave the sums of R^2: over stretches of kAfTileCols columns (rows x tiles) and of kAfProjectionRows rows (one row
// of sums for each).  False for an R so tall that one thread would have too many of them to add up for a column: steps of four layers
// of 16384 x 512 at rank 64 with the pass over R / without it 195 / 172 us, of 32768 x 512 356 / 368, of 65536 x 512 650 / 681.
constexpr int kAfProjectionRows = 64, kAfProjectionTallest = 256 * kAfProjectionRows;
struct AdafactorSquares {
  float *row, *col;
  int tiles;
};
bool adafactor_squares(const AdafactorItem& item, AdafactorSquares* out);
size_t adafactor_scratch_bytes(int64_t rows, int64_t cols);
galore_status_t launch_adafactor(const AdafactorItem& item, int n_planes, bool early, cudaStream_t st);

// Several layers in the same launches (every reduction stays inside its layer and keeps its order: a
// layer's result does not depend on what it is grouped with).  All items share the number of planes of N.
constexpr int kAdafactorGroup = 32;
template <int CAP>
struct AdafactorArgs {
  AdafactorItem item[CAP];
  int tile_end[CAP];     // running totals of the statistics pass's tiles
  int vec_end[CAP];      // running totals of the 256-entry blocks of v_row | v_col
  float beta2t[CAP];
  int count;
};
using AdafactorGroup = AdafactorArgs<kAdafactorGroup>;
galore_status_t adafactor_group_add(AdafactorGroup& g, const AdafactorItem& item);
galore_status_t launch_adafactor_group(const AdafactorGroup& g, int n_planes, bool early, cudaStream_t st);

}  // namespace galore
