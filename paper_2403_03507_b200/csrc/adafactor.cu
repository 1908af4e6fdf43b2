// Adafactor with first-order statistics on the compact gradient R (rows x cols):
//   v_row <- b2 v_row + (1 - b2) mean_j (R^2 + eps_1),  v_col likewise along columns,  b2 = 1 - t^-0.8
//   U = R / sqrt(v_row v_col^T / mean(v_row)),  U <- U / max(1, rms(U) / d)
//   M <- beta1 M + (1 - beta1) U,  N = M
// Four passes, each a plain streaming kernel, every reduction in a fixed order (run-to-run identical):
//   1. sums the split-K partials of R and leaves per-tile row and column sums of R^2 (the projection of a batch on the tensor
//      path leaves them itself: the pass is left out),
//   2. folds those into v_row, v_col (one thread per entry), with 1 / sqrt of each and the blocks' sums of v_row,
//   3. sum of (R / sqrt(v_row v_col^T))^2 over a fixed set of parts, one per warp,
//   4. the clipped update, the momentum and N; the scalar sqrt(mean(v_row)) that pass 2 cannot know yet enters here.
// A small matrix is bound by the latency of the four launches: loops over partial sums keep
// their loads in flight together (a 1152 x 958 matrix at rank 80: pass 1 and 2 took 25 us one load after another).
// R is r x n (or m x r) fp32, a small matrix beside G and W; the passes are bound by its HBM traffic.
#include "adafactor.cuh"

#include <cuda_bf16.h>

#include "launch.cuh"

namespace galore {
namespace {

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// every thread of a 256-thread CTA gets the sum
__device__ __forceinline__ double block_sum_256d(double v, double* red) {
  v = warp_sum_d(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
#pragma unroll
  for (int i = 0; i < 8; ++i) s += red[i];
  return s;
}

struct AfLayout {
  float* rowpart;    // rows x tiles_c
  float* colpart;    // tiles_r x cols
  float* a_row;      // rows: rsqrt(v_row)
  float* b_col;      // cols: rsqrt(v_col)        (U = sqrt(mean(v_row)) R a_row b_col^T)
  double* sums;      // kAfSumBlocks partial sums of (U / sqrt(mean(v_row)))^2
  double* row_sums;  // sums of v_row over blocks of 256 entries
  int tile_rows, tiles_r, tiles_c;
};
__host__ __device__ inline AfLayout af_layout(const AdafactorItem& it) {
  const int rows = it.rows, cols = it.cols;
  float* const scratch = it.scratch;
  AfLayout a;
  a.tile_rows = it.tile_rows;
  a.tiles_r = it.tiles_r;
  a.tiles_c = (cols + kAfTileCols - 1) / kAfTileCols;
  a.sums = reinterpret_cast<double*>(scratch);
  a.row_sums = a.sums + kAfSumBlocks + 8;
  a.rowpart = scratch + 2 * (kAfSumBlocks + 8 + (rows + 255) / 256 * 2);
  // every section starts on a 16-byte boundary
  a.colpart = a.rowpart + ((size_t)rows * a.tiles_c + 3) / 4 * 4;
  a.a_row = a.colpart + ((size_t)a.tiles_r * cols + 3) / 4 * 4;
  a.b_col = a.a_row + (rows + 3) / 4 * 4;
  return a;
}

// item whose running total first exceeds b, and b's position inside it; every lane looks at one of them (one after the other
// in every CTA of the statistics: 82 us for half of the LLaMA-1B set, 75 so)
static_assert(kAdafactorGroup <= 32, "one lane per item");
template <int CAP>
__device__ __forceinline__ int find_item(const int* end, int count, int b, int& local) {
  if constexpr (CAP == 1) {
    local = b;
    return 0;
  }
  const int lane = threadIdx.x & 31;
  const int mine = lane < count ? end[lane] : 0x7fffffff;
  const int i = __popc(__ballot_sync(0xffffffffu, mine <= b));
  local = b - (i ? end[i - 1] : 0);
  return i;
}

// Warp w of the CTA takes the rows w, w + 4, ... of the tile; a lane holds four neighbouring columns
// (one 16-byte load when the rows allow it).  Row sums by warp shuffle, column sums in the lanes'
// registers, combined across the four warps in a fixed order.
template <int CAP>
__global__ void __launch_bounds__(kAfTileCols) af_stats_kernel(const __grid_constant__ AdafactorArgs<CAP> g) {
  {
    const int first = (int)(blockIdx.x * blockDim.x + threadIdx.x), stride = (int)(gridDim.x * blockDim.x);
    for (int i = 0; i < (CAP == 1 ? 1 : g.count); ++i) plane_split_part(g.item[i].split, first, stride);
  }
  grid_dependency_wait();
  grid_launch_dependents();
  __shared__ float cs[kAfTileCols / 32][kAfTileCols];
  int tile;
  const AdafactorItem& it = g.item[find_item<CAP>(g.tile_end, g.count, blockIdx.x, tile)];
  const AfLayout a = af_layout(it);
  const int tile_r = tile / a.tiles_c, tile_c = tile % a.tiles_c;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r0 = tile_r * a.tile_rows, c0 = tile_c * kAfTileCols + 4 * lane;
  const bool vec = (it.r_ld % 4) == 0 && (it.split_stride % 4) == 0 && ((uintptr_t)it.Rpart & 15) == 0 && c0 + 3 < it.cols;
  float col[4] = {0.f, 0.f, 0.f, 0.f};
  // the four columns of one row: the sum of the K slices, written back when there are several
  auto load_row = [&](int row, float (&v)[4]) {
    v[0] = v[1] = v[2] = v[3] = 0.f;
    if (row >= it.rows) return;
    const int64_t at = (int64_t)row * it.r_ld + c0;
    if (vec) {
      float4 x = *reinterpret_cast<const float4*>(it.Rpart + at);
      for (int s0 = 1; s0 < it.splits; s0 += 4) {          // four slices in flight, added in order
        float4 y[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (s0 + k < it.splits) y[k] = *reinterpret_cast<const float4*>(it.Rpart + at + (s0 + k) * it.split_stride);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (s0 + k < it.splits) { x.x += y[k].x; x.y += y[k].y; x.z += y[k].z; x.w += y[k].w; }
      }
      if (it.splits > 1) *reinterpret_cast<float4*>(it.Rpart + at) = x;
      v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (c0 + k < it.cols) {
          float x = it.Rpart[at + k];
          for (int s = 1; s < it.splits; ++s) x += it.Rpart[at + k + s * it.split_stride];
          if (it.splits > 1) it.Rpart[at + k] = x;
          v[k] = x;
        }
    }
  };
  constexpr int kWarps = kAfTileCols / 32, kFlight = 4;      // four rows of a warp in flight
  for (int i = warp; i < a.tile_rows; i += kWarps * kFlight) {
    float v[kFlight][4];
#pragma unroll
    for (int u = 0; u < kFlight; ++u) load_row(r0 + i + u * kWarps, v[u]);
#pragma unroll
    for (int u = 0; u < kFlight; ++u) {
      const int row = r0 + i + u * kWarps;
      float row_sum = 0.f;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float sq = v[u][k] * v[u][k];
        col[k] += sq;
        row_sum += sq;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) row_sum += __shfl_xor_sync(0xffffffffu, row_sum, o);
      if (lane == 0 && row < it.rows) a.rowpart[(size_t)row * a.tiles_c + tile_c] = row_sum;
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) cs[warp][4 * lane + k] = col[k];
  __syncthreads();
  const int c = tile_c * kAfTileCols + threadIdx.x;
  if (c < it.cols) {
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < kAfTileCols / 32; ++w) sum += cs[w][threadIdx.x];
    a.colpart[(size_t)tile_r * it.cols + c] = sum;
  }
}

// sum of `count` floats `step` apart, eight loads in flight, added in order
__device__ __forceinline__ double af_sum(const float* __restrict__ x, int count, size_t step) {
  double s = 0.0;
  for (int k0 = 0; k0 < count; k0 += 8) {
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = k0 + k < count ? x[(size_t)(k0 + k) * step] : 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += (double)v[k];
  }
  return s;
}

// pass 2: entries 0 .. rows-1 are v_row (in blocks of 256 of their own), the next cols entries v_col
template <int CAP>
__global__ void __launch_bounds__(256) af_vectors_kernel(const __grid_constant__ AdafactorArgs<CAP> g) {
  __shared__ double red[8];
  grid_dependency_wait();
  grid_launch_dependents();
  int blk;
  const int which = find_item<CAP>(g.vec_end, g.count, blockIdx.x, blk);
  const AdafactorItem& it = g.item[which];
  const float beta2t = g.beta2t[which];
  const AfLayout a = af_layout(it);
  const int row_blocks = (it.rows + 255) / 256;
  if (blk < row_blocks) {
    const int i = blk * 256 + threadIdx.x;
    float v = 0.f;
    if (i < it.rows) {
      const float mean = (float)(af_sum(a.rowpart + (size_t)i * a.tiles_c, a.tiles_c, 1) / (double)it.cols) + kAdafactorEps1;
      v = fmaf(beta2t, it.v_row[i], (1.f - beta2t) * mean);
      it.v_row[i] = v;
      a.a_row[i] = rsqrtf(v);
    }
    const double s = block_sum_256d((double)v, red);
    if (threadIdx.x == 0) a.row_sums[blk] = s;
  } else {
    const int j = (blk - row_blocks) * 256 + threadIdx.x;
    if (j < it.cols) {
      const float mean = (float)(af_sum(a.colpart + j, a.tiles_r, (size_t)it.cols) / (double)it.rows) + kAdafactorEps1;
      const float v = fmaf(beta2t, it.v_col[j], (1.f - beta2t) * mean);
      it.v_col[j] = v;
      a.b_col[j] = rsqrtf(v);
    }
  }
}

// rows of R in four-column groups where its rows are 16-byte aligned, the ragged end one by one
struct AfRowWalk {
  bool vec;
  int cols4;
};
__device__ __forceinline__ AfRowWalk af_walk(const AdafactorItem& it, bool with_state) {
  AfRowWalk w;
  w.vec = (it.r_ld % 4) == 0 && ((uintptr_t)it.Rpart & 15) == 0;
  if (with_state) w.vec = w.vec && (it.s_ld % 4) == 0 && (it.n_ld % 4) == 0 && (it.n_plane % 4) == 0 && ((uintptr_t)it.M & 15) == 0 && ((uintptr_t)it.Nout & 15) == 0;
  w.cols4 = w.vec ? (it.cols & ~3) : 0;
  return w;
}

// Pass 3: partial sums of U^2.  A part is a row, or a stretch of one where there are few rows, or every kAfSumBlocks-th row
// where there are many; a warp adds up a part, with eight 16-byte loads in flight.  (A CTA per part, with its barriers, took
// 61 us for half of the LLaMA-1B set, this 50.  The other way round the update: 148 x 6 CTAs in one wave, two rows in flight,
// took 151 us, one CTA per row 124.)
constexpr int kRmsThreads = 128;
template <int CAP>
__global__ void __launch_bounds__(kRmsThreads) af_rms_kernel(const __grid_constant__ AdafactorArgs<CAP> g) {
  grid_dependency_wait();
  grid_launch_dependents();
  const AdafactorItem& it = g.item[blockIdx.y];
  const AfLayout a = af_layout(it);
  const AfRowWalk w = af_walk(it, false);
  const int lane = threadIdx.x & 31;
  const int part = (int)(blockIdx.x * (kRmsThreads / 32) + (threadIdx.x >> 5));
  if (part >= kAfSumBlocks) return;
  const int stretches = it.rows >= kAfSumBlocks ? 1 : min(kAfSumBlocks / it.rows, (it.cols + 127) / 128);
  const int stretch = ((it.cols + stretches - 1) / stretches + 127) / 128 * 128;
  const int c0 = (part % stretches) * stretch, c1 = min(it.cols, c0 + stretch), v1 = min(c1, w.cols4);
  double s = 0.0;
  // (rows * stretches <= kAfSumBlocks unless stretches is 1: a second round only then)
  for (int row = part / stretches; row < it.rows; row += kAfSumBlocks / stretches) {
    const float ar = a.a_row[row];
    const float* R = it.Rpart + (int64_t)row * it.r_ld;
    for (int c = c0 + 4 * lane; c < v1; c += 8 * 128) {
      float4 x[8], b[8];
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (c + 128 * k < v1) {
          x[k] = *reinterpret_cast<const float4*>(R + c + 128 * k);
          b[k] = *reinterpret_cast<const float4*>(a.b_col + c + 128 * k);
        }
      float sum = 0.f;                        // at most 32 terms
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (c + 128 * k < v1) {
          const float u0 = x[k].x * ar * b[k].x, u1 = x[k].y * ar * b[k].y, u2 = x[k].z * ar * b[k].z, u3 = x[k].w * ar * b[k].w;
          sum += u0 * u0 + u1 * u1 + u2 * u2 + u3 * u3;
        }
      s += (double)sum;
    }
    float sum = 0.f;
    for (int c = max(c0, w.cols4) + lane; c < c1; c += 32) {
      const float u = R[c] * ar * a.b_col[c];
      sum += u * u;
    }
    s += (double)sum;
  }
  s = warp_sum_d(s);
  if (lane == 0) a.sums[part] = s;
}

// PL = 1: four values rounded to bf16, 3: their three planes
template <int PL>
__device__ __forceinline__ void af_store4(__nv_bfloat16* dst, int64_t plane, float m0, float m1, float m2, float m3) {
#pragma unroll
  for (int p = 0; p < PL; ++p, dst += plane) {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(m0, m1), hi = __floats2bfloat162_rn(m2, m3);
    uint2 v;
    v.x = *reinterpret_cast<const uint32_t*>(&lo);
    v.y = *reinterpret_cast<const uint32_t*>(&hi);
    *reinterpret_cast<uint2*>(dst) = v;
    m0 -= __uint_as_float(v.x << 16);
    m1 -= __uint_as_float(v.x & 0xffff0000u);
    m2 -= __uint_as_float(v.y << 16);
    m3 -= __uint_as_float(v.y & 0xffff0000u);
  }
}

// pass 4
template <int PL, int CAP>
__global__ void __launch_bounds__(256) af_update_kernel(const __grid_constant__ AdafactorArgs<CAP> g) {
  grid_dependency_wait();
  grid_launch_dependents();
  __shared__ double red[8];
  const AdafactorItem& it = g.item[blockIdx.y];
  const AfLayout a = af_layout(it);
  double s = 0.0, sr = 0.0;
  for (int i = threadIdx.x; i < kAfSumBlocks; i += 256) s += a.sums[i];
  for (int i = threadIdx.x; i < (it.rows + 255) / 256; i += 256) sr += a.row_sums[i];
  s = block_sum_256d(s, red);
  const double mean_r = block_sum_256d(sr, red) / (double)it.rows;
  const float rms = (float)sqrt(s * mean_r / ((double)it.rows * (double)it.cols));
  const float shrink = (float)sqrt(mean_r) / fmaxf(1.f, rms / kAdafactorClip);
  const float b1 = it.beta1, omb1 = 1.f - it.beta1;
  const AfRowWalk w = af_walk(it, true);
  __nv_bfloat16* N = it.Nout;
  for (int row = blockIdx.x; row < it.rows; row += gridDim.x) {
    const float ar = a.a_row[row] * shrink;
    const float* R = it.Rpart + (int64_t)row * it.r_ld;
    float* M = it.M + (int64_t)row * it.s_ld;
    __nv_bfloat16* Nr = N + (int64_t)row * it.n_ld;
    for (int c = 4 * threadIdx.x; c < w.cols4; c += 4 * 256) {
      const float4 x = *reinterpret_cast<const float4*>(R + c);
      const float4 b = *reinterpret_cast<const float4*>(a.b_col + c);
      float4 m = *reinterpret_cast<const float4*>(M + c);
      m.x = fmaf(b1, m.x, omb1 * (x.x * ar * b.x));
      m.y = fmaf(b1, m.y, omb1 * (x.y * ar * b.y));
      m.z = fmaf(b1, m.z, omb1 * (x.z * ar * b.z));
      m.w = fmaf(b1, m.w, omb1 * (x.w * ar * b.w));
      *reinterpret_cast<float4*>(M + c) = m;
      af_store4<PL>(Nr + c, it.n_plane, m.x, m.y, m.z, m.w);
    }
    for (int c = w.cols4 + threadIdx.x; c < it.cols; c += 256) {
      const float m = fmaf(b1, M[c], omb1 * (R[c] * ar * a.b_col[c]));
      M[c] = m;
      float x = m;
#pragma unroll
      for (int p = 0; p < PL; ++p) {
        const __nv_bfloat16 h = __float2bfloat16_rn(x);
        Nr[c + p * it.n_plane] = h;
        x -= __bfloat162float(h);
      }
    }
  }
}

}  // namespace

// the division stays out of the kernels (every CTA lays its item's scratch out)
static void set_tiles(AdafactorItem& it) {
  it.tile_rows = it.squares_ready ? kAfProjectionRows : af_tile_rows(it.rows, it.cols);
  it.tiles_r = (int)ceil_div(it.rows, it.tile_rows);
}

size_t adafactor_scratch_bytes(int64_t rows, int64_t cols) {
  const int least = rows <= kAfProjectionTallest ? std::min(af_tile_rows(rows, cols), kAfProjectionRows) : af_tile_rows(rows, cols);
  const int64_t tiles_r = ceil_div(rows, least), tiles_c = ceil_div(cols, kAfTileCols);
  return align_up((size_t)(2 * (kAfSumBlocks + 8 + ceil_div(rows, 256) * 2) + rows * tiles_c + tiles_r * cols + rows + cols + 16) * sizeof(float), 256);
}

bool adafactor_squares(const AdafactorItem& item, AdafactorSquares* out) {
  if (item.rows > kAfProjectionTallest) return false;
  AdafactorItem it = item;
  it.squares_ready = true;
  set_tiles(it);
  const AfLayout a = af_layout(it);
  *out = AdafactorSquares{a.rowpart, a.colpart, a.tiles_c};
  return true;
}

galore_status_t adafactor_group_add(AdafactorGroup& g, const AdafactorItem& it) {
  if (g.count >= kAdafactorGroup) return GALORE_ERR_INVALID_ARG;
  if (it.rows <= 0 || it.cols <= 0 || !it.Rpart || !it.M || !it.v_row || !it.v_col || !it.Nout || !it.scratch || it.splits < 1)
    return GALORE_ERR_INVALID_ARG;
  const int i = g.count;
  g.item[i] = it;
  set_tiles(g.item[i]);
  g.beta2t[i] = (float)(1.0 - pow(it.t, -kAdafactorDecay));
  if (it.squares_ready && (it.splits != 1 || it.split.src)) return GALORE_ERR_INVALID_ARG;      // the pass adds slices and splits P too
  const int tiles = it.squares_ready ? 0 : (int)(g.item[i].tiles_r * ceil_div(it.cols, kAfTileCols));
  const int blocks = (int)(ceil_div(it.rows, 256) + ceil_div(it.cols, 256));
  g.tile_end[i] = (i ? g.tile_end[i - 1] : 0) + tiles;
  g.vec_end[i] = (i ? g.vec_end[i - 1] : 0) + blocks;
  g.count = i + 1;
  return GALORE_OK;
}

template <int PL, int CAP>
static galore_status_t launch_passes(const AdafactorArgs<CAP>& g, bool early, cudaStream_t st) {
  const int n = g.count;
  if (g.tile_end[n - 1] > 0)      // (an item whose sums are ready has no tiles)
    GALORE_TRY(launch_kernel(af_stats_kernel<CAP>, dim3((unsigned)g.tile_end[n - 1]), kAfTileCols, 0, 1, early, st, g));
  GALORE_TRY(launch_kernel(af_vectors_kernel<CAP>, dim3((unsigned)g.vec_end[n - 1]), 256, 0, 1, early, st, g));
  const unsigned parts = (unsigned)ceil_div(kAfSumBlocks, kRmsThreads / 32);
  GALORE_TRY(launch_kernel(af_rms_kernel<CAP>, dim3(parts, (unsigned)n), kRmsThreads, 0, 1, early, st, g));
  return launch_kernel(af_update_kernel<PL, CAP>, dim3(kAfSumBlocks, (unsigned)n), 256, 0, 1, early, st, g);
}

galore_status_t launch_adafactor_group(const AdafactorGroup& g, int n_planes, bool early, cudaStream_t st) {
  if (g.count <= 0) return GALORE_OK;
  if (g.count > 1)
    return n_planes == 3 ? launch_passes<3, kAdafactorGroup>(g, early, st) : launch_passes<1, kAdafactorGroup>(g, early, st);
  AdafactorArgs<1> one;
  one.item[0] = g.item[0];
  one.tile_end[0] = g.tile_end[0];
  one.vec_end[0] = g.vec_end[0];
  one.beta2t[0] = g.beta2t[0];
  one.count = 1;
  return n_planes == 3 ? launch_passes<3, 1>(one, early, st) : launch_passes<1, 1>(one, early, st);
}

galore_status_t launch_adafactor(const AdafactorItem& it, int n_planes, bool early, cudaStream_t st) {
  AdafactorGroup g;
  g.count = 0;
  GALORE_TRY(adafactor_group_add(g, it));
  return launch_adafactor_group(g, n_planes, early, st);
}

}  // namespace galore
