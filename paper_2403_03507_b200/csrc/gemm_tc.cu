// Projection of the GaLore step on the 5th-generation tensor cores (sm_100a):
// bf16 operands staged in shared memory by TMA, tcgen05.mma with fp32
// accumulators in tensor memory, an epilogue that stores split-K partial sums
// of R (Algorithm 1: R = P^T G resp. G Q).  The products of the refresh's power
// steps are problems of the same kernel.
//
// With one K slice per output tile the projection's epilogue also runs Adam on its tile of R
// (moment update, bias correction, Eq. 15, 8-bit dequantisation and requantisation of the moments)
// and writes the normalised update N for the back-projection: R never reaches memory.
//
// One persistent CTA per SM:
//   warp 0        TMA producer: fills a ring of kStages shared-memory stages
//   warp 1        MMA issuer (one lane) and owner of the tensor-memory allocation
//   warps 2..     epilogue (four warps, sixteen when it runs Adam): tcgen05.ld of a finished
//                 accumulator, then global memory
//   last warp     with fp32 moments: TMA loads and stores of the moments through a ring in shared memory
// Two accumulators of kBN columns alternate, so the epilogue of one tile runs
// under the MMAs of the next.  Work units are (tile_m, tile_n, K slice); the
// K slices of one output tile go to separate partial buffers that the Adam
// kernel sums in a fixed order, so results do not depend on scheduling.
//
// Every wait on an mbarrier is bounded by a clock limit; when it runs out the
// CTA latches GALORE_DEV_WAIT_EXPIRED, lets its outstanding copies land,
// releases tensor memory and returns.
#include "gemm_tc.cuh"

#include <cudaTypedefs.h>

#include "adam.cuh"
#include "launch.cuh"
#include "tc_ptx.cuh"

#include <algorithm>
#include <atomic>
#include <memory>
#include <new>

namespace galore {

namespace {

constexpr int kBM = 128;          // rows of an output tile = TMEM lanes
constexpr int kBN = 256;          // columns of an output tile = TMEM columns per accumulator (single products with up to 128: 128)
constexpr int kBK = 64;           // K per stage: 64 bf16 = one 128-byte swizzle row
constexpr int kUmmaK = 16;
constexpr uint32_t kTmemCols = 512;
constexpr int kABytes = kBM * kBK * 2;            // 16 KiB: the 128 rows of A one CTA stages per k-block

// EPI_ADAM_F32 / EPI_ADAM_Q8: the projection with Adam on its output tile (fp32 / 8-bit moments).
// EPI_DRAIN: EPI_PARTIAL with shorter chains.  The tensor core's accumulator rounds towards zero; here it is added to fp32 sums in
// the epilogue's registers after every few k-blocks (R of 2048 x 5461 at rank 512: after each one 9e-8 from 64 bits, in one
// accumulator 8e-7).
// EPI_STATS: EPI_PARTIAL with Adafactor's statistics, the sums of R^2 over 128 columns of a row and over 64 rows of a column (added
// up in fp64 by the pass behind; over 128 rows a column's sum was further from fp64 than before).  They hide under the next
// tile's MMAs: eight layers of LLaMA-1B size 361 -> 387 us, and the pass over R for them took 147.
enum { EPI_PARTIAL = 0, EPI_ADAM_F32 = 1, EPI_ADAM_Q8 = 2, EPI_DRAIN = 3, EPI_STATS = 4 };
constexpr bool epi_is_adam(int epi) { return epi == EPI_ADAM_F32 || epi == EPI_ADAM_Q8; }
// Adam is instruction-heavy (about 70 per element with 8-bit moments) and every element is a chain
// of dependent lookups and arithmetic: sixteen epilogue warps, four per quarter of the accumulator's
// lanes with 64 columns each, give every scheduler of the SM four warps to switch between while the
// tensor cores work on the next tile (eight warps of 128 columns each ran three times longer than
// the MMAs of a tile).
// Sixteen as well (64 columns each) where accumulators are drained after every k-block: a pair's MMAs take 512 cycles for one.
constexpr int epi_warps(int epi, int bn) { return epi == EPI_PARTIAL || epi == EPI_STATS ? 4 : (epi == EPI_DRAIN ? bn / 16 : 16); }
constexpr int epi_threads(int epi, int bn) { return 64 + 32 * epi_warps(epi, bn) + (epi == EPI_ADAM_F32 ? 32 : 0); }   // + producer, MMA, moments
// behind the ring and the barriers: the tables of the 8-bit code, or the column sums of two tiles by quarters of the rows
constexpr int epi_smem(int epi) { return epi == EPI_ADAM_Q8 ? (int)sizeof(Q8Tables) : (epi == EPI_STATS ? 2 * 4 * kBN * 4 : 0); }

// A piece of a moment: 32 rows x 64 columns, as two boxes of 32 x 32 (128 bytes a row).  It belongs to the four epilogue warps
// that can read its rows of the accumulator, 16 columns each, and so does its slot: a warp that waited for a slot's next
// phase but one would find the wrong parity.
constexpr int kMomentRows = 32, kMomentCols = 64, kBoxCols = 32;
constexpr int kBoxBytes = kMomentRows * kBoxCols * 4;
constexpr int kMomentBytes = kMomentRows * kMomentCols * 4;
// CTAS = 1: one CTA computes a 128 x 256 tile.  CTAS = 2: a cluster of two CTAs computes 256 x 256
// with cta_group::2 MMAs; each CTA stages its own 128 rows of A and half (128 columns) of B, so a
// k-block costs 32 KiB of shared-memory fill per CTA instead of 48 and the ring holds 6 stages.
// With fp32 moments the ring gives up a stage or two for pieces of M and V.  Read and written by the epilogue's lanes, a row
// each, they kept the epilogue at 28 to 38 thousand cycles a tile against 21 of the MMAs, which waited; through the ring it
// is out of the way and the operands' latency bounds the tile (eight layers of LLaMA-1B size at rank 512: 611 -> 523 us of
// 392 for the bytes).  Pieces of 128 rows x 32 columns with 5 / 4 / 3 stages: 529 / 541 / 596 us; rows of 64 bytes
// (16 columns): 595 and more; 32 x 32 with 6 stages: 566.
template <int CTAS, int EPI, int BN>
struct Geo {
  static constexpr int kTileM = kBM * CTAS;
  static constexpr int kBNcta = BN / CTAS;
  static constexpr int kBBytes = kBNcta * kBK * 2;
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr bool kMoments = EPI == EPI_ADAM_F32;
  static constexpr int kStages = kMoments ? (CTAS == 1 ? 3 : 5) : 192 * 1024 / kStageBytes;
  static constexpr int kSlots = kMoments ? 4 : 0;              // pieces of M and of V, one per quarter of the rows
  static constexpr int kRingBytes = kStages * kStageBytes + kSlots * 2 * kMomentBytes;
  static constexpr int kSmemBytes = kRingBytes + 1024 /* alignment slack */ + 256 /* barriers */;
};

constexpr int kMaxGroup = 32;     // problems one launch can carry (its arguments travel as kernel parameters)

struct TcParams {
  int M, N, K;
  int tile_m;                 // rows of a work unit: 128 (one CTA) or 256 (CTA pair)
  int a_mn, b_mn;             // operand majors in shared memory: 1 = M/N contiguous, 0 = K contiguous
  int tiles_m, tiles_n, splits;
  int kblocks_total, kblocks_per_split;
  int drain;                  // EPI_DRAIN: k-blocks per accumulator
  int m_fast;                 // 1: consecutive units walk tile_m first (B panel shared), 0: tile_n first
  // EPI_PARTIAL
  float* part;
  int64_t ld_part, split_stride;
  float *row_sq, *col_sq;     // EPI_STATS: rows x sq_tiles, ceil(rows / 64) x columns
  int sq_tiles;
  int vec32;                  // the partial buffer's base and row pitch are 32-byte aligned
  int32_t* status;
  // EPI_ADAM_*: the state of the layer (rows x cols of the output, row pitch ld_s) and where N goes
  uint8_t *Mc, *Vc;           // 8-bit codes with (fp32 moments travel by their tensor maps)
  float *Mam, *Vam;           // one absmax per tile of q_rows x 64 state elements, tile (I, J) at I * q_tiles_c + J
  int64_t ld_s;
  int q_rows, q_tiles_c;
  __nv_bfloat16* Nout;
  int64_t ld_n;
  int adam_vec;               // bases and pitches of the codes and of N allow wide accesses
  AdamParams ap;
};

// One launch = up to CAP independent problems; work units are numbered across them.  (A single matrix travels
// in a capacity of one: the launch copies its parameters, 14 KiB at the full capacity.)
template <int CAP>
struct TcArgs {
  CUtensorMap map_a[CAP];
  CUtensorMap map_b[CAP];
  TcParams p[CAP];
  int unit_end[CAP];          // running total of units: problem i owns [unit_end[i-1], unit_end[i])
  int count;
  Q8TablePtrs q8;             // EPI_ADAM_Q8: the code tables in global memory
  CUtensorMap map_m[CAP];     // EPI_ADAM_F32: the moments
  CUtensorMap map_v[CAP];
};
using TcGroup = TcArgs<kMaxGroup>;

// ---- descriptors ------------------------------------------------------------------------
// Shared-memory operand descriptor, 128-byte swizzle, tile base 1024-byte aligned.
//  K-major  : rows of 64 bf16 (128 B); 8-row groups 1024 B apart (stride offset); leading offset unused.
//  MN-major : 64-element (128 B) runs along M/N, one per k; 8-k groups 1024 B apart (stride offset);
//             the next 64 elements of M/N start kBK * 128 B further on (leading offset).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, bool mn_major) {
  const uint64_t lbo = mn_major ? (uint64_t)((kBK * 128) >> 4) : 1ull;
  const uint64_t sbo = 1024 >> 4;
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | (lbo << 16) | (sbo << 32) | (1ull << 46) | (2ull << 61);
}

// Instruction descriptor: fp32 accumulate, bf16 x bf16, majors, N, M.
__host__ __device__ constexpr uint32_t instr_desc(int a_mn, int b_mn, int tile_m, int tile_n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
         ((uint32_t)(tile_n >> 3) << 17) | ((uint32_t)(tile_m >> 4) << 24);
}

struct Unit {
  int m0, n0, split, kb_begin, kb_end;
};

template <int BN, int CAP>
__device__ __forceinline__ Unit decode_unit(const TcArgs<CAP>& g, int u, GroupCursor& cursor) {
  u = cursor.seek<CAP>(g, u);
  const TcParams& p = g.p[cursor.pi];
  int tm, tn, s;
  if (p.m_fast) {
    tm = u % p.tiles_m;
    s = (u / p.tiles_m) % p.splits;
    tn = u / (p.tiles_m * p.splits);
  } else {
    tn = u % p.tiles_n;
    s = (u / p.tiles_n) % p.splits;
    tm = u / (p.tiles_n * p.splits);
  }
  Unit w;
  w.m0 = tm * p.tile_m;
  w.n0 = tn * BN;
  w.split = s;
  w.kb_begin = s * p.kblocks_per_split;
  w.kb_end = min(p.kblocks_total, w.kb_begin + p.kblocks_per_split);
  return w;
}

// ---- epilogues ----------------------------------------------------------------------------

// thread owns row `row`, columns [col0, col0 + 32) of the tile
__device__ __forceinline__ void epi_partial(const TcParams& p, const Unit& w, int row, int col0, const uint32_t (&v)[32]) {
  if (row >= p.M) return;
  float* dst = p.part + (int64_t)w.split * p.split_stride + (int64_t)row * p.ld_part + col0;
  if (col0 + 32 <= p.N && p.vec32) {
#pragma unroll
    for (int j = 0; j < 32; j += 8)
      st_global_32B(dst + j, make_uint4(v[j], v[j + 1], v[j + 2], v[j + 3]), make_uint4(v[j + 4], v[j + 5], v[j + 6], v[j + 7]));
  } else if (col0 + 32 <= p.N && (p.ld_part & 3) == 0) {
#pragma unroll
    for (int j = 0; j < 32; j += 4)
      *reinterpret_cast<float4*>(dst + j) = make_float4(__uint_as_float(v[j]), __uint_as_float(v[j + 1]),
                                                        __uint_as_float(v[j + 2]), __uint_as_float(v[j + 3]));
  } else {
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (col0 + j < p.N) dst[j] = __uint_as_float(v[j]);
  }
}

__device__ __forceinline__ float tree_sum(const float (&x)[32]) {
  float t[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) t[j] = x[j] + x[j + 16];
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) {
#pragma unroll
    for (int j = 0; j < o; ++j) t[j] += t[j + o];
  }
  return t[0];
}
// lane l's share of 32 columns that each lane holds one row of: the sum of column l
__device__ __forceinline__ float column_sum(float (&x)[32]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int j = 0; j < o; ++j) {
      const bool up = (lane & o) != 0;
      const float keep = up ? x[j + o] : x[j], send = up ? x[j] : x[j + o];
      x[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  return x[0];
}

// ---- Adam in the projection's epilogue ----------------------------------------------------------
// The thread owns row `row` of R and the kAdamCols columns from col0 on (Algorithm 1, the update
// block on its part of R; Eq. 15 for N), and walks them kAdamChunk at a time.  Rows and columns
// outside the matrix hold exact zeros in the accumulator (TMA fills out-of-range operand elements
// with zeros).
constexpr int kAdamCols = kStateTileCols;    // 64: columns per epilogue warp = width of a quantisation block

// fp32 moments: eight columns of the thread's row of a box, M at `row` and V kMomentBytes further on; `first` is the 16-byte
// chunk they begin with, `sw` the row's part of TMA's 128-byte swizzle.
__device__ __forceinline__ bool epi_adam_f32(const AdamParams& ap, uint32_t row, uint32_t first, uint32_t sw, const uint32_t (&acc)[8],
                                             int valid, __nv_bfloat16* __restrict__ n_out) {
  const uint32_t at0 = row + ((first ^ sw) << 4), at1 = row + (((first + 1u) ^ sw) << 4);
  const uint4 m0 = ld_shared_16B(at0), m1 = ld_shared_16B(at1), v0 = ld_shared_16B(at0 + kMomentBytes), v1 = ld_shared_16B(at1 + kMomentBytes);
  uint32_t m[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w}, v[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
  float n[8];
  uint32_t top = 0u;      // largest bit pattern among the new second moments (all >= 0): a non-finite r shows here
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float r = __uint_as_float(acc[j]);
    const float mj = adam_m(__uint_as_float(m[j]), r, ap), vj = adam_v(__uint_as_float(v[j]), r, ap);
    n[j] = adam_normalised(mj, vj, ap);
    m[j] = __float_as_uint(mj);
    v[j] = __float_as_uint(vj);
    top = max(top, v[j]);
  }
  st_shared_16B(at0, make_uint4(m[0], m[1], m[2], m[3]));
  st_shared_16B(at1, make_uint4(m[4], m[5], m[6], m[7]));
  st_shared_16B(at0 + kMomentBytes, make_uint4(v[0], v[1], v[2], v[3]));
  st_shared_16B(at1 + kMomentBytes, make_uint4(v[4], v[5], v[6], v[7]));
  if (valid >= 8) {
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(n[2 * j], n[2 * j + 1]);
      w[j] = *reinterpret_cast<const uint32_t*>(&h);
    }
    *reinterpret_cast<uint4*>(n_out) = make_uint4(w[0], w[1], w[2], w[3]);
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (j < valid) n_out[j] = __float2bfloat16_rn(n[j]);
  }
  return top >= 0x7f800000u;
}

// eight old codes of one moment, columns [c, c + 8) of the thread's stretch: one 8-byte load, or byte by
// byte with the code of zero outside the matrix
__device__ __forceinline__ uint2 ld_codes8(const uint8_t* row, int c, int ncols, bool vec, uint32_t zero_code) {
  if (vec) return *reinterpret_cast<const uint2*>(row + c);
  uint32_t w[2] = {0u, 0u};
#pragma unroll
  for (int k = 0; k < 8; ++k) w[k >> 2] |= (c + k < ncols ? (uint32_t)row[c + k] : zero_code) << (8 * (k & 3));
  return make_uint2(w[0], w[1]);
}

// 8-bit moments.  A quantisation block is a tile of q_rows x 64 state elements: q_rows lanes of this
// warp hold all of it, so its absmax is a warp-shuffle reduction.  Two passes over the accumulator:
// the first finds the block's absmax of the updated moments, the second recomputes them (the same
// instructions, hence the same bits), writes N and the new codes.  Both walk the thread's 64
// columns eight at a time in loops that are NOT unrolled: sixteen warps at different points of a
// fully unrolled body (about 5000 instructions) spent most of their time waiting for instruction
// fetch, and the old codes kept in registers across both passes spilled.  The codes are read once
// per pass instead, the second time from L2.
__device__ __forceinline__ bool epi_adam_q8(const TcParams& p, int row, int col0, uint32_t t_addr, uint32_t accf,
                                            uint32_t acc_phase, volatile int* abort_flag, const Q8Tables& t, bool& ok) {
  constexpr int CH = 8;
  const bool row_ok = row < p.M;
  const int ncols = row_ok ? max(0, min(kAdamCols, p.N - col0)) : 0;
  const bool vec = p.adam_vec != 0 && ncols == kAdamCols;
  const AdamParams ap = p.ap;
  const int64_t so = (int64_t)row * p.ld_s + col0;
  uint8_t* __restrict__ Mrow = p.Mc + so;
  uint8_t* __restrict__ Vrow = p.Vc + so;
  __nv_bfloat16* __restrict__ Nrow = p.Nout + (int64_t)row * p.ld_n + col0;
  const int tile = ncols > 0 ? (row / p.q_rows) * p.q_tiles_c + col0 / kAdamCols : 0;
  // the old codes and the block's old absmax do not depend on the MMAs: asked for now, they arrive
  // while the tile is computed
  if (ncols > 0) {
    prefetch_l2(Mrow);
    prefetch_l2(Vrow);
  }
  const float am_m = ncols > 0 ? p.Mam[tile] : 0.f, am_v = ncols > 0 ? p.Vam[tile] : 0.f;
  // the decision is taken by the warp as a whole: what follows is warp-synchronous
  if (!__all_sync(0xffffffffu, mbar_wait(accf, acc_phase, abort_flag))) { ok = false; return false; }
  tc_fence_after();
  const int wcols = __reduce_max_sync(0xffffffffu, ncols);       // columns any lane of the warp has
  if (wcols == 0) return false;                                  // the warp's part of the tile lies outside the matrix

  // Both passes are software-pipelined by one chunk: the next chunk's accumulator columns and old
  // codes are asked for before the current chunk's arithmetic, which is a chain of dependent
  // shared-memory lookups per element.
  // ---- pass 1: absmax of the updated moments over the block
  float mx_m = 0.f;
  uint32_t mx_vb = 0u;          // v >= 0: bit order is value order; a NaN or an infinity ends up on top
  {
    uint2 nm = ld_codes8(Mrow, 0, ncols, vec, 127u), nv = ld_codes8(Vrow, 0, ncols, vec, 0u);
    uint32_t nacc[CH];
    tmem_ld_32x8(t_addr, nacc);
#pragma unroll 1
    for (int c = 0; c < wcols; c += CH) {
      const uint2 cm = nm, cv = nv;
      uint32_t acc[CH];
      tmem_ld_wait();
#pragma unroll
      for (int j = 0; j < CH; ++j) acc[j] = nacc[j];
      if (c + CH < wcols) {
        tmem_ld_32x8(t_addr + (uint32_t)(c + CH), nacc);
        nm = ld_codes8(Mrow, c + CH, ncols, vec, 127u);
        nv = ld_codes8(Vrow, c + CH, ncols, vec, 0u);
      }
#pragma unroll
      for (int j = 0; j < CH; ++j) {
        const float r = __uint_as_float(acc[j]);
        const uint32_t im = ((j < 4 ? cm.x : cm.y) >> (8 * (j & 3))) & 0xffu, iv = ((j < 4 ? cv.x : cv.y) >> (8 * (j & 3))) & 0xffu;
        const float m = adam_m(__fmul_rn(t.code_s[im], am_m), r, ap);
        const float v = adam_v(__fmul_rn(t.code_u[iv], am_v), r, ap);
        mx_m = fmaxf(mx_m, fabsf(m));
        mx_vb = max(mx_vb, __float_as_uint(v));
      }
    }
  }
  for (int o = 1; o < p.q_rows; o <<= 1) {      // the q_rows lanes of the block (a power of two up to 32)
    mx_m = fmaxf(mx_m, __shfl_xor_sync(0xffffffffu, mx_m, o));
    mx_vb = max(mx_vb, __shfl_xor_sync(0xffffffffu, mx_vb, o));
  }
  const bool bad = mx_vb >= 0x7f800000u;
  const float mx_v = __uint_as_float(mx_vb);
  // an all-zero block: with 0 in place of the reciprocal every y' is 0 and takes the code of zero
  const float inv_m = mx_m != 0.f ? 1.0f / mx_m : 0.f, inv_v = mx_v != 0.f ? 1.0f / mx_v : 0.f;

  // ---- pass 2: N and the new codes, eight elements at a time with one (rare) branch to the exact search
  {
    uint2 nm = ld_codes8(Mrow, 0, ncols, vec, 127u), nv = ld_codes8(Vrow, 0, ncols, vec, 0u);
    uint32_t nacc[CH];
    tmem_ld_32x8(t_addr, nacc);
#pragma unroll 1
    for (int c = 0; c < wcols; c += CH) {
      const uint2 cm = nm, cv = nv;
      uint32_t acc[CH];
      tmem_ld_wait();
#pragma unroll
      for (int j = 0; j < CH; ++j) acc[j] = nacc[j];
      if (c + CH < wcols) {
        tmem_ld_32x8(t_addr + (uint32_t)(c + CH), nacc);
        nm = ld_codes8(Mrow, c + CH, ncols, vec, 127u);
        nv = ld_codes8(Vrow, c + CH, ncols, vec, 0u);
      }
      float xm[CH], xv[CH];
      uint32_t nw[CH / 2];
#pragma unroll
      for (int j = 0; j < CH; j += 2) {
        float n[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int e = j + k;
          const float r = __uint_as_float(acc[e]);
          const uint32_t im = ((e < 4 ? cm.x : cm.y) >> (8 * (e & 3))) & 0xffu, iv = ((e < 4 ? cv.x : cv.y) >> (8 * (e & 3))) & 0xffu;
          xm[e] = adam_m(__fmul_rn(t.code_s[im], am_m), r, ap);
          xv[e] = adam_v(__fmul_rn(t.code_u[iv], am_v), r, ap);
          n[k] = adam_normalised(xm[e], xv[e], ap);
        }
        const __nv_bfloat162 h = __floats2bfloat162_rn(n[0], n[1]);
        nw[j >> 1] = *reinterpret_cast<const uint32_t*>(&h);
      }
      uint32_t pm[2] = {0u, 0u}, pv[2] = {0u, 0u}, need = 0u;     // need: bit e for M value e, bit 8 + e for V value e
#pragma unroll
      for (int e = 0; e < CH; ++e) {
        bool ex_m, ex_v;
        const uint32_t km = q8_encode_fast<true>(xm[e], inv_m, t.enc_s, ex_m) & 0xffu;
        const uint32_t kv = q8_encode_fast<false>(xv[e], inv_v, t.enc_u, ex_v) & 0xffu;
        pm[e >> 2] |= km << (8 * (e & 3));
        pv[e >> 2] |= kv << (8 * (e & 3));
        need |= ((ex_m ? 1u : 0u) << e) | ((ex_v ? 1u : 0u) << (8 + e));
      }
      if (need != 0u) {                         // about one value in 4000: the quotient by IEEE division, searched exactly
#pragma unroll
        for (int e = 0; e < CH; ++e) {
          if (need & (1u << e)) {
            const uint32_t k = (uint32_t)q8_encode(__fdiv_rn(xm[e], mx_m), t.mid_s) & 0xffu;
            pm[e >> 2] = (pm[e >> 2] & ~(0xffu << (8 * (e & 3)))) | (k << (8 * (e & 3)));
          }
          if (need & (0x100u << e)) {
            const uint32_t k = (uint32_t)q8_encode(__fdiv_rn(xv[e], mx_v), t.mid_u) & 0xffu;
            pv[e >> 2] = (pv[e >> 2] & ~(0xffu << (8 * (e & 3)))) | (k << (8 * (e & 3)));
          }
        }
      }
      if (vec) {
        *reinterpret_cast<uint2*>(Mrow + c) = make_uint2(pm[0], pm[1]);
        *reinterpret_cast<uint2*>(Vrow + c) = make_uint2(pv[0], pv[1]);
        *reinterpret_cast<uint4*>(Nrow + c) = make_uint4(nw[0], nw[1], nw[2], nw[3]);
      } else {
#pragma unroll
        for (int j = 0; j < CH; ++j)
          if (c + j < ncols) {
            Mrow[c + j] = (uint8_t)(pm[j >> 2] >> (8 * (j & 3)));
            Vrow[c + j] = (uint8_t)(pv[j >> 2] >> (8 * (j & 3)));
            reinterpret_cast<uint16_t*>(Nrow)[c + j] = (uint16_t)(nw[j >> 1] >> (16 * (j & 1)));
          }
      }
    }
  }
  if (ncols > 0 && (row % p.q_rows) == 0) {     // the first lane of each block stores its absmax
    p.Mam[tile] = mx_m;
    p.Vam[tile] = mx_v;
  }
  return bad;
}

// ---- the kernel -------------------------------------------------------------------------------

template <int EPI, int CTAS, int CAP, int BN>
__global__ void __launch_bounds__(epi_threads(EPI, BN), 1)
gemm_tc_kernel(const __grid_constant__ TcArgs<CAP> g) {
  using G = Geo<CTAS, EPI, BN>;
  constexpr int kEpiWarps = epi_warps(EPI, BN);
  constexpr int kStages = G::kStages;
  constexpr int kStageBytes = G::kStageBytes;
  extern __shared__ uint8_t smem_raw[];
  // stage ring, 1024-byte aligned for the 128-byte swizzle
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t ring = (raw_addr + 1023u) & ~1023u;
  uint8_t* ring_ptr = smem_raw + (ring - raw_addr);
  uint64_t* bars = reinterpret_cast<uint64_t*>(ring_ptr + G::kRingBytes);
  // bars[0..S) full, [S..2S) empty, [2S..2S+2) accumulator full, [2S+2..2S+4) accumulator empty, then a piece of
  // the moments loaded and updated.
  // In a CTA pair the full and accumulator-empty barriers that count are the leader's (rank 0).
  const uint32_t bar_base = smem_u32(bars);
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (kStages + s); };
  auto accf_bar = [&](int a) { return bar_base + 8u * (2 * kStages + a); };
  auto acce_bar = [&](int a) { return bar_base + 8u * (2 * kStages + 2 + a); };
  auto mvfull_bar = [&](int s) { return bar_base + 8u * (2 * kStages + 4 + s); };
  auto mvdone_bar = [&](int s) { return bar_base + 8u * (2 * kStages + 4 + G::kSlots + s); };
  const uint32_t sq_bar = bar_base + 8u * (2 * kStages + 4 + 2 * G::kSlots);        // EPI_STATS: the column sums of a tile are in place
  constexpr int kBars = 2 * kStages + 5 + 2 * G::kSlots;
  static_assert(kBars * 8 + 16 <= 256, "barrier space");
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(bars + kBars);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + kBars + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int total_units = g.unit_end[g.count - 1];
  const uint32_t rank = CTAS == 2 ? cluster_ctarank() : 0u;
  const int team = blockIdx.x / CTAS;               // CTA or CTA pair that walks the units together
  const int teams = gridDim.x / CTAS;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(accf_bar(a), 1);
      mbar_init(acce_bar(a), kEpiWarps * CTAS);     // one arrival per epilogue warp of the group, from every CTA
    }
    mbar_init(sq_bar, kEpiWarps);
    for (int s = 0; s < G::kSlots; ++s) {
      mbar_init(mvfull_bar(s), 1);
      mbar_init(mvdone_bar(s), kEpiWarps / 4);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    if (CTAS == 2) {
      tmem_alloc_pair(smem_u32((const void*)tmem_slot), kTmemCols);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(smem_u32((const void*)tmem_slot), kTmemCols);
      tmem_relinquish();
    }
  }
  // the 8-bit code tables follow the barriers (256 bytes after the ring)
  Q8Tables* q8t = reinterpret_cast<Q8Tables*>(ring_ptr + G::kRingBytes + 256);
  float* const col_sums = reinterpret_cast<float*>(ring_ptr + G::kRingBytes + 256);
  if constexpr (EPI == EPI_ADAM_Q8) q8_tables_fill(*q8t, g.q8, (int)threadIdx.x, epi_threads(EPI, BN));
  tc_fence_before();
  __syncthreads();
  if (CTAS == 2) cluster_sync_all();                // the peer's barriers exist before anyone signals them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  grid_dependency_wait();
  grid_launch_dependents();

  if (warp == 0) {
    // ================= TMA producer (every CTA loads its own share) =================
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      long long issued = 0;
      bool ok = true;
      GroupCursor cursor;
      for (int u = team; u < total_units && ok; u += teams) {
        const Unit w = decode_unit<BN>(g, u, cursor);
        const int pi = cursor.pi;
        const bool A_MN = g.p[pi].a_mn != 0, B_MN = g.p[pi].b_mn != 0;
        const CUtensorMap* map_a = &g.map_a[pi];
        const CUtensorMap* map_b = &g.map_b[pi];
        const int m0 = w.m0 + (int)rank * kBM;               // this CTA's rows of A
        const int n0 = w.n0 + (int)rank * G::kBNcta;         // this CTA's columns of B
        for (int kb = w.kb_begin; kb < w.kb_end; ++kb) {
          if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag)) { ok = false; break; }
          const uint32_t a_dst = ring + stage * kStageBytes;
          const uint32_t b_dst = a_dst + kABytes;
          const uint32_t fbar = CTAS == 2 ? map_to_cta(full_bar(stage), 0) : full_bar(stage);
          if (rank == 0) mbar_arrive_expect_tx(full_bar(stage), CTAS * kStageBytes);
          const int k0 = kb * kBK;
          auto load = [&](uint32_t dst, const CUtensorMap* map, int x, int y) {
            if (CTAS == 2) tma_load_2d_pair(dst, map, x, y, fbar);
            else tma_load_2d(dst, map, x, y, fbar);
          };
          if (A_MN) {
#pragma unroll
            for (int j = 0; j < kBM / 64; ++j) load(a_dst + j * (kBK * 128), map_a, m0 + 64 * j, k0);
          } else {
            load(a_dst, map_a, k0, m0);
          }
          if (B_MN) {
#pragma unroll
            for (int j = 0; j < G::kBNcta / 64; ++j) load(b_dst + j * (kBK * 128), map_b, n0 + 64 * j, k0);
          } else {
            load(b_dst, map_b, k0, n0);
          }
          ++issued;
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok && CTAS == 1) {
        // let the copies that are still in flight land before the CTA goes away
        int s = stage;
        uint32_t ph = phase;
        const long long pending = issued < kStages ? issued : kStages;
        for (long long i = 0; i < pending; ++i) {
          if (--s < 0) { s = kStages - 1; ph ^= 1u; }
          const long long t0 = clock64();
          while (!mbar_try_wait(full_bar(s), ph) && clock64() - t0 < kWaitLimitCycles) {}
        }
      }
    }
  } else if (warp == 1) {
    // ================= MMA issuer (the leader CTA of a pair issues for both) =================
    if (lane == 0 && rank == 0) {
      int stage = 0;
      uint32_t phase = 0;
      int acc = 0;
      uint32_t acc_phase = 0;
      bool ok = true;
      GroupCursor cursor;
      for (int u = team; u < total_units && ok; u += teams) {
        const Unit w = decode_unit<BN>(g, u, cursor);
        const int pi = cursor.pi;
        const bool A_MN = g.p[pi].a_mn != 0, B_MN = g.p[pi].b_mn != 0;
        const uint32_t idesc = instr_desc(g.p[pi].a_mn, g.p[pi].b_mn, G::kTileM, BN);
        const int drain = EPI == EPI_DRAIN ? g.p[pi].drain : 0;
        int done = 0;                                 // k-blocks in the accumulator
        for (int kb = w.kb_begin; kb < w.kb_end; ++kb) {
          const bool fresh = done == 0;
          if (fresh && !mbar_wait<CTAS == 2>(acce_bar(acc), acc_phase ^ 1u, abort_flag)) { ok = false; break; }
          if (!mbar_wait(full_bar(stage), phase, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint32_t a_addr = ring + stage * kStageBytes;
          const uint32_t b_addr = a_addr + kABytes;
          const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
          const uint64_t a_desc = smem_desc(a_addr, A_MN);
          const uint64_t b_desc = smem_desc(b_addr, B_MN);
#pragma unroll
          for (int k = 0; k < kBK / kUmmaK; ++k) {
            // K-major: 16 bf16 = 32 B along the swizzled row; MN-major: 16 k = two 8-k groups of 1024 B
            const uint64_t a_adv = (uint64_t)((A_MN ? k * 2048 : k * 32) >> 4);
            const uint64_t b_adv = (uint64_t)((B_MN ? k * 2048 : k * 32) >> 4);
            const uint32_t accum = (!fresh || k > 0) ? 1u : 0u;
            if (CTAS == 2) umma_bf16_pair(d_tmem, a_desc + a_adv, b_desc + b_adv, idesc, accum);
            else umma_bf16(d_tmem, a_desc + a_adv, b_desc + b_adv, idesc, accum);
          }
          // stage reusable (in both CTAs of a pair) once these MMAs have read it
          if (CTAS == 2) umma_commit_pair(empty_bar(stage));
          else umma_commit(empty_bar(stage));
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
          ++done;
          if ((EPI == EPI_DRAIN && done == drain) || kb + 1 == w.kb_end) {           // accumulator complete
            done = 0;
            if (CTAS == 2) umma_commit_pair(accf_bar(acc));
            else umma_commit(accf_bar(acc));
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
          }
        }
      }
    }
  } else if (G::kMoments && warp == 2 + kEpiWarps) {
    // ================= M and V: into the ring, and back once the epilogue has updated a piece =================
    if constexpr (G::kMoments) {
      if (lane == 0) {
        const uint32_t mring = ring + kStages * kStageBytes;
        int px[4] = {}, py[4] = {}, pp[4] = {-1, -1, -1, -1};   // what the slots hold
        uint32_t phase = 0;                           // of the pieces in the slots
        bool ok = true;
        auto store = [&](int q) {                     // the piece goes back; its slot may be written once the copies have read it
          if (!mbar_wait(mvdone_bar(q), phase, abort_flag)) return false;
          uint32_t src = mring + (uint32_t)q * 2u * kMomentBytes;
          const TcParams& p = g.p[pp[q]];
          if (py[q] < p.M)
            for (int x = px[q]; x < px[q] + kMomentCols && x < p.N; x += kBoxCols, src += kBoxBytes) {
              tma_store_2d(&g.map_m[pp[q]], x, py[q], src);
              tma_store_2d(&g.map_v[pp[q]], x, py[q], src + kMomentBytes);
            }
          bulk_commit();
          return true;
        };
        GroupCursor cursor;
        for (int u = team; u < total_units && ok; u += teams) {
          const Unit w = decode_unit<BN>(g, u, cursor);
          const int pi = cursor.pi;
          const int row0 = w.m0 + (int)rank * kBM, N = g.p[pi].N;
          for (int c = 0; c < BN && w.n0 + c < N && ok; c += kMomentCols) {
            const bool first = pp[0] < 0;
            for (int q = 0; q < 4; ++q) {
              if (!first) {
                if (!store(q)) { ok = false; break; }
                bulk_wait_read<0>();
              }
              px[q] = w.n0 + c;
              py[q] = row0 + kMomentRows * q;
              pp[q] = pi;
              const uint32_t dst = mring + (uint32_t)q * 2u * kMomentBytes;
              const int boxes = min(kMomentCols, N - px[q] + kBoxCols - 1) / kBoxCols;
              mbar_arrive_expect_tx(mvfull_bar(q), (uint32_t)boxes * 2u * kBoxBytes);
              for (int i = 0; i < boxes; ++i) tma_load_2d(dst + i * kBoxBytes, &g.map_m[pi], px[q] + i * kBoxCols, py[q], mvfull_bar(q));
              for (int i = 0; i < boxes; ++i)
                tma_load_2d(dst + kMomentBytes + i * kBoxBytes, &g.map_v[pi], px[q] + i * kBoxCols, py[q], mvfull_bar(q));
            }
            if (!first) phase ^= 1u;
          }
        }
        for (int q = 0; q < 4 && ok && pp[0] >= 0; ++q) ok = store(q);
        bulk_wait_read<0>();                          // the ring stays until the last store has read it
      }
    }
  } else {
    // ================= epilogue =================
    const int quarter = warp & 3;                   // TMEM lanes 32*quarter .. +31 belong to this warp
    int acc = 0;
    uint32_t acc_phase = 0;
    uint32_t mv_phase = 0, sq_phase = 0;
    bool ok = true;
    auto release_acc = [&]() {                        // accumulator free for the MMA warp (the leader's)
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (rank == 0) mbar_arrive(acce_bar(acc));
        else mbar_arrive_remote(map_to_cta(acce_bar(acc), 0));
      }
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    };
    GroupCursor cursor;
    for (int u = team; u < total_units && ok; u += teams) {
      const Unit w = decode_unit<BN>(g, u, cursor);
      const int pi = cursor.pi;
      const TcParams& p = g.p[pi];
      const int row = w.m0 + (int)rank * kBM + quarter * 32 + lane;
      const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * BN);
      if constexpr (EPI == EPI_ADAM_F32) {
        // the four warps of a quarter share its pieces, 16 columns each
        const int part = 16 * ((warp - 2) >> 2);
        const uint32_t sw = (uint32_t)lane & 7u;
        const AdamParams ap = p.ap;
        __nv_bfloat16* const n_row = p.Nout + (int64_t)row * p.ld_n;
        const uint32_t at = ring + kStages * kStageBytes + (uint32_t)quarter * 2u * kMomentBytes + (uint32_t)(part / kBoxCols) * kBoxBytes + (uint32_t)lane * 128u;
        if (!__all_sync(0xffffffffu, mbar_wait(accf_bar(acc), acc_phase, abort_flag))) { ok = false; break; }
        tc_fence_after();
        bool bad = false;
        for (int c = 0; c < BN && w.n0 + c < p.N; c += kMomentCols, mv_phase ^= 1u) {
          if (!__all_sync(0xffffffffu, mbar_wait(mvfull_bar(quarter), mv_phase, abort_flag))) { ok = false; break; }
          const int col0 = w.n0 + c + part;
          if (col0 < p.N) {
#pragma unroll 1
            for (int h = 0; h < 16; h += 8) {
              uint32_t v[8];
              tmem_ld_32x8(t_row + (uint32_t)(c + part + h), v);
              tmem_ld_wait();
#pragma unroll
              for (int j = 0; j < 8; ++j) asm volatile("" : "+r"(v[j]));          // not read before the wait
              const int valid = row < p.M ? p.N - (col0 + h) : 0;
              bad |= epi_adam_f32(ap, at, (uint32_t)(part % kBoxCols + h) >> 2, sw, v, valid, n_row + col0 + h);
            }
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(mvdone_bar(quarter));
        }
        if (!ok) break;
        if (bad) atomicOr(p.status, GALORE_DEV_NONFINITE);
      } else if constexpr (EPI == EPI_ADAM_Q8) {
        // warps 2..5 take the first 64 columns of the tile, warps 6..9 the next 64, and so on
        const int part = (warp - 2) >> 2;
        const int col0 = w.n0 + part * kAdamCols;
        const bool bad = epi_adam_q8(p, row, col0, t_row + (uint32_t)(part * kAdamCols), accf_bar(acc), acc_phase, abort_flag, *q8t, ok);
        if (!ok) break;
        if (bad) atomicOr(p.status, GALORE_DEV_NONFINITE);
      } else if constexpr (EPI == EPI_DRAIN) {
        const int part = 64 * ((warp - 2) >> 2);      // 64 columns a warp
        float sum[64];
#pragma unroll
        for (int j = 0; j < 64; ++j) sum[j] = 0.f;
#pragma unroll 1
        for (int kb = w.kb_begin; kb < w.kb_end; kb += p.drain) {
          if (!__all_sync(0xffffffffu, mbar_wait(accf_bar(acc), acc_phase, abort_flag))) { ok = false; break; }
          tc_fence_after();
          const uint32_t t = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * BN + part);
#pragma unroll
          for (int c = 0; c < 64; c += 16) {
            uint32_t v[16];
            tmem_ld_32x16(t + (uint32_t)c, v);
            tmem_ld_wait();
            add_acc(sum + c, v);
          }
          release_acc();
        }
        if (!ok) break;
#pragma unroll
        for (int c = 0; c < 64; c += 32) {
          if (w.n0 + part + c >= p.N) break;
          uint32_t v[32];
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(sum[c + j]);
          epi_partial(p, w, row, w.n0 + part + c, v);
        }
        continue;
      } else if constexpr (EPI == EPI_STATS) {
        if (!__all_sync(0xffffffffu, mbar_wait(accf_bar(acc), acc_phase, abort_flag))) { ok = false; break; }
        tc_fence_after();
        float* const sums = col_sums + sq_phase * (4 * BN);
        float row_lo = 0.f, row_hi = 0.f;             // (halves of a stretch: a balanced tree)
#pragma unroll 1
        for (int c = 0; c < BN && w.n0 + c < p.N; c += 32) {
          uint32_t v[32];
          tmem_ld_32x32(t_row + (uint32_t)c, v);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 32; ++j) asm volatile("" : "+r"(v[j]));          // not read before the wait
          epi_partial(p, w, row, w.n0 + c, v);
          float sq[32];                               // (rows and columns outside the matrix are zeros)
#pragma unroll
          for (int j = 0; j < 32; ++j) sq[j] = __uint_as_float(v[j]) * __uint_as_float(v[j]);
          if (c & 64) row_hi += tree_sum(sq);
          else row_lo += tree_sum(sq);
          sums[quarter * BN + c + lane] = column_sum(sq);
          if ((c & 127) == 96 || w.n0 + c + 32 >= p.N) {
            if (row < p.M && p.row_sq) p.row_sq[(int64_t)row * p.sq_tiles + (w.n0 + c) / 128] = row_lo + row_hi;
            row_lo = row_hi = 0.f;
          }
        }
        release_acc();
        __syncwarp();
        if (lane == 0) mbar_arrive(sq_bar);
        if (!__all_sync(0xffffffffu, mbar_wait(sq_bar, sq_phase, abort_flag))) { ok = false; break; }
        sq_phase ^= 1u;                               // the other half: a warp may be a tile ahead
        const int m0 = w.m0 + (int)rank * kBM;
        for (int c = (warp - 2) * 32 + lane; c < BN; c += 128)
          if (w.n0 + c < p.N && p.row_sq) {
            float* const dst = p.col_sq + (int64_t)(m0 / 64) * p.N + w.n0 + c;
            if (m0 < p.M) dst[0] = sums[c] + sums[BN + c];
            if (m0 + 64 < p.M) dst[p.N] = sums[2 * BN + c] + sums[3 * BN + c];
          }
        continue;
      } else {
        if (!mbar_wait(accf_bar(acc), acc_phase, abort_flag)) { ok = false; break; }
        tc_fence_after();
#pragma unroll 1
        for (int c = 0; c < BN; c += 32) {
          if (w.n0 + c >= p.N) break;                 // columns past the matrix: nothing to write
          uint32_t v[32];
          tmem_ld_32x32(t_row + (uint32_t)c, v);
          tmem_ld_wait();
          epi_partial(p, w, row, w.n0 + c, v);
        }
      }
      release_acc();
    }
  }

  if ((CTAS == 2 || G::kMoments) && *abort_flag) {    // gave up: let copies that are still in flight land
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000LL) {}
  }
  tc_fence_before();
  __syncthreads();
  if (CTAS == 2) cluster_sync_all();                  // neither CTA leaves while the peer may still signal it
  if (threadIdx.x == 0 && *abort_flag) atomicOr(g.p[0].status, GALORE_DEV_WAIT_EXPIRED);
  if (warp == 1) {
    tc_fence_after();
    if (CTAS == 2) tmem_dealloc_pair(tmem_base, kTmemCols);
    else tmem_dealloc(tmem_base, kTmemCols);
  }
}

// ---- host side --------------------------------------------------------------------------------------

std::atomic<PFN_cuTensorMapEncodeTiled_v12000> g_encode{nullptr};

galore_status_t ensure_encode() {
  if (g_encode.load(std::memory_order_acquire)) return GALORE_OK;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  GALORE_CUDA_TRY(cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres));
  if (!fn || qres != cudaDriverEntryPointSuccess) return GALORE_ERR_CUDA;
  g_encode.store((PFN_cuTensorMapEncodeTiled_v12000)fn, std::memory_order_release);
  return GALORE_OK;
}

}  // namespace

galore_status_t tensor_encode(CUtensorMap* map, const void* base, int32_t dtype, int64_t rows, int64_t cols, int64_t ld,
                              int box_rows, int box_cols, bool swizzle) {
  GALORE_TRY(ensure_encode());
  const int64_t es = (int64_t)dtype_size(dtype);
  if (((uintptr_t)base & 15) || (ld * es) % 16) return GALORE_ERR_ALIGNMENT;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)(ld * es)};
  cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1u, 1u};
  CUresult r = g_encode.load(std::memory_order_relaxed)(
      map, dtype == GALORE_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base), dims,
      strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
      CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    note_cuda_error(cudaErrorInvalidValue, "cuTensorMapEncodeTiled");
    return GALORE_ERR_CUDA;
  }
  return GALORE_OK;
}

namespace {
// bf16 operand of the kernel above: 64 columns per box
galore_status_t make_map(CUtensorMap* map, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
  return tensor_encode(map, base, GALORE_BF16, rows, cols, ld, box_rows, 64);
}
}  // namespace

int tensor_sm_count() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 148;
  }
  return sms;
}

galore_status_t CudaOrder::capturing(cudaStream_t st, bool* on) {
  cudaStreamCaptureStatus c = cudaStreamCaptureStatusNone;
  GALORE_CUDA_TRY(cudaStreamIsCapturing(st, &c));
  *on = c != cudaStreamCaptureStatusNone;
  return GALORE_OK;
}
galore_status_t CudaOrder::wait(cudaStream_t st, cudaEvent_t e) {
  GALORE_CUDA_TRY(cudaStreamWaitEvent(st, e, 0));
  return GALORE_OK;
}
galore_status_t CudaOrder::create(cudaEvent_t* e) {
  GALORE_CUDA_TRY(cudaEventCreateWithFlags(e, cudaEventDisableTiming));
  return GALORE_OK;
}
galore_status_t CudaOrder::record(cudaEvent_t e, cudaStream_t st) {
  GALORE_CUDA_TRY(cudaEventRecord(e, st));
  return GALORE_OK;
}

LaunchOrder<CudaOrder>& launch_order() {
  static LaunchOrder<CudaOrder> order;
  return order;
}

namespace {

template <int EPI, int CTAS, int CAP, int BN = kBN>
galore_status_t launch_tc_variant(const TcArgs<CAP>& g, bool early, cudaStream_t st) {
  constexpr int smem = Geo<CTAS, EPI, BN>::kSmemBytes + epi_smem(EPI);
  static_assert(smem <= 227 * 1024, "shared memory of one CTA");
  static std::atomic<uint64_t> configured{0};
  auto kern = gemm_tc_kernel<EPI, CTAS, CAP, BN>;
  GALORE_TRY(allow_smem(configured, (const void*)kern, smem));
  const int units = g.unit_end[g.count - 1];
  if (units <= 0) return GALORE_OK;
  const int teams = std::min(units, tensor_sm_count() / CTAS);
  return launch_kernel(kern, dim3((unsigned)(teams * CTAS)), epi_threads(EPI, BN), smem, CTAS, early, st, g);
}

// every problem of a group was tiled for the same variant (TcParams::tile_m)
template <int EPI>
galore_status_t launch_tc(const TcGroup& g, bool early, cudaStream_t st) {
  if (g.count < 1 || g.count > kMaxGroup) return GALORE_ERR_INVALID_ARG;
  for (int i = 1; i < g.count; ++i)
    if (g.p[i].tile_m != g.p[0].tile_m) return GALORE_ERR_INVALID_ARG;
  const bool pair = g.p[0].tile_m == 2 * kBM;
  if (g.count == 1) {
    TcArgs<1> one;
    one.map_a[0] = g.map_a[0];
    one.map_b[0] = g.map_b[0];
    one.p[0] = g.p[0];
    one.unit_end[0] = g.unit_end[0];
    one.count = 1;
    one.q8 = g.q8;
    one.map_m[0] = g.map_m[0];
    one.map_v[0] = g.map_v[0];
    if constexpr (EPI == EPI_DRAIN || EPI == EPI_PARTIAL)
      // (the group's units are the same; a K-major B comes in boxes of 256 rows, more than this kernel's stages hold)
      if (!pair && g.p[0].N <= 128 && g.p[0].b_mn) return launch_tc_variant<EPI, 1, 1, 128>(one, early, st);
    return pair ? launch_tc_variant<EPI, 2, 1>(one, early, st) : launch_tc_variant<EPI, 1, 1>(one, early, st);
  }
  if constexpr (EPI == EPI_DRAIN) return GALORE_ERR_INVALID_ARG;      // single matrices only
  else return pair ? launch_tc_variant<EPI, 2, kMaxGroup>(g, early, st) : launch_tc_variant<EPI, 1, kMaxGroup>(g, early, st);
}

// appends one problem to a group
void group_add(TcGroup& g, const CUtensorMap& ma, const CUtensorMap& mb, const TcParams& p) {
  const int i = g.count++;
  g.map_a[i] = ma;
  g.map_b[i] = mb;
  g.p[i] = p;
  g.unit_end[i] = (i > 0 ? g.unit_end[i - 1] : 0) + p.tiles_m * p.tiles_n * p.splits;
}

void fill_tiles(TcParams& p, int M, int N, int K, int splits, int ctas) {
  p.M = M; p.N = N; p.K = K;
  p.tile_m = kBM * ctas;
  p.tiles_m = (int)ceil_div(M, p.tile_m);
  p.tiles_n = (int)ceil_div(N, kBN);
  p.kblocks_total = (int)ceil_div(K, kBK);
  if (splits < 1) splits = 1;
  p.kblocks_per_split = (int)ceil_div(p.kblocks_total, splits);
  p.splits = (int)ceil_div(p.kblocks_total, p.kblocks_per_split);
}

// K slices that fill the last wave of CTAs best, keeping at least 4 k-blocks per slice
int fill_splits(int64_t M, int64_t N, int64_t K, int ctas) {
  const int64_t tiles = ceil_div(M, kBM * ctas) * ceil_div(N, kBN);
  const int kblocks = (int)ceil_div(K, kBK);
  const int sms = 148 / ctas;
  int best = 1;
  double best_score = -1.0;
  for (int s = 1; s <= 8; ++s) {
    const int per = (int)ceil_div(kblocks, s);
    if (s > 1 && per < 4) break;
    const int eff_s = (int)ceil_div(kblocks, per);
    if (eff_s != s) continue;
    const int64_t units = tiles * s;
    const double fill = (double)units / (double)(ceil_div(units, sms) * sms);
    // each extra slice costs one more partial buffer to write and read back
    const double score = fill - 0.02 * (s - 1);
    if (score > best_score + 1e-9) { best_score = score; best = s; }
  }
  return best;
}

// K slices of a single product (EPI_DRAIN) with a kernel behind it that reads the partial results: the least of waves x (k-blocks x
// time of one + time of a unit) plus the slices' round trip.  Microseconds a k-block, fitted to steps in 1 to 7 slices of 2048 x 2048 and
// 2048 x 5461 at rank 512, 4096 x 11008 at 1024, 11008 x 4096 and 4096 x 11008 at 128: pairs 0.33, single CTAs 0.35, with tiles
// of 128 columns 0.25.  (2048 x 5461, 8-bit moments: 58.9 us unsliced, 61.4 in three, 68.1 in five, which fill the machine best.)
// Half a microsecond less is the least that the fit can tell: below it the slices that fill the machine stay.  (Steps in the one / the
// other: 3008 x 1183 at rank 80 predicted 3.40 / 3.39, measured 20.4 / 21.7; 1216 x 2816 at 192 4.80 / 4.69, 21.3 / 22.3; 1344 x 2816 at 184
// 5.17 / 4.89, 22.0 / 22.5; 3840 x 2432 at 632 15.9 / 15.4, 55.8 / 54.5; 1920 x 2267 at 256 6.32 / 5.51, 29.3 / 28.5; the 19
// sizes measured above the line all gained.)
// codes: 8-bit moments, whose codes at a threshold show the last bit of R.  Only slices that leave R's bits as they are: those that
// fill the machine, or one, whose accumulators are drained where those slices end and added in their order.
int time_splits(int64_t M, int64_t N, int64_t K, int ctas, bool codes) {
  const int64_t tiles = ceil_div(M, kBM * ctas) * ceil_div(N, kBN);
  const int kblocks = (int)ceil_div(K, kBK);
  const double block = ctas == 2 ? 0.33 : (N <= 128 ? 0.25 : 0.35);
  auto us = [&](int s) {
    return (double)ceil_div(tiles * s, 148 / ctas) * (ceil_div(kblocks, s) * block + 1.1) + s * (0.1 + (double)(M * N) * 4.0 / 6.0e6);
  };
  const int fill = fill_splits(M, N, K, ctas);
  int best = fill;
  double best_us = us(fill) - 0.5;
  for (int s = 1; s <= (codes ? 1 : 8); ++s) {
    const int per = (int)ceil_div(kblocks, s);
    if (s > 1 && per < 4) break;
    if ((int)ceil_div(kblocks, per) != s) continue;
    if (us(s) < best_us) { best_us = us(s); best = s; }
  }
  return best;
}

}  // namespace

bool tensor_path_eligible(const galore_config_t& c) {
  return c.g_dtype == GALORE_BF16 && c.p_dtype == GALORE_BF16 && (c.rank % 8) == 0;
}

// CTA pairs (256-row tiles) whenever every GEMM of the layer has at least 256 rows
int tensor_ctas(const galore_config_t& c) { return c.rank >= 256 ? 2 : 1; }

int tensor_proj_splits(const galore_config_t& c, bool left) {
  const int ctas = tensor_ctas(c);
  return left ? fill_splits(c.rank, c.n, c.m, ctas) : fill_splits(c.m, c.rank, c.n, ctas);
}
int tensor_chain_blocks(int64_t K, int splits) { return (int)ceil_div(ceil_div(K, kBK), std::max(1, splits)); }
int tensor_step_splits(const galore_config_t& c, bool left) {
  const int ctas = tensor_ctas(c);
  const bool codes = c.state_fmt == GALORE_STATE_Q8_BLOCK;
  return left ? time_splits(c.rank, c.n, c.m, ctas, codes) : time_splits(c.m, c.rank, c.n, ctas, codes);
}

galore_status_t tensor_plan_init(TensorPlan* plan, const galore_config_t& c, bool left, void* P) {
  plan->ready = false;
  plan->ctas = tensor_ctas(c);
  const int64_t r = c.rank;
  if (left) {
    // A = P^T, MN-major from P (m x r)
    GALORE_TRY(make_map(&plan->map_p_proj, P, c.m, r, r, 64));
  } else {
    // B = Q (n x r), MN-major
    GALORE_TRY(make_map(&plan->map_p_proj, P, c.n, r, r, 64));
  }
  plan->ready = true;
  return GALORE_OK;
}

bool tensor_operands_aligned(const galore_config_t& c, const void* W, int64_t ldw, const void* G, int64_t ldg) {
  if (((uintptr_t)G & 15) || (ldg % 8)) return false;
  if ((uintptr_t)W & 15) return false;
  return c.w_dtype == GALORE_BF16 ? (ldw % 8) == 0 : (ldw % 4) == 0;
}

// ---- problems -----------------------------------------------------------------------------------

// R partials <- P^T G (left) / G Q (right)
static galore_status_t project_problem(const TensorPlan* plan, const galore_config_t& c, bool left, const void* G,
                                       int64_t ldg, float* part, int64_t ld_part, int splits, int32_t* status,
                                       TcParams* p, CUtensorMap* ma, CUtensorMap* mb) {
  if (!plan->ready) return GALORE_ERR_STATE;
  const int r = c.rank;
  *p = TcParams{};
  p->status = status;
  p->part = part;
  p->ld_part = ld_part;
  p->vec32 = (((uintptr_t)part & 31) == 0 && (ld_part % 8) == 0) ? 1 : 0;
  if (left) {
    // A = P^T, M/N-major from P; B = G, M/N-major.  G is the big operand: units sharing a G panel run together
    fill_tiles(*p, r, (int)c.n, (int)c.m, splits, plan->ctas);
    p->split_stride = (int64_t)r * ld_part;
    p->m_fast = 1;
    p->a_mn = 1;
    p->b_mn = 1;
    *ma = plan->map_p_proj;
    return make_map(mb, G, c.m, c.n, ldg, 64);
  }
  // A = G, K-major; B = Q, M/N-major
  fill_tiles(*p, (int)c.m, r, (int)c.n, splits, plan->ctas);
  p->split_stride = (int64_t)c.m * ld_part;
  p->m_fast = 0;
  p->a_mn = 0;
  p->b_mn = 1;
  *mb = plan->map_p_proj;
  return make_map(ma, G, c.m, c.n, ldg, kBM);
}

// the Adam part of a projection problem
static galore_status_t set_adam(TcParams* p, const TcAdamArgs& a) {
  if (a.state_fmt == GALORE_STATE_Q8_BLOCK &&
      (a.q_block < 256 || a.q_block > 2048 || (a.q_block & (a.q_block - 1)) != 0)) return GALORE_ERR_INVALID_ARG;
  p->Mc = a.Mc; p->Vc = a.Vc; p->Mam = a.Mam; p->Vam = a.Vam;
  p->ld_s = a.ld_s;
  p->q_rows = a.q_block / kStateTileCols;
  p->q_tiles_c = (int)ceil_div(p->N, kStateTileCols);
  p->Nout = (__nv_bfloat16*)a.Nout;
  p->ld_n = a.ld_n;
  p->ap = a.ap;
  // 8-byte accesses to the codes, 16-byte stores of N
  const uintptr_t bases = (uintptr_t)a.Nout | (uintptr_t)a.Mc | (uintptr_t)a.Vc;
  p->adam_vec = ((bases & 31) == 0 && (a.ld_s % 32) == 0 && (a.ld_n % 16) == 0) ? 1 : 0;
  return GALORE_OK;
}

static galore_status_t launch_project_adam(const TcGroup& g, int32_t state_fmt, bool early, cudaStream_t st) {
  if (state_fmt == GALORE_STATE_F32) return launch_tc<EPI_ADAM_F32>(g, early, st);
  return launch_tc<EPI_ADAM_Q8>(g, early, st);
}

// ---- groups: many layers per launch ------------------------------------------------------------------

struct TensorGroup {
  TcGroup g;
};

TensorGroup* tensor_group_new() {
  TensorGroup* t = new (std::nothrow) TensorGroup;
  if (t) t->g.count = 0;
  return t;
}
void tensor_group_free(TensorGroup* t) { delete t; }
void tensor_group_reset(TensorGroup* t) { t->g.count = 0; }
int tensor_group_capacity() { return kMaxGroup; }

galore_status_t tensor_group_add_project(TensorGroup* t, const TensorPlan* plan, const galore_config_t& c, bool left,
                                         const void* G, int64_t ldg, float* part, int64_t ld_part, int splits,
                                         int32_t* status) {
  if (t->g.count >= kMaxGroup) return GALORE_ERR_BUFFER_TOO_SMALL;
  TcParams p;
  CUtensorMap ma, mb;
  GALORE_TRY(project_problem(plan, c, left, G, ldg, part, ld_part, splits, status, &p, &ma, &mb));
  group_add(t->g, ma, mb, p);
  return GALORE_OK;
}

galore_status_t tensor_group_add_project_adam(TensorGroup* t, const TensorPlan* plan, const galore_config_t& c, bool left,
                                              const void* G, int64_t ldg, const TcAdamArgs& adam, int32_t* status) {
  if (t->g.count >= kMaxGroup) return GALORE_ERR_BUFFER_TOO_SMALL;
  TcParams p;
  CUtensorMap ma, mb;
  GALORE_TRY(project_problem(plan, c, left, G, ldg, nullptr, 0, 1, status, &p, &ma, &mb));
  GALORE_TRY(set_adam(&p, adam));
  if (adam.state_fmt == GALORE_STATE_F32) {
    GALORE_TRY(tensor_encode(&t->g.map_m[t->g.count], adam.M, GALORE_F32, p.M, p.N, adam.ld_s, kMomentRows, kBoxCols));
    GALORE_TRY(tensor_encode(&t->g.map_v[t->g.count], adam.V, GALORE_F32, p.M, p.N, adam.ld_s, kMomentRows, kBoxCols));
    if (((uintptr_t)adam.Nout & 15) || (adam.ld_n % 8)) return GALORE_ERR_ALIGNMENT;
  }
  group_add(t->g, ma, mb, p);
  return GALORE_OK;
}

galore_status_t tensor_group_launch_project_adam(TensorGroup* t, int32_t state_fmt, bool early, cudaStream_t st) {
  if (t->g.count == 0) return GALORE_OK;
  if (state_fmt == GALORE_STATE_Q8_BLOCK) GALORE_TRY(q8_table_ptrs(&t->g.q8));
  return launch_project_adam(t->g, state_fmt, early, st);
}

// A plain GEMM problem for the group: C (M x N, fp32, leading dimension ldc) = op(A) op(B), bf16
// operands.  a_mn = 1: A is stored K rows x M contiguous, 0: M rows x K contiguous; b_mn likewise
// (K x N contiguous resp. N x K contiguous).  All problems of a group must have M on the same side
// of 256 (they share the tile shape).
galore_status_t tensor_group_add_gemm(TensorGroup* t, const void* A, int64_t lda, int a_mn, const void* B, int64_t ldb,
                                      int b_mn, int M, int N, int K, float* C, int64_t ldc, int32_t* status) {
  if (t->g.count >= kMaxGroup) return GALORE_ERR_BUFFER_TOO_SMALL;
  const int ctas = M >= 2 * kBM ? 2 : 1;
  TcParams p = {};
  p.status = status;
  p.part = C;
  p.ld_part = ldc;
  p.split_stride = 0;
  p.vec32 = (((uintptr_t)C & 31) == 0 && (ldc % 8) == 0) ? 1 : 0;
  p.a_mn = a_mn ? 1 : 0;
  p.b_mn = b_mn ? 1 : 0;
  p.m_fast = 1;
  fill_tiles(p, M, N, K, 1, ctas);
  CUtensorMap ma, mb;
  if (a_mn) GALORE_TRY(make_map(&ma, A, K, M, lda, 64));
  else GALORE_TRY(make_map(&ma, A, M, K, lda, kBM));
  if (b_mn) GALORE_TRY(make_map(&mb, B, K, N, ldb, 64));
  else GALORE_TRY(make_map(&mb, B, N, K, ldb, kBN / ctas));
  group_add(t->g, ma, mb, p);
  return GALORE_OK;
}

void tensor_group_want_squares(TensorGroup* t, float* row_sq, float* col_sq, int tiles) {
  TcParams& p = t->g.p[t->g.count - 1];
  p.row_sq = row_sq;
  p.col_sq = col_sq;
  p.sq_tiles = tiles;
}
galore_status_t tensor_group_launch_project(TensorGroup* t, bool early, cudaStream_t st) {
  if (t->g.count == 0) return GALORE_OK;
  for (int i = 0; i < t->g.count; ++i)
    if (t->g.p[i].row_sq) return launch_tc<EPI_STATS>(t->g, early, st);
  return launch_tc<EPI_PARTIAL>(t->g, early, st);
}
galore_status_t tensor_group_launch_project_drained(TensorGroup* t, int blocks, bool early, cudaStream_t st) {
  if (t->g.count != 1 || blocks < 1) return GALORE_ERR_INVALID_ARG;
  t->g.p[0].drain = blocks;
  return blocks < t->g.p[0].kblocks_per_split ? launch_tc<EPI_DRAIN>(t->g, early, st) : launch_tc<EPI_PARTIAL>(t->g, early, st);
}

}  // namespace galore
