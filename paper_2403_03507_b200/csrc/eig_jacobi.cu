// Block one-sided Jacobi for the symmetric eigenproblem of the Rayleigh-Ritz step (Eq. 12-13).
//
// The rows of X (initially H) are made mutually orthogonal by plane rotations, as in the Hestenes
// method; at convergence X = Theta V^T.  Rows are grouped in blocks of 32.  One round pairs the
// blocks by a round-robin schedule; for every pair of blocks
//   1. the 64 x 64 Gram matrix of its rows is formed (fp64 tensor-core MMA, columns split over CTAs),
//   2. one cyclic sweep of rotations is run on that Gram matrix in shared memory, which is exactly
//      the sequence of rotations the 64 rows themselves would receive, accumulated into a 64 x 64
//      orthogonal matrix,
//   3. the accumulated rotation is applied to the 64 rows (again an fp64 MMA product).
// All blocks meet once per sweep; a sweep without any rotation ends the iteration.  Compared with
// rotating two rows per CTA and round, the matrix is read and written twice per block round instead
// of once per row round: 32 times less traffic for the same rotations.
#include "eig_jacobi.cuh"

#include <algorithm>

#include "gemm_dmma.cuh"
#include "launch.cuh"

namespace galore {
namespace {

constexpr int kBlockRows = 32;
constexpr int kPairRows = 64;
// Columns summed by one CTA of the Gram kernel: 256, or 64 where that leaves only a few CTAs, each with eight 32-column tiles
// one after the other (with 256 the Gram matrices of b = 256, four pairs, take 11 us, the longest part of them in one chain).
// By the block's size alone.
__host__ __device__ constexpr int gram_chunk(int b) { return b <= 512 ? 64 : 256; }
constexpr int kApplyCols = 128;   // columns transformed by one CTA of the apply kernel
constexpr int kGramLd = 36;       // shared-memory row strides, all = 4 mod 16 doubles: the 8 x 4 operand
constexpr int kRotLd = 68;        // fragments of the fp64 MMA then fall on distinct banks
constexpr int kApplyHalf = 64;    // columns in shared memory at a time
constexpr int kHalfLd = 68;

// Round-robin tournament of n players (n even): in `round`, position k meets position n - 1 - k.
__host__ __device__ __forceinline__ int rr_player(int pos, int round, int n) {
  if (pos == 0) return 0;
  const int m = n - 1;
  int v = (pos - 1 - round) % m;
  if (v < 0) v += m;
  return 1 + v;
}

struct BlockPair {
  int I, J;   // I < J
  __device__ __forceinline__ int row(int l) const { return l < kBlockRows ? I * kBlockRows + l : J * kBlockRows + (l - kBlockRows); }
};
__device__ __forceinline__ BlockPair block_pair(int pair, int round, int nblk) {
  int I = rr_player(pair, round, nblk), J = rr_player(nblk - 1 - pair, round, nblk);
  if (I > J) { const int t = I; I = J; J = t; }
  return BlockPair{I, J};
}

// part[(pair * chunks + chunk)] (64 x 64) = rows(pair)[:, chunk] rows(pair)[:, chunk]^T
// In the first round of a sweep its upper triangle, later the products of the two blocks with each other alone: those within a
// block the sweep kernel has carried along since (eight 1280 x 1280 matrices: 40 -> 26 us a round).
__global__ void __launch_bounds__(128) jb_gram_kernel(const double* X, int b, int nblk, int round, int chunks,
                                                      double* __restrict__ part, const SlotList slots) {
  grid_dependency_wait();
  grid_launch_dependents();
  __shared__ __align__(16) double Xs[2][kPairRows][kGramLd];
  const int pair = blockIdx.x, chunk = blockIdx.y;
  {
    const int64_t shift = (int64_t)slots.id[blockIdx.z] * slots.bytes;     // blockIdx.z: workspace slot
    X = slot_ptr(X, shift);
    part = slot_ptr(part, shift);
  }
  const BlockPair bp = block_pair(pair, round, nblk);
  if (bp.I * kBlockRows >= b) return;                 // both blocks are padding
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  const bool cross = round > 0;                       // warp (wy, wx): 16 x 16 of the 32 x 32 products of the two blocks
  const int wy = warp >> 1, wx = warp & 1;
  // The Gram matrix is symmetric and the sweep reads its upper triangle only: of the 8 x 8 grid of 8 x 8
  // tiles the 36 with tile row <= tile column are formed.  Warps 0 and 3 take the upper halves of the two
  // diagonal 32 x 32 quadrants (10 tiles each), warps 1 and 2 the two column halves of the off-diagonal one.
  const bool diagonal = warp == 0 || warp == 3;
  const int rb = warp == 3 ? 1 : 0, cb = rb;                     // the diagonal quadrant of warps 0 and 3
  const int jbase = warp == 2 ? 2 : 0;                           // first tile column of warps 1 and 2
  const int c_begin = chunk * gram_chunk(b);
  const int c_end = min(b, c_begin + gram_chunk(b));
  const int tiles = (c_end - c_begin + 31) / 32;
  const bool vec = (b & 1) == 0;

  double acc[4][4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;

  double2 stage[8];
  auto fetch = [&](int tile) {
    const int c0 = c_begin + tile * 32;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int id = tid + 128 * i;
      const int l = id >> 4, col = c0 + (id & 15) * 2;
      const int row = bp.row(l);
      double2 v = make_double2(0.0, 0.0);
      if (row < b) {
        const double* src = X + (int64_t)row * b + col;
        if (vec && col + 1 < c_end) {
          v = *reinterpret_cast<const double2*>(src);
        } else {
          if (col < c_end) v.x = src[0];
          if (col + 1 < c_end) v.y = src[1];
        }
      }
      stage[i] = v;
    }
  };
  auto stash = [&](int buf) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int id = tid + 128 * i;
      *reinterpret_cast<double2*>(&Xs[buf][id >> 4][(id & 15) * 2]) = stage[i];
    }
  };

  fetch(0);
  stash(0);
  __syncthreads();
  for (int tile = 0; tile < tiles; ++tile) {
    const int buf = tile & 1;
    if (tile + 1 < tiles) fetch(tile + 1);
    if (cross) {
#pragma unroll
      for (int ks = 0; ks < 8; ++ks) {
        double a[2], bb[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) a[i] = Xs[buf][wy * 16 + i * 8 + g][ks * 4 + t];
#pragma unroll
        for (int j = 0; j < 2; ++j) bb[j] = Xs[buf][32 + wx * 16 + j * 8 + g][ks * 4 + t];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int j = 0; j < 2; ++j) dmma_m8n8k4(acc[i][j], a[i], bb[j]);
      }
    } else if (diagonal) {     // upper half of a diagonal quadrant: tiles (i, j) with i <= j
#pragma unroll
      for (int ks = 0; ks < 8; ++ks) {
        double a[4], bb[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = Xs[buf][rb * 32 + i * 8 + g][ks * 4 + t];
#pragma unroll
        for (int j = 0; j < 4; ++j) bb[j] = Xs[buf][cb * 32 + j * 8 + g][ks * 4 + t];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = i; j < 4; ++j) dmma_m8n8k4(acc[i][j], a[i], bb[j]);
      }
    } else {                   // two of the four tile columns of the off-diagonal quadrant (kept in acc[.][0..1])
#pragma unroll
      for (int ks = 0; ks < 8; ++ks) {
        double a[4], bb[2];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = Xs[buf][i * 8 + g][ks * 4 + t];
#pragma unroll
        for (int j = 0; j < 2; ++j) bb[j] = Xs[buf][32 + (jbase + j) * 8 + g][ks * 4 + t];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 2; ++j) dmma_m8n8k4(acc[i][j], a[i], bb[j]);
      }
    }
    if (tile + 1 < tiles) stash(buf ^ 1);
    __syncthreads();
  }

  double* out = part + ((int64_t)pair * chunks + chunk) * (kPairRows * kPairRows);
  if (cross) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int r = wy * 16 + i * 8 + g, c = 32 + wx * 16 + j * 8 + 2 * t;
        *reinterpret_cast<double2*>(out + r * kPairRows + c) = make_double2(acc[i][j][0], acc[i][j][1]);
      }
  } else if (diagonal) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = i; j < 4; ++j) {
        const int r = rb * 32 + i * 8 + g, c = cb * 32 + j * 8 + 2 * t;
        *reinterpret_cast<double2*>(out + r * kPairRows + c) = make_double2(acc[i][j][0], acc[i][j][1]);
      }
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int r = i * 8 + g, c = 32 + (jbase + j) * 8 + 2 * t;
        *reinterpret_cast<double2*>(out + r * kPairRows + c) = make_double2(acc[i][j][0], acc[i][j][1]);
      }
  }
}

// One cyclic sweep over the 64 rows of a block pair, run on their Gram matrix A, with the rotations
// accumulated into Rot (Rot <- R Rot, so that the rows themselves become Rot x rows).
//
// The 64 rows sit at the 64 positions of a round-robin table; slot k pairs position k (its f) and 63 - k
// (its g).  After every round the rows move on by one position (position 0 stays), and the data moves with
// them: a round reads one shared-memory copy of A and writes the other at the next positions, so every
// address a thread touches is the same in all rounds and is computed once.  After the 63 rounds of a
// sweep all rows are back where they started.
//   * The 32 rotations of a round split A into 2 x 2 blocks (f, g of slot u x f, g of slot v) that
//     transform independently, B <- R_u B R_v^T.  Of (u, v) and (v, u) the one with v - u mod 32 <= 16 is
//     kept.  The entries of a kind (f f, f g, g f, g g) lie in rows of equal v - u, column u, and a warp
//     takes a row: what it reads is contiguous, and so is what it writes, one position on, except at the
//     ends of the table.  8 warps hold two rows each.
//   * Rot lives in the registers of 8 warps.  A thread holds 4 slots (8 rows) of two columns; moving on by
//     one position is a renaming of registers, with one entry of a column passed up and one down to the
//     lanes that hold the neighbouring slots.
//   * One warp keeps the squared norms (the diagonal of A) and the product of every slot's two rows in registers and
//     computes the next round's rotations.  The product that a rotation needs is worked out from the old A and the
//     current rotations again, so the rotations of round t + 1 are found while the other warps apply those of round t,
//     and a round has a single barrier.
//   * The angle is computed in single precision (after scaling by the exponent of the larger of
//     aqq - app and 2 apq) and (c, s) are then renormalised in double precision: the rotation is
//     orthogonal to double rounding, its angle accurate to about 1e-7.
// own: the products within each block (32 x 32 of a block, upper triangle), read after the first round of the sweep and
// written in every one.  flags[pair] = rotations applied (0: Rot is the identity and is not written).
//
// What bounds it: 63 rounds one after the other, each about 600 shared-memory wavefronts (half of them reads, then the writes) and,
// beside them, the latency of an angle.  56 registers: two CTAs on an SM, for groups of more than 148 pairs.  (A off the diagonal in
// single precision: half the wavefronts, 3.52 instead of 3.73 ms for the refresh of 512 x 1376 at rank 128, 116.8 instead of 119.5 ms
// for eight 4096 x 4096 at 1024.  Not taken: the sums it holds are fp64 ones.)
constexpr int kSweepRounds = kPairRows - 1;
constexpr int kSlots = kPairRows / 2;
constexpr int kBlockWarps = 8;                                // blocks with u != v: rows 1 .. 16
constexpr int kRotWarps = 8;                                  // Rot, 8 columns each
constexpr int kAngleWarp = kBlockWarps + kRotWarps;
constexpr int kSweepThreads = (kAngleWarp + 1) * 32;
constexpr int kLaneSlots = 4;                                 // slots of Rot in one thread
constexpr int kLaneGroups = kSlots / kLaneSlots;              // lanes that share a column of Rot
constexpr int kLaneCols = 32 / kLaneGroups;
constexpr int kKindRows = kSlots / 2 + 1;                     // rows of a kind of entry: v - u = 0 .. 16
constexpr int kKindSize = kKindRows * kSlots;
constexpr int kPackedSize = 4 * kKindSize;                    // one copy of A
constexpr int kLoads = (kPairRows * kPairRows + kSweepThreads - 1) / kSweepThreads;

__host__ __device__ __forceinline__ int next_position(int pos) { return pos == 0 ? 0 : (pos == kPairRows - 1 ? 1 : pos + 1); }
__host__ __device__ __forceinline__ int slot_of(int pos) { return pos < kSlots ? pos : kPairRows - 1 - pos; }
// where the entry of positions p and q (in either order) is kept in a copy of A
__host__ __device__ __forceinline__ int packed_offset(int p, int q) {
  int u = slot_of(p), v = slot_of(q);
  int gu = p >= kSlots, gv = q >= kSlots;
  int d = (v - u) & (kSlots - 1);
  const bool other = d == 0 ? gu > gv : (d > kSlots / 2 || (d == kSlots / 2 && u >= kSlots / 2));
  if (other) {
    int t = u; u = v; v = t;
    t = gu; gu = gv; gv = t;
    d = (kSlots - d) & (kSlots - 1);
  }
  return ((gu * 2 + gv) * kKindRows + d) * kSlots + u;
}

struct BlockWrites {
  int at[4];       // where (fu, fv), (fu, gv), (gu, fv), (gu, gv) go, one position on
};
__device__ __forceinline__ BlockWrites block_writes(int u, int v) {
  const int nfu = next_position(u), ngu = next_position(kPairRows - 1 - u);
  const int nfv = next_position(v), ngv = next_position(kPairRows - 1 - v);
  return BlockWrites{{packed_offset(nfu, nfv), packed_offset(nfu, ngv), packed_offset(ngu, nfv), packed_offset(ngu, ngv)}};
}
struct BlockValues {
  double a0, a1, a2, a3;
};
// B <- R_u B R_v^T for one 2 x 2 block
__device__ __forceinline__ void block_write(const BlockWrites& t, const double2 ru, const double2 rv, const BlockValues& b, double* An) {
  const double r00 = ru.x * b.a0 - ru.y * b.a2, r01 = ru.x * b.a1 - ru.y * b.a3;
  const double r10 = ru.y * b.a0 + ru.x * b.a2, r11 = ru.y * b.a1 + ru.x * b.a3;
  An[t.at[0]] = rv.x * r00 - rv.y * r01;
  An[t.at[1]] = rv.y * r00 + rv.x * r01;
  An[t.at[2]] = rv.x * r10 - rv.y * r11;
  An[t.at[3]] = rv.y * r10 + rv.x * r11;
}

// 1 / sqrt(x) of a normal number
__device__ __forceinline__ float rsqrt_normal(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// the rotation that annihilates apq; {1, 0} when the pair is orthogonal to the tolerance.  Every lane computes the angle and
// selects at the end: the latency of this function is on the path of every round, and a branch would put the test in front.
__device__ __forceinline__ double2 jacobi_rotation(double app, double aqq, double apq, double tol2, int& applied) {
  // tan(2 phi) = 2 apq / (aqq - app), |phi| <= pi/4.  With h = hypot(d, o): cos(2 phi) = |d| / h,
  // c = sqrt((1 + |d|/h) / 2), s = sign(d) o / (2 h c).
  const double d = aqq - app, o = 2.0 * apq;
  const int ex = max(__double2hiint(d) & 0x7fffffff, __double2hiint(o) & 0x7fffffff) >> 20;    // the larger exponent
  const double sc = __hiloint2double((2046 - ex) << 20, 0);
  const float df = (float)(d * sc), of = (float)(o * sc);
  const float rh = rsqrt_normal(fmaf(df, df, of * of));
  const float v = fmaf(0.5f * fabsf(df), rh, 0.5f);
  const float rc = rsqrt_normal(v);
  const float c0 = v * rc, s0 = (d >= 0.0 ? 0.5f : -0.5f) * of * rh * rc;
  const double c = (double)c0, s = (double)s0;
  const double eps = fma(c, c, fma(s, s, -1.0));          // c0^2 + s0^2 = 1 + eps, |eps| ~ 1e-7
  const double fix = fma(eps, fma(eps, 0.375, -0.5), 1.0);  // (1 + eps)^-1/2 to O(eps^3)
  const bool turn = apq != 0.0 && apq * apq > tol2 * app * aqq && ex >= 1 && ex <= 2045 && s0 != 0.0f;
  applied += turn;
  return turn ? make_double2(c * fix, s * fix) : make_double2(1.0, 0.0);
}

__global__ void __launch_bounds__(kSweepThreads, 2) jb_sweep_kernel(const double* part, int chunks, int b, int nblk,
                                                                 int round, double tol, double* own, double* __restrict__ rot_out,
                                                                 int* __restrict__ flags, int* __restrict__ rotations,
                                                                 const SlotList slots) {
  grid_dependency_wait();
  grid_launch_dependents();
  {
    const int64_t shift = (int64_t)slots.id[blockIdx.y] * slots.bytes;     // blockIdx.y: workspace slot
    part = slot_ptr(part, shift);
    own = slot_ptr(own, shift);
    rot_out = slot_ptr(rot_out, shift);
    flags = slot_ptr(flags, shift);
    rotations = slot_ptr(rotations, shift);
  }
  __shared__ double A0[kPackedSize], A1[kPackedSize];     // the Gram matrix off the diagonal, even rounds and odd ones
  __shared__ double diag[kPairRows];
  __shared__ double2 cs[2][kSlots];               // the rotations of the current round and of the next
  __shared__ double2 cs_rot[2][kSlots + kLaneGroups];     // the same for the warps of Rot, which read eight slots, 4 apart, at once
  __shared__ int total;
  const int pair = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const BlockPair bp = block_pair(pair, round, nblk);
  if (bp.I * kBlockRows >= b) {
    if (tid == 0) flags[pair] = 0;
    return;
  }
  const double* src = part + (int64_t)pair * chunks * (kPairRows * kPairRows);
  // where the products of rows r and c of one block are carried
  auto own_at = [&](int r, int c) { return own + (int64_t)(r < kBlockRows ? bp.I : bp.J) * (kBlockRows * kBlockRows) + (r % kBlockRows) * kBlockRows + c % kBlockRows; };
  // entries r <= c of the partial matrices (what lies below the diagonal is not written)
  double sum[kLoads];
#pragma unroll
  for (int i = 0; i < kLoads; ++i) {
    const int idx = tid + kSweepThreads * i, r = idx >> 6, c = idx & 63;
    sum[i] = round > 0 && idx < kPairRows * kPairRows && r <= c && (r < kBlockRows) == (c < kBlockRows) ? *own_at(r, c) : 0.0;
  }
  for (int c = 0; c < chunks; c += 2) {     // two partial matrices in flight
    double v[2][kLoads];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const double* sc = src + (int64_t)(c + j) * (kPairRows * kPairRows);
#pragma unroll
      for (int i = 0; i < kLoads; ++i) {
        const int idx = tid + kSweepThreads * i, r = idx >> 6, col = idx & 63;
        const bool summed = round == 0 ? r <= col : r < kBlockRows && col >= kBlockRows;
        v[j][i] = (c + j < chunks && idx < kPairRows * kPairRows && summed) ? sc[idx] : 0.0;
      }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int i = 0; i < kLoads; ++i) sum[i] += v[j][i];
  }
#pragma unroll
  for (int i = 0; i < kLoads; ++i) {
    const int idx = tid + kSweepThreads * i, r = idx >> 6, c = idx & 63;
    if (idx < kPairRows * kPairRows && r == c) diag[r] = sum[i];
  }
  const double tol2 = tol * tol;
  __syncthreads();
  // A pair that is orthogonal already (every pair of the last sweep) keeps its rows: no rotation of the 63 rounds would be
  // applied.
  bool any = false;
#pragma unroll
  for (int i = 0; i < kLoads; ++i) {
    const int idx = tid + kSweepThreads * i, r = idx >> 6, c = idx & 63;
    if (idx < kPairRows * kPairRows && r < c) {
      any |= sum[i] * sum[i] > tol2 * diag[r] * diag[c];
      A0[packed_offset(r, c)] = sum[i];
    }
  }
  if (!__syncthreads_or(any)) {
    if (tid == 0) flags[pair] = 0;
    if (round == 0) {
#pragma unroll
      for (int i = 0; i < kLoads; ++i) {
        const int idx = tid + kSweepThreads * i, r = idx >> 6, c = idx & 63;
        if (idx < kPairRows * kPairRows && r <= c && (r < kBlockRows) == (c < kBlockRows)) *own_at(r, c) = sum[i];
      }
    }
    return;
  }
  // A round starts with a barrier: the copy of A it reads and its rotations are complete, and nobody reads any longer what
  // it writes.
  auto round_barrier = [] { asm volatile("bar.sync 1, %0;" ::"n"(kSweepThreads) : "memory"); };
  if (warp < kBlockWarps) {
    const int d0 = 1 + warp, d1 = 1 + kBlockWarps + warp;
    const int v0 = (lane + d0) & (kSlots - 1), v1 = (lane + d1) & (kSlots - 1);
    const BlockWrites w0 = block_writes(lane, v0), w1 = block_writes(lane, v1);
    const bool second = d1 < kSlots / 2 || lane < kSlots / 2;      // half of row 16 says it all
    for (int rr = 0; rr < kSweepRounds; ++rr) {
      const double* A = (rr & 1 ? A1 : A0) + d0 * kSlots + lane;
      double* An = rr & 1 ? A0 : A1;
      const double2* cur = cs[rr & 1];
      round_barrier();
      const double2 ru = cur[lane], rv0 = cur[v0];
      const BlockValues b0{A[0], A[kKindSize], A[2 * kKindSize], A[3 * kKindSize]};
      const double2 rv1 = cur[v1];
      const double* B = A + kBlockWarps * kSlots;
      const BlockValues b1{B[0], B[kKindSize], B[2 * kKindSize], B[3 * kKindSize]};
      block_write(w0, ru, rv0, b0, An);
      if (second) block_write(w1, ru, rv1, b1, An);
    }
    round_barrier();
  } else if (warp < kAngleWarp) {
    // lane: columns col and col + 4 of the warp's 8, slots 4 q .. 4 q + 3 with q = lane / 4
    const int q = lane / kLaneCols, col = (warp - kBlockWarps) * 2 * kLaneCols + lane % kLaneCols;
    double F[2][kLaneSlots], G[2][kLaneSlots];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int k = 0; k < kLaneSlots; ++k) {
        F[j][k] = q * kLaneSlots + k == col + kLaneCols * j ? 1.0 : 0.0;
        G[j][k] = kPairRows - 1 - (q * kLaneSlots + k) == col + kLaneCols * j ? 1.0 : 0.0;
      }
    for (int rr = 0; rr < kSweepRounds; ++rr) {
      const double2* cur = cs_rot[rr & 1] + q * (kLaneSlots + 1);
      round_barrier();
      double nf[2][kLaneSlots], ng[2][kLaneSlots];
#pragma unroll
      for (int k = 0; k < kLaneSlots; ++k) {
        const double2 r = cur[k];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          nf[j][k] = r.x * F[j][k] - r.y * G[j][k];
          ng[j][k] = r.y * F[j][k] + r.x * G[j][k];
        }
      }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const double below = __shfl_up_sync(0xffffffffu, nf[j][kLaneSlots - 1], kLaneCols);
        const double above = __shfl_down_sync(0xffffffffu, ng[j][0], kLaneCols);
        F[j][0] = q == 0 ? nf[j][0] : below;                              // position 0 stays
        F[j][1] = q == 0 ? ng[j][0] : nf[j][0];                           // position 63 goes on to 1
#pragma unroll
        for (int k = 2; k < kLaneSlots; ++k) F[j][k] = nf[j][k - 1];
#pragma unroll
        for (int k = 0; k + 1 < kLaneSlots; ++k) G[j][k] = ng[j][k + 1];
        G[j][kLaneSlots - 1] = q == kLaneGroups - 1 ? nf[j][kLaneSlots - 1] : above;    // position 31 goes on to 32
      }
    }
    round_barrier();
    if (total != 0) {                                                     // all rows are back at their own positions
      double* out = rot_out + (int64_t)pair * (kPairRows * kPairRows) + col;
#pragma unroll
      for (int k = 0; k < kLaneSlots; ++k) {
        const int slot = q * kLaneSlots + k;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          out[slot * kPairRows + kLaneCols * j] = F[j][k];
          out[(kPairRows - 1 - slot) * kPairRows + kLaneCols * j] = G[j][k];
        }
      }
    }
  } else {
    // Lane k: slot k, its two squared norms and the product of its rows, and its rotation in the next round.  The rows that
    // will be at positions k and 63 - k are now row f or g of slot s1 and of slot s2.
    const int s1 = lane <= 1 ? 0 : lane - 1, s2 = lane == 31 ? 31 : lane + 1;
    const bool g1 = lane == 1, g2 = lane != 31;
    const int x0 = packed_offset(s1, s2), x1 = packed_offset(s1, kPairRows - 1 - s2),
              x2 = packed_offset(kPairRows - 1 - s1, s2), x3 = packed_offset(kPairRows - 1 - s1, kPairRows - 1 - s2);
    const int left = packed_offset(next_position(lane), next_position(kPairRows - 1 - lane));    // where the slot's own product goes
    const int rot_at = lane + lane / kLaneSlots;
    int applied = 0;
    double f = diag[lane], g = diag[kPairRows - 1 - lane], o = A0[kKindSize + lane];
    double2 own_rot = jacobi_rotation(f, g, o, tol2, applied);
    cs[0][lane] = own_rot;
    cs_rot[0][rot_at] = own_rot;
    for (int rr = 0; rr < kSweepRounds; ++rr) {
      const double* A = rr & 1 ? A1 : A0;
      double* An = rr & 1 ? A0 : A1;
      const double2* cur = cs[rr & 1];
      round_barrier();
      const double2 r1 = cur[s1], r2 = cur[s2];
      const double y0 = A[x0], y1 = A[x1], y2 = A[x2], y3 = A[x3];
      // this round's rotation of the slot's own two rows
      const double c = own_rot.x, sn = own_rot.y;
      const double fn = c * (c * f - sn * o) - sn * (c * o - sn * g), gn = sn * (sn * f + c * o) + c * (sn * o + c * g);
      An[left] = c * (sn * f + c * o) - sn * (sn * o + c * g);
      // the rows move on
      const double f_up = __shfl_up_sync(0xffffffffu, fn, 1), g_down = __shfl_down_sync(0xffffffffu, gn, 1), g_first = __shfl_sync(0xffffffffu, gn, 0);
      f = lane == 0 ? fn : (g1 ? g_first : f_up);
      g = g2 ? g_down : fn;
      const double p1 = g1 ? r1.y : r1.x, q1 = g1 ? r1.x : -r1.y;
      const double p2 = g2 ? r2.y : r2.x, q2 = g2 ? r2.x : -r2.y;
      o = p2 * (p1 * y0 + q1 * y2) + q2 * (p1 * y1 + q1 * y3);
      if (rr + 1 < kSweepRounds) {
        own_rot = jacobi_rotation(f, g, o, tol2, applied);
        cs[(rr + 1) & 1][lane] = own_rot;
        cs_rot[(rr + 1) & 1][rot_at] = own_rot;
      }
    }
    for (int k = 16; k > 0; k >>= 1) applied += __shfl_xor_sync(0xffffffffu, applied, k);
    if (lane == 0) {
      total = applied;
      flags[pair] = applied;
      if (applied) atomicAdd(rotations, applied);
    }
    diag[lane] = f;
    diag[kPairRows - 1 - lane] = g;
    round_barrier();
  }
  // all rows are back at their own positions: the products within the blocks, for the rounds to come
  const double* A = kSweepRounds & 1 ? A1 : A0;
  for (int idx = tid; idx < kPairRows * kBlockRows; idx += kSweepThreads) {
    const int r = idx >> 5, c = (idx & 31) + (r & ~(kBlockRows - 1));
    if (r <= c) *own_at(r, c) = r == c ? diag[r] : A[packed_offset(r, c)];
  }
}

// rows(pair)[:, cols] <- Rot rows(pair)[:, cols]  for X (blockIdx.z = 0) and, if present, Vt (blockIdx.z = 1)
// A CTA owns 128 columns and takes them in two halves of 64: while the first half is multiplied the second
// is already on its way from global memory into registers, and with one half in shared memory three CTAs
// fit on an SM.  Warp (wy, wx) forms rows 32 wy .. + 32, columns 16 wx .. + 16 of a half.
__global__ void __launch_bounds__(256) jb_apply_kernel(double* __restrict__ X, double* __restrict__ Vt, int b, int nblk, int round,
                                                       const double* rot, const int* flags,
                                                       const SlotList slots, int matrices) {
  grid_dependency_wait();
  grid_launch_dependents();
  extern __shared__ __align__(16) double jb_smem[];
  double(*Rs)[kRotLd] = reinterpret_cast<double(*)[kRotLd]>(jb_smem);
  double(*Xs)[kHalfLd] = reinterpret_cast<double(*)[kHalfLd]>(jb_smem + kPairRows * kRotLd);
  const int pair = blockIdx.x;
  const int which = blockIdx.z % matrices;                                  // 0: X, 1: Vt
  {
    const int64_t shift = (int64_t)slots.id[blockIdx.z / matrices] * slots.bytes;
    X = slot_ptr(X, shift);
    Vt = Vt ? slot_ptr(Vt, shift) : Vt;
    rot = slot_ptr(rot, shift);
    flags = slot_ptr(flags, shift);
  }
  if (flags[pair] == 0) return;
  const BlockPair bp = block_pair(pair, round, nblk);
  double* M = which ? Vt : X;
  const int c0 = blockIdx.y * kApplyCols;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int wy = warp >> 2, wx = warp & 3;
  const bool vec = (b & 1) == 0;
  const double* rsrc = rot + (int64_t)pair * (kPairRows * kPairRows);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int id = tid + 256 * i;
    const int l = id >> 5, m2 = (id & 31) * 2;
    *reinterpret_cast<double2*>(&Rs[l][m2]) = *reinterpret_cast<const double2*>(rsrc + l * kPairRows + m2);
  }
  double2 stage[8];
  auto fetch = [&](int half) {             // 64 rows x 64 columns: row id / 32, columns 2 (id % 32) of the half
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int id = tid + 256 * i;
      const int l = id >> 5, cl = (id & 31) * 2;
      const int row = bp.row(l), col = c0 + half * kApplyHalf + cl;
      double2 v = make_double2(0.0, 0.0);
      if (row < b) {
        const double* src = M + (int64_t)row * b + col;
        if (vec && col + 1 < b) {
          v = *reinterpret_cast<const double2*>(src);
        } else {
          if (col < b) v.x = src[0];
          if (col + 1 < b) v.y = src[1];
        }
      }
      stage[i] = v;
    }
  };
  auto stash = [&]() {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int id = tid + 256 * i;
      *reinterpret_cast<double2*>(&Xs[id >> 5][(id & 31) * 2]) = stage[i];
    }
  };
  fetch(0);
  stash();
  __syncthreads();
  const bool second = c0 + kApplyHalf < b;        // the second half holds columns of the matrix
  for (int half = 0; half < 2; ++half) {
    if (half == 0 && second) fetch(1);
    double acc[4][2][2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;
#pragma unroll 4
    for (int ks = 0; ks < kPairRows / 4; ++ks) {
      double a[4], bb[2];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = Rs[wy * 32 + i * 8 + g][ks * 4 + t];
#pragma unroll
      for (int j = 0; j < 2; ++j) bb[j] = Xs[ks * 4 + t][wx * 16 + j * 8 + g];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) dmma_m8n8k4(acc[i][j], a[i], bb[j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int row = bp.row(wy * 32 + i * 8 + g);
      if (row >= b) continue;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int col = c0 + half * kApplyHalf + wx * 16 + j * 8 + 2 * t;
        double* dst = M + (int64_t)row * b + col;
        if (vec && col + 1 < b) {
          *reinterpret_cast<double2*>(dst) = make_double2(acc[i][j][0], acc[i][j][1]);
        } else {
          if (col < b) dst[0] = acc[i][j][0];
          if (col + 1 < b) dst[1] = acc[i][j][1];
        }
      }
    }
    if (half == 1 || !second) break;
    __syncthreads();                               // every warp has read the first half
    stash();
    __syncthreads();
  }
}

struct JacobiGeometry {
  int nblk, pairs, chunks, col_tiles;
};
JacobiGeometry jacobi_geometry(int b) {
  JacobiGeometry g;
  g.nblk = std::max(2, (int)ceil_div(b, kBlockRows));
  g.nblk += g.nblk & 1;
  g.pairs = g.nblk / 2;
  g.chunks = (int)ceil_div(b, gram_chunk(b));
  g.col_tiles = (int)ceil_div(b, kApplyCols);
  return g;
}

size_t own_bytes(const JacobiGeometry& g) { return align_up((size_t)g.nblk * kBlockRows * kBlockRows * sizeof(double), 256); }
constexpr size_t kApplySmem = (size_t)(kPairRows * kRotLd + kPairRows * kHalfLd) * sizeof(double);

}  // namespace

size_t jacobi_scratch_bytes(int b) {
  const JacobiGeometry g = jacobi_geometry(b);
  const size_t tile = (size_t)kPairRows * kPairRows * sizeof(double);
  return align_up((size_t)g.pairs * g.chunks * tile, 256) + align_up((size_t)g.pairs * tile, 256) +
         align_up((size_t)g.pairs * sizeof(int), 256) + own_bytes(g);
}

galore_status_t jacobi_eigh(double* X, double* Vt, int b, void* scratch, int* counter, double tol, int max_sweeps,
                            int* sweeps_out, cudaStream_t st, const SlotList* slot_list) {
  const SlotList all = slot_list ? *slot_list : single_slot();
  for (int i = 0; i < all.n; ++i)
    if (sweeps_out) sweeps_out[i] = 0;
  if (b < 2) return GALORE_OK;
  const JacobiGeometry g = jacobi_geometry(b);
  const size_t tile = (size_t)kPairRows * kPairRows * sizeof(double);
  char* p = (char*)scratch;
  double* part = (double*)p;
  p += align_up((size_t)g.pairs * g.chunks * tile, 256);
  double* rot = (double*)p;
  p += align_up((size_t)g.pairs * tile, 256);
  int* flags = (int*)p;
  p += align_up((size_t)g.pairs * sizeof(int), 256);
  double* own = (double*)p;

  // per device, so set on every call rather than once per process
  GALORE_CUDA_TRY(cudaFuncSetAttribute(jb_apply_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kApplySmem));

  // Slots leave the list as they converge (a sweep without a rotation), so every problem sees exactly
  // the sweeps it would see on its own.
  SlotList live = all;
  int where[kMaxSlots];                       // position of live.id[i] in the caller's list
  for (int i = 0; i < all.n; ++i) where[i] = i;
  const int matrices = Vt ? 2 : 1;
  int sweeps = 0;
  while (sweeps < max_sweeps && live.n > 0) {
    for (int i = 0; i < live.n; ++i)
      GALORE_CUDA_TRY(cudaMemsetAsync(slot_ptr(counter, (int64_t)live.id[i] * live.bytes), 0, sizeof(int), st));
    for (int round = 0; round < g.nblk - 1; ++round) {
      // Three dependent launches of a few microseconds each: every one is set up while the one before it runs (with the
      // other products of the refresh launched so, and 64 columns a CTA above: 512 x 1376 fp32 at rank 128 4.60 -> 3.96 ms,
      // eight 4096 x 4096 at rank 1024 127.8 -> 125.1 ms).
      GALORE_TRY(launch_kernel(jb_gram_kernel, dim3(g.pairs, g.chunks, live.n), 128, 0, 1, true, st, (const double*)X, b, g.nblk, round,
                               g.chunks, part, live));
      GALORE_TRY(launch_kernel(jb_sweep_kernel, dim3(g.pairs, live.n), kSweepThreads, 0, 1, true, st, (const double*)part,
                               g.chunks, b, g.nblk, round, tol, own, rot, flags, counter, live));
      GALORE_TRY(launch_kernel(jb_apply_kernel, dim3(g.pairs, g.col_tiles, matrices * live.n), 256, kApplySmem, 1, true, st, X, Vt, b,
                               g.nblk, round, (const double*)rot, (const int*)flags, live, matrices));
    }
    ++sweeps;
    int rot_count[kMaxSlots] = {};
    for (int i = 0; i < live.n; ++i)
      GALORE_CUDA_TRY(cudaMemcpyAsync(&rot_count[i], slot_ptr(counter, (int64_t)live.id[i] * live.bytes), sizeof(int),
                                      cudaMemcpyDeviceToHost, st));
    GALORE_CUDA_TRY(cudaStreamSynchronize(st));
    int kept = 0;
    for (int i = 0; i < live.n; ++i) {
      if (sweeps_out) sweeps_out[where[i]] = sweeps;
      if (rot_count[i] != 0) {
        live.id[kept] = live.id[i];
        where[kept] = where[i];
        ++kept;
      }
    }
    live.n = kept;
  }
  return GALORE_OK;
}

}  // namespace galore
