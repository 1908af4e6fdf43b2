// What the kernels of split operands share: bf16 tiles in shared memory, work units, register hand-over.
#pragma once

#include "gemm_split.cuh"
#include "tc_ptx.cuh"

namespace galore {

constexpr int kSplitK = 64;                              // K of one tile in shared memory
constexpr int kTileBytes = 128 * kSplitK * 2;            // one bf16 tile of either operand
constexpr int kStageLd = 33;                             // epilogue transposition: 32 x 32 floats per warp

// K-major and MN-major tiles as in the bf16 kernels: 128-byte swizzle, 8-row groups 1024 bytes apart; MN-major
// operands continue kSplitK * 128 bytes further on after 64 elements of M / N.
__device__ __forceinline__ uint64_t split_desc(uint32_t addr, bool mn) {
  const uint64_t lbo = mn ? (uint64_t)((kSplitK * 128) >> 4) : 1ull;
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | (lbo << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// fp32 accumulate, bf16 x bf16; tiles of m x n
__device__ __forceinline__ uint32_t split_idesc(int a_mn, int b_mn, int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(m >> 4) << 24);
}

struct SplitUnit {
  int pi, m0, n0, slice, kb, kb_end;
};
template <int TILE, class Args>
__device__ __forceinline__ SplitUnit split_unit(const Args& g, int u, GroupCursor& cursor) {
  SplitUnit w;
  u = cursor.seek<Args::kCapacity>(g, u);
  w.pi = cursor.pi;
  const SplitProblem& p = g.p[w.pi];
  int tm, tn;
  if (p.m_fast) {
    tm = u % p.tiles_m;
    w.slice = (u / p.tiles_m) % p.splits;
    tn = u / (p.tiles_m * p.splits);
  } else {
    tn = u % p.tiles_n;
    w.slice = (u / p.tiles_n) % p.splits;
    tm = u / (p.tiles_n * p.splits);
  }
  w.m0 = tm * TILE;
  w.n0 = tn * TILE;
  w.kb = w.slice * p.kblocks_per_split;
  w.kb_end = min(p.kblocks, w.kb + p.kblocks_per_split);
  return w;
}

__device__ __forceinline__ uint32_t pack_bf16(float x0, float x1) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
  return *reinterpret_cast<const uint32_t*>(&h);
}

template <int R>
__device__ __forceinline__ void regs_up() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(R)); }
template <int R>
__device__ __forceinline__ void regs_down() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(R)); }

}  // namespace galore
