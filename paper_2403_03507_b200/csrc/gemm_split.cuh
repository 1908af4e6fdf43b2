// fp32-accurate and alignment-free products on the tensor cores: interface.
//
// C(i, j) = sum_k A(i, k) * B(k, j) for fp32 or bf16 operands of any leading dimension and either
// storage order.  An fp32 operand is carried as three bf16 numbers (8 + 8 + 8 significand bits: the
// value itself, nothing is lost), a bf16 operand as itself, so the products keep fp32's precision.  That
// holds for 2^-110 <= |x| <= 3.39e38, the largest bf16: below, the last number loses bits; a larger value
// enters as an infinity, and the step reports it as non-finite.
#pragma once

#include "common.cuh"

namespace galore {

constexpr int kSplitGroup = 32;      // problems one launch can carry

struct SplitOperand {
  const void* base;
  int64_t ld;          // elements between consecutive rows of the storage
  int mn;              // 1: M (resp. N) is the contiguous direction, 0: K is
  int aligned;         // base and rows on 16-byte boundaries: vector loads
};
struct SplitProblem {
  int M, N, K;
  SplitOperand a, b;
  int tiles_m, tiles_n, splits;
  int kblocks, kblocks_per_split;
  int m_fast;          // consecutive units walk M first (they share a panel of B), else N first
  // C (fp32) of K slice s at C + s * split_stride
  float* C;
  int64_t ldc, split_stride;
  int32_t* status;
};
template <int CAP>
struct SplitArgs {
  static constexpr int kCapacity = CAP;
  SplitProblem p[CAP];
  int unit_end[CAP];
  int count;
};
using SplitGroup = SplitArgs<kSplitGroup>;

// operand X(i, k) = base[i * s_mn + k * s_k]; one of the strides is 1
SplitOperand split_operand(const void* base, int32_t dtype, int64_t s_mn, int64_t s_k);
// K slices that balance filling the machine against the traffic of the partial results
int split_choose_slices(int64_t M, int64_t N, int64_t K);
double split_store_us(int64_t M, int64_t N, int64_t K, int slices);      // what one such product takes in 128 x 128 tiles
// Of a group of products, unsliced: its tiles of 128 x 128 and of 256 x 256 and the most blocks of 64 of K; may_pair: fp32 operands,
// all on 16-byte boundaries
struct SplitTiles {
  int64_t singles = 0, pairs = 0, blocks = 0;
  bool may_pair = true;
};
double split_group_us(const SplitTiles& t);
int split_effective_slices(int64_t K, int slices);
galore_status_t split_group_add_store(SplitGroup& g, int M, int N, int K, const SplitOperand& a, const SplitOperand& b, int splits,
                                      float* C, int64_t ldc, int64_t split_stride, int32_t* status);
// All problems of a group share the operand types.  pairs: fp32 operands may take the tiles of CTA pairs, where the group's
// size makes them the faster ones (their sums round differently); false: a problem's bits do not depend on its group.
galore_status_t launch_split_store(const SplitGroup& g, int32_t a_dtype, int32_t b_dtype, bool pairs, bool early, cudaStream_t st);
// the same for fp32 operands on 16-byte boundaries, by CTA pairs (gemm_split_pair.cu); taken false: this build cannot, nothing is launched
galore_status_t launch_split_pair(const SplitGroup& g, bool early, bool* taken, cudaStream_t st);

}  // namespace galore
