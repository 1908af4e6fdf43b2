// Products with fp32 FMA: the projection of layers with fp32 W, G and Adam moments.  Interface.
//
// C(i, j) = sum_k A(i, k) * B(k, j),  A(i, k) = A[i * sAi + k * sAk],  B(k, j) = B[k * sBk + j * sBj], any leading
// dimension and either storage order.  Every element of a K slice is one chain of fmaf in the order of k, whatever the tile.
#pragma once

#include "common.cuh"

namespace galore {

constexpr int kFmaGroup = 32;        // problems one launch can carry

struct FmaProblem {
  int M, N, K;
  const void *A, *B;
  int64_t sAi, sAk, sBk, sBj;
  int kchunk, splits;                // K slices of kchunk elements
  float* C;                          // slice s at C + s * split_stride
  int64_t ldc, split_stride;
};
template <int CAP>
struct FmaArgs {
  FmaProblem p[CAP];
  int unit_end[CAP];                 // running totals of CTAs (tiles x K slices)
  int count;
};
using FmaGroup = FmaArgs<kFmaGroup>;

// Slices of K for an M x N result: enough CTAs to fill the machine when the result is small.
int fma_choose_slices(int64_t M, int64_t N, int64_t K);
// slices that a request for `slices` gives (they are multiples of 16 elements long)
int fma_effective_slices(int64_t K, int slices);
// microseconds of a group of products, unsliced, with `tiles` of 128 x 128 and K up to k
double fma_group_us(int64_t tiles, int64_t k);
galore_status_t fma_group_add(FmaGroup& g, const FmaProblem& problem, int slices);
// All problems share the operand types.  early: see launch.cuh.
galore_status_t launch_fma_group(const FmaGroup& g, int32_t a_dtype, int32_t b_dtype, bool early, cudaStream_t st);

}  // namespace galore
