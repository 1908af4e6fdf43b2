// The weight update that closes Algorithm 1 as one tensor-core kernel:
//   W <- keep W - scale P N (left) resp. W <- keep W - scale N Q^T (right).
// The product never exists in memory.  P and N are bf16, or fp32 values carried as three bf16 planes
// (hi + mid + lo holds all 24 significand bits); W is fp32 or bf16 with any leading dimension.
#pragma once

#include "common.cuh"

namespace galore {

constexpr int kApplyGroup = 32;      // problems one launch can carry

// `planes` bf16 matrices of `rows` rows below each other, rows of `ld` elements on 16-byte boundaries
struct PlaneMatrix {
  const void* base;
  int64_t rows, ld;
  int planes;          // 1 or 3
};
struct ApplyItem {
  int m, n, r;
  bool left;
  PlaneMatrix P;       // m x r (left) or n x r (right)
  PlaneMatrix N;       // r x n (left) or m x r (right)
  void* W;
  int64_t ldw;
  float scale, keep;
  int32_t* status;
};
struct ApplyGroup {
  ApplyItem item[kApplyGroup];
  int count = 0;
};
// Tiles of a group's updates: 256 x 256 per CTA pair, 128 x 128 per CTA; the most k-blocks of one, all products of planes
struct ApplyTiles {
  int64_t pairs = 0, singles = 0, blocks = 0;
  bool aligned = true;       // W's rows lie on 16-byte boundaries
  bool direct = false;       // single tiles would read and write them from registers
  void add(int m, int n, int r, int p_planes, int n_planes, bool w_aligned);
};
// microseconds of a group's update with operands of several planes
double apply_group_us(const ApplyTiles& t, int32_t w_dtype);
galore_status_t apply_group_add(ApplyGroup& g, const ApplyItem& item);
// early: the kernel before this one on the stream lets its successor start (griddepcontrol.launch_dependents) and does not
// write W.  All items share the type of W.
galore_status_t launch_apply_group(const ApplyGroup& g, int32_t w_dtype, bool early, cudaStream_t st);

}  // namespace galore
