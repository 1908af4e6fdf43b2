// tcgen05 / TMEM / TMA projection kernels (bf16 operands, fp32 accumulation): interface.
#pragma once

#include <cuda.h>

#include <utility>

#include "common.cuh"
#include "launch_order.h"
#include "q8_code.cuh"

namespace galore {

// What the projection needs to run Adam on its output (Algorithm 1's update block and Eq. 15 in the
// epilogue): the layer's moments and where the normalised update goes.
struct TcAdamArgs {
  int32_t state_fmt;          // galore_state_fmt_t
  float *M, *V;               // fp32 moments (rows of ld_s floats), or
  uint8_t *Mc, *Vc;           // 8-bit codes (rows of ld_s bytes) with
  float *Mam, *Vam;           // one absmax per tile of q_block / 64 rows x 64 columns
  int64_t ld_s;
  int q_block;
  void* Nout;                 // bf16, leading dimension ld_n
  int64_t ld_n;
  AdamParams ap;
};

// Per-layer launch state of the tensor-core path: the tensor map of the projector, which the library owns.  The map
// of G is encoded per call.
struct TensorPlan {
  bool ready = false;
  int ctas = 1;               // 1: 128-row tiles per CTA; 2: 256-row tiles per CTA pair (cta_group::2)
  CUtensorMap map_p_proj;     // projector as an operand of the projection
};

// bf16 G and P, rank a multiple of 8 (16-byte rows for TMA).
bool tensor_path_eligible(const galore_config_t& cfg);
int tensor_proj_splits(const galore_config_t& cfg, bool left);       // K slices that fill the machine
int tensor_chain_blocks(int64_t K, int splits);                       // 64 of K that one accumulator of such a slice sums
int tensor_step_splits(const galore_config_t& cfg, bool left);       // those a layer's own step takes (drained accumulators)
int tensor_ctas(const galore_config_t& cfg);
galore_status_t tensor_plan_init(TensorPlan* plan, const galore_config_t& cfg, bool left, void* P);
// G and W usable by this path: 16-byte aligned bases and rows.
bool tensor_operands_aligned(const galore_config_t& cfg, const void* W, int64_t ldw, const void* G, int64_t ldg);
// ---- groups: up to tensor_group_capacity() layers per launch ------------------------------------
struct TensorGroup;   // opaque, host memory
TensorGroup* tensor_group_new();
void tensor_group_free(TensorGroup* t);
void tensor_group_reset(TensorGroup* t);
int tensor_group_capacity();
// the layer's projection with its R partials going to `part` (leading dimension ld_part, `splits` K slices)
galore_status_t tensor_group_add_project(TensorGroup* t, const TensorPlan* plan, const galore_config_t& cfg, bool left,
                                         const void* G, int64_t ldg, float* part, int64_t ld_part, int splits,
                                         int32_t* status);
// the layer's projection with Adam in its epilogue; launch with tensor_group_launch_project_adam
// (all layers of the group have the same state format)
galore_status_t tensor_group_add_project_adam(TensorGroup* t, const TensorPlan* plan, const galore_config_t& cfg, bool left,
                                              const void* G, int64_t ldg, const TcAdamArgs& adam, int32_t* status);
galore_status_t tensor_group_launch_project_adam(TensorGroup* t, int32_t state_fmt, bool early, cudaStream_t st);
// a plain GEMM: C (M x N fp32, ldc) = op(A) op(B), bf16 operands; *_mn = 1 when the operand is stored
// with M (resp. N) contiguous, 0 when K is contiguous.  Launch with tensor_group_launch_project.
galore_status_t tensor_group_add_gemm(TensorGroup* t, const void* A, int64_t lda, int a_mn, const void* B, int64_t ldb,
                                      int b_mn, int M, int N, int K, float* C, int64_t ldc, int32_t* status);
galore_status_t tensor_group_launch_project(TensorGroup* t, bool early, cudaStream_t st);
// The problem added last (one K slice) leaves the sums of R^2 as well: over stretches of 128 columns, rows x tiles, and over
// stretches of 64 rows, one row of sums for each
void tensor_group_want_squares(TensorGroup* t, float* row_sq, float* col_sq, int tiles);
// one layer's projection, its accumulators added to fp32 sums after every `blocks` times 64 of K
galore_status_t tensor_group_launch_project_drained(TensorGroup* t, int blocks, bool early, cudaStream_t st);

struct CudaOrder {
  using Status = galore_status_t;
  using Stream = cudaStream_t;
  using Event = cudaEvent_t;
  static Status capturing(Stream st, bool* on);
  static Status wait(Stream st, Event e);
  static Status create(Event* e);
  static Status record(Event e, Stream st);
};
LaunchOrder<CudaOrder>& launch_order();
// Runs `launch` (which queues kernels that allocate tensor memory on st) after every such kernel queued before it,
// whatever their streams; see launch_order.h.  The entry points call it, once around all their launches.
template <class F>
galore_status_t tensor_launch_in_order(cudaStream_t st, F&& launch) {
  int dev = 0;
  GALORE_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= LaunchOrder<CudaOrder>::kDevices) return GALORE_ERR_INVALID_ARG;
  return launch_order().run(dev, st, std::forward<F>(launch));
}
int tensor_sm_count();
// a matrix of rows x cols elements (cols contiguous) with boxes of box_rows x box_cols, 128-byte swizzle or none
galore_status_t tensor_encode(CUtensorMap* map, const void* base, int32_t dtype, int64_t rows, int64_t cols, int64_t ld,
                              int box_rows, int box_cols, bool swizzle = true);

}  // namespace galore
