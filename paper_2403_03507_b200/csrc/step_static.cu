// galore_step_static: one fp32 GaLore-Adam step whose scratch memory lives inside the library.
//
// The regular entry points take a caller-allocated workspace for the two intermediates of a step
// (the split-K partial sums of the projected gradient R and the normalised update N).  Some
// callers have no way of providing one: a host framework may own every byte of device memory
// through its own pool and forbid plug-ins from calling cudaMalloc; an allocation may be
// unacceptable at the call site because cudaMalloc/cudaFree synchronise the whole device; or the
// code runs on a thread that is not allowed to touch the allocator at all.  For those callers the
// intermediates are placed in one fixed array that is part of the loaded module.
//
// The array is shared by every call in the process (per device) and keeps whatever the previous
// call left in it.  Nothing in it needs to start at zero except the word that collects this call's
// status bits, which each call clears itself (a second word accumulates them across calls until
// galore_static_status() reads it); every other byte that is read has been written earlier in the
// same call.  Two
// calls whose GPU work overlaps (different streams, or different host threads) would both write
// the array and race: callers serialise them.
#include <algorithm>
#include <mutex>

#include "adam.cuh"
#include "common.cuh"
#include "gemm_apply.cuh"
#include "gemm_fma.cuh"
#include "gemm_tc.cuh"

namespace galore {

constexpr size_t kStaticScratchBytes = GALORE_STATIC_SCRATCH_BYTES;

// Device storage.  In host code this name is only a handle for the symbol, not an address a
// kernel can use: the device address is looked up once per device with cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

static std::mutex g_static_mutex;
static void* g_static_ptr[64] = {};

// Device address of the array on the current device (looked up on the first call per device).
static galore_status_t static_scratch(void** out) {
  int dev = 0;
  GALORE_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return GALORE_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lock(g_static_mutex);
  if (!g_static_ptr[dev]) {
    void* p = nullptr;
    GALORE_CUDA_TRY(cudaGetSymbolAddress(&p, g_static_scratch));
    g_static_ptr[dev] = p;
  }
  *out = g_static_ptr[dev];
  return GALORE_OK;
}

// the bits of this call (word 0) are added to the word that only galore_static_status() clears (word 1)
__global__ void fold_status_kernel(int32_t* words) {
  if (words[0]) atomicOr(words + 1, words[0]);
}

// the stream, if one is given, must live on the device whose array is about to be used
static galore_status_t check_stream_device(cudaStream_t st) {
  if (!st || st == cudaStreamLegacy || st == cudaStreamPerThread) return GALORE_OK;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  GALORE_CUDA_TRY(cudaStreamIsCapturing(st, &capture));
  if (capture != cudaStreamCaptureStatusNone) return GALORE_OK;      // a captured stream does not tell its device
  int cur = 0, dev = 0;
  GALORE_CUDA_TRY(cudaGetDevice(&cur));
  GALORE_CUDA_TRY(cudaStreamGetDevice(st, &dev));
  return dev == cur ? GALORE_OK : GALORE_ERR_INVALID_ARG;
}

}  // namespace galore

using namespace galore;

extern "C" galore_status_t galore_static_status(int32_t* flags, void* stream) {
  if (!flags) return GALORE_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  GALORE_TRY(check_stream_device(st));
  void* base = nullptr;
  GALORE_TRY(static_scratch(&base));
  int32_t f = 0;
  GALORE_CUDA_TRY(cudaMemcpyAsync(&f, (int32_t*)base + 1, sizeof(f), cudaMemcpyDeviceToHost, st));
  GALORE_CUDA_TRY(cudaMemsetAsync((int32_t*)base + 1, 0, sizeof(f), st));
  GALORE_CUDA_TRY(cudaStreamSynchronize(st));
  *flags = f;
  return GALORE_OK;
}

extern "C" galore_status_t galore_step_static(int64_t m, int64_t n, int32_t rank, int32_t side, float alpha,
                                               double beta1, double beta2, double eps, int64_t completed_steps,
                                               const float* P, float* M, float* V, float* W, int64_t ldw,
                                               const float* G, int64_t ldg, float lr, int32_t* device_flags,
                                               void* stream) {
  if (!P || !M || !V || !W || !G) return GALORE_ERR_INVALID_ARG;
  if (m <= 0 || n <= 0 || m > 0x7fffffff || n > 0x7fffffff) return GALORE_ERR_SHAPE;
  if (rank < 1 || rank > (m < n ? m : n)) return GALORE_ERR_SHAPE;
  if (ldw < n || ldg < n || completed_steps < 0) return GALORE_ERR_INVALID_ARG;
  if (side < GALORE_SIDE_AUTO || side > GALORE_SIDE_RIGHT) return GALORE_ERR_INVALID_ARG;
  if (!(beta1 >= 0.0 && beta1 < 1.0) || !(beta2 >= 0.0 && beta2 < 1.0) || !(eps >= 0.0)) return GALORE_ERR_INVALID_ARG;
  const bool left = side == GALORE_SIDE_AUTO ? (m <= n) : (side == GALORE_SIDE_LEFT);
  const int r = rank;
  const int64_t wide = left ? n : m;           // the side of G that the state spans
  if (256 + 2 * align_up((size_t)r * wide * 4, 256) > kStaticScratchBytes) return GALORE_ERR_BUFFER_TOO_SMALL;

  cudaStream_t st = (cudaStream_t)stream;
  GALORE_TRY(check_stream_device(st));
  void* base = nullptr;
  GALORE_TRY(static_scratch(&base));
  int32_t* status = (int32_t*)base;
  GALORE_CUDA_TRY(cudaMemsetAsync(status, 0, sizeof(int32_t), st));   // this call's bits: the one part that must start at zero

  // The step is independent along the wide side: where the array does not hold the intermediates of the whole matrix it
  // is done in strips.  Layout inside the array: [status words 256 B][R partials][planes of N][planes of P, whole or a
  // range of rows].  The K slices are those that the regular path gives the whole matrix, so that the moments agree bit for
  // bit; fewer where even the narrowest strip would not hold them.
  const AdamParams ap = make_adam_params(beta1, beta2, eps, (double)(completed_steps + 1));
  const float scale = lr * alpha;
  const int64_t d = left ? m : n, ldp = ((int64_t)r + 7) / 8 * 8;
  const size_t room = kStaticScratchBytes - 256, plane_row = 6 * (size_t)ldp;
  const size_t p_least = std::min<size_t>((size_t)d, 256) * plane_row + 256;
  auto r_bytes = [&](int64_t rows, int64_t cols, int splits) { return align_up((size_t)splits * rows * ((cols + 7) / 8 * 8) * 4, 256); };
  auto n_bytes = [&](int64_t rows, int64_t cols) { return align_up((size_t)rows * ((cols + 15) / 16 * 16) * 6, 256); };
  auto rows_of = [&](int64_t w) { return left ? (int64_t)r : w; };
  auto cols_of = [&](int64_t w) { return left ? w : (int64_t)r; };
  auto need = [&](int64_t w, int splits) { return r_bytes(rows_of(w), cols_of(w), splits) + n_bytes(rows_of(w), cols_of(w)) + p_least; };
  auto strip_of = [&](int splits) {
    int64_t strip = wide;
    for (int64_t parts = 2; strip > 256 && need(strip, splits) > room; ++parts) strip = align_up(ceil_div(wide, parts), 256);
    return strip;
  };
  int splits = fma_choose_slices(rows_of(wide), cols_of(wide), d);
  while (splits > 1 && need(strip_of(splits), splits) > room) splits = fma_effective_slices(d, splits - 1);
  const int64_t strip = strip_of(splits);
  if (need(strip, splits) > room) return GALORE_ERR_BUFFER_TOO_SMALL;
  float* const Rpart = (float*)((char*)base + 256);
  __nv_bfloat16* const Nbuf = (__nv_bfloat16*)((char*)Rpart + r_bytes(rows_of(strip), cols_of(strip), splits));
  __nv_bfloat16* const planes = (__nv_bfloat16*)((char*)Nbuf + n_bytes(rows_of(strip), cols_of(strip)));
  const size_t p_room = (size_t)((char*)base + kStaticScratchBytes - (char*)planes);
  // rows of P whose planes fit; a range of them updates that range of W's rows (left) or columns (right)
  int64_t p_rows = (int64_t)std::min<size_t>((size_t)d, p_room / plane_row);
  if (p_rows < d) p_rows = p_rows / 256 * 256;

  const galore_status_t queued = tensor_launch_in_order(st, [&]() -> galore_status_t {
    for (int64_t w0 = 0; w0 < wide; w0 += strip) {
      const int64_t w = std::min(strip, wide - w0);
      const int64_t srows = rows_of(w), scols = cols_of(w), scols_all = cols_of(wide), ld = (scols + 7) / 8 * 8, ldn = (scols + 15) / 16 * 16;
      const float* Gs = left ? G + w0 : G + w0 * ldg;
      float* Ws = left ? W + w0 : W + w0 * ldw;
      const int64_t state_at = left ? w0 : w0 * scols_all;
      FmaProblem proj = left ? FmaProblem{r, (int)w, (int)m, P, Gs, 1, r, ldg, 1} : FmaProblem{(int)w, r, (int)n, Gs, P, ldg, 1, r, 1};
      proj.C = Rpart; proj.ldc = ld; proj.split_stride = srows * ld;
      FmaGroup g;
      g.count = 0;
      GALORE_TRY(fma_group_add(g, proj, splits));
      GALORE_TRY(launch_fma_group(g, GALORE_F32, GALORE_F32, false, st));

      AdamItem item = {};
      item.Rpart = Rpart; item.splits = g.p[0].splits; item.split_stride = srows * ld;
      item.rows = (int)srows; item.cols = (int)scols;
      item.r_ld = ld; item.n_ld = ldn;
      item.s_ld = scols_all;                     // the caller's arrays are packed
      item.M = M + state_at; item.V = V + state_at;
      item.Nout = Nbuf; item.n_plane = srows * ldn;
      item.p = ap; item.status = status;
      GALORE_TRY(launch_adam(item, GALORE_STATE_F32, 2048, 3, false, st));

      for (int64_t p0 = 0; p0 < d; p0 += p_rows) {
        const int64_t rows = std::min(p_rows, d - p0);
        GALORE_TRY(launch_plane_split(PlaneSplit{P + p0 * r, planes, GALORE_F32, (int)rows, r, (int)ldp, 3}, st));
        ApplyItem a = {};
        a.m = (int)(left ? rows : w); a.n = (int)(left ? w : rows); a.r = r;
        a.left = left;
        a.P = PlaneMatrix{planes, rows, ldp, 3};
        a.N = PlaneMatrix{Nbuf, srows, ldn, 3};
        a.W = left ? Ws + p0 * ldw : Ws + p0;
        a.ldw = ldw;
        a.scale = scale; a.keep = 1.0f;
        a.status = status;
        ApplyGroup back;
        GALORE_TRY(apply_group_add(back, a));
        GALORE_TRY(launch_apply_group(back, GALORE_F32, false, st));
      }
    }
    return GALORE_OK;
  });
  if (queued < 0) return queued;

  fold_status_kernel<<<1, 1, 0, st>>>(status);
  GALORE_LAUNCH_CHECK();

  if (device_flags) {   // optional: wait for the step and report what the kernels latched
    int32_t f = 0;
    GALORE_CUDA_TRY(cudaMemcpyAsync(&f, status, sizeof(f), cudaMemcpyDeviceToHost, st));
    GALORE_CUDA_TRY(cudaStreamSynchronize(st));
    *device_flags = f;
  }
  return GALORE_OK;
}
