// fp32 matrices as three bf16 planes: hi + mid + lo holds an fp32 value exactly (8 + 8 + 8 significand
// bits; for 2^-110 <= |x| <= 3.39e38).  The planes lie below one another, as operands of the weight update (gemm_apply.cuh).
#pragma once

#include "common.cuh"

namespace galore {

// dst (planes x rows x ld) <- src (rows x cols, packed), `planes` = 3 for fp32, 1 (a copy in aligned rows) for bf16
struct PlaneSplit {
  const void* src;       // null: nothing to do
  __nv_bfloat16* dst;
  int32_t dtype;
  int rows, cols;
  int ld;                // a multiple of 8
  int planes;
};

// eight values -> their planes, 16 bytes each
__device__ __forceinline__ void plane_pack(const float (&x)[8], uint4& hi, uint4& mid, uint4& lo) {
  uint32_t* const h = reinterpret_cast<uint32_t*>(&hi);
  uint32_t* const m = reinterpret_cast<uint32_t*>(&mid);
  uint32_t* const l = reinterpret_cast<uint32_t*>(&lo);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(x[2 * j], x[2 * j + 1]);
    h[j] = *reinterpret_cast<const uint32_t*>(&a);
    const float r0 = x[2 * j] - __uint_as_float(h[j] << 16), r1 = x[2 * j + 1] - __uint_as_float(h[j] & 0xffff0000u);
    const __nv_bfloat162 b = __floats2bfloat162_rn(r0, r1);
    m[j] = *reinterpret_cast<const uint32_t*>(&b);
    const __nv_bfloat162 c = __floats2bfloat162_rn(r0 - __uint_as_float(m[j] << 16), r1 - __uint_as_float(m[j] & 0xffff0000u));
    l[j] = *reinterpret_cast<const uint32_t*>(&c);
  }
}

// this thread's share of one matrix: groups of eight columns first, first + stride, ...
__device__ __forceinline__ void plane_split_part(const PlaneSplit& s, int first, int stride) {
  if (!s.src) return;
  const int groups = s.ld / 8, total = s.rows * groups;
  const int64_t plane = (int64_t)s.rows * s.ld;
  for (int i = first; i < total; i += stride) {
    const int row = i / groups, c = (i - row * groups) * 8;
    const int64_t at = (int64_t)row * s.cols + c;
    float x[8];
    if (s.dtype == GALORE_F32) {
      const float* src = (const float*)s.src + at;
      if (c + 8 <= s.cols && (s.cols & 3) == 0 && ((uintptr_t)s.src & 15) == 0) {
        const float4 a = *reinterpret_cast<const float4*>(src), b = *reinterpret_cast<const float4*>(src + 4);
        x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
        x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = c + j < s.cols ? src[j] : 0.f;
      }
    } else {
      const __nv_bfloat16* src = (const __nv_bfloat16*)s.src + at;
#pragma unroll
      for (int j = 0; j < 8; ++j) x[j] = c + j < s.cols ? __bfloat162float(src[j]) : 0.f;
    }
    uint4 hi, mid, lo;
    plane_pack(x, hi, mid, lo);
    __nv_bfloat16* dst = s.dst + (int64_t)row * s.ld + c;
    *reinterpret_cast<uint4*>(dst) = hi;
    if (s.planes == 3) {
      *reinterpret_cast<uint4*>(dst + plane) = mid;
      *reinterpret_cast<uint4*>(dst + 2 * plane) = lo;
    }
  }
}
// the same as a launch of its own
galore_status_t launch_plane_split(const PlaneSplit& s, cudaStream_t st);

}  // namespace galore
