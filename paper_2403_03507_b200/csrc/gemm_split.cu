// Products with fp32 operands (or bf16 operands whose rows TMA cannot address) on the 5th-generation
// tensor cores.
//
// x = hi + mid + lo with three bf16 numbers holds an fp32 value exactly (24 significand bits; gemm_split.cuh has the range), so
//   a b = ah bh + (ah bm + am bh) + (ah bl + am bm + al bh) + O(2^-26) |a b|
// and six tcgen05 products of bf16 operands replace one fp32 product (three when one operand is bf16
// already, one when both are).  The dropped terms lie below fp32's own rounding of a product.
//
// Accumulation: the leading products go to one TMEM accumulator, all smaller ones to a second, and
// after every k-block (kChunk) both are added to an fp32 sum in the epilogue warps' registers.  The
// tensor core's accumulator rounds towards zero: the short chains keep that below the rounding of an
// ordinary fp32 sum.
//
// Measured: 32 fp32 gradients of 512 x 1024 at rank 96 44 us, 28 of 512 x 1408 at 128 62 us, eight of 2048 x 2048 at 512 250 us.  (Groups
// that fill the machine with the tiles of CTA pairs run in gemm_split_pair.cu, the last of these in 179 us; packed bf16 rows of long
// products are copied for TMA, api.cu.)  What bounds it: the conversion
// of the operands (about twelve instructions per element, each element of a tile once) and the latency of the one
// stage of loads the producers hold in registers.
//
// One persistent CTA per SM, 128 x 128 tiles, 64 of K per stage:
//   warps 0..7    epilogue: four quarters of the TMEM lanes x two halves of the columns
//   warps 8..23   producers: load the operands from global memory in whatever layout and alignment
//                 they have, split them and store the bf16 tiles in the 128-byte swizzle the MMAs read.
//                 The loads of the next stage are issued while the current one is converted.
//   warp 24       MMA issuer (one lane), owner of the TMEM allocation; its warpgroup and the
//                 producers' give registers to the epilogue's
#include "gemm_split.cuh"

#include <algorithm>

#include "gemm_tc.cuh"
#include "launch.cuh"
#include "split_tiles.cuh"

namespace galore {

namespace {

constexpr int kM = 128, kN = 128;
constexpr int kEpiWarps = 8, kProducerWarps = 16;
constexpr int kProducers = 32 * kProducerWarps;
constexpr int kMmaWarp = kEpiWarps + kProducerWarps;
constexpr int kThreads = 32 * (kMmaWarp + 4);
constexpr int kChunksEach = 1024 / kProducers;           // chunks of 8 elements a producer thread takes of each operand's tile
// registers per thread: 896 threads start with 72 each; 2 x 104 + 4 x 64 + 40 = 7 x 72 over the seven warpgroups
constexpr int kLaunchRegs = 72, kEpiRegs = 104, kProducerRegs = 64, kMmaRegs = 40;
static_assert(kEpiWarps == 8 && kProducerWarps == 16 && 2 * kEpiRegs + 4 * kProducerRegs + kMmaRegs <= 7 * kLaunchRegs, "register split");
static_assert(kEpiRegs >= kLaunchRegs && kProducerRegs <= kLaunchRegs && kMmaRegs <= kLaunchRegs,
              "setmaxnreg.inc only goes up, .dec only down: the other direction is an illegal instruction");
constexpr int kTiles = 12;                               // bf16 tiles in shared memory: stages x splits
constexpr int kSmemBytes = kTiles * kTileBytes + kEpiWarps * 32 * kStageLd * 4 + 1024 + 256;
constexpr int kChunk = 1;                                // k-blocks per accumulator
constexpr uint32_t kTmem = 512;                          // two buffers x (leading, corrections) x 128 columns

template <typename T>
constexpr int splits_of() { return sizeof(T) == 4 ? 3 : 1; }

// ---- producer ------------------------------------------------------------------------------------
// A stage's tile of an operand is 1024 chunks of 8 elements along the contiguous direction; a thread
// takes two of them, `step` storage rows apart.  K-major: 128 rows (M or N) x 8 chunks; MN-major: 64
// rows (k) x 16 chunks.
struct ChunkPos {
  int outer, fast, step;      // first storage row, first element, rows between a thread's chunks
  uint32_t smem, smem_step;   // where the chunk goes inside the tile
};
__device__ __forceinline__ ChunkPos chunk_pos(int tid, bool mn) {
  ChunkPos c;
  if (mn) {
    const int ch = tid & 15;
    c.outer = tid >> 4;
    c.fast = ch * 8;
    c.step = kProducers / 16;
    c.smem = (uint32_t)((ch >> 3) * (kSplitK * 128) + c.outer * 128 + (((ch & 7) ^ (c.outer & 7)) << 4));
  } else {
    const int ch = tid & 7;
    c.outer = tid >> 3;
    c.fast = ch * 8;
    c.step = kProducers / 8;
    c.smem = (uint32_t)(c.outer * 128 + ((ch ^ (c.outer & 7)) << 4));
  }
  c.smem_step = (uint32_t)c.step * 128u;         // the step is a multiple of 8: the swizzle phase stays
  return c;
}

// where the thread's chunks of one operand lie for one stage
struct ChunkSrc {
  const char* ptr;       // first chunk
  int64_t step;          // bytes between its chunks
  int rows;              // storage rows from the first chunk's row to the end of the matrix
  int valid;             // elements of the chunk inside the matrix along the contiguous direction
};

// raw bits of a chunk.  fp32: eight words.  bf16 on 16-byte boundaries: four words; otherwise the two
// aligned 16-byte vectors that hold it (both contain elements of the chunk), shifted when it is converted.
template <typename T>
__device__ __forceinline__ void load_chunk(uint32_t (&raw)[8], const char* ptr, int valid, bool aligned) {
  if (valid >= 8) {
    if constexpr (sizeof(T) == 4) {
      if (aligned) {
        const uint4 a = *reinterpret_cast<const uint4*>(ptr), b = *reinterpret_cast<const uint4*>(ptr + 16);
        raw[0] = a.x; raw[1] = a.y; raw[2] = a.z; raw[3] = a.w;
        raw[4] = b.x; raw[5] = b.y; raw[6] = b.z; raw[7] = b.w;
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) raw[j] = reinterpret_cast<const uint32_t*>(ptr)[j];
      }
    } else {
      const char* base = reinterpret_cast<const char*>((uintptr_t)ptr & ~(uintptr_t)15);
      const uint4 a = *reinterpret_cast<const uint4*>(base);
      raw[0] = a.x; raw[1] = a.y; raw[2] = a.z; raw[3] = a.w;
      if (!aligned && base != ptr) {
        const uint4 b = *reinterpret_cast<const uint4*>(base + 16);
        raw[4] = b.x; raw[5] = b.y; raw[6] = b.z; raw[7] = b.w;
      }
    }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) raw[j] = 0u;
    if (valid > 0) {
      if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (j < valid) raw[j] = reinterpret_cast<const uint32_t*>(ptr)[j];
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (j < valid) raw[j >> 1] |= (uint32_t) reinterpret_cast<const uint16_t*>(ptr)[j] << (16 * (j & 1));
      }
    }
  }
}

__device__ __forceinline__ void st_shared_16B(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
// chunk -> its bf16 tiles, kTileBytes apart.  shift: byte offset of the chunk inside its first aligned vector (bf16)
template <typename T>
__device__ __forceinline__ void store_chunk(uint32_t dst, const uint32_t (&raw)[8], uint32_t shift) {
  if constexpr (sizeof(T) == 4) {
    uint32_t h[4], m[4], l[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float x0 = __uint_as_float(raw[2 * j]), x1 = __uint_as_float(raw[2 * j + 1]);
      h[j] = pack_bf16(x0, x1);
      const float r0 = x0 - __uint_as_float(h[j] << 16), r1 = x1 - __uint_as_float(h[j] & 0xffff0000u);
      m[j] = pack_bf16(r0, r1);
      l[j] = pack_bf16(r0 - __uint_as_float(m[j] << 16), r1 - __uint_as_float(m[j] & 0xffff0000u));
    }
    st_shared_16B(dst, h[0], h[1], h[2], h[3]);
    st_shared_16B(dst + kTileBytes, m[0], m[1], m[2], m[3]);
    st_shared_16B(dst + 2 * kTileBytes, l[0], l[1], l[2], l[3]);
  } else {
    if (shift == 0u) {
      st_shared_16B(dst, raw[0], raw[1], raw[2], raw[3]);
    } else {
      const uint4 x = bytes_from(make_uint4(raw[0], raw[1], raw[2], raw[3]), make_uint4(raw[4], raw[5], raw[6], raw[7]), shift);
      st_shared_16B(dst, x.x, x.y, x.z, x.w);
    }
  }
}

// one operand's position for one stage
template <typename T>
__device__ __forceinline__ ChunkSrc chunk_src(const SplitOperand& op, const ChunkPos& c, int mn0, int k0, int mn_size, int k_size) {
  const int o0 = (op.mn ? k0 : mn0) + c.outer, f0 = (op.mn ? mn0 : k0) + c.fast;
  ChunkSrc s;
  s.ptr = (const char*)op.base + ((int64_t)o0 * op.ld + f0) * (int64_t)sizeof(T);
  s.step = (int64_t)c.step * op.ld * (int64_t)sizeof(T);
  s.rows = (op.mn ? k_size : mn_size) - o0;
  s.valid = (op.mn ? mn_size : k_size) - f0;
  return s;
}

// ---- the kernel ------------------------------------------------------------------------------------

template <typename TA, typename TB, int CAP>
__global__ void __launch_bounds__(kThreads, 1) gemm_split_kernel(const __grid_constant__ SplitArgs<CAP> g) {
  constexpr int SA = splits_of<TA>(), SB = splits_of<TB>();
  constexpr int kStages = kTiles / (SA + SB);
  constexpr int kStageBytes = (SA + SB) * kTileBytes;
  constexpr bool kCorr = SA + SB > 2;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t ring = (raw_addr + 1023u) & ~1023u;
  uint8_t* ring_ptr = smem_raw + (ring - raw_addr);
  float* staging = reinterpret_cast<float*>(ring_ptr + kTiles * kTileBytes);
  uint64_t* bars = reinterpret_cast<uint64_t*>(staging + kEpiWarps * 32 * kStageLd);
  const uint32_t bar_base = smem_u32(bars);
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (kStages + s); };
  auto accf_bar = [&](int a) { return bar_base + 8u * (2 * kStages + a); };
  auto acce_bar = [&](int a) { return bar_base + 8u * (2 * kStages + 2 + a); };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(bars + 2 * kStages + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + 2 * kStages + 5);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int total_units = g.unit_end[g.count - 1];

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full_bar(s), kProducerWarps);
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(accf_bar(a), 1);
      mbar_init(acce_bar(a), kEpiWarps);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    tmem_alloc(smem_u32((const void*)tmem_slot), kTmem);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  grid_dependency_wait();
  grid_launch_dependents();

  if (warp >= kEpiWarps && warp < kMmaWarp) {
    // ================= producers =================
    regs_down<kProducerRegs>();
    const int tid = (int)threadIdx.x - 32 * kEpiWarps;
    int u = blockIdx.x;
    if (u < total_units) {
      GroupCursor cursor;
      SplitUnit w = split_unit<kM>(g, u, cursor);
      uint32_t ra[kChunksEach][8], rb[kChunksEach][8];
      ChunkPos ca = chunk_pos(tid, g.p[w.pi].a.mn != 0), cb = chunk_pos(tid, g.p[w.pi].b.mn != 0);
      // shifts of the chunks in the registers (bf16 operands off the 16-byte boundaries)
      uint32_t sha = 0u, sha_step = 0u, shb = 0u, shb_step = 0u;
      auto src_a = [&]() { return chunk_src<TA>(g.p[w.pi].a, ca, w.m0, w.kb * kSplitK, g.p[w.pi].M, g.p[w.pi].K); };
      auto src_b = [&]() { return chunk_src<TB>(g.p[w.pi].b, cb, w.n0, w.kb * kSplitK, g.p[w.pi].N, g.p[w.pi].K); };
      auto fetch = [&]<typename T>(T, uint32_t (&raw)[8], const ChunkSrc& s, int i, int step, bool aligned) {
        load_chunk<T>(raw, s.ptr + i * s.step, i * step < s.rows ? s.valid : 0, aligned);
      };
      auto shift_of = [](const ChunkSrc& s, bool aligned, uint32_t& sh, uint32_t& st) {
        const bool shifted = !aligned && s.valid >= 8;
        sh = shifted ? (uint32_t)(uintptr_t)s.ptr & 15u : 0u;
        st = shifted ? (uint32_t)s.step & 15u : 0u;
      };
      {
        const ChunkSrc sa = src_a(), sb = src_b();
        const bool al_a = g.p[w.pi].a.aligned != 0, al_b = g.p[w.pi].b.aligned != 0;
#pragma unroll
        for (int i = 0; i < kChunksEach; ++i) fetch(TA(), ra[i], sa, i, ca.step, al_a);
#pragma unroll
        for (int i = 0; i < kChunksEach; ++i) fetch(TB(), rb[i], sb, i, cb.step, al_b);
        shift_of(sa, al_a, sha, sha_step);
        shift_of(sb, al_b, shb, shb_step);
      }
      int stage = 0;
      uint32_t phase = 0;
      for (;;) {
        const uint32_t dst_a = ring + (uint32_t)(stage * kStageBytes) + ca.smem;
        const uint32_t dst_b = ring + (uint32_t)(stage * kStageBytes + SA * kTileBytes) + cb.smem;
        const uint32_t sst_a = ca.smem_step, sst_b = cb.smem_step;
        const uint32_t c_sha = sha, c_sha_step = sha_step, c_shb = shb, c_shb_step = shb_step;
        // the stage after this one
        bool more = true;
        if (++w.kb == w.kb_end) {
          u += gridDim.x;
          more = u < total_units;
          if (more) {
            w = split_unit<kM>(g, u, cursor);
            ca = chunk_pos(tid, g.p[w.pi].a.mn != 0);
            cb = chunk_pos(tid, g.p[w.pi].b.mn != 0);
          }
        }
        ChunkSrc sa = {}, sb = {};
        bool al_a = false, al_b = false;
        if (more) {
          sa = src_a();
          sb = src_b();
          al_a = g.p[w.pi].a.aligned != 0;
          al_b = g.p[w.pi].b.aligned != 0;
          shift_of(sa, al_a, sha, sha_step);
          shift_of(sb, al_b, shb, shb_step);
        }
        if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag)) break;
#pragma unroll
        for (int i = 0; i < kChunksEach; ++i) {
          store_chunk<TA>(dst_a + i * sst_a, ra[i], (c_sha + i * c_sha_step) & 15u);
          if (more) fetch(TA(), ra[i], sa, i, ca.step, al_a);
        }
#pragma unroll
        for (int i = 0; i < kChunksEach; ++i) {
          store_chunk<TB>(dst_b + i * sst_b, rb[i], (c_shb + i * c_shb_step) & 15u);
          if (more) fetch(TB(), rb[i], sb, i, cb.step, al_b);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(full_bar(stage));
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
        if (!more) break;
      }
    }
  } else if (warp >= kMmaWarp) {
    // ================= MMA issuer =================
    regs_down<kMmaRegs>();
    if (warp == kMmaWarp && lane == 0) {
      int stage = 0, acc = 0;
      uint32_t phase = 0, acc_phase = 0;
      bool ok = true;
      GroupCursor cursor;
      for (int u = blockIdx.x; u < total_units && ok; u += gridDim.x) {
        const SplitUnit w = split_unit<kM>(g, u, cursor);
        const bool a_mn = g.p[w.pi].a.mn != 0, b_mn = g.p[w.pi].b.mn != 0;
        const uint32_t idesc = split_idesc(a_mn, b_mn, kM, kN);
        for (int kb = w.kb; kb < w.kb_end && ok;) {
          if (!mbar_wait(acce_bar(acc), acc_phase ^ 1u, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint32_t lead = tmem_base + (uint32_t)(acc * 2 * kN), corr = lead + kN;
          const int end = min(w.kb_end, kb + kChunk);
          uint32_t acc_lead = 0u, acc_corr = 0u;
          for (; kb < end; ++kb) {
            if (!mbar_wait(full_bar(stage), phase, abort_flag)) { ok = false; break; }
            tc_fence_after();
            const uint32_t a_addr = ring + (uint32_t)(stage * kStageBytes), b_addr = a_addr + SA * kTileBytes;
#pragma unroll
            for (int k = 0; k < kSplitK / 16; ++k) {
              const uint64_t a_adv = (uint64_t)((a_mn ? k * 2048 : k * 32) >> 4), b_adv = (uint64_t)((b_mn ? k * 2048 : k * 32) >> 4);
#pragma unroll
              for (int i = 0; i < SA; ++i)
#pragma unroll
                for (int j = 0; j < SB; ++j) {
                  if (i + j > 2) continue;
                  const uint64_t ad = split_desc(a_addr + i * kTileBytes, a_mn) + a_adv;
                  const uint64_t bd = split_desc(b_addr + j * kTileBytes, b_mn) + b_adv;
                  if (i + j == 0) {
                    umma_bf16(lead, ad, bd, idesc, acc_lead);
                    acc_lead = 1u;
                  } else {
                    umma_bf16(corr, ad, bd, idesc, acc_corr);
                    acc_corr = 1u;
                  }
                }
            }
            umma_commit(empty_bar(stage));
            if (++stage == kStages) { stage = 0; phase ^= 1u; }
          }
          if (ok) umma_commit(accf_bar(acc));
          if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
      }
    }
  } else {
    // ================= epilogue =================
    regs_up<kEpiRegs>();
    const int quarter = warp & 3, half = warp >> 2;
    float* const sm = staging + warp * 32 * kStageLd;
    int acc = 0;
    uint32_t acc_phase = 0;
    bool ok = true;
    GroupCursor cursor;
    for (int u = blockIdx.x; u < total_units && ok; u += gridDim.x) {
      const SplitUnit w = split_unit<kM>(g, u, cursor);
      const SplitProblem& p = g.p[w.pi];
      float sum[64];
#pragma unroll
      for (int j = 0; j < 64; ++j) sum[j] = 0.f;
#pragma unroll 1
      for (int kb = w.kb; kb < w.kb_end; kb += kChunk) {
        if (!__all_sync(0xffffffffu, mbar_wait(accf_bar(acc), acc_phase, abort_flag))) { ok = false; break; }
        tc_fence_after();
        const uint32_t t = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * 2 * kN + half * 64);
#pragma unroll
        for (int c = 0; c < 64; c += 16) {
          uint32_t x[16], y[16];
          tmem_ld_32x16(t + (uint32_t)c, x);
          if constexpr (kCorr) tmem_ld_32x16(t + (uint32_t)(kN + c), y);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            asm volatile("" : "+r"(x[j]));            // not read before the wait
            float v = __uint_as_float(x[j]);
            if constexpr (kCorr) {
              asm volatile("" : "+r"(y[j]));
              v += __uint_as_float(y[j]);
            }
            sum[c + j] += v;
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acce_bar(acc));
        if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
      }
      if (!ok) break;
      const int r0 = w.m0 + quarter * 32;
      const int rows = min(32, p.M - r0);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int c0 = w.n0 + half * 64 + c * 32;
        if (rows <= 0 || c0 >= p.N) continue;         // the same for the whole warp
        // through shared memory: a lane holds a row of the tile, the accesses below run along rows
#pragma unroll
        for (int j = 0; j < 32; ++j) sm[lane * kStageLd + j] = sum[c * 32 + j];
        __syncwarp();
        float* dst = p.C + (int64_t)w.slice * p.split_stride + (int64_t)r0 * p.ldc + c0 + lane;
        if (c0 + lane < p.N) {
#pragma unroll
          for (int r = 0; r < 32; ++r)
            if (r < rows) dst[(int64_t)r * p.ldc] = sm[r * kStageLd + lane];
        }
        __syncwarp();
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) atomicOr(g.p[0].status, GALORE_DEV_WAIT_EXPIRED);
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmem);
  }
}

template <typename TA, typename TB, int CAP>
galore_status_t launch_split_variant(const SplitArgs<CAP>& g, bool early, cudaStream_t st) {
  const int units = g.unit_end[g.count - 1];
  if (units <= 0) return GALORE_OK;
  auto kern = gemm_split_kernel<TA, TB, CAP>;
  static_assert(kSmemBytes <= 227 * 1024, "shared memory of one CTA");
  static std::atomic<uint64_t> configured{0};
  static std::atomic<int> registers{0};
  if (registers.load(std::memory_order_relaxed) == 0) {
    cudaFuncAttributes attr;
    GALORE_CUDA_TRY(cudaFuncGetAttributes(&attr, kern));
    registers.store(attr.numRegs, std::memory_order_relaxed);
  }
  // setmaxnreg moves registers inside what the CTA was launched with: less than kLaunchRegs would leave it waiting, more
  // would make a step the wrong way
  if (registers.load(std::memory_order_relaxed) != kLaunchRegs) {
    note_cuda_error(cudaErrorInvalidConfiguration, "gemm_split_kernel: its register split needs a build with 72 registers a thread");
    return GALORE_ERR_CUDA;
  }
  GALORE_TRY(allow_smem(configured, (const void*)kern, kSmemBytes));
  return launch_kernel(kern, dim3((unsigned)std::min(units, tensor_sm_count())), kThreads, kSmemBytes, 1, early, st, g);
}

template <typename TA, typename TB>
galore_status_t launch_split(const SplitGroup& g, bool early, cudaStream_t st) {
  if (g.count < 1) return GALORE_OK;
  if (g.count > 1) return launch_split_variant<TA, TB, kSplitGroup>(g, early, st);
  SplitArgs<1> one;
  one.p[0] = g.p[0];
  one.unit_end[0] = g.unit_end[0];
  one.count = 1;
  return launch_split_variant<TA, TB, 1>(one, early, st);
}

galore_status_t add_problem(SplitGroup& g, SplitProblem& p, int splits) {
  if (g.count >= kSplitGroup) return GALORE_ERR_BUFFER_TOO_SMALL;
  if (p.M <= 0 || p.N <= 0 || p.K <= 0) return GALORE_ERR_SHAPE;
  p.tiles_m = (int)ceil_div(p.M, kM);
  p.tiles_n = (int)ceil_div(p.N, kN);
  p.kblocks = (int)ceil_div(p.K, kSplitK);
  p.kblocks_per_split = (int)ceil_div(p.kblocks, std::max(1, splits));
  p.splits = (int)ceil_div(p.kblocks, p.kblocks_per_split);
  p.m_fast = p.tiles_m <= p.tiles_n ? 1 : 0;         // neighbours share the panel of the larger operand
  const int64_t before = g.count ? g.unit_end[g.count - 1] : 0, units = (int64_t)p.tiles_m * p.tiles_n * p.splits;
  if (before + units >= ((int64_t)1 << 31)) return GALORE_ERR_SHAPE;
  g.p[g.count] = p;
  g.unit_end[g.count] = (int)(before + units);
  g.count += 1;
  return GALORE_OK;
}

}  // namespace

SplitOperand split_operand(const void* base, int32_t dtype, int64_t s_mn, int64_t s_k) {
  SplitOperand o;
  o.base = base;
  o.mn = s_k == 1 ? 0 : 1;
  o.ld = s_k == 1 ? s_mn : s_k;
  o.aligned = (((uintptr_t)base | (uintptr_t)(o.ld * (int64_t)dtype_size(dtype))) & 15) == 0 ? 1 : 0;
  return o;
}

int split_effective_slices(int64_t K, int slices) {
  const int64_t kb = ceil_div(K, kSplitK);
  return (int)ceil_div(kb, ceil_div(kb, std::max(1, slices)));
}

namespace {
// Microseconds of `units` work units of kb k-blocks: waves x (k-blocks x time of a k-block + fixed time of a unit).  A k-block
// of 128 x 128 on one SM takes 1.75 us (the producers' loads, whatever the number of planes: 512 x 5461 x 2048 of unaligned bf16
// in 1 to 5 slices 115 / 86 / 77 / 74 / 73 us, 128 x 1376 x 512 of fp32 in 1, 2, 4: 19.9 / 12.9 / 9.5 us).  A pair's, of 256 x 256,
// takes 2.85 us (256 x 4096 x K in groups of 144 tiles: 65.7 us at K = 512, 378 at 4096).
double split_us(int64_t units, int64_t kb, bool pair) {
  return (double)ceil_div(units, pair ? 74 : 148) * (pair ? (double)kb * 2.85 + 2.5 : (double)kb * 1.75 + 0.6);
}
int64_t split_units(int64_t M, int64_t N, int64_t slices, int tile) { return ceil_div(M, tile) * ceil_div(N, tile) * slices; }
}  // namespace

// The time of the launch plus that of reading back the partial results: the Adam kernel behind it reads a slice at 4.8 TB/s.
// (With 0.6 us a k-block for bf16 512 x 5461 x 2048 was cut in two: 153 us a step instead of 146.)
int split_choose_slices(int64_t M, int64_t N, int64_t K) {
  const int64_t kb = ceil_div(K, kSplitK);
  int best = 1;
  double best_us = 1e30;
  for (int s = 1; s <= 16; ++s) {
    if (split_effective_slices(K, s) != s) continue;
    const double us = split_us(split_units(M, N, s, 128), ceil_div(kb, s), false) + s * (0.35 + (double)(M * N) * 4.0 / 4.8e6);
    if (us < best_us) {
      best_us = us;
      best = s;
    }
  }
  return best;
}

double split_store_us(int64_t M, int64_t N, int64_t K, int slices) {
  return split_us(split_units(M, N, slices, 128), ceil_div(ceil_div(K, kSplitK), slices), false);
}

// The kernel is the one that launch_split_store takes.  Its time, measured in groups of 8 to 32 matrices with K of 384 to 2048, is 1.75 us a
// block + 3.6 us for every wave of single tiles (768 x 2048 at rank 256: 8 / 16 / 32 of them 58 / 107 / 181 us), 2.85 + 0.6 us of pairs
// (47 / 81 / 151 us), and about 10 us a launch.
double split_group_us(const SplitTiles& t) {
  const bool pair = t.may_pair && split_us(t.pairs, t.blocks, true) < split_us(t.singles, t.blocks, false);
  const double block = (double)t.blocks;
  return 10.0 + (pair ? (double)ceil_div(t.pairs, 74) * (2.85 * block + 0.6) : (double)ceil_div(t.singles, 148) * (1.75 * block + 3.6));
}

galore_status_t split_group_add_store(SplitGroup& g, int M, int N, int K, const SplitOperand& a, const SplitOperand& b, int splits,
                                      float* C, int64_t ldc, int64_t split_stride, int32_t* status) {
  SplitProblem p = {};
  p.M = M; p.N = N; p.K = K;
  p.a = a; p.b = b;
  p.C = C; p.ldc = ldc; p.split_stride = split_stride;
  p.status = status;
  return add_problem(g, p, splits);
}

galore_status_t launch_split_store(const SplitGroup& g, int32_t a_dtype, int32_t b_dtype, bool pairs, bool early, cudaStream_t st) {
  const bool ab = a_dtype == GALORE_BF16, bb = b_dtype == GALORE_BF16;
  if (ab && bb) return launch_split<__nv_bfloat16, __nv_bfloat16>(g, early, st);
  if (ab) return launch_split<__nv_bfloat16, float>(g, early, st);
  if (bb) return launch_split<float, __nv_bfloat16>(g, early, st);
  if (pairs) {
    int64_t single = 0, pair = 0, kb = 0;
    for (int i = 0; i < g.count && pairs; ++i) {
      const SplitProblem& p = g.p[i];
      pairs = p.a.aligned && p.b.aligned;
      single += split_units(p.M, p.N, p.splits, 128);
      pair += split_units(p.M, p.N, p.splits, 256);
      kb = std::max<int64_t>(kb, p.kblocks_per_split);
    }
    if (pairs && split_us(pair, kb, true) < split_us(single, kb, false)) {
      bool taken = false;
      GALORE_TRY(launch_split_pair(g, early, &taken, st));
      if (taken) return GALORE_OK;
    }
  }
  return launch_split<float, float>(g, early, st);
}

}  // namespace galore
