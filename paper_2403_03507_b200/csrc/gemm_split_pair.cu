// Products of fp32 operands on CTA pairs (cta_group::2): 256 x 256 tiles for groups large enough to fill the machine with them.
//
// The arithmetic is that of gemm_split.cu: six products of bf16 planes for one fp32 product; leading products and corrections
// in accumulators of their own, the leading ones added to fp32 sums in registers after every 64 of K, before their rounding
// towards zero can pile up.  The corrections, 2^-8 of that, are added after every kCorrBlocks blocks only: 512 columns of
// tensor memory hold one accumulator of each kind, and the leading one is drained while the corrections of its
// block are formed.
//
// What bounds the 128 x 128 tiles of gemm_split.cu is shared memory: 192 KiB read by the MMAs and 96 KiB of planes written per 64
// of K, and the loads beside them.  In a pair's tile an SM reads the same for twice the flops and converts an element for twice
// as many.  Operands arrive by TMA as they are, three half-blocks of K ahead, so that no thread waits for memory.
// Eight layers of the LLaMA-130M set at rank 256: projections 245 -> 174 us, the call 553 -> 492 us.  A block of 64 takes 2.85 us
// (1.3 PFLOP/s of plane products; without the conversion, or with half the products, little less), a launch about 15 us more.
// The sums are nearer to 64 bits than those of the smaller tiles (R of 448 x 2304, 768 x 2048, 1024 x 2816 at rank 256 and 3000 x 3000 at 512:
// 8.03e-8, 9.1e-8, 9.8e-8 and 1.41e-7 against 8.33e-8, 9.3e-8, 1.00e-7 and 1.42e-7); with leading products and corrections in one
// accumulator they were not (768 x 2048: 9.75e-8).
//
// One persistent CTA per SM:
//   warps 0..7    epilogue: four quarters of the TMEM lanes x two halves of the columns
//   warps 8..15   converters: fp32 from the raw ring, three bf16 planes to the tiles the MMAs read
//   warp 16       MMA issuer (one lane of the leader CTA), owner of the TMEM allocation
//   warp 17       TMA producer (one lane); warps 18 and 19 only give their registers away
#include "gemm_split.cuh"

#include <algorithm>

#include "gemm_tc.cuh"
#include "launch.cuh"
#include "split_tiles.cuh"

namespace galore {

namespace {

constexpr int kTile = 256, kRows = 128;                  // tile of a pair; rows (or columns) of an operand one CTA stages
constexpr int kHalf = 32;                                // K of a half-block: what is loaded, converted and drained at a time
constexpr int kEpiWarps = 8, kConvertWarps = 8;
constexpr int kMmaWarp = kEpiWarps + kConvertWarps, kLoadWarp = kMmaWarp + 1;
constexpr int kThreads = 32 * (kMmaWarp + 4);
// registers per thread: 640 threads start with 96 each; 2 x 160 + 2 x 64 + 32 = 5 x 96 over the five warpgroups
constexpr int kLaunchRegs = 96, kEpiRegs = 160, kConvertRegs = 64, kOtherRegs = 32;
static_assert(2 * kEpiRegs + 2 * kConvertRegs + kOtherRegs <= 5 * kLaunchRegs, "register split");
constexpr int kRawBytes = 2 * kRows * kHalf * 4;         // both operands
constexpr int kRawStages = 3;
constexpr int kPlaneBytes = 6 * kTileBytes;              // 64 of K of both operands, as two halves that are filled in turn
constexpr int kSmemBytes = kPlaneBytes + kRawStages * kRawBytes + kEpiWarps * 32 * kStageLd * 4 + 1024 + 256;
static_assert(kSmemBytes <= 227 * 1024, "shared memory of one CTA");
constexpr uint32_t kTmem = 512;                          // the leading products, then the corrections
constexpr int kCorrBlocks = 8;

template <int CAP>
struct PairArgs {
  static constexpr int kCapacity = CAP;
  CUtensorMap map_a[CAP], map_b[CAP];
  SplitProblem p[CAP];
  int unit_end[CAP];
  int count;
};

// after this block of a tile's K the corrections are added, with the leading products of the block
__device__ __forceinline__ bool corrections_due(int kb, int blocks) { return kb % kCorrBlocks == kCorrBlocks - 1 || kb == blocks - 1; }

// four fp32 values -> eight bytes of each plane, kTileBytes apart
__device__ __forceinline__ void convert_quad(uint32_t dst, const uint4& raw) {
  const uint32_t x[4] = {raw.x, raw.y, raw.z, raw.w};
  uint32_t h[2], m[2], l[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const float x0 = __uint_as_float(x[2 * j]), x1 = __uint_as_float(x[2 * j + 1]);
    h[j] = pack_bf16(x0, x1);
    const float r0 = x0 - __uint_as_float(h[j] << 16), r1 = x1 - __uint_as_float(h[j] & 0xffff0000u);
    m[j] = pack_bf16(r0, r1);
    l[j] = pack_bf16(r0 - __uint_as_float(m[j] << 16), r1 - __uint_as_float(m[j] & 0xffff0000u));
  }
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dst), "r"(h[0]), "r"(h[1]) : "memory");
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dst + kTileBytes), "r"(m[0]), "r"(m[1]) : "memory");
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dst + 2 * kTileBytes), "r"(l[0]), "r"(l[1]) : "memory");
}

// A converter thread takes four quads of each operand's 128 x 32 half-block, 4096 raw bytes apart.
//   MN-major: 32 rows (k) of 128 floats; a warp takes a row, its next one eight further on.
//   K-major: 128 rows (M or N) of 32 floats; a warp takes four rows, those of a half-warp four apart: their 64 bytes of
//   plane then lie in different halves of the banks.  Its next rows come 32 further on.
struct QuadPos {
  uint32_t raw, dst, step;     // in the raw half-block; in the tile's first half; between its quads
  uint32_t half;               // XOR (K-major) resp. sum (MN-major) that leads to the second half
};
__device__ __forceinline__ QuadPos quad_pos(int warp, int lane, bool mn) {
  QuadPos q;
  if (mn) {
    const int k = warp, c = (lane & 15) >> 1;
    q.raw = (uint32_t)(k * 512 + lane * 16);
    q.dst = (uint32_t)((lane >> 4) * (kSplitK * 128) + k * 128 + ((c ^ (k & 7)) << 4) + (lane & 1) * 8);
    q.step = 8 * 128;
    q.half = kHalf * 128;      // no carry: bit 12, and what lies above it is a multiple of 8192
  } else {
    const int rr = lane >> 3, j = lane & 7;
    const int row = (rr & 1) * 4 + (rr >> 1) * 8 + (warp & 3) + (warp >> 2) * 16;
    q.raw = (uint32_t)(row * 128 + j * 16);
    q.dst = (uint32_t)(row * 128 + (((j >> 1) ^ (row & 7)) << 4) + (j & 1) * 8);
    q.step = 32 * 128;
    q.half = 64;               // bit 6 of the swizzled address
  }
  return q;
}

template <int CAP>
__global__ void __launch_bounds__(kThreads, 1) gemm_split_pair_kernel(const __grid_constant__ PairArgs<CAP> g) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t planes = (raw_addr + 1023u) & ~1023u;
  uint8_t* const base_ptr = smem_raw + (planes - raw_addr);
  const uint32_t raw_ring = planes + kPlaneBytes;
  float* staging = reinterpret_cast<float*>(base_ptr + kPlaneBytes + kRawStages * kRawBytes);
  uint64_t* bars = reinterpret_cast<uint64_t*>(staging + kEpiWarps * 32 * kStageLd);
  const uint32_t bar_base = smem_u32(bars);
  // raw stages full / empty (each CTA its own), halves of the planes full / empty, accumulator full / empty; the
  // half-full and accumulator-empty barriers that count are the leader's
  auto rawf_bar = [&](int s) { return bar_base + 8u * s; };
  auto rawe_bar = [&](int s) { return bar_base + 8u * (kRawStages + s); };
  auto full_bar = [&](int h) { return bar_base + 8u * (2 * kRawStages + h); };
  auto empty_bar = [&](int h) { return bar_base + 8u * (2 * kRawStages + 2 + h); };
  const uint32_t accf_bar = bar_base + 8u * (2 * kRawStages + 4), acce_bar = accf_bar + 8u;
  constexpr int kBars = 2 * kRawStages + 6;
  static_assert(kBars * 8 + 16 <= 256, "barrier space");
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(bars + kBars);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + kBars + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int total_units = g.unit_end[g.count - 1];
  const uint32_t rank = cluster_ctarank();
  const int team = blockIdx.x / 2, teams = gridDim.x / 2;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kRawStages; ++s) {
      mbar_init(rawf_bar(s), 1);
      mbar_init(rawe_bar(s), kConvertWarps);
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(full_bar(h), kConvertWarps * 2);
      mbar_init(empty_bar(h), 1);
    }
    mbar_init(accf_bar, 1);
    mbar_init(acce_bar, kEpiWarps * 2);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    tmem_alloc_pair(smem_u32((const void*)tmem_slot), kTmem);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                                 // the peer's barriers exist before anyone signals them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  grid_dependency_wait();
  grid_launch_dependents();

  if (warp >= kMmaWarp) {
    regs_down<kOtherRegs>();
    if (warp == kLoadWarp && lane == 0) {
      // ================= TMA producer =================
      int stage = 0;
      uint32_t phase = 0;
      long long issued = 0;
      bool ok = true;
      GroupCursor cursor;
      for (int u = team; u < total_units && ok; u += teams) {
        const SplitUnit w = split_unit<kTile>(g, u, cursor);
        const bool a_mn = g.p[w.pi].a.mn != 0, b_mn = g.p[w.pi].b.mn != 0;
        const int m0 = w.m0 + (int)rank * kRows, n0 = w.n0 + (int)rank * kRows;
        for (int k0 = w.kb * kSplitK; k0 < w.kb_end * kSplitK; k0 += kHalf) {
          if (!mbar_wait(rawe_bar(stage), phase ^ 1u, abort_flag)) { ok = false; break; }
          const uint32_t dst = raw_ring + (uint32_t)stage * kRawBytes;
          mbar_arrive_expect_tx(rawf_bar(stage), kRawBytes);
          tma_load_2d(dst, &g.map_a[w.pi], a_mn ? m0 : k0, a_mn ? k0 : m0, rawf_bar(stage));
          tma_load_2d(dst + kRawBytes / 2, &g.map_b[w.pi], b_mn ? n0 : k0, b_mn ? k0 : n0, rawf_bar(stage));
          ++issued;
          if (++stage == kRawStages) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok) {                                      // let the copies that are still in flight land
        const long long pending = issued < kRawStages ? issued : kRawStages;
        for (long long i = 0; i < pending; ++i) {
          if (--stage < 0) { stage = kRawStages - 1; phase ^= 1u; }
          const long long t0 = clock64();
          while (!mbar_try_wait(rawf_bar(stage), phase) && clock64() - t0 < kWaitLimitCycles) {}
        }
      }
    } else if (warp == kMmaWarp && lane == 0 && rank == 0) {
      // ================= MMA issuer =================
      uint32_t phase = 0;                             // of the halves, and of the accumulator: one block after the other
      bool ok = true;
      GroupCursor cursor;
      for (int u = team; u < total_units && ok; u += teams) {
        const SplitUnit w = split_unit<kTile>(g, u, cursor);
        const bool a_mn = g.p[w.pi].a.mn != 0, b_mn = g.p[w.pi].b.mn != 0;
        const uint32_t idesc = split_idesc(a_mn, b_mn, kTile, kTile);
        const uint64_t a_step = (uint64_t)((a_mn ? 2048 : 32) >> 4), b_step = (uint64_t)((b_mn ? 2048 : 32) >> 4);
        const int blocks = w.kb_end - w.kb;
        for (int kb = 0; kb < blocks && ok; ++kb, phase ^= 1u) {
          const bool closing = corrections_due(kb, blocks), fresh = kb % kCorrBlocks == 0;
          // The leading products come last in the first half and first in the second: between them the accumulator is
          // drained.  Where the epilogue reads the corrections as well, they come first in the second half.
          for (int half = 0; half < 2; ++half) {
            if (half == 0 && fresh && !mbar_wait<true>(acce_bar, phase ^ 1u, abort_flag)) { ok = false; break; }
            if (!mbar_wait<true>(full_bar(half), phase, abort_flag)) { ok = false; break; }
            tc_fence_after();
            const uint64_t a_desc = split_desc(planes, a_mn) + (uint64_t)(2 * half) * a_step;
            const uint64_t b_desc = split_desc(planes + 3 * kTileBytes, b_mn) + (uint64_t)(2 * half) * b_step;
            auto lead = [&]() {
              umma_bf16_pair(tmem_base, a_desc, b_desc, idesc, (uint32_t)half);
              umma_bf16_pair(tmem_base, a_desc + a_step, b_desc + b_step, idesc, 1u);
              if (half == 1) umma_commit_pair(accf_bar);
            };
            const bool first = half == 1 && !closing;
            if (first) lead();
            uint32_t accumulate = fresh && half == 0 ? 0u : 1u;
            // planes i of A and order - i of B (rolled up: registers)
#pragma unroll 1
            for (int order = 2; order >= 1; --order)
#pragma unroll 1
              for (int i = 0; i <= order; ++i) {
                const uint64_t ad = a_desc + (uint64_t)((i * kTileBytes) >> 4), bd = b_desc + (uint64_t)(((order - i) * kTileBytes) >> 4);
                umma_bf16_pair(tmem_base + kTile, ad, bd, idesc, accumulate);
                accumulate = 1u;
                umma_bf16_pair(tmem_base + kTile, ad + a_step, bd + b_step, idesc, accumulate);
              }
            if (!first) {
              if (half == 0 && !fresh) {
                if (!mbar_wait<true>(acce_bar, phase ^ 1u, abort_flag)) { ok = false; break; }
                tc_fence_after();
              }
              lead();
            }
            umma_commit_pair(empty_bar(half));        // reusable, in both CTAs, once these MMAs have read it
          }
        }
      }
    }
  } else if (warp >= kEpiWarps) {
    // ================= converters =================
    regs_down<kConvertRegs>();
    int stage = 0, half = 0;
    uint32_t raw_phase = 0, phase = 0;
    bool ok = true;
    int majors = -1;
    GroupCursor cursor;
    for (int u = team; u < total_units && ok; u += teams) {
      const SplitUnit w = split_unit<kTile>(g, u, cursor);
      // a half of a K-major tile lies in both halves of an MN-major one
      const int m = g.p[w.pi].a.mn * 2 + g.p[w.pi].b.mn;
      if (majors >= 0 && m != majors && !__all_sync(0xffffffffu, mbar_wait(empty_bar(1), phase ^ 1u, abort_flag))) { ok = false; break; }
      majors = m;
      const QuadPos qa = quad_pos(warp - kEpiWarps, lane, g.p[w.pi].a.mn != 0), qb = quad_pos(warp - kEpiWarps, lane, g.p[w.pi].b.mn != 0);
      for (int n = 2 * (w.kb_end - w.kb); n > 0; --n) {
        if (!__all_sync(0xffffffffu, mbar_wait(rawf_bar(stage), raw_phase, abort_flag))) { ok = false; break; }
        const uint32_t src = raw_ring + (uint32_t)stage * kRawBytes;
        uint4 va[4], vb[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) va[i] = ld_shared_16B(src + qa.raw + i * 4096);
#pragma unroll
        for (int i = 0; i < 4; ++i) vb[i] = ld_shared_16B(src + kRawBytes / 2 + qb.raw + i * 4096);
        if (!__all_sync(0xffffffffu, mbar_wait(empty_bar(half), phase ^ 1u, abort_flag))) { ok = false; break; }
        const uint32_t da = planes + (qa.dst ^ (half ? qa.half : 0u)), db = planes + 3 * kTileBytes + (qb.dst ^ (half ? qb.half : 0u));
#pragma unroll
        for (int i = 0; i < 4; ++i) convert_quad(da + i * qa.step, va[i]);
#pragma unroll
        for (int i = 0; i < 4; ++i) convert_quad(db + i * qb.step, vb[i]);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(rawe_bar(stage));
          if (rank == 0) mbar_arrive(full_bar(half));
          else mbar_arrive_remote(map_to_cta(full_bar(half), 0));
        }
        if (++stage == kRawStages) { stage = 0; raw_phase ^= 1u; }
        half ^= 1;
        if (half == 0) phase ^= 1u;
      }
    }
  } else {
    // ================= epilogue =================
    regs_up<kEpiRegs>();
    constexpr int kCols = kTile / 2;                  // columns of the tile one warp sums
    const int quarter = warp & 3, part = warp >> 2;
    float* const sm = staging + warp * 32 * kStageLd;
    const uint32_t t = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(part * kCols);
    uint32_t phase = 0;
    bool ok = true;
    GroupCursor cursor;
    for (int u = team; u < total_units && ok; u += teams) {
      const SplitUnit w = split_unit<kTile>(g, u, cursor);
      const SplitProblem& p = g.p[w.pi];
      float sum[kCols];
#pragma unroll
      for (int j = 0; j < kCols; ++j) sum[j] = 0.f;
      const int blocks = w.kb_end - w.kb;
#pragma unroll 1
      for (int kb = 0; kb < blocks; ++kb, phase ^= 1u) {
        if (!__all_sync(0xffffffffu, mbar_wait(accf_bar, phase, abort_flag))) { ok = false; break; }
        tc_fence_after();
        const bool closing = corrections_due(kb, blocks);
#pragma unroll
        for (int c = 0; c < kCols; c += 8) {
          uint32_t x[8], y[8];
          tmem_ld_32x8(t + (uint32_t)c, x);
          if (closing) tmem_ld_32x8(t + (uint32_t)(kTile + c), y);
          tmem_ld_wait();
          if (closing) {
            float v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(x[j]);
            add_acc(v, y);
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = __float_as_uint(v[j]);
          }
          add_acc(sum + c, x);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {                              // accumulator free for the MMA warp (the leader's)
          if (rank == 0) mbar_arrive(acce_bar);
          else mbar_arrive_remote(map_to_cta(acce_bar, 0));
        }
      }
      if (!ok) break;
      const int r0 = w.m0 + (int)rank * kRows + quarter * 32;
      const int rows = min(32, p.M - r0);
#pragma unroll
      for (int c = 0; c < kCols / 32; ++c) {
        const int c0 = w.n0 + part * kCols + c * 32;
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

  if (*abort_flag) {                                  // gave up: let copies, MMAs and signals that are still in flight land
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000LL) {}
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                                 // neither CTA leaves while the peer may still signal it
  if (threadIdx.x == 0 && *abort_flag) atomicOr(g.p[0].status, GALORE_DEV_WAIT_EXPIRED);
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, kTmem);
  }
}

// a 128 x 32 half-block of the operand per copy, rows as they lie in memory
galore_status_t operand_map(CUtensorMap* map, const SplitOperand& o, int mn_size, int K) {
  return o.mn ? tensor_encode(map, o.base, GALORE_F32, K, mn_size, o.ld, kHalf, kRows, false)
              : tensor_encode(map, o.base, GALORE_F32, mn_size, K, o.ld, kRows, kHalf, false);
}

template <int CAP>
galore_status_t launch_pair(const SplitGroup& g, bool early, bool* taken, cudaStream_t st) {
  auto kern = gemm_split_pair_kernel<CAP>;
  static std::atomic<uint64_t> configured{0};
  static std::atomic<int> registers{0};
  if (registers.load(std::memory_order_relaxed) == 0) {
    cudaFuncAttributes attr;
    GALORE_CUDA_TRY(cudaFuncGetAttributes(&attr, kern));
    registers.store(attr.numRegs, std::memory_order_relaxed);
  }
  // setmaxnreg moves registers inside what the CTA was launched with: less than kLaunchRegs would leave it waiting, more
  // would make a step the wrong way.  A build that gave another number leaves the group to the tiles of one CTA.
  *taken = registers.load(std::memory_order_relaxed) == kLaunchRegs;
  if (!*taken) return GALORE_OK;
  PairArgs<CAP> args;
  args.count = g.count;
  int64_t units = 0;
  for (int i = 0; i < g.count; ++i) {
    SplitProblem& p = args.p[i];
    p = g.p[i];
    GALORE_TRY(operand_map(&args.map_a[i], p.a, p.M, p.K));
    GALORE_TRY(operand_map(&args.map_b[i], p.b, p.N, p.K));
    p.tiles_m = (int)ceil_div(p.M, kTile);
    p.tiles_n = (int)ceil_div(p.N, kTile);
    p.m_fast = p.tiles_m <= p.tiles_n ? 1 : 0;
    units += (int64_t)p.tiles_m * p.tiles_n * p.splits;
    if (units >= ((int64_t)1 << 31)) return GALORE_ERR_SHAPE;
    args.unit_end[i] = (int)units;
  }
  GALORE_TRY(allow_smem(configured, (const void*)kern, kSmemBytes));
  const int teams = (int)std::min<int64_t>(units, tensor_sm_count() / 2);
  return launch_kernel(kern, dim3((unsigned)(teams * 2)), kThreads, kSmemBytes, 2, early, st, args);
}

}  // namespace

galore_status_t launch_split_pair(const SplitGroup& g, bool early, bool* taken, cudaStream_t st) {
  return g.count == 1 ? launch_pair<1>(g, early, taken, st) : launch_pair<kSplitGroup>(g, early, taken, st);
}

}  // namespace galore
