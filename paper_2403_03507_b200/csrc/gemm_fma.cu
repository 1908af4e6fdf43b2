// Products with fp32 FMA.
//
// Why they stand beside the faster split products (gemm_split.cuh), whose sums are nearer to the exact ones: with both moments
// young, Eq. 15 is N = r / (|r| + eps), and an r that the sum over K all but cancels hands its rounding to N undamped.  An
// fp32 W shows that: for 512 x 1376 at rank 128 two sums that differ in their last bits gave weights 8.5e-5 apart in 1 of 40
// runs (each 1.6e-5 to 6.9e-5 from those of a product in 64 bits).  Such layers therefore keep one fixed order of their
// sums: fmaf over k, slice after slice.  A bf16 W or 8-bit moments round far above the difference, and Adafactor's
// factored second moment does not vanish with a single r: there the split products carry the projection.
//
// What bounds it: the FMA rate of a 128 x 128 tile of 256 threads for large matrices; for small ones latency.  fp32 operands on
// 16-byte boundaries whose rows lie along the tile, or A's along K, are copied to shared memory asynchronously, several steps of 16 k ahead (a small
// result's whole slice at once: five waits for memory become one).  512 x 1376 at rank 128: 25.0 -> 20.1 us a step, 1376 x 512
// 25.0 -> 20.3; 2048 x 5464 and 5461 x 2048 at rank 512 650 -> 417 and 439, 11008 x 4096 at 128 990 -> 540.  Others go through
// registers, one step ahead: copies of four bytes were slower.
#include "gemm_fma.cuh"

#include <algorithm>
#include <type_traits>

#include "launch.cuh"
#include "tc_ptx.cuh"

namespace galore {

namespace {

constexpr int kBK = 16;
constexpr int kThreads = 256;
// steps of 16 k in shared memory: 42.5 KiB of a small tile's, 66 KiB of a large one's
constexpr int stages(bool async, int bm) { return !async ? 1 : (bm == 64 ? 5 : 4); }
constexpr int smem_bytes(bool async, int bm, int bn) { return stages(async, bm) * kBK * (bm + bn + 8) * 4; }

enum { FMA_LOADED = 0, FMA_COLUMNS = 1, FMA_ROWS = 2 };
// Operands that can be copied ahead: four elements along the tile at a time, A's also along K (FMA_ROWS).
__host__ __device__ inline bool fma_copied(const FmaProblem& p, int mode) {
  return mode != FMA_LOADED && (mode == FMA_ROWS ? p.sAk : p.sAi) == 1 && p.sBj == 1 && (((uintptr_t)p.A | (uintptr_t)p.B) & 15) == 0 &&
         (((mode == FMA_ROWS ? p.sAi : p.sAk) | p.sBk) & 3) == 0;
}

// BM x BN tile, TM x TN elements a thread in groups of four.  A kernel for each kind of A, as both in one, or a bound on the registers
// that is not the one a kind does best with, cost the others: 512 x 1376 at rank 128 22.9 instead of 20.2 us a step, 2048 x 5461 of
// rows off 16 bytes 632 instead of 548, 2048 x 5464 425 instead of 417.
template <typename TA, typename TB, int BM, int BN, int TM, int TN, int CAP, int MODE>
__global__ void __launch_bounds__(kThreads, BM == 64 ? 2 : (MODE == FMA_COLUMNS ? 0 : 1)) gemm_fma_kernel(const __grid_constant__ FmaArgs<CAP> g) {
  static_assert((BM / TM) * (BN / TN) == kThreads, "one micro-tile a thread");
  constexpr int LA = BM * kBK / kThreads, LB = BN * kBK / kThreads;      // elements of a tile each thread fetches
  constexpr bool kRows = MODE == FMA_ROWS;
  constexpr int kStages = stages(MODE != FMA_LOADED, BM);
  extern __shared__ __align__(16) float fma_smem[];
  float(*const As)[kBK][BM + 4] = reinterpret_cast<float(*)[kBK][BM + 4]>(fma_smem);
  float(*const Bs)[kBK][BN + 4] = reinterpret_cast<float(*)[kBK][BN + 4]>(fma_smem + kStages * kBK * (BM + 4));
  grid_dependency_wait();
  grid_launch_dependents();
  GroupCursor cursor;
  int local = cursor.seek<CAP>(g, (int)blockIdx.x);
  const FmaProblem& p = g.p[cursor.pi];
  const int tiles_n = (p.N + BN - 1) / BN, tiles_m = (p.M + BM - 1) / BM;
  const int n0 = (local % tiles_n) * BN;
  local /= tiles_n;
  const int m0 = (local % tiles_m) * BM, slice = local / tiles_m;
  const int k_begin = slice * p.kchunk, k_end = min(p.K, k_begin + p.kchunk);
  const TA* A = (const TA*)p.A;
  const TB* B = (const TB*)p.B;
  const int64_t sAi = p.sAi, sAk = p.sAk, sBk = p.sBk, sBj = p.sBj;
  const int M = p.M, N = p.N;

  const int tid = threadIdx.x;
  const int tx = tid % (BN / TN), ty = tid / (BN / TN);
  const bool a_kfast = (sAk == 1);   // consecutive threads walk the contiguous direction
  const bool b_kfast = (sBk == 1);

  float acc[TM][TN];
#pragma unroll
  for (int u = 0; u < TM; ++u)
#pragma unroll
    for (int v = 0; v < TN; ++v) acc[u][v] = 0.f;

  auto multiply = [&](const float (*As)[BM + 4], const float (*Bs)[BN + 4]) {
#pragma unroll
    for (int k = 0; k < kBK; ++k) {
      float a[TM], b[TN];
#pragma unroll
      for (int u = 0; u < TM; ++u) a[u] = As[k][(u / 4) * (BM / (TM / 4)) + ty * 4 + (u % 4)];
#pragma unroll
      for (int v = 0; v < TN; ++v) b[v] = Bs[k][(v / 4) * (BN / (TN / 4)) + tx * 4 + (v % 4)];
#pragma unroll
      for (int u = 0; u < TM; ++u)
#pragma unroll
        for (int v = 0; v < TN; ++v) acc[u][v] = fmaf(a[u], b[v], acc[u][v]);
    }
  };
  // A's rows along K: four k of a row in 16 bytes, the fours of a row moved round by its place (a warp reads two rows, four apart)
  auto a_four = [&](float* stage, int i, int four) { return stage + i * kBK + ((four ^ (i >> 2)) & 3) * 4; };
  auto multiply_rows = [&](float* As, const float (*Bs)[BN + 4]) {
#pragma unroll
    for (int four = 0; four < kBK / 4; ++four) {
      float4 a[TM];
#pragma unroll
      for (int u = 0; u < TM; ++u) a[u] = *reinterpret_cast<const float4*>(a_four(As, (u / 4) * (BM / (TM / 4)) + ty * 4 + (u % 4), four));
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        float b[TN];
#pragma unroll
        for (int v = 0; v < TN; ++v) b[v] = Bs[4 * four + k][(v / 4) * (BN / (TN / 4)) + tx * 4 + (v % 4)];
#pragma unroll
        for (int u = 0; u < TM; ++u) {
          const float au = k == 0 ? a[u].x : k == 1 ? a[u].y : k == 2 ? a[u].z : a[u].w;
#pragma unroll
          for (int v = 0; v < TN; ++v) acc[u][v] = fmaf(au, b[v], acc[u][v]);
        }
      }
    }
  };
  bool copied = false;
  if constexpr (MODE != FMA_LOADED) copied = fma_copied(p, MODE);
  if (copied) {
    // 16 k of one operand in runs of four; zeros outside the matrix
    auto copy = [&]<int BX, class Tile>(std::integral_constant<int, BX>, Tile dst, const float* X, int64_t s_k, int x0, int X_size, int k0) {
#pragma unroll
      for (int e = 0; e < BX * kBK / 4 / kThreads; ++e) {
        const int idx = tid + e * kThreads, x = idx % (BX / 4) * 4, k = idx / (BX / 4);
        const int valid = k0 + k < k_end ? min(4, max(0, X_size - x0 - x)) : 0;
        const float* src = valid ? X + (int64_t)(k0 + k) * s_k + x0 + x : X;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(&dst[k][x])), "l"(src), "r"(valid * 4) : "memory");
      }
    };
    const int steps = (k_end - k_begin + kBK - 1) / kBK;
    auto request = [&](int step) {                    // (an empty group behind the last step: the count of groups stays)
      if (step < steps) {
        if constexpr (kRows) {
          const int k0 = k_begin + step * kBK;
#pragma unroll
          for (int e = 0; e < BM * kBK / 4 / kThreads; ++e) {
            const int idx = tid + e * kThreads, four = idx % (kBK / 4), i = idx / (kBK / 4);
            const int valid = m0 + i < M ? min(4, max(0, k_end - k0 - 4 * four)) : 0;
            const float* src = valid ? (const float*)A + (int64_t)(m0 + i) * sAi + k0 + 4 * four : (const float*)A;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(a_four(&As[step % kStages][0][0], i, four))), "l"(src), "r"(valid * 4) : "memory");
          }
        } else {
          copy(std::integral_constant<int, BM>(), As[step % kStages], (const float*)A, sAk, m0, M, k_begin + step * kBK);
        }
        copy(std::integral_constant<int, BN>(), Bs[step % kStages], (const float*)B, sBk, n0, N, k_begin + step * kBK);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int step = 0; step < kStages - 1; ++step) request(step);
    for (int step = 0; step < steps; ++step) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
      __syncthreads();                                // the step's copies of all threads are in, the stage to be filled has been read
      request(step + kStages - 1);
      if constexpr (kRows) multiply_rows(&As[step % kStages][0][0], Bs[step % kStages]);
      else multiply(As[step % kStages], Bs[step % kStages]);
    }
  } else {
    float ra[LA], rb[LB];
    auto fetch = [&](int k0) {
#pragma unroll
      for (int e = 0; e < LA; ++e) {
        const int idx = tid + e * kThreads;
        const int i = a_kfast ? idx / kBK : idx % BM;
        const int k = a_kfast ? idx % kBK : idx / BM;
        const int gi = m0 + i, gk = k0 + k;
        ra[e] = (gi < M && gk < k_end) ? cvt<float>(A[(int64_t)gi * sAi + (int64_t)gk * sAk]) : 0.f;
      }
#pragma unroll
      for (int e = 0; e < LB; ++e) {
        const int idx = tid + e * kThreads;
        const int j = b_kfast ? idx / kBK : idx % BN;
        const int k = b_kfast ? idx % kBK : idx / BN;
        const int gj = n0 + j, gk = k0 + k;
        rb[e] = (gj < N && gk < k_end) ? cvt<float>(B[(int64_t)gk * sBk + (int64_t)gj * sBj]) : 0.f;
      }
    };
    auto stash = [&]() {
#pragma unroll
      for (int e = 0; e < LA; ++e) {
        const int idx = tid + e * kThreads;
        As[0][a_kfast ? idx % kBK : idx / BM][a_kfast ? idx / kBK : idx % BM] = ra[e];
      }
#pragma unroll
      for (int e = 0; e < LB; ++e) {
        const int idx = tid + e * kThreads;
        Bs[0][b_kfast ? idx % kBK : idx / BN][b_kfast ? idx / kBK : idx % BN] = rb[e];
      }
    };
    if (k_begin < k_end) fetch(k_begin);
    for (int k0 = k_begin; k0 < k_end; k0 += kBK) {
      __syncthreads();
      stash();
      __syncthreads();
      if (k0 + kBK < k_end) fetch(k0 + kBK);
      multiply(As[0], Bs[0]);
    }
  }
  // a thread's columns come in runs of four: one 16-byte store where the rows allow it
  float* const C = p.C + (int64_t)slice * p.split_stride;
  const bool vec = (((uintptr_t)C & 15) == 0) && (p.ldc % 4) == 0;
#pragma unroll
  for (int u = 0; u < TM; ++u) {
    const int i = m0 + (u / 4) * (BM / (TM / 4)) + ty * 4 + (u % 4);
    if (i >= M) continue;
#pragma unroll
    for (int vg = 0; vg < TN / 4; ++vg) {
      const int j = n0 + vg * (BN / (TN / 4)) + tx * 4;
      float* dst = C + (int64_t)i * p.ldc + j;
      if (j + 3 < N && vec) {
        *reinterpret_cast<float4*>(dst) = make_float4(acc[u][4 * vg], acc[u][4 * vg + 1], acc[u][4 * vg + 2], acc[u][4 * vg + 3]);
      } else {
#pragma unroll
        for (int v = 0; v < 4; ++v)
          if (j + v < N) dst[v] = acc[u][4 * vg + v];
      }
    }
  }
}

// Results below 96 tiles of 128 x 128 are cut into 64 x 64.
bool small_result(int64_t M, int64_t N) { return M * N < (int64_t)128 * 128 * 96; }

template <typename TA, typename TB, int BM, int TM, int MODE, int CAP>
galore_status_t launch_mode(const FmaArgs<CAP>& g, bool early, cudaStream_t st) {
  constexpr int smem = smem_bytes(MODE != FMA_LOADED, BM, BM);
  auto kern = gemm_fma_kernel<TA, TB, BM, BM, TM, TM, CAP, MODE>;
  static std::atomic<uint64_t> configured{0};
  GALORE_TRY(allow_smem(configured, (const void*)kern, smem));
  return launch_kernel(kern, dim3((unsigned)g.unit_end[g.count - 1]), kThreads, smem, 1, early, st, g);
}
// (a problem of a group that does not fit its kernel's copies is loaded there)
template <typename TA, typename TB, int BM, int TM, int CAP>
galore_status_t launch_tiles(const FmaArgs<CAP>& g, bool early, cudaStream_t st) {
  if constexpr (sizeof(TA) == 4 && sizeof(TB) == 4) {
    int columns = 0, rows = 0;
    for (int i = 0; i < g.count; ++i) {
      columns += fma_copied(g.p[i], FMA_COLUMNS) ? 1 : 0;
      rows += fma_copied(g.p[i], FMA_ROWS) ? 1 : 0;
    }
    if (rows > columns) return launch_mode<TA, TB, BM, TM, FMA_ROWS>(g, early, st);
    if (columns > 0) return launch_mode<TA, TB, BM, TM, FMA_COLUMNS>(g, early, st);
  }
  return launch_mode<TA, TB, BM, TM, FMA_LOADED>(g, early, st);
}

template <typename TA, typename TB>
galore_status_t launch_typed(const FmaGroup& g, bool early, cudaStream_t st) {
  if (g.count > 1) return launch_tiles<TA, TB, 128, 8, kFmaGroup>(g, early, st);
  FmaArgs<1> one;
  const FmaProblem& p = one.p[0] = g.p[0];
  one.count = 1;
  const bool small = small_result(p.M, p.N);
  const int64_t t = small ? 64 : 128;
  one.unit_end[0] = (int)(ceil_div(p.M, t) * ceil_div(p.N, t) * p.splits);
  if (small) return launch_tiles<TA, TB, 64, 4, 1>(one, early, st);
  return launch_tiles<TA, TB, 128, 8, 1>(one, early, st);
}

int chunk_of(int64_t K, int slices) { return (int)(std::max<int64_t>(1, ceil_div(ceil_div(K, std::max(1, slices)), kBK)) * kBK); }

}  // namespace

int fma_effective_slices(int64_t K, int slices) { return (int)ceil_div(std::max<int64_t>(1, K), chunk_of(K, slices)); }

int fma_choose_slices(int64_t M, int64_t N, int64_t K) {
  const int64_t t = small_result(M, N) ? 64 : 128;
  const int64_t tiles = ceil_div(M, t) * ceil_div(N, t);
  int64_t want = std::min<int64_t>(16, std::max<int64_t>(1, ceil_div(2 * 148, tiles)));
  want = std::min<int64_t>(want, std::max<int64_t>(1, K / 64));
  return fma_effective_slices(K, (int)want);
}

// 28 matrices of 512 x 1376 at rank 128, 196 tiles: 145 us in two waves; 784 of 1024 x 2752 at rank 512: 1.6 ms in six
double fma_group_us(int64_t tiles, int64_t k) { return (double)ceil_div(tiles, 148) * (double)k * 0.14; }

galore_status_t fma_group_add(FmaGroup& g, const FmaProblem& problem, int slices) {
  if (g.count >= kFmaGroup) return GALORE_ERR_BUFFER_TOO_SMALL;
  FmaProblem p = problem;
  if (p.M <= 0 || p.N <= 0 || p.K <= 0) return GALORE_ERR_SHAPE;
  p.kchunk = chunk_of(p.K, slices);
  p.splits = fma_effective_slices(p.K, slices);
  const int64_t ctas = ceil_div(p.M, 128) * ceil_div(p.N, 128) * p.splits;
  const int64_t before = g.count ? g.unit_end[g.count - 1] : 0;
  if (before + 4 * ctas >= ((int64_t)1 << 31)) return GALORE_ERR_SHAPE;
  g.p[g.count] = p;
  g.unit_end[g.count] = (int)(before + ctas);
  g.count += 1;
  return GALORE_OK;
}

galore_status_t launch_fma_group(const FmaGroup& g, int32_t a_dtype, int32_t b_dtype, bool early, cudaStream_t st) {
  if (g.count < 1) return GALORE_OK;
  const bool ab = a_dtype == GALORE_BF16, bb = b_dtype == GALORE_BF16;
  if (ab && bb) return GALORE_ERR_INVALID_ARG;       // the split products are as exact
  if (ab) return launch_typed<__nv_bfloat16, float>(g, early, st);
  if (bb) return launch_typed<float, __nv_bfloat16>(g, early, st);
  return launch_typed<float, float>(g, early, st);
}

}  // namespace galore
