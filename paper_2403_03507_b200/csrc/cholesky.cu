// T = L^-1 with C = L L^T for b x b matrices (b up to a few thousand), 64 columns at a time.
//
// The elimination that turns C into L turns the identity into L^-1, so both run side by side.  With
// J the block column of a step and Linv = L_JJ^-1:
//   L_i  = C_iJ Linv^T                      for every block row i below J
//   C_ij = C_ij - L_i L_j^T                 J < j <= i
//   T_Jj = Linv B_Jj,  B_ij = B_ij - L_i T_Jj    j <= J (B starts as the identity, T_JJ = Linv)
// B is kept transposed, which makes every product a row-times-row one: no operand is transposed on its
// way into shared memory.  A CTA owns one 64 x 64 tile (i, j); the one of the next diagonal block goes
// on to factor it and to invert its factor.  Where the tiles of a step fit the machine at once, a CTA
// forms the L_i, L_j or T_Jj it needs itself (three 64^3 products instead of one, but one launch per
// step); otherwise a launch before it leaves them in T, the L_i in the part above the diagonal.
//
// What bounds it: for a few blocks the chain of launches, about half of each the 64 x 64 factorisation (with a
// panel's rows in one warp's registers, its inverse beside the next panel and fp64 updates on the MMA unit a launch of four blocks in
// fp64 takes 24.9 us at least instead of 32.9, the refresh of 512 x 1376 at rank 128 3.54 ms instead of 3.69); for many the
// FMA rate.
#include "cholesky.cuh"

#include <algorithm>

#include "gemm_dmma.cuh"
#include "launch.cuh"

namespace galore {

namespace {

constexpr int kB = kCholBlock;
// Rows of the matrix being factored, and of the factorisation's scratch: walked by column as well (65, 67: neighbouring rows on
// distinct banks), and with doubles by the 8 x 4 fragments of the MMA (67: two of them on a bank at most).
template <typename S>
constexpr int kLdF = sizeof(S) == 8 ? 67 : 65;
template <typename S>
constexpr int kLdW = sizeof(S) == 8 ? 35 : 33;
template <typename S>
constexpr size_t kFactorBytes = (2 * 64 * kLdF<S> + 32 * kLdW<S>) * sizeof(S);
constexpr int kThreads = 256;
constexpr int kOwnTiles = 40;           // tiles of a step up to which every CTA forms its own L_i, L_j, T_Jj

// shared-memory rows of a tile: 16-byte aligned; fp32: neighbouring rows four banks apart, fp64: 4 mod 16 doubles, so that the
// 8 x 4 operand fragments of the MMA fall on distinct banks
template <typename S>
constexpr int kLd = 68;
template <typename S>
using Tile = S (*)[kLd<S>];
template <typename S>
constexpr int chol_smem(int tiles) { return tiles * kB * kLd<S> * (int)sizeof(S); }

// ---- factor and inverse of one 64 x 64 block ---------------------------------------------------------
// acc = the sum over 4 KS of P(i, k) Q(k, j), an 8 x 8 tile of a warp; p and q lead to the lane's elements of the first step
template <int KS>
__device__ __forceinline__ void warp_tile(double (&acc)[2], const double* p, int p_k, const double* q, int q_k) {
  acc[0] = acc[1] = 0.0;
#pragma unroll
  for (int ks = 0; ks < KS; ++ks) dmma_m8n8k4(acc, p[4 * ks * p_k], q[4 * ks * q_k]);
}

// A (lower triangle, rows of kLdF) <- L, X (rows of kLdF) <- L^-1 with zeros above the diagonal; W: 32 rows of kLdW of
// scratch, rdiag: 64 values.  By panels of 16 columns: one warp factors the panel, two rows in each lane's registers (no
// barrier inside), another inverts the diagonal sub-block of the panel before, then all 256 threads update the rest.  In fp64 the
// update and the products of the inverse run on the MMA unit: as scalar code they were bound by their loads from shared memory.
template <typename S>
__device__ __forceinline__ void factor_block(S (*A)[kLdF<S>], S (*X)[kLdF<S>], S (*W)[kLdW<S>], S* rdiag, int32_t* status) {
  constexpr bool kMma = sizeof(S) == 8;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, t = lane & 3;
  for (int e = tid; e < kB * kB; e += kThreads) X[e >> 6][e & 63] = S(0);
  // the inverse of the diagonal sub-block at o, a column per lane
  auto invert = [&](int o) {
    if (lane >= 16) return;
    S s[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) s[k] = k == lane ? S(1) : S(0);
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      s[r] *= rdiag[o + r];
#pragma unroll
      for (int k = r + 1; k < 16; ++k) s[k] = fma(-A[o + k][o + r], s[r], s[k]);
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) X[o + k][o + lane] = s[k];
  };
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int o = 16 * p;
    if (warp == 0) {
      // rows o + lane and o + 32 + lane of the panel
      const bool one = o + lane < kB, two = o + 32 + lane < kB;
      S r[16], q[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        r[k] = one && k <= lane ? A[o + lane][o + k] : S(0);
        q[k] = o < 32 && two ? A[o + 32 + lane][o + k] : S(0);
      }
      // The chain from pivot to pivot is rsqrt, multiply, fma: every lane works out the next pivot for itself, from values
      // that were passed on before the root was known.  No branch in it, so that the updates fill the waits.
      bool bad = false;
      S piv = __shfl_sync(0xffffffffu, r[0], 0);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const bool unusable = !(piv > S(0));       // not positive definite: go on with a usable pivot, latch the fact
        bad |= unusable;
        piv = unusable ? (S)fabs(piv) + S(1e-30) : piv;
        S raw = S(0), next = S(1);
        if (j < 15) {
          raw = __shfl_sync(0xffffffffu, r[j], j + 1);
          next = __shfl_sync(0xffffffffu, r[j + 1], j + 1);
        }
        const S rs = rsqrt(piv);
        const S l = (lane == j ? piv : (lane > j ? r[j] : S(0))) * rs;
        const S l1 = raw * rs;
        r[j] = l;
        q[j] *= rs;
        piv = fma(-l1, l1, next);
        if (lane == j) rdiag[o + j] = rs;
        // the column, by way of shared memory: fewer instructions than a shuffle per value
        S* const column = W[4 * (j & 1)];            // rows 0 and 4: 16-byte aligned for either type
        if (lane < 16) column[lane] = l;
        __syncwarp();
        constexpr int V = 16 / (int)sizeof(S);
#pragma unroll
        for (int k0 = 0; k0 < 16; k0 += V) {
          if (k0 + V - 1 <= j) continue;
          alignas(16) S c[V];
          *reinterpret_cast<uint4*>(c) = *reinterpret_cast<const uint4*>(column + k0);
#pragma unroll
          for (int k = 0; k < V; ++k)
            if (k0 + k > j) {
              r[k0 + k] = fma(-l, c[k], r[k0 + k]);
              if (o < 32) q[k0 + k] = fma(-q[j], c[k], q[k0 + k]);
            }
        }
      }
      if (bad && lane == 0) atomicOr(status, GALORE_DEV_CHOLESKY);
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        if (one && k <= lane) A[o + lane][o + k] = r[k];
        if (o < 32 && two) A[o + 32 + lane][o + k] = q[k];
      }
    } else if (warp == 1 && p > 0) {
      invert(o - 16);
    }
    __syncthreads();
    if (p < 3) {
      // A[rest][rest] -= L L^T, lower part
      if constexpr (kMma) {
        const int n = 6 - 2 * p;           // tiles of 8
        for (int tile = warp; tile < n * (n + 1) / 2; tile += kThreads / 32) {
          int ti = 0, tj = tile;
          while (tj > ti) tj -= ++ti;
          double acc[2];
          warp_tile<4>(acc, &A[o + 16 + 8 * ti + g][o + t], 1, &A[o + 16 + 8 * tj + g][o + t], 1);
          double* dst = &A[o + 16 + 8 * ti + g][o + 16 + 8 * tj + 2 * t];
          dst[0] -= acc[0];
          dst[1] -= acc[1];
        }
      } else {
        // thread (ty, tx) owns rows ty + 16 u, columns tx + 16 v
        constexpr int kMost = 3;
        const int per = 3 - p, ty = tid >> 4, tx = tid & 15;
        S acc[kMost][kMost];
#pragma unroll
        for (int u = 0; u < kMost; ++u)
#pragma unroll
          for (int v = 0; v < kMost; ++v) acc[u][v] = S(0);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          S x[kMost], y[kMost];
#pragma unroll
          for (int u = 0; u < kMost; ++u)
            if (u < per) {
              x[u] = A[o + 16 + ty + 16 * u][o + k];
              y[u] = A[o + 16 + tx + 16 * u][o + k];
            }
#pragma unroll
          for (int u = 0; u < kMost; ++u)
#pragma unroll
            for (int v = 0; v <= u; ++v)
              if (u < per) acc[u][v] = fma(x[u], y[v], acc[u][v]);
        }
#pragma unroll
        for (int u = 0; u < kMost; ++u)
#pragma unroll
          for (int v = 0; v <= u; ++v)
            if (u < per && (u > v || ty >= tx)) A[o + 16 + ty + 16 * u][o + 16 + tx + 16 * v] -= acc[u][v];
      }
      __syncthreads();
    }
  }
  // ---- the rest of the inverse: the sub-blocks merged pairwise, T21 = -T22 (L21 T11)
  if (warp == 1) invert(48);
  __syncthreads();
  if constexpr (kMma) {
    {                                    // two pairs of 16: a tile of 8 x 8 per warp
      const int pair = warp >> 2, o = 32 * pair, i = 8 * ((warp >> 1) & 1), j = 8 * (warp & 1);
      double acc[2];
      warp_tile<4>(acc, &A[o + 16 + i + g][o + t], 1, &X[o + t][o + j + g], kLdF<S>);
      W[16 * pair + i + g][j + 2 * t] = acc[0];
      W[16 * pair + i + g][j + 2 * t + 1] = acc[1];
      __syncthreads();
      warp_tile<4>(acc, &X[o + 16 + i + g][o + 16 + t], 1, &W[16 * pair + t][j + g], kLdW<S>);
      X[o + 16 + i + g][o + j + 2 * t] = -acc[0];
      X[o + 16 + i + g][o + j + 2 * t + 1] = -acc[1];
      __syncthreads();
    }
    {                                    // the pair of 32: two tiles per warp, side by side
      const int i = 8 * (warp >> 1), j = 16 * (warp & 1);
      double acc[2][2];
#pragma unroll
      for (int v = 0; v < 2; ++v) warp_tile<8>(acc[v], &A[32 + i + g][t], 1, &X[t][j + 8 * v + g], kLdF<S>);
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        W[i + g][j + 8 * v + 2 * t] = acc[v][0];
        W[i + g][j + 8 * v + 2 * t + 1] = acc[v][1];
      }
      __syncthreads();
#pragma unroll
      for (int v = 0; v < 2; ++v) warp_tile<8>(acc[v], &X[32 + i + g][32 + t], 1, &W[t][j + 8 * v + g], kLdW<S>);
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        X[32 + i + g][j + 8 * v + 2 * t] = -acc[v][0];
        X[32 + i + g][j + 8 * v + 2 * t + 1] = -acc[v][1];
      }
    }
  } else {
    {                                    // two pairs of 16: thread (pair, r, c-pair)
      const int pair = tid >> 7, o = 32 * pair, r = (tid >> 3) & 15, c = (tid & 7) * 2;
      S w0 = S(0), w1 = S(0);
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const S l = A[o + 16 + r][o + k];
        w0 = fma(l, X[o + k][o + c], w0);
        w1 = fma(l, X[o + k][o + c + 1], w1);
      }
      W[16 * pair + r][c] = w0;
      W[16 * pair + r][c + 1] = w1;
      __syncthreads();
      S t0 = S(0), t1 = S(0);
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const S x = X[o + 16 + r][o + 16 + k];
        t0 = fma(-x, W[16 * pair + k][c], t0);
        t1 = fma(-x, W[16 * pair + k][c + 1], t1);
      }
      X[o + 16 + r][o + c] = t0;
      X[o + 16 + r][o + c + 1] = t1;
      __syncthreads();
    }
    {                                    // the pair of 32: thread owns rows ty, ty + 16 and columns tx, tx + 16
      const int ty = tid >> 4, tx = tid & 15;
      S w[2][2] = {{S(0), S(0)}, {S(0), S(0)}};
#pragma unroll 8
      for (int k = 0; k < 32; ++k) {
        const S a0 = A[32 + ty][k], a1 = A[48 + ty][k], x0 = X[k][tx], x1 = X[k][16 + tx];
        w[0][0] = fma(a0, x0, w[0][0]); w[0][1] = fma(a0, x1, w[0][1]);
        w[1][0] = fma(a1, x0, w[1][0]); w[1][1] = fma(a1, x1, w[1][1]);
      }
      W[ty][tx] = w[0][0]; W[ty][16 + tx] = w[0][1];
      W[16 + ty][tx] = w[1][0]; W[16 + ty][16 + tx] = w[1][1];
      __syncthreads();
      S u[2][2] = {{S(0), S(0)}, {S(0), S(0)}};
#pragma unroll 8
      for (int k = 0; k < 32; ++k) {
        const S a0 = X[32 + ty][32 + k], a1 = X[48 + ty][32 + k], x0 = W[k][tx], x1 = W[k][16 + tx];
        u[0][0] = fma(-a0, x0, u[0][0]); u[0][1] = fma(-a0, x1, u[0][1]);
        u[1][0] = fma(-a1, x0, u[1][0]); u[1][1] = fma(-a1, x1, u[1][1]);
      }
      X[32 + ty][tx] = u[0][0]; X[32 + ty][16 + tx] = u[0][1];
      X[48 + ty][tx] = u[1][0]; X[48 + ty][16 + tx] = u[1][1];
    }
  }
  __syncthreads();
}

// ---- tiles -------------------------------------------------------------------------------------------
// dst <- the rows x cols part of a 64 x 64 tile that exists, zeros elsewhere
template <typename S>
__device__ __forceinline__ void load_tile(Tile<S> dst, const S* __restrict__ src, int64_t ld, int rows, int cols) {
  constexpr int V = 16 / (int)sizeof(S), kPerRow = kB / V, kEach = kB * kPerRow / kThreads;
  if (cols == kB && ((uintptr_t)src & 15) == 0 && (ld % V) == 0) {
    uint4 v[kEach];
#pragma unroll
    for (int it = 0; it < kEach; ++it) {
      const int e = (int)threadIdx.x + kThreads * it, r = e / kPerRow, c = (e % kPerRow) * V;
      v[it] = r < rows ? *reinterpret_cast<const uint4*>(src + (int64_t)r * ld + c) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int it = 0; it < kEach; ++it) {
      const int e = (int)threadIdx.x + kThreads * it;
      *reinterpret_cast<uint4*>(&dst[e / kPerRow][(e % kPerRow) * V]) = v[it];
    }
  } else {
    S v[16];
#pragma unroll
    for (int it = 0; it < 16; ++it) {
      const int e = (int)threadIdx.x + kThreads * it, r = e >> 6, c = e & 63;
      v[it] = r < rows && c < cols ? src[(int64_t)r * ld + c] : S(0);
    }
#pragma unroll
    for (int it = 0; it < 16; ++it) {
      const int e = (int)threadIdx.x + kThreads * it;
      dst[e >> 6][e & 63] = v[it];
    }
  }
}
// Row and column of the 64 x 64 result that acc[u][v] of this thread holds.
template <typename S>
__device__ __forceinline__ int acc_row(int u) {
  if constexpr (sizeof(S) == 4) return (int)(threadIdx.x >> 4) + 16 * u;
  return (int)(threadIdx.x >> 7) * 32 + 8 * u + (int)((threadIdx.x & 31) >> 2);
}
template <typename S>
__device__ __forceinline__ int acc_col(int v) {
  if constexpr (sizeof(S) == 4) return (int)(threadIdx.x & 15) + 16 * v;
  return (int)((threadIdx.x >> 5) & 3) * 16 + 8 * (v >> 1) + 2 * (int)(threadIdx.x & 3) + (v & 1);
}
// acc[u][v] = sum_k P[row][k] Q[col][k]: fp32 a 4 x 4 micro-tile per thread, fp64 32 x 16 per warp on the MMA unit
// (as the micro-tile 7.4 thousand cycles, of which the shared memory took the larger part)
__device__ __forceinline__ void product(float (&acc)[4][4], Tile<float> P, Tile<float> Q) {
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[u][v] = 0.0f;
#pragma unroll 4
  for (int k = 0; k < kB; k += 4) {
    alignas(16) float x[4][4], y[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      *reinterpret_cast<uint4*>(x[u]) = *reinterpret_cast<const uint4*>(&P[acc_row<float>(u)][k]);
      *reinterpret_cast<uint4*>(y[u]) = *reinterpret_cast<const uint4*>(&Q[acc_col<float>(u)][k]);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = fma(x[u][e], y[v][e], acc[u][v]);
  }
}
__device__ __forceinline__ void product(double (&acc)[4][4], Tile<double> P, Tile<double> Q) {
  const int m0 = (int)(threadIdx.x >> 7) * 32 + (int)((threadIdx.x & 31) >> 2);
  const int n0 = (int)((threadIdx.x >> 5) & 3) * 16 + (int)((threadIdx.x & 31) >> 2), t = threadIdx.x & 3;
  double d[4][2][2];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) d[u][v][0] = d[u][v][1] = 0.0;
#pragma unroll 4
  for (int k = 0; k < kB; k += 4) {
    double x[4], y[2];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = P[m0 + 8 * u][k + t];
#pragma unroll
    for (int v = 0; v < 2; ++v) y[v] = Q[n0 + 8 * v][k + t];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 2; ++v) dmma_m8n8k4(d[u][v], x[u], y[v]);
  }
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[u][v] = d[u][v >> 1][v & 1];
}
// once every thread has read the buffer it receives acc
template <typename S>
__device__ __forceinline__ void keep(Tile<S> dst, const S (&acc)[4][4]) {
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) dst[acc_row<S>(u)][acc_col<S>(v)] = acc[u][v];
  __syncthreads();
}

template <typename S>
struct CholArgs {
  S *C, *T, *B, *slabs;
  int b, col;
  int32_t* status;
  __device__ __forceinline__ void shift(int64_t bytes) {
    C = slot_ptr(C, bytes);
    T = slot_ptr(T, bytes);
    B = slot_ptr(B, bytes);
    slabs = slot_ptr(slabs, bytes);
    status = slot_ptr(status, bytes);
  }
  __device__ __forceinline__ int size(int blk) const { return min(kB, b - blk * kB); }
  __device__ __forceinline__ S* tile(S* X, int r, int c) const { return X + (int64_t)r * kB * b + (int64_t)c * kB; }
  __device__ __forceinline__ S* slab(int blk) const { return slabs + (int64_t)blk * kB * kB; }
};

// T_Jj (its transpose in X) to its place, zeros to the place opposite to it
template <typename S>
__device__ __forceinline__ void store_row_tile(const CholArgs<S>& a, Tile<S> X, int j, bool transposed) {
  const int rows = a.size(a.col), cols = a.size(j);
  for (int e = threadIdx.x; e < kB * kB; e += kThreads) {
    const int r = e >> 6, c = e & 63;
    if (r < rows && c < cols) a.tile(a.T, a.col, j)[(int64_t)r * a.b + c] = transposed ? X[c][r] : X[r][c];
    if (j < a.col && r < cols && c < rows) a.tile(a.T, j, a.col)[(int64_t)r * a.b + c] = S(0);
  }
}

// The L_i and T_Jj of one step, a tile per CTA: blockIdx.x = j <= col: T_Jj; > col: L_i, kept in T above the diagonal
// (place (col, i)) until step i writes its zeros there.
template <typename S>
__global__ void __launch_bounds__(kThreads) chol_panel_kernel(const CholArgs<S> args, const SlotList slots) {
  extern __shared__ __align__(16) unsigned char chol_raw[];
  CholArgs<S> a = args;
  a.shift((int64_t)slots.id[blockIdx.y] * slots.bytes);
  Tile<S> P = reinterpret_cast<Tile<S>>(chol_raw), Q = P + kB;
  const int t = (int)blockIdx.x, col = a.col;
  grid_dependency_wait();
  grid_launch_dependents();
  load_tile<S>(Q, a.slab(col), kB, kB, kB);
  if (t == col) {
    __syncthreads();
    store_row_tile<S>(a, Q, col, false);
    return;
  }
  S acc[4][4];
  if (t < col) {                         // (T_Jj)^T = B^T Linv^T
    load_tile<S>(P, a.tile(a.B, t, col), a.b, kB, a.size(col));
    __syncthreads();
    product(acc, P, Q);
    keep<S>(P, acc);
    store_row_tile<S>(a, P, t, true);
  } else {                               // L_i
    load_tile<S>(P, a.tile(a.C, t, col), a.b, a.size(t), a.size(col));
    __syncthreads();
    product(acc, P, Q);
    keep<S>(P, acc);
    const int rows = a.size(t);
    S* dst = a.tile(a.T, col, t);        // as 64 rows (k) x the block's columns: transposed
    for (int e = threadIdx.x; e < kB * kB; e += kThreads) {
      const int k = e >> 6, r = e & 63;
      if (r < rows) dst[(int64_t)k * a.b + r] = P[r][k];
    }
  }
}

// dst[r][k] <- src[k][r]: an L_i as the panel kernel left it
template <typename S>
__device__ __forceinline__ void load_panel(Tile<S> dst, const S* __restrict__ src, int64_t ld, int rows) {
  S v[16];
#pragma unroll
  for (int it = 0; it < 16; ++it) {
    const int e = (int)threadIdx.x + kThreads * it, k = e >> 6, r = e & 63;
    v[it] = r < rows ? src[(int64_t)k * ld + r] : S(0);
  }
#pragma unroll
  for (int it = 0; it < 16; ++it) {
    const int e = (int)threadIdx.x + kThreads * it;
    dst[e & 63][e >> 6] = v[it];
  }
}

// One step; col = -1: only the first diagonal block is factored.  blockIdx.x: tile (i, j), i > col, j <= i, the next
// diagonal block first; blockIdx.y: slot.  (The last step has no tiles: its T_Jj come from the panel kernel.)
// OWN: the CTA forms its L_i, L_j or T_Jj itself, else the panel kernel has.
template <typename S, bool OWN>
__global__ void __launch_bounds__(kThreads) chol_update_kernel(const CholArgs<S> args, const SlotList slots) {
  extern __shared__ __align__(16) unsigned char chol_raw[];
  __shared__ S rdiag[kB];
  CholArgs<S> a = args;
  a.shift((int64_t)slots.id[blockIdx.y] * slots.bytes);
  Tile<S> P = reinterpret_cast<Tile<S>>(chol_raw), Q = P + kB, Linv = Q + kB;
  const int col = a.col;
  int i, j;
  {
    int t = (int)blockIdx.x;
    i = col + 1;
    while (t >= i + 1) { t -= i + 1; ++i; }
    j = i - t;
  }
  grid_dependency_wait();
  grid_launch_dependents();
  S acc[4][4], old[4][4];
  // what the product is taken from, on its way while it is formed
  const int rows = j > col ? a.size(i) : a.size(j), cols = j > col ? a.size(j) : a.size(i);
  S* dst = j > col ? a.tile(a.C, i, j) : a.tile(a.B, j, i);
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int r = acc_row<S>(u), c = acc_col<S>(v);
      old[u][v] = j != col && r < rows && c < cols ? dst[(int64_t)r * a.b + c] : S(0);
    }
  if (col >= 0) {
    if constexpr (OWN) {
      load_tile<S>(Linv, a.slab(col), kB, kB, kB);
      load_tile<S>(P, a.tile(a.C, i, col), a.b, a.size(i), a.size(col));
      if (j > col && j < i) load_tile<S>(Q, a.tile(a.C, j, col), a.b, a.size(j), a.size(col));
      else if (j < col) load_tile<S>(Q, a.tile(a.B, j, col), a.b, kB, a.size(col));
      __syncthreads();
      product(acc, P, Linv);          // L_i
      keep<S>(P, acc);
      if (j != col && j < i) {           // L_j, or (T_Jj)^T = B^T Linv^T
        product(acc, Q, Linv);
        keep<S>(Q, acc);
      }
      if (j == col) {                    // (T_JJ)^T
        for (int e = threadIdx.x; e < kB * kB; e += kThreads) Q[e & 63][e >> 6] = Linv[e >> 6][e & 63];
        __syncthreads();
      }
      if (j <= col && i == col + 1) store_row_tile<S>(a, Q, j, true);      // one CTA per column tile
    } else {
      load_panel<S>(P, a.tile(a.T, col, i), a.b, a.size(i));
      if (j > col && j < i) load_panel<S>(Q, a.tile(a.T, col, j), a.b, a.size(j));
      else if (j <= col) load_panel<S>(Q, a.tile(a.T, col, j), a.b, a.size(j));        // T_Jj as [k][c]: Q[c][k]
      __syncthreads();
    }
    if (j > col) product(acc, P, j == i ? P : Q);
    else product(acc, Q, P);          // (B_ij)^T
  }
  if (i == col + 1 && j == i) {          // the next diagonal block: factored at once, its inverse goes to its slab
    S(*A)[kLdF<S>] = reinterpret_cast<S(*)[kLdF<S>]>(chol_raw);
    S(*X)[kLdF<S>] = A + kB;
    S(*W)[kLdW<S>] = reinterpret_cast<S(*)[kLdW<S>]>(X + kB);
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int r = acc_row<S>(u), c = acc_col<S>(v);
        S x = r == c ? S(1) : S(0);
        if (r < rows && c < rows) x = c <= r ? old[u][v] - (col >= 0 ? acc[u][v] : S(0)) : S(0);
        A[r][c] = x;
      }
    __syncthreads();
    factor_block<S>(A, X, W, rdiag, a.status);
    S* out = a.slab(i);
    for (int e = threadIdx.x; e < kB * kB; e += kThreads) out[e] = X[e >> 6][e & 63];
    return;
  }
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int r = acc_row<S>(u), c = acc_col<S>(v);
      if (r < rows && c < cols) dst[(int64_t)r * a.b + c] = old[u][v] - acc[u][v];
    }
}

}  // namespace

template <typename S>
galore_status_t cholesky_inverse_factor(S* C, S* T, S* B, S* slabs, int b, int32_t* flags, const SlotList& slots, cudaStream_t st) {
  if (b < 1 || slots.n < 1) return GALORE_OK;
  static_assert(kFactorBytes<S> <= chol_smem<S>(3), "the factorisation uses the tiles' space");
  static std::atomic<uint64_t> configured[3] = {};
  const int own_smem = chol_smem<S>(3), tile_smem = std::max(chol_smem<S>(2), (int)kFactorBytes<S>);
  GALORE_TRY(allow_smem(configured[0], (const void*)chol_update_kernel<S, true>, own_smem));
  GALORE_TRY(allow_smem(configured[1], (const void*)chol_update_kernel<S, false>, tile_smem));
  GALORE_TRY(allow_smem(configured[2], (const void*)chol_panel_kernel<S>, tile_smem));
  const int blocks = (int)ceil_div(b, kB);
  CholArgs<S> args{C, T, B, slabs, b, 0, flags};
  for (int col = -1; col < blocks; ++col) {
    args.col = col;
    int tiles = 1;
    if (col >= 0 && col < blocks - 1) tiles = blocks * (blocks + 1) / 2 - (col + 1) * (col + 2) / 2;      // sum of i + 1 over i > col
    const dim3 grid((unsigned)tiles, (unsigned)slots.n), row((unsigned)blocks, (unsigned)slots.n);
    // by the tiles of one matrix, not of the group: a matrix is factored the same way whatever it is grouped with
    const bool own = tiles <= kOwnTiles;
    if (col == blocks - 1) {
      GALORE_TRY(launch_kernel(chol_panel_kernel<S>, row, kThreads, tile_smem, 1, true, st, args, slots));
    } else if (own) {
      GALORE_TRY(launch_kernel(chol_update_kernel<S, true>, grid, kThreads, own_smem, 1, true, st, args, slots));
    } else {
      GALORE_TRY(launch_kernel(chol_panel_kernel<S>, row, kThreads, tile_smem, 1, true, st, args, slots));
      GALORE_TRY(launch_kernel(chol_update_kernel<S, false>, grid, kThreads, tile_smem, 1, true, st, args, slots));
    }
  }
  return GALORE_OK;
}
template galore_status_t cholesky_inverse_factor<float>(float*, float*, float*, float*, int, int32_t*, const SlotList&, cudaStream_t);
template galore_status_t cholesky_inverse_factor<double>(double*, double*, double*, double*, int, int32_t*, const SlotList&, cudaStream_t);

}  // namespace galore
