// FP32 GEMM tiles of the element network's training (forward, backward and update of three dense
// layers on a minibatch), with everything that follows a product done in its epilogue: bias and
// ReLU, the squared error and its gradient, the ReLU mask of the backward pass, the bias gradient
// and the Adam update.
//
// The products are small (a minibatch of some hundred rows against 256 to 518 columns: 17 to 68
// MFMA each), so what bounds them is how many SMs work and how long one K loop takes, not the FMA
// rate.  Two tile shapes, each 256 threads, operands brought by 4-byte cp.async (rows of n^3 + 6
// values keep no wider alignment) into a ring of K slices of 32:
//   * GemmSmall, 32 x 16 outputs, the K slice split over 4 groups of 64 threads whose sums are
//     added in a fixed order through shared memory: 128 blocks for a 256 x 256 product, a K loop
//     a quarter as long per thread;
//   * GemmLarge, 64 x 64 outputs, no split: for products with a tile for every SM.
// A step at n^3 = 512 and 256 rows takes 68 us in six launches (0.44 GFLOP: 6 us at the FP32 rate).
// Operands are read from shared memory four values at a time along whichever of their two
// directions is contiguous in memory (KC: the K direction).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "sem_internal.h"
#include "sem_tma.cuh"

namespace mlpg {

constexpr int GT = 256, BK = 32;

template <int BM_, int BN_, int TM_, int TN_, int KS_, int ST_>
struct GemmCfg {
  static constexpr int BM = BM_, BN = BN_, TM = TM_, TN = TN_, KS = KS_, ST = ST_;
  static constexpr int MT = BM / TM, NTH = BN / TN;  // threads of one K group along m and n
  static_assert(MT * NTH * KS == GT && BK % (4 * KS) == 0, "thread layout of the tile");
  // operand slices: [rows][BK + 4] when K is contiguous, else [BK][cols + 4] (16-byte row starts)
  static constexpr int A_SZ = (BM * (BK + 4) > BK * (BM + 4)) ? BM * (BK + 4) : BK * (BM + 4);
  static constexpr int B_SZ = (BN * (BK + 4) > BK * (BN + 4)) ? BN * (BK + 4) : BK * (BN + 4);
  static constexpr int SMEM = ST * (A_SZ + B_SZ);  // floats
  static_assert(KS * (BM + 1) * BN <= SMEM, "partial sums fit in the operand ring");
};
using GemmSmall = GemmCfg<32, 16, 4, 2, 4, 4>;
using GemmLarge = GemmCfg<64, 64, 4, 4, 1, 2>;

// what happens to a finished product
enum Epilogue {
  EP_FWD,   // C = act(v + bias)
  EP_MSE,   // o = v + bias: C = 2 (o - T) inv, *loss += sum (o - T)^2 inv
  EP_MASK,  // C = H > 0 ? v : 0
  EP_GRAD   // gradient of a weight matrix (and of its bias: column sums of B), Adam update
};

struct GemmArgs {
  int M, N, K;
  const float *A, *B;  // op(A)[m][k] = TA ? A[k lda + m] : A[m lda + k]; op(B)[k][n] = TB ? B[n ldb + k] : B[k ldb + n]
  int lda, ldb;
  const float *bias;  // FWD, MSE
  float *C;           // row length N; may be NULL for GRAD
  int relu;           // FWD
  const float *aux;   // MSE: targets T; MASK: activations H
  double *loss;       // MSE
  float inv;          // MSE
  float *zero_loss;   // the loss (two words) to be cleared by a launch that precedes its sum, or NULL
  // GRAD: parameters and moments of the weights (NULL w: no update), and of the bias
  float *w, *m, *v;
  float *Cb, *wb, *mb, *vb;
  float lr, c1, c2;
};

__device__ __forceinline__ void cp_async4(float *dst, const float *src, bool ok) {
  const int n = ok ? 4 : 0;  // 0: the word is zero filled and src is not read
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(n) : "memory");
}

// Adam (Kingma & Ba): m = b1 m + (1-b1) g; v = b2 v + (1-b2) g^2; w -= lr mhat / (sqrt(vhat) + eps)
__device__ __forceinline__ void adam(float g, float *w, float *m, float *v, float lr, float c1, float c2) {
  constexpr float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float mi = b1 * *m + (1.f - b1) * g;
  const float vi = b2 * *v + (1.f - b2) * g * g;
  *m = mi;
  *v = vi;
  *w -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// one operand slice: rows r0.. of `rows` (m or n), k0.. of K.  KC: K is the contiguous direction
template <int BR, bool KC>
__device__ __forceinline__ void load_slice(float *s, const float *p, int ld, int r0, int rows, int k0, int K) {
  constexpr int N = BR * BK / GT;
  static_assert(BR * BK % GT == 0, "whole passes over the slice");
#pragma unroll
  for (int it = 0; it < N; ++it) {
    const int q = threadIdx.x + it * GT;
    const int kk = KC ? q % BK : q / BR, rr = KC ? q / BK : q % BR;
    const int k = k0 + kk, r = r0 + rr;
    const bool ok = r < rows && k < K;
    const float *src = ok ? p + (KC ? (size_t)r * ld + k : (size_t)k * ld + r) : p;
    cp_async4(KC ? s + rr * (BK + 4) + kk : s + kk * (BR + 4) + rr, src, ok);
  }
}

// v[i][j] = operand value at row r + i, k + j (j < 4) from a slice
template <int BR, int T, bool KC>
__device__ __forceinline__ void read_frag(const float *s, int r, int k, float (&v)[T][4]) {
  if constexpr (KC) {
#pragma unroll
    for (int i = 0; i < T; ++i) {
      const float4 f = *reinterpret_cast<const float4 *>(s + (r + i) * (BK + 4) + k);
      v[i][0] = f.x, v[i][1] = f.y, v[i][2] = f.z, v[i][3] = f.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float *row = s + (k + j) * (BR + 4) + r;
      if constexpr (T == 4) {
        const float4 f = *reinterpret_cast<const float4 *>(row);
        v[0][j] = f.x, v[1][j] = f.y, v[2][j] = f.z, v[3][j] = f.w;
      } else {
        const float2 f = *reinterpret_cast<const float2 *>(row);
        v[0][j] = f.x, v[1][j] = f.y;
      }
    }
  }
}

template <typename C, bool TA, bool TB, int EP>
__device__ __forceinline__ void gemm_tile(const GemmArgs &g, int tile, float *sm) {
  constexpr int BM = C::BM, BN = C::BN, TM = C::TM, TN = C::TN, KS = C::KS, ST = C::ST, KG = BK / KS;
  const int ntn = (g.N + BN - 1) / BN;
  const int m0 = (tile / ntn) * BM, n0 = (tile % ntn) * BN;
  const int tid = threadIdx.x, grp = tid / (C::MT * C::NTH), t = tid % (C::MT * C::NTH);
  // thread's outputs: rows tm.., columns tn..  (the n index runs fastest over the lanes)
  const int tm = (t / C::NTH) * TM, tn = (t % C::NTH) * TN;
  float *sA = sm, *sB = sm + ST * C::A_SZ;
  float acc[TM][TN] = {}, bsum[TN] = {};
  const bool sums = EP == EP_GRAD && m0 == 0 && tm == 0;
  const int nk = (g.K + BK - 1) / BK;
  auto fetch = [&](int c) {
    if (c < nk) {
      load_slice<BM, !TA>(sA + (c % ST) * C::A_SZ, g.A, g.lda, m0, g.M, c * BK, g.K);
      load_slice<BN, TB>(sB + (c % ST) * C::B_SZ, g.B, g.ldb, n0, g.N, c * BK, g.K);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int c = 0; c < ST - 1; ++c) fetch(c);
  for (int c = 0; c < nk; ++c) {
    asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
    __syncthreads();  // slice c is complete, and every thread is done with the slot that is refilled now
    fetch(c + ST - 1);
    const float *a = sA + (c % ST) * C::A_SZ, *b = sB + (c % ST) * C::B_SZ;
#pragma unroll
    for (int kk = 0; kk < KG; kk += 4) {
      const int k = grp * KG + kk;
      float va[TM][4], vb[TN][4];
      read_frag<BM, TM, !TA>(a, tm, k, va);
      read_frag<BN, TN, TB>(b, tn, k, vb);
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int x = 0; x < TM; ++x)
#pragma unroll
          for (int y = 0; y < TN; ++y) acc[x][y] = fmaf(va[x][j], vb[y][j], acc[x][y]);
      if (sums) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int y = 0; y < TN; ++y) bsum[y] += vb[y][j];
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // the groups' sums, added in group order; row BM holds the column sums of B
  constexpr int PS = (BM + 1) * BN;
#pragma unroll
  for (int x = 0; x < TM; ++x)
#pragma unroll
    for (int y = 0; y < TN; ++y) sm[grp * PS + (tm + x) * BN + tn + y] = acc[x][y];
  if (sums) {
#pragma unroll
    for (int y = 0; y < TN; ++y) sm[grp * PS + BM * BN + tn + y] = bsum[y];
  }
  __syncthreads();
  double lacc = 0.0;
#pragma unroll
  for (int it = 0; it < BM * BN / GT; ++it) {
    const int q = tid + it * GT, m = m0 + q / BN, n = n0 + q % BN;
    if (m >= g.M || n >= g.N) continue;
    float val = sm[q];
#pragma unroll
    for (int s = 1; s < KS; ++s) val += sm[s * PS + q];
    const size_t o = (size_t)m * g.N + n;
    if constexpr (EP == EP_FWD) {
      val += g.bias[n];
      g.C[o] = g.relu ? fmaxf(val, 0.f) : val;
    } else if constexpr (EP == EP_MSE) {
      const float d = val + g.bias[n] - g.aux[o];
      g.C[o] = 2.f * d * g.inv;
      lacc += (double)d * d;
    } else if constexpr (EP == EP_MASK) {
      g.C[o] = g.aux[o] > 0.f ? val : 0.f;
    } else {
      if (g.C) g.C[o] = val;
      if (g.w) adam(val, g.w + o, g.m + o, g.v + o, g.lr, g.c1, g.c2);
    }
  }
  if constexpr (EP == EP_MSE) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lacc += __shfl_xor_sync(0xffffffffu, lacc, o);
    if ((tid & 31) == 0) atomicAdd(g.loss, lacc * (double)g.inv);
  }
  if constexpr (EP == EP_GRAD) {
    if (m0 == 0 && tid < BN && n0 + tid < g.N) {
      const int n = n0 + tid;
      float val = sm[BM * BN + tid];
#pragma unroll
      for (int s = 1; s < KS; ++s) val += sm[s * PS + BM * BN + tid];
      if (g.Cb) g.Cb[n] = val;
      if (g.wb) adam(val, g.wb + n, g.mb + n, g.vb + n, g.lr, g.c1, g.c2);
    }
  }
}

template <typename C, bool TA, bool TB, int EP>
__global__ void __launch_bounds__(GT) k_gemm(const __grid_constant__ GemmArgs g) {
  __shared__ __align__(16) float sm[C::SMEM];
  if (g.zero_loss && blockIdx.x == 0 && threadIdx.x < 2) g.zero_loss[threadIdx.x] = 0.f;
  gemm_tile<C, TA, TB, EP>(g, blockIdx.x, sm);
}

// two independent products in one launch: the first n0 blocks work on g0, the others on g1
template <typename C, bool TA0, bool TB0, int EP0, bool TA1, bool TB1, int EP1>
__global__ void __launch_bounds__(GT) k_gemm_pair(const __grid_constant__ GemmArgs g0,
                                                  const __grid_constant__ GemmArgs g1, int n0) {
  __shared__ __align__(16) float sm[C::SMEM];
  if ((int)blockIdx.x < n0)
    gemm_tile<C, TA0, TB0, EP0>(g0, blockIdx.x, sm);
  else
    gemm_tile<C, TA1, TB1, EP1>(g1, (int)blockIdx.x - n0, sm);
}

template <typename C>
int tiles(const GemmArgs &g) {
  return ((g.M + C::BM - 1) / C::BM) * ((g.N + C::BN - 1) / C::BN);
}

// The 64 x 64 tile from one tile per SM (152) on, the split 32 x 16 tile below: with fewer large
// tiles than SMs the rest of the chip idles.
inline bool use_large(int large_tiles) { return large_tiles >= SEM_SMS; }

template <bool TA, bool TB, int EP>
sem_status gemm(const GemmArgs &g, cudaStream_t s) {
  if (use_large(tiles<GemmLarge>(g)))
    k_gemm<GemmLarge, TA, TB, EP><<<tiles<GemmLarge>(g), GT, 0, s>>>(g);
  else
    k_gemm<GemmSmall, TA, TB, EP><<<tiles<GemmSmall>(g), GT, 0, s>>>(g);
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

template <bool TA0, bool TB0, int EP0, bool TA1, bool TB1, int EP1>
sem_status gemm_pair(const GemmArgs &g0, const GemmArgs &g1, cudaStream_t s) {
  if (use_large(tiles<GemmLarge>(g0) + tiles<GemmLarge>(g1))) {
    const int n0 = tiles<GemmLarge>(g0);
    k_gemm_pair<GemmLarge, TA0, TB0, EP0, TA1, TB1, EP1><<<n0 + tiles<GemmLarge>(g1), GT, 0, s>>>(g0, g1, n0);
  } else {
    const int n0 = tiles<GemmSmall>(g0);
    k_gemm_pair<GemmSmall, TA0, TB0, EP0, TA1, TB1, EP1><<<n0 + tiles<GemmSmall>(g1), GT, 0, s>>>(g0, g1, n0);
  }
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

}  // namespace mlpg
