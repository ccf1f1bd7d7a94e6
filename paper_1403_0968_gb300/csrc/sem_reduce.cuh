// Deterministic block and grid reductions in FP64.
//
// A kernel that contributes to a dot product writes one FP64 partial per block; the block that
// finishes last (a ticket taken with atomicAdd after a memory fence) sums every partial in a
// fixed order and runs a small epilogue on the result.  The order of additions depends only on
// the grid size, so repeated solves give bit-identical scalars.
#pragma once

#include <cuda_runtime.h>

#include "sem_internal.h"

// Sum of v over the block (all threads must call; result valid in every thread).
template <int NT>
__device__ __forceinline__ double block_sum(double v, double *s_red /* >= 32 */) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int NW = (NT + 31) / 32;
  __syncthreads();
  if (lane == 0) s_red[warp] = v;
  __syncthreads();
  double t = 0.0;
  if (warp == 0) {
    t = lane < NW ? s_red[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) s_red[0] = t;
  }
  __syncthreads();
  t = s_red[0];
  __syncthreads();
  return t;
}

// FP32 -> FP64, exact, on the integer pipeline: GB300 runs FP64 instructions, conversions included,
// at about two lanes per cycle per SM, so a warp-wide one takes 16 cycles of the whole SM
__device__ __forceinline__ double widen_f64(float f) {
  const unsigned int b = __float_as_uint(f);
  const unsigned int ex = (b >> 23) & 0xFFu;
  if (ex == 0u) return (b << 1) ? (double)f : 0.0;  // zero; a subnormal takes the conversion
  const unsigned long long e64 = ex == 0xFFu ? 0x7FFull : (unsigned long long)(ex + 896u);
  return __longlong_as_double((long long)(((unsigned long long)(b & 0x80000000u) << 32) | (e64 << 52) |
                                          ((unsigned long long)(b & 0x7FFFFFu) << 29)));
}
__device__ __forceinline__ double widen_f64(double v) { return v; }

// Sum in FP64 of n values in shared memory by one warp (fixed order; result in every lane).  n / 32
// + 5 FP64 additions per warp, where block_sum spends 5 on every warp of the block: the sums of the
// CG step took longer than its vector updates that way (update kernel at 1.4e6 nodes 22 us).
template <typename T>
__device__ __forceinline__ double warp_sum(const T *s, int n) {
  const int lane = threadIdx.x & 31;
  double v = 0.0;
  for (int q = lane; q < n; q += 32) v += widen_f64(s[q]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum of nparts partials in global memory by one warp (L2 loads, fixed order; result in every lane).
__device__ __forceinline__ double warp_sum_partials(const double *partials, int nparts) {
  const int lane = threadIdx.x & 31;
  double v0 = 0.0, v1 = 0.0, v2 = 0.0, v3 = 0.0;
  int q = lane;
  for (; q + 96 < nparts; q += 128) {
    const double a = __ldcg(partials + q), b = __ldcg(partials + q + 32), c = __ldcg(partials + q + 64),
                 d = __ldcg(partials + q + 96);
    v0 += a, v1 += b, v2 += c, v3 += d;
  }
  for (; q < nparts; q += 32) v0 += __ldcg(partials + q);
  double v = (v0 + v1) + (v2 + v3);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Two-level sum of one value per block by one warp of each block (v: this block's, in lane 0): the
// groups of 256 blocks and then the groups are added in order by the warp that comes last.  Returns
// true in every lane of the very last one, with the total.  Called before the block's scatter: the
// fences then have no writes to wait for, and the block's other warps need not wait at all.
__device__ __forceinline__ bool warp_publish_2level(double v, double *partials, double *gpartials,
                                                    unsigned int *gtickets, unsigned int *ticket, double *total) {
  const unsigned int group = blockIdx.x / 256u, ngroups = (gridDim.x + 255u) / 256u;
  const unsigned int gsize = (gridDim.x - group * 256u) < 256u ? (gridDim.x - group * 256u) : 256u;
  const int lane = threadIdx.x & 31;
  int last = 0;
  if (lane == 0) {
    partials[blockIdx.x] = v;
    __threadfence();
    last = atomicAdd(&gtickets[group], 1u) == gsize - 1u;
  }
  // a shuffle alone does not order the lanes' memory accesses: the other lanes' loads come after lane 0's ticket
  __syncwarp();
  if (!__shfl_sync(0xffffffffu, last, 0)) return false;
  __threadfence();
  const double gsum = warp_sum_partials(partials + group * 256u, (int)gsize);
  if (lane == 0) {
    gtickets[group] = 0u;
    gpartials[group] = gsum;
    __threadfence();
    last = atomicAdd(ticket, 1u) == ngroups - 1u;
  }
  __syncwarp();
  if (!__shfl_sync(0xffffffffu, last, 0)) return false;
  __threadfence();
  *total = warp_sum_partials(gpartials, (int)ngroups);
  return true;
}

// p^T A p -> the CG step length, by one thread
__device__ __forceinline__ void cg_set_alpha(SemScalars *S, double pAp) {
  S->pAp = pAp;
  if (!(pAp > 0.0) || !isfinite(pAp) || !isfinite(S->rz)) {
    S->breakdown = 1;
    S->alpha = 0.0;
  } else {
    S->alpha = S->rz / pAp;
  }
  S->counter[0] = 0;
}

// Writes this block's partial; returns true in every thread of the one block that arrives last.
// `nparts` = number of blocks contributing.  The ticket counter is reset by the last block.
template <int NT>
__device__ __forceinline__ bool publish_partial(double v, double *partials, unsigned int *ticket, double *s_red,
                                                int *s_flag) {
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = v;
    __threadfence();
    const unsigned int t = atomicAdd(ticket, 1u);
    *s_flag = (t == gridDim.x - 1);
  }
  __syncthreads();
  const bool last = *s_flag != 0;
  if (last) __threadfence();
  return last;
}

// Called by every thread of the last block: fixed-order sum of partials[0..nparts).  The loads go
// to L2 (ld.global.cg: coherent with the other blocks' fenced stores, not cached in L1) and are
// independent, so many are in flight at once; four accumulators keep the order fixed.
template <int NT>
__device__ __forceinline__ double final_sum(const double *partials, int nparts, double *s_red) {
  double v0 = 0.0, v1 = 0.0, v2 = 0.0, v3 = 0.0;
  int q = threadIdx.x;
  for (; q + 3 * NT < nparts; q += 4 * NT) {
    v0 += __ldcg(partials + q);
    v1 += __ldcg(partials + q + NT);
    v2 += __ldcg(partials + q + 2 * NT);
    v3 += __ldcg(partials + q + 3 * NT);
  }
  for (; q < nparts; q += NT) v0 += __ldcg(partials + q);
  return block_sum<NT>((v0 + v1) + (v2 + v3), s_red);
}

// Two-level variant for grids of up to 256 * 4096 blocks: blocks are grouped by 256; the last
// block of each group (a ticket per group) sums the group's partials in order into gpartials[group];
// the block that completes the last group sums the group results in order.  Returns true in every
// thread of that final block, with the total in *total.  Deterministic for a given grid size.
// gtickets: one zeroed counter per group (reset here); ticket: the final counter (reset by caller).
template <int NT>
__device__ __forceinline__ bool publish_partial_2level(double v, double *partials, double *gpartials,
                                                       unsigned int *gtickets, unsigned int *ticket, double *s_red,
                                                       int *s_flag, double *total) {
  const unsigned int group = blockIdx.x / 256u, ngroups = (gridDim.x + 255u) / 256u;
  const unsigned int gsize = (gridDim.x - group * 256u) < 256u ? (gridDim.x - group * 256u) : 256u;
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = v;
    __threadfence();
    *s_flag = (atomicAdd(&gtickets[group], 1u) == gsize - 1u);
  }
  __syncthreads();
  if (*s_flag == 0) return false;
  __threadfence();
  const double gsum = final_sum<NT>(partials + group * 256u, (int)gsize, s_red);
  if (threadIdx.x == 0) {
    gtickets[group] = 0u;
    gpartials[group] = gsum;
    __threadfence();
    *s_flag = (atomicAdd(ticket, 1u) == ngroups - 1u);
  }
  __syncthreads();
  if (*s_flag == 0) return false;
  __threadfence();
  *total = final_sum<NT>(gpartials, (int)ngroups, s_red);
  return true;
}
