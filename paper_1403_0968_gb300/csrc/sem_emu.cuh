// FP64-accurate operator apply in double-float arithmetic (SEM_FP64_EMU).
//
// Same operator and the same five-phase element schedule as the FP64/FP32 kernel
// (sem_apply_kernel.cuh; arXiv 1403.0968 §4.2.1, sum-factorised stiffness display), but every
// value is carried as an unevaluated pair of FP32 numbers (hi, lo) with |lo| <= ulp(hi)/2, because
// GB300 executes FP64 FMAs at 1/61 of the FP32 rate.  Inputs and outputs stay FP64:
//   * u (FP64) is scaled per element by an exact power of two, 2^(1023 - e) with e the largest
//     biased FP64 exponent among the element's gathered values, so that the element's largest
//     |u| lies in [1, 2) whatever the scale of u; y_e is scaled back by the inverse power of two
//     when it is rebuilt as FP64 (exact).  The scaled value is split into (hi, lo) by bit
//     manipulation: hi keeps the top 24 significand bits, lo the next 24 (integer instructions,
//     not FP64 conversions);
//   * the factors are stored as (hi, lo) pairs by set-up, D as (hi, lo) launch parameters;
//   * each sum  sum_m a_m b_m  is formed with exact products (p = a_hi b_hi and its FMA
//     remainder, the published TwoProduct transformation) and Knuth's TwoSum on the high parts;
//     every low-order term goes into one FP32 compensation, and the pair is renormalised at the
//     end (Fast2Sum).  The error is about 2^-44 of the sum of |terms| per output (double-float
//     accuracy after Dekker 1971 / Ogita-Rump-Oishi 2005);
//   * y = hi + lo is rebuilt as FP64 (one FP64 add per node) and scatter-added with FP64 atomics.
// Accuracy: u of any FP64 magnitude (FP64 subnormals are flushed to zero).  Within an element,
// entries smaller than 2^-74 of its largest |u| keep FP32 relative accuracy and entries below
// 2^-126 of it are flushed: absolute errors below 2^-98 of the element's largest |u|.  The
// factors must lie within 2^-60 .. 2^60 (checked at set-up, which refuses SEM_FEAT_EMU otherwise),
// so that every intermediate product keeps its low word in the FP32 normal range.
//
// This header holds the kernel and its launcher; sem_emu_*.cu instantiate the launcher for ranges of
// orders (to spread the compile time over translation units) and sem_emu.cu dispatches by order.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "sem_internal.h"
#include "sem_reduce.cuh"
#include "sem_tma.cuh"

namespace semu {

// ---- double <-> double-float conversions (integer pipeline) ----
// biased FP64 exponent of u (0 for zeros and subnormals)
__device__ __forceinline__ int f64_biased_exp(double u) {
  return (int)(((unsigned int)(__double_as_longlong(u) >> 32) >> 20) & 0x7FFu);
}

// 2^k as a double, for -1022 <= k <= 1023
__device__ __forceinline__ double exp2i(int k) { return __longlong_as_double((long long)(k + 1023) << 52); }

// atomicMax of v into *slot for the element this thread belongs to: a warp whose lanes all belong
// to one element reduces first and issues one atomic (a shared-memory atomic from every lane to
// the same address would serialise 32 ways)
__device__ __forceinline__ void element_max(int *slot, int v, int es) {
  const int es0 = __shfl_sync(0xffffffffu, es, 0), es31 = __shfl_sync(0xffffffffu, es, 31);
  if (es0 == es31) {
    v = __reduce_max_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) atomicMax(slot, v);
  } else {
    atomicMax(slot, v);
  }
}

// element coordinates (ex, ey, ez) of element e of an sx x sy x sz box, in 32-bit arithmetic when
// the element count allows (64-bit division costs several times more instructions)
__device__ __forceinline__ void box_coords(int64_t e, int sx, int sy, int64_t E, int64_t &ex, int64_t &ey,
                                           int64_t &ez) {
  if (E <= 0x7fffffffll) {
    const uint32_t e32 = (uint32_t)e, exy = e32 / (uint32_t)sx;
    ex = e32 - exy * (uint32_t)sx;
    ey = exy % (uint32_t)sy;
    ez = exy / (uint32_t)sy;
  } else {
    const int64_t exy = e / sx;
    ex = e - exy * sx;
    ey = exy % sy;
    ez = exy / sy;
  }
}

// (hi, lo) of u * 2^shift (exact scaling; shift chosen so that the result is below 2); FP64
// subnormals and results below 2^-126 are flushed to zero
__device__ __forceinline__ float2 split_f64(double u, int shift) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(u);
  const unsigned int hw = (unsigned int)(b >> 32), lw = (unsigned int)b;
  const int ex0 = (int)((hw >> 20) & 0x7FFu);
  const int ex = ex0 == 0 ? 0 : ex0 + shift;
  const unsigned int sign = hw & 0x80000000u;
  float h = 0.0f, l = 0.0f;
  if (ex >= 897 && ex <= 1150) {
    const unsigned int m23 = ((hw & 0xFFFFFu) << 3) | (lw >> 29);  // significand bits 51..29
    h = __uint_as_float(sign | ((unsigned int)(ex - 896) << 23) | m23);
    const unsigned int mlo = lw & 0x1FFFFFFFu;  // significand bits 28..0, weight 2^(ex-1075)
    if (mlo != 0u && ex >= 949) {
      const float scale = __uint_as_float((unsigned int)(ex - 948) << 23);
      l = __uint_as_float(__float_as_uint(__fmul_rn(__uint2float_rn(mlo), scale)) | sign);
    }
  } else if (ex > 1150) {
    h = __double2float_rn(u);  // overflow, inf or nan (not expected on this path)
  }
  return make_float2(h, l);
}

__device__ __forceinline__ double f32_as_f64(float f) {
  const unsigned int b = __float_as_uint(f);
  const unsigned int ex = (b >> 23) & 0xFFu;
  if (ex == 0u) return 0.0;
  const unsigned long long e64 = ex == 0xFFu ? 0x7FFull : (unsigned long long)(ex + 896u);
  const unsigned long long r =
      ((unsigned long long)(b & 0x80000000u) << 32) | (e64 << 52) | ((unsigned long long)(b & 0x7FFFFFu) << 29);
  return __longlong_as_double((long long)r);
}

__device__ __forceinline__ double df_to_f64(float2 v) { return f32_as_f64(v.x) + f32_as_f64(v.y); }

// ---- double-float dot-product accumulation: (s, c) += (dh + dl) * (v.x + v.y) ----
__device__ __forceinline__ void dacc_first(float &s, float &c, float dh, float dl, float2 v) {
  s = __fmul_rn(dh, v.x);
  float e = __fmaf_rn(dh, v.x, -s);
  e = __fmaf_rn(dh, v.y, e);
  c = __fmaf_rn(dl, v.x, e);
}

__device__ __forceinline__ void dacc(float &s, float &c, float dh, float dl, float2 v) {
  const float p = __fmul_rn(dh, v.x);
  float e = __fmaf_rn(dh, v.x, -p);
  e = __fmaf_rn(dh, v.y, e);
  e = __fmaf_rn(dl, v.x, e);
  const float t = __fadd_rn(s, p);  // TwoSum(s, p)
  const float z = __fsub_rn(t, s);
  const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));
  s = t;
  c = __fadd_rn(c, __fadd_rn(err, e));
}

// (s, c) += v
__device__ __forceinline__ void dadd(float &s, float &c, float2 v) {
  const float t = __fadd_rn(s, v.x);
  const float z = __fsub_rn(t, s);
  const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(v.x, z));
  s = t;
  c = __fadd_rn(c, __fadd_rn(err, v.y));
}

__device__ __forceinline__ float2 dnorm(float s, float c) {
  const float h = __fadd_rn(s, c);
  return make_float2(h, __fsub_rn(c, __fsub_rn(h, s)));
}

// (s1 + c1) + sgn (s2 + c2), normalised
__device__ __forceinline__ float2 dcombine(float s1, float c1, float s2, float c2, bool minus) {
  if (minus) {
    s2 = -s2;
    c2 = -c2;
  }
  const float t = __fadd_rn(s1, s2);
  const float z = __fsub_rn(t, s1);
  const float err = __fadd_rn(__fsub_rn(s1, __fsub_rn(t, z)), __fsub_rn(s2, z));
  return dnorm(t, __fadd_rn(__fadd_rn(c1, c2), err));
}

// v[a] + sgn v[b] as an (unnormalised) pair: TwoSum of the high parts, low parts added
__device__ __forceinline__ float2 dpm(float2 va, float2 vb, bool minus) {
  const float bx = minus ? -vb.x : vb.x, by = minus ? -vb.y : vb.y;
  const float t = __fadd_rn(va.x, bx);
  const float z = __fsub_rn(t, va.x);
  const float err = __fadd_rn(__fsub_rn(va.x, __fsub_rn(t, z)), __fsub_rn(bx, z));
  return make_float2(t, __fadd_rn(__fadd_rn(va.y, by), err));
}

// ---- the same operations on two independent values at once (packed FP32, f32x2) ----
// Two FP32 operations per instruction at the scalar rate per lane: the packed forms halve the issue
// slots and round exactly as the scalar ones.
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }

// (s, c) = (dh + dl) * (vh + vl) for both halves
__device__ __forceinline__ void dacc2_first(float2 &s, float2 &c, float2 dh, float2 dl, float2 vh, float2 vl) {
  s = __fmul2_rn(dh, vh);
  float2 e = __ffma2_rn(dh, vh, neg2(s));
  e = __ffma2_rn(dh, vl, e);
  c = __ffma2_rn(dl, vh, e);
}

// (s, c) += (dh + dl) * (vh + vl)
__device__ __forceinline__ void dacc2(float2 &s, float2 &c, float2 dh, float2 dl, float2 vh, float2 vl) {
  const float2 p = __fmul2_rn(dh, vh);
  float2 e = __ffma2_rn(dh, vh, neg2(p));
  e = __ffma2_rn(dh, vl, e);
  e = __ffma2_rn(dl, vh, e);
  const float2 t = __fadd2_rn(s, p);  // TwoSum(s, p)
  const float2 z = sub2(t, s);
  const float2 err = __fadd2_rn(sub2(s, sub2(t, z)), sub2(p, z));
  s = t;
  c = __fadd2_rn(c, __fadd2_rn(err, e));
}

template <int NP>
struct DPair {
  float hi[NP * NP], lo[NP * NP];  // D[i][m] at i * NP + m
};

// Even-odd form of a centro-antisymmetric line operator M (M[N-i][N-m] = -M[i][m], true for the
// GLL derivative matrix and its transpose): with e_m = v_m + v_{N-m}, o_m = v_m - v_{N-m} (m < H),
//   p_i = sum_m A+[i][m] o_m,  q_i = sum_m A-[i][m] e_m,  out_i = p_i + q_i,  out_{N-i} = p_i - q_i,
// A+-[i][m] = (M[i][m] +- M[N-i][m]) / 2, H = n / 2.  Two H x H products replace one n x n
// product; for odd n the middle node adds one column and one row of H terms (see df_line).
template <int NP>
struct EvenOdd {
  static constexpr int H = NP / 2 > 0 ? NP / 2 : 1;
  // pairs (A+, A-)[i][m] at i * H + m, high and low words, for M = D (index 0) and M = D^T (index 1)
  float2 hi[2][H * H], lo[2][H * H];
};

template <int NP>
struct EmuParams {
  int64_t E;
  int sx, sy, sz;
  int64_t gxs, gys, gzs;
  int bc;
  const double *u;
  double *y;
  const float *Gf;  // [E][gs12]: factor f hi at 2f n3 + p, lo at (2f+1) n3 + p
  int64_t gs;
  const float *wJa;  // [E][2][n3] or NULL
  const int32_t *glo;
  const uint8_t *mask;
  double *partials;
  double *gpartials;
  unsigned int *gtickets;
  SemScalars *scal;
  int *err;             // set to 1 if a bounded wait gave up
  uint32_t wait_polls;  // polls of the staged copy's barrier before the wait gives up
  DPair<NP> D;
  EvenOdd<NP> EO;
};

// Forms of the kernel by problem size (emu_form): fuller blocks for a chip full of them, one or two elements
// per block without register floors, and the same in scalar arithmetic.
enum EmuForm { EMU_FULL, EMU_SMALL, EMU_SCALAR };

// Whether an order runs its line products and factor scaling in packed form (DOT: with the fused
// reduction of a CG step, whose registers come on top).  Measured, GDOF/s at 1.6e7 nodes, scalar /
// packed: plain N = 2 59 / 57, 4 52 / 51, 10 32 / 30, 7 42 / 44.5, 11 20.6 / 24.6, 15 17 / 21; DOT
// N = 5 43 / 37, 6 36 / 36, 7 42 / 40, 8 35.5 / 28, 9 27 / 30, 15 14.5 / 21.
__host__ __device__ constexpr bool emu_packed(int NP, bool dot, EmuForm form) {
  if (form == EMU_SCALAR) return false;
  return NP == 4 || NP == 10 || NP >= 12 || (!dot && NP >= 6 && NP <= 9);
}
// whether the even and odd parts of a line are formed together too (N = 15, whose 128 registers do not hold
// both, one after the other: 20% faster in the build the choice was made in)
__host__ __device__ constexpr bool emu_packed_parts(int NP) { return NP <= 14; }

// out = M v for one line, M = D (TRANS false) or D^T (TRANS true), in double-float: the odd part
// (p_i, from o) and the even part (q_i, from e), accumulated together in the two halves of packed
// operations or one after the other.  Odd n adds the middle node mid = N / 2: M[i][mid] v_mid joins
// q_i (mirrored with a sign like q), and the middle row, M[mid][mid] = 0 and
// M[mid][N-m] = -M[mid][m], is sum_m M[mid][m] o_m.
template <int NP, bool TRANS, bool PK>
__device__ __forceinline__ void df_line(const EmuParams<NP> &P, const float2 (&v)[NP], float2 (&out)[NP]) {
  constexpr int H = NP / 2, MID = NP / 2, T = TRANS ? 1 : 0;
  const float2 *ah = P.EO.hi[T], *al = P.EO.lo[T];
  float2 oeh[H], oel[H];  // (o, e): high words, low words
#pragma unroll
  for (int m = 0; m < H; ++m) {
    const float2 va = v[m], vb = v[NP - 1 - m];
    if constexpr (PK && emu_packed_parts(NP)) {  // va - vb and va + vb at once, as dpm
      const float2 a2 = make_float2(va.x, va.x), b2 = make_float2(-vb.x, vb.x);
      const float2 t = __fadd2_rn(a2, b2), z = sub2(t, a2);
      const float2 err = __fadd2_rn(sub2(a2, sub2(t, z)), sub2(b2, z));
      oeh[m] = t;
      oel[m] = __fadd2_rn(__fadd2_rn(make_float2(va.y, va.y), make_float2(-vb.y, vb.y)), err);
    } else {
      const float2 e = dpm(va, vb, false), o = dpm(va, vb, true);
      oeh[m] = make_float2(o.x, e.x);
      oel[m] = make_float2(o.y, e.y);
    }
  }
#pragma unroll
  for (int i = 0; i < H; ++i) {
    float2 s, c;
    if constexpr (PK) {
      dacc2_first(s, c, ah[i * H], al[i * H], oeh[0], oel[0]);
#pragma unroll
      for (int m = 1; m < H; ++m) dacc2(s, c, ah[i * H + m], al[i * H + m], oeh[m], oel[m]);
    } else {
      dacc_first(s.x, c.x, ah[i * H].x, al[i * H].x, make_float2(oeh[0].x, oel[0].x));
      dacc_first(s.y, c.y, ah[i * H].y, al[i * H].y, make_float2(oeh[0].y, oel[0].y));
#pragma unroll
      for (int m = 1; m < H; ++m) {
        dacc(s.x, c.x, ah[i * H + m].x, al[i * H + m].x, make_float2(oeh[m].x, oel[m].x));
        dacc(s.y, c.y, ah[i * H + m].y, al[i * H + m].y, make_float2(oeh[m].y, oel[m].y));
      }
    }
    if constexpr (NP % 2 == 1) {
      const int qm = TRANS ? MID * NP + i : i * NP + MID;  // M[i][mid]
      dacc(s.y, c.y, P.D.hi[qm], P.D.lo[qm], v[MID]);
    }
    out[i] = dcombine(s.x, c.x, s.y, c.y, false);
    out[NP - 1 - i] = dcombine(s.x, c.x, s.y, c.y, true);
  }
  if constexpr (NP % 2 == 1) {
    float s, c;
    dacc_first(s, c, P.D.hi[TRANS ? MID : MID * NP], P.D.lo[TRANS ? MID : MID * NP], make_float2(oeh[0].x, oel[0].x));
#pragma unroll
    for (int m = 1; m < H; ++m) {
      const int q = TRANS ? m * NP + MID : MID * NP + m;  // M[mid][m]
      dacc(s, c, P.D.hi[q], P.D.lo[q], make_float2(oeh[m].x, oel[m].x));
    }
    out[MID] = dnorm(s, c);
  }
}

// elements per block: with the factor block staged, and with factors read directly (there the block's
// last warp is filled up as far as shared memory lets two blocks or more onto an SM: N = 5 with 7
// elements 48 GDOF/s against 46 with 5, 6 with 5 43 / 36 with 3, 8 with 3 36.5 / 33.5 with 1, 9 with
// 3 31.6 / 29.6 with 1)
__host__ __device__ constexpr int emu_eb_staged(int NP) {
  return NP <= 2 ? 32 : NP == 3 ? 14 : NP == 4 ? 8 : NP == 5 ? 5 : NP == 6 ? 3 : NP <= 8 ? 2 : 1;
}
__host__ __device__ constexpr int emu_eb(int NP, EmuForm form) {
  return form != EMU_FULL ? emu_eb_staged(NP) : NP == 6 ? 7 : NP == 7 ? 5 : (NP == 9 || NP == 10) ? 3 : NP == 12 ? 2 : emu_eb_staged(NP);
}

template <int NP, bool STAGE, bool DOT, EmuForm FORM>
struct EmuCfg {
  static constexpr int NP2 = NP * NP, NP3 = NP2 * NP, EB = emu_eb(NP, STAGE ? EMU_SMALL : FORM), NT = NP2 * EB;
  static constexpr int RS = NP | 1, PS = NP * RS, BUF = NP * PS;
  static constexpr int GS = (12 * NP3 + 3) / 4 * 4;  // factor block of one element (floats)
  // byte offsets: [factor block (TMA, offset 0)] [value buffers] [reduction slots, mbarrier]
  static constexpr size_t BUF_OFF = STAGE ? (size_t)EB * GS * sizeof(float) : 0;
  static constexpr size_t RED_OFF = (BUF_OFF + (size_t)EB * 3 * BUF * sizeof(float2) + 15) / 16 * 16;
  // reduction slots (one double per thread with the fused reduction), mbarrier, per-element exponent
  // maxima (EB ints)
  static constexpr size_t RED_SIZE = DOT ? ((size_t)NT * 8 + 15) / 16 * 16 : 0;
  static constexpr size_t SMEM = RED_OFF + RED_SIZE + 16 + (size_t)EB * 4;
};
// the factor block can be staged in shared memory by one bulk (TMA) copy when it fits
__host__ __device__ constexpr bool emu_stage_fits(int NP) {
  return (size_t)emu_eb_staged(NP) * ((12 * NP * NP * NP + 3) / 4 * 4 * sizeof(float) +
                                      3 * NP * NP * (NP | 1) * sizeof(float2)) <= 112 * 1024;
}

// Blocks per SM the register allocation is held to; 0 = no floor (an explicit 1 lets the compiler
// take far more registers).  Measured for the packed forms over floors of 0..7.
__host__ __device__ constexpr int emu_min_blocks(int NP, bool stage, bool dot, EmuForm form) {
  if (form == EMU_SMALL) return 0;
  if (stage || form == EMU_SCALAR) return NP == 10 ? 4 : NP == 11 ? 3 : NP >= 12 ? 2 : 0;
  if (dot) return NP == 4 ? 7 : NP == 10 || NP >= 12 ? 2 : 0;
  return NP == 4 ? 7 : NP == 6 || NP == 7 ? 4 : NP == 8 ? 5 : NP == 9 || NP == 11 ? 3 : NP >= 10 ? 2 : 0;
}

// How the line products of phases 1 and 3 are laid out in code: 0 three inlined line products per
// phase; 2 the r- and s-lines through one loop body, the t-line (the thread's column, in
// registers) inlined; 3 all three directions through one loop body (the t-line read from shared
// memory).  The loops shorten the code (fewer instruction-fetch stalls) at some addressing cost.
// Packed forms, GDOF/s at 1.6e7 nodes, modes 0 / 2 / 3: N = 3 61 / 59 / 55, 5 48 / 47 / 45, 6 41 / 43 /
// 40, 7 41.5 / 44.5 / 40, 8 34.5 / 36.5 / 35, 9 31.6 / 31.0 / 30.8, 11 23.5 / 24.6 / 23.7, 12 23.5 / 19 /
// 19, 13 16 / 17 / 20; mode 3 also leads at N = 14 and 15 (20.5 and 21.3 as chosen here).
__host__ __device__ constexpr int emu_loop_mode(int NP, EmuForm form) {
  if (form == EMU_SCALAR) return NP == 7 || NP == 10 ? 0 : 2;
  return NP >= 14 ? 3 : (NP == 7 || NP == 8 || NP == 9 || NP == 11 || NP == 12) ? 2 : 0;
}

// the block's factors asked for in L2 at its start by one bulk prefetch (one element per block and
// two blocks per SM leave the loads exposed: N = 13 16.9 -> 19.9 GDOF/s, 15 +8%; slower below)
__host__ __device__ constexpr bool emu_prefetch(int NP) { return NP >= 14; }

template <int NP, bool BOXM, bool STAGE, bool DOT, EmuForm FORM>
__global__ void __launch_bounds__(EmuCfg<NP, STAGE, DOT, FORM>::NT, emu_min_blocks(NP, STAGE, DOT, FORM)) k_apply_emu(const EmuParams<NP> P) {
  using C = EmuCfg<NP, STAGE, DOT, FORM>;
  constexpr int N = NP - 1, NP2 = C::NP2, NP3 = C::NP3, EB = C::EB, NT = C::NT, RS = C::RS, PS = C::PS,
                BUF = C::BUF, GS = C::GS;
  constexpr bool PK = emu_packed(NP, DOT, FORM);
  extern __shared__ __align__(128) unsigned char smem_raw[];
  static_assert(C::BUF_OFF % 16 == 0 && C::RED_OFF % 16 == 0, "shared-memory alignment");
  float *sG = reinterpret_cast<float *>(smem_raw);  // TMA destination: 16-byte aligned at offset 0
  float2 *sbuf = reinterpret_cast<float2 *>(smem_raw + C::BUF_OFF);
  double *s_red = reinterpret_cast<double *>(smem_raw + C::RED_OFF);
  uint64_t *bar = reinterpret_cast<uint64_t *>(smem_raw + C::RED_OFF + C::RED_SIZE);
  int *s_emax = reinterpret_cast<int *>(bar + 2);  // [EB] largest biased FP64 exponent of each element's u

  if constexpr (DOT) {  // a step of a solve: nothing to do once the iteration has stopped
    dependent_wait();
    if (P.scal->converged || P.scal->breakdown) return;
  }
  const int tid = threadIdx.x;
  const int es = tid / NP2, t2 = tid - es * NP2, a = t2 % NP, b = t2 / NP;
  if (t2 == 0) s_emax[es] = 1;
  const int64_t e0 = (int64_t)blockIdx.x * EB;
  const int64_t e = e0 + es;
  const bool active = e < P.E;
  float2 *su = sbuf + es * 3 * BUF, *sr = su + BUF, *ss = sr + BUF;
  if constexpr (STAGE) {
    if (tid == 0) mbar_init(bar, 1);
  }
  __syncthreads();  // s_emax initialised (and the mbarrier)
  if constexpr (STAGE) {
    if (tid == 0) {
      const int64_t nel = (P.E - e0) < EB ? (P.E - e0) : EB;
      tma_load_1d(sG, P.Gf + e0 * P.gs, (uint32_t)(nel * P.gs * sizeof(float)), bar);
    }
  }

  if constexpr (!STAGE && emu_prefetch(NP)) {
    if (tid == 0) {
      const int64_t nel = (P.E - e0) < EB ? (P.E - e0) : EB;
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(P.Gf + e0 * P.gs),
                   "r"((uint32_t)(nel * P.gs * sizeof(float)))
                   : "memory");
    }
  }

  // ---- phase 0: gather and split u ----
  int64_t gbase = 0;
  uint32_t dirbits = 0;
  float2 uc[NP];
  double ud[NP];
  if constexpr (BOXM) {
    const int64_t plane = P.gxs * P.gys;
    if (active) {
      int64_t ex, ey, ez;
      box_coords(e, P.sx, P.sy, P.E, ex, ey, ez);
      const int64_t I = ex * N + a, J = ey * N + b;
      gbase = I + P.gxs * (J + P.gys * (ez * N));
      if (P.bc == SEM_BC_BOX) {
        if (I == 0 || I == P.gxs - 1 || J == 0 || J == P.gys - 1) dirbits = (1u << NP) - 1u;
        if (ez == 0) dirbits |= 1u;
        if (ez == P.sz - 1) dirbits |= 1u << N;
      }
    } else {
      dirbits = (1u << NP) - 1u;
    }
    const double *up = P.u + gbase;
#pragma unroll
    for (int k = 0; k < NP; ++k) ud[k] = ((dirbits >> k) & 1u) ? 0.0 : up[k * plane];
  } else {
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      int64_t g = 0;
      bool d = !active;
      if (active) {
        if (P.glo) {
          g = P.glo[e * NP3 + t2 + NP2 * k];
        } else {
          const int64_t ex = e % P.sx, ey = (e / P.sx) % P.sy, ez = e / ((int64_t)P.sx * P.sy);
          g = (ex * N + a) + P.gxs * ((ey * N + b) + P.gys * (ez * N + k));
        }
        if (P.bc == SEM_BC_BOX) {
          const int64_t I = g % P.gxs, J = (g / P.gxs) % P.gys, K = g / (P.gxs * P.gys);
          d = I == 0 || J == 0 || K == 0 || I == P.gxs - 1 || J == P.gys - 1 || K == P.gzs - 1;
        } else if (P.bc == SEM_BC_MASK) {
          d = P.mask[g] != 0;
        }
      }
      dirbits |= (d ? 1u : 0u) << k;
      ud[k] = d ? 0.0 : P.u[g];
    }
  }
  // element scale: the largest exponent over the element's gathered values
  {
    int emx = 1;
#pragma unroll
    for (int k = 0; k < NP; ++k) emx = max(emx, f64_biased_exp(ud[k]));
    element_max(&s_emax[es], emx, es);
  }
  __syncthreads();
  const int shift = 1023 - s_emax[es];  // u * 2^shift has its element maximum in [1, 2)
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    uc[k] = split_f64(ud[k], shift);
    su[k * PS + b * RS + a] = uc[k];
  }
  __syncthreads();

  // ---- phase 1: gradients ----
  float2 wt[NP];
  if constexpr (emu_loop_mode(NP, FORM) == 3) {
    // direction 0: the r-line (j = a, k = b) into sr, 1: the s-line (i = a, k = b) into ss, 2: the
    // t-line (the column) into registers; the same base and stride address input and output
#pragma unroll 1
    for (int dir = 0; dir < 3; ++dir) {
      const int ib = dir == 0 ? b * PS + a * RS : dir == 1 ? b * PS + a : b * RS + a;
      const int is = dir == 0 ? 1 : dir == 1 ? RS : PS;
      float2 row[NP], out[NP];
#pragma unroll
      for (int m = 0; m < NP; ++m) row[m] = su[ib + m * is];
      df_line<NP, false, PK>(P, row, out);
      if (dir == 2) {
#pragma unroll
        for (int k = 0; k < NP; ++k) wt[k] = out[k];
      } else {
        float2 *dst = dir == 0 ? sr : ss;
#pragma unroll
        for (int i = 0; i < NP; ++i) dst[ib + i * is] = out[i];
      }
    }
  } else if constexpr (emu_loop_mode(NP, FORM) == 2) {
    // the t-line (the column, in registers) inlined; the r-line (j = a, k = b) into sr and the
    // s-line (i = a, k = b) into ss through one loop body (the same base and stride address input
    // and output)
    df_line<NP, false, PK>(P, uc, wt);  // u_t of the column
#pragma unroll 1
    for (int dir = 0; dir < 2; ++dir) {
      const int ib = dir == 0 ? b * PS + a * RS : b * PS + a;
      const int is = dir == 0 ? 1 : RS;
      float2 *dst = dir == 0 ? sr : ss;
      float2 row[NP], out[NP];
#pragma unroll
      for (int m = 0; m < NP; ++m) row[m] = su[ib + m * is];
      df_line<NP, false, PK>(P, row, out);
#pragma unroll
      for (int i = 0; i < NP; ++i) dst[ib + i * is] = out[i];
    }
  } else {
    df_line<NP, false, PK>(P, uc, wt);  // u_t of the column
    float2 row[NP], out[NP];
#pragma unroll
    for (int m = 0; m < NP; ++m) row[m] = su[b * PS + a * RS + m];
    df_line<NP, false, PK>(P, row, out);
#pragma unroll
    for (int i = 0; i < NP; ++i) sr[b * PS + a * RS + i] = out[i];
#pragma unroll
    for (int m = 0; m < NP; ++m) row[m] = su[b * PS + m * RS + a];
    df_line<NP, false, PK>(P, row, out);
#pragma unroll
    for (int j = 0; j < NP; ++j) ss[b * PS + j * RS + a] = out[j];
  }

  // ---- phase 2: geometric factors ----
  bool ok = true;
  if constexpr (STAGE) ok = mbar_wait(bar, 0, P.wait_polls);
  if (__syncthreads_or(!ok)) {
    // record the timeout, wait (bounded) for this block's own copy, leave without scattering
    if (tid == 0) {
      if (P.err) atomicOr(P.err, 1);
      mbar_wait(bar, 0);
    }
    return;
  }
  const float *Ge = STAGE ? (sG + es * GS + t2) : (P.Gf + (active ? e : 0) * P.gs + t2);
  auto load_g = [&](int k, float(&gh)[6], float(&gl)[6]) {
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      gh[f] = (STAGE || active) ? Ge[(2 * f) * NP3 + k * NP2] : 0.f;
      gl[f] = (STAGE || active) ? Ge[(2 * f + 1) * NP3 + k * NP2] : 0.f;
    }
  };
  // two nodes of the column at a time, one in each half of the packed operations
  constexpr int KP = PK ? NP / 2 * 2 : 0;
#pragma unroll
  for (int k = 0; k < KP; k += 2) {
    const int q0 = k * PS + b * RS + a, q1 = q0 + PS;
    float g0h[6], g0l[6], g1h[6], g1l[6];
    load_g(k, g0h, g0l);
    load_g(k + 1, g1h, g1l);
    const float2 r0 = sr[q0], r1 = sr[q1], s0 = ss[q0], s1 = ss[q1], t0 = wt[k], t1 = wt[k + 1];
    const float2 vh[3] = {make_float2(r0.x, r1.x), make_float2(s0.x, s1.x), make_float2(t0.x, t1.x)};
    const float2 vl[3] = {make_float2(r0.y, r1.y), make_float2(s0.y, s1.y), make_float2(t0.y, t1.y)};
    constexpr int F[3][3] = {{0, 1, 2}, {1, 3, 4}, {2, 4, 5}};
    float2 w0[3], w1[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      float2 s, c;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const float2 gh = make_float2(g0h[F[r][d]], g1h[F[r][d]]), gl = make_float2(g0l[F[r][d]], g1l[F[r][d]]);
        if (d == 0)
          dacc2_first(s, c, gh, gl, vh[d], vl[d]);
        else
          dacc2(s, c, gh, gl, vh[d], vl[d]);
      }
      w0[r] = dnorm(s.x, c.x);
      w1[r] = dnorm(s.y, c.y);
    }
    sr[q0] = w0[0], sr[q1] = w1[0];
    ss[q0] = w0[1], ss[q1] = w1[1];
    wt[k] = w0[2], wt[k + 1] = w1[2];
  }
#pragma unroll
  for (int k = KP; k < NP; ++k) {  // one node at a time: the last of an odd column, or all
    const int q = k * PS + b * RS + a;
    float gh[6], gl[6];
    load_g(k, gh, gl);
    const float2 ur = sr[q], us = ss[q], ut = wt[k];
    float s, c;
    dacc_first(s, c, gh[0], gl[0], ur);
    dacc(s, c, gh[1], gl[1], us);
    dacc(s, c, gh[2], gl[2], ut);
    sr[q] = dnorm(s, c);
    dacc_first(s, c, gh[1], gl[1], ur);
    dacc(s, c, gh[3], gl[3], us);
    dacc(s, c, gh[4], gl[4], ut);
    ss[q] = dnorm(s, c);
    dacc_first(s, c, gh[2], gl[2], ur);
    dacc(s, c, gh[4], gl[4], us);
    dacc(s, c, gh[5], gl[5], ut);
    wt[k] = dnorm(s, c);
  }
  float2 yt[NP];
  if constexpr (emu_loop_mode(NP, FORM) == 3) {
    __syncthreads();
    // ---- phase 3: transposed contractions: 0 the r-line of sr, 1 the s-line of ss (in place),
    // 2 the column w_t in registers ----
#pragma unroll 1
    for (int dir = 0; dir < 3; ++dir) {
      const int ib = dir == 0 ? b * PS + a * RS : dir == 1 ? b * PS + a : 0;
      const int is = dir == 0 ? 1 : dir == 1 ? RS : 0;
      float2 *buf = dir == 1 ? ss : sr;
      float2 row[NP], out[NP];
#pragma unroll
      for (int m = 0; m < NP; ++m) row[m] = dir == 2 ? wt[m] : buf[ib + m * is];
      df_line<NP, true, PK>(P, row, out);
      if (dir == 2) {
#pragma unroll
        for (int k = 0; k < NP; ++k) yt[k] = out[k];
      } else {
#pragma unroll
        for (int i = 0; i < NP; ++i) buf[ib + i * is] = out[i];
      }
    }
  } else if constexpr (emu_loop_mode(NP, FORM) == 2) {
    df_line<NP, true, PK>(P, wt, yt);  // D^T w_t of the column
    __syncthreads();
    // ---- phase 3: transposed contractions: 0 the r-line of sr, 1 the s-line of ss (in place) ----
#pragma unroll 1
    for (int dir = 0; dir < 2; ++dir) {
      const int ib = dir == 0 ? b * PS + a * RS : b * PS + a;
      const int is = dir == 0 ? 1 : RS;
      float2 *buf = dir == 0 ? sr : ss;
      float2 row[NP], out[NP];
#pragma unroll
      for (int m = 0; m < NP; ++m) row[m] = buf[ib + m * is];
      df_line<NP, true, PK>(P, row, out);
#pragma unroll
      for (int i = 0; i < NP; ++i) buf[ib + i * is] = out[i];
    }
  } else {
    df_line<NP, true, PK>(P, wt, yt);  // D^T w_t of the column
    __syncthreads();

    // ---- phase 3: transposed r and s contractions ----
    float2 row[NP], out[NP];
#pragma unroll
    for (int m = 0; m < NP; ++m) row[m] = sr[b * PS + a * RS + m];
    df_line<NP, true, PK>(P, row, out);
#pragma unroll
    for (int i = 0; i < NP; ++i) sr[b * PS + a * RS + i] = out[i];
#pragma unroll
    for (int m = 0; m < NP; ++m) row[m] = ss[b * PS + m * RS + a];
    df_line<NP, true, PK>(P, row, out);
#pragma unroll
    for (int j = 0; j < NP; ++j) ss[b * PS + j * RS + a] = out[j];
  }
  __syncthreads();

  // ---- phase 4: assemble, convert to FP64, scatter ----
  const int64_t plane = P.gxs * P.gys;
  const bool ij_interior = (a > 0) && (a < N) && (b > 0) && (b < N) && !P.glo;
  const double unscale = exp2i(-shift);  // undoes the element's scaling of u (exact)
  auto node_of = [&](int k) -> int64_t {
    if constexpr (BOXM) {
      return gbase + k * plane;
    } else {
      if (P.glo) return P.glo[e * NP3 + t2 + NP2 * k];
      const int64_t ex = e % P.sx, ey = (e / P.sx) % P.sy, ez = e / ((int64_t)P.sx * P.sy);
      return (ex * N + a) + P.gxs * ((ey * N + b) + P.gys * (ez * N + k));
    }
  };
  if constexpr (DOT) {
    // (u, y) of this column in double-float; the scaled values carry the element's scale twice.  One
    // warp adds the block's values and publishes them before its scatter.
    float dps = 0.f, dpc = 0.f;
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      const int q = k * PS + b * RS + a;
      float s = yt[k].x, c = yt[k].y;
      dadd(s, c, sr[q]);
      dadd(s, c, ss[q]);
      if (P.wJa && active) {
        const int64_t o = e * 2 * NP3 + t2 + NP2 * k;
        dacc(s, c, P.wJa[o], P.wJa[o + NP3], uc[k]);
      }
      yt[k] = dnorm(s, c);
      if (!((dirbits >> k) & 1u)) dacc(dps, dpc, uc[k].x, uc[k].y, yt[k]);
    }
    s_red[tid] = df_to_f64(dnorm(dps, dpc)) * unscale * unscale;
    __syncthreads();
    if (tid < 32) {
      double pAp;
      if (warp_publish_2level(warp_sum(s_red, NT), P.partials, P.gpartials, P.gtickets, &P.scal->counter[0], &pAp) &&
          tid == 0)
        cg_set_alpha(P.scal, pAp);
    }
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      if ((dirbits >> k) & 1u) continue;
      const double yd = df_to_f64(yt[k]) * unscale;
      if (ij_interior && k > 0 && k < N)
        P.y[node_of(k)] = yd;
      else
        atomicAdd(P.y + node_of(k), yd);
    }
  } else {
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      const int q = k * PS + b * RS + a;
      float s = yt[k].x, c = yt[k].y;
      dadd(s, c, sr[q]);
      dadd(s, c, ss[q]);
      if (P.wJa && active) {
        const int64_t o = e * 2 * NP3 + t2 + NP2 * k;
        dacc(s, c, P.wJa[o], P.wJa[o + NP3], uc[k]);
      }
      const float2 yk = dnorm(s, c);
      if ((dirbits >> k) & 1u) continue;
      const int64_t g = node_of(k);
      const double yd = df_to_f64(yk) * unscale;
      if (ij_interior && k > 0 && k < N)
        P.y[g] = yd;
      else
        atomicAdd(P.y + g, yd);
    }
  }
}

template <int NP, bool BOXM, bool STAGE, bool DOT, EmuForm FORM>
sem_status launch_k(const EmuParams<NP> &p, cudaStream_t s) {
  using C = EmuCfg<NP, STAGE, DOT, FORM>;
  const unsigned grid = (unsigned)((p.E + C::EB - 1) / C::EB);
  if (p.partials && grid > SEM_MAX_PARTIALS) return sem_fail(SEM_ERR_INVALID, "too many elements for fused dot");
  static std::atomic<unsigned long long> attr_done;
  const cudaError_t e = set_smem_limit_once(k_apply_emu<NP, BOXM, STAGE, DOT, FORM>, C::SMEM, attr_done);
  if (e != cudaSuccess) return sem_fail(SEM_ERR_CUDA, std::string("emu attributes: ") + cudaGetErrorString(e));
  if constexpr (DOT)
    SEM_CUDA_TRY(launch_dependent(k_apply_emu<NP, BOXM, STAGE, DOT, FORM>, grid, C::NT, C::SMEM, s, p));
  else
    k_apply_emu<NP, BOXM, STAGE, DOT, FORM><<<grid, C::NT, C::SMEM, s>>>(p);
  return SEM_OK;
}

// Which form a problem of E elements takes.  The fuller blocks of EMU_FULL (and their register floors, which
// spill) serve a chip full of blocks; a few blocks, or a last wave that is nearly empty, want smaller ones and
// a short chain of instructions per thread.  The limits are elements per SM; plain applies, us, full / small /
// scalar (caches warm):
//   N = 6   128 elements 13.5 / 10.7 / 11.0, 1200 18.1 / 15.5 / 15.2, 1728 22.8 / 23.3 / 20.0, 2160 23.1 / 26.5 / 28.0
//   N = 7   288 9.9 / 10.8 / 11.3, 729 14.7 / 14.2 / 13.9, 1200 17.9 / 20.8 / 17.3, 1573 24.0 / 25.4 / 26.4
//   N = 8   128 17.2 / 12.7 / 12.2, 576 23.7 / 17.4 / 15.9, 729 24.0 / 24.8 / 20.0, 891 24.2 / 26.7 / 27.0, 972 31.0 full
//   N = 9   128 21.9 / 12.0 / 15.0, 441 22.7 / 19.8 / 18.8, 729 32.4 / 31.4 / 35.8, 1200 49.4 / 48.9 / 51.8 (1000:
//           47.2 full, 42.7 scalar; two blocks of the scalar form fill an SM four at a time)
//   N = 11  128 31.0 / 16.4 / 20.0, 288 31.6 / 30.3 / 26.8, 441 44.7 / 44.1 / 42.3 (caches cold 54 / 58 / 64), 576 47.9 /
//           57.6 / 49.8, 729 74.5 / 71.9 / 66.5, 891 78.0 / 91.5 / 76.0
// The kernel of a CG step has its own order (an iteration, us): N = 6 27 elements 26.1 / 25.1 / 27.2, 1000 35.6 / 34.5 /
// 35.3, N = 8 27 30.9 / 29.8 / 29.9, 729 43.5 / 44.1 / 44.0, 1000 53.4 / 55.7 / 55.7, N = 9 1000 85.7 / 74.3 / 78.2, 2535
// 154.6 / 151.4 / 165.6 (explicit numbering, 2744: 240 full, 306 small), N = 11 200 55.2 / 53.4 / 46.9, 441 74.8 / 74.5 / 79.1,
// 1000 137 / 165 / 157 (explicit numbering, 216: 80 small, 66 scalar; 729: 177 full, 162 scalar).
__host__ __device__ constexpr bool emu_has(int NP, EmuForm form, bool dot) {
  return form == EMU_FULL || (form == EMU_SMALL ? NP == 10 || NP == 12 || (dot && NP == 7)
                                                : NP == 9 || NP == 12 || (!dot && (NP == 7 || NP == 8 || NP == 10)));
}
inline EmuForm emu_form(int NP, int64_t E, bool dot, bool boxm) {
  const int64_t S = SEM_SMS;
  switch (NP) {
    case 7: return dot ? (E <= 10 * S ? EMU_SMALL : EMU_FULL) : E <= 13 * S ? EMU_SCALAR : EMU_FULL;
    case 8: return !dot && E > 3 * S && E <= 8 * S ? EMU_SCALAR : EMU_FULL;
    case 9: return E <= 5 * S || (!dot && E > 6 * S && E <= 8 * S) ? EMU_SCALAR : EMU_FULL;
    case 10:
      if (E > (dot && boxm ? 20 : dot ? 6 : 8) * S) return EMU_FULL;
      return !dot && (E - 1) / (2 * S) % 2 == 1 ? EMU_SCALAR : EMU_SMALL;
    case 12:
      if (E <= S) return EMU_SMALL;
      if (E <= 2 * S || (dot && !boxm && E <= 6 * S)) return EMU_SCALAR;
      if (E <= 4 * S) return dot ? EMU_SMALL : EMU_FULL;
      return !dot && E <= 6 * S ? EMU_SCALAR : EMU_FULL;
    default: return EMU_FULL;
  }
}

template <int NP, bool STAGE, EmuForm FORM>
sem_status launch_b(const EmuParams<NP> &p, bool boxm, bool dot, cudaStream_t s) {
  if (dot) {
    if constexpr (emu_has(NP, FORM, true))
      return boxm ? launch_k<NP, true, STAGE, true, FORM>(p, s) : launch_k<NP, false, STAGE, true, FORM>(p, s);
  } else {
    if constexpr (emu_has(NP, FORM, false))
      return boxm ? launch_k<NP, true, STAGE, false, FORM>(p, s) : launch_k<NP, false, STAGE, false, FORM>(p, s);
  }
  return sem_fail(SEM_ERR_INVALID, "emu apply: form not built");  // emu_form asks for no such form
}

template <int NP>
sem_status launch_emu(const sem_handle *h, const double *u, double *y, double *partials, SemScalars *scal,
                      cudaStream_t s) {
  EmuParams<NP> p;
  p.E = h->E;
  p.sx = h->box[0];
  p.sy = h->box[1];
  p.sz = h->box[2];
  p.gxs = (int64_t)h->box[0] * h->N + 1;
  p.gys = (int64_t)h->box[1] * h->N + 1;
  p.gzs = (int64_t)h->box[2] * h->N + 1;
  p.bc = h->bc;
  p.u = u;
  p.y = y;
  p.Gf = h->Gemu;
  p.gs = h->gs12;
  p.wJa = h->wJaemu;
  p.glo = h->structured ? nullptr : h->glo;
  p.mask = h->mask;
  p.partials = partials;
  p.gpartials = h->gpartials;
  p.gtickets = h->gtickets;
  p.scal = scal;
  p.err = &h->scal->error;
  p.wait_polls = h->wait_polls;
  for (int q = 0; q < NP * NP; ++q) {
    p.D.hi[q] = h->Dhih[q];
    p.D.lo[q] = h->Dloh[q];
  }
  constexpr int H = EvenOdd<NP>::H;
  auto split = [](double x, float &hi, float &lo) {
    hi = (float)x;
    lo = (float)(x - (double)hi);
  };
  for (int t = 0; t < 2; ++t)  // M = D, D^T; pairs (i, N - i), i < H = n / 2, for even and odd n
    for (int i = 0; i < H && NP >= 2; ++i)
      for (int m = 0; m < H; ++m) {
        const double *D = h->D64h;
        const int N = NP - 1, q = i * H + m;
        const double u = t == 0 ? D[i * NP + m] : D[m * NP + i], v = t == 0 ? D[(N - i) * NP + m] : D[m * NP + (N - i)];
        split(0.5 * (u + v), p.EO.hi[t][q].x, p.EO.lo[t][q].x);
        split(0.5 * (u - v), p.EO.hi[t][q].y, p.EO.lo[t][q].y);
      }
  if (partials && !scal) return sem_fail(SEM_ERR_INVALID, "fused dot needs the solver scalars");
  const bool boxm = p.glo == nullptr && p.bc != SEM_BC_MASK;
  // variant 0: factor block staged by TMA when it fits; other variants read factors directly, and so
  // does the automatic choice (-1) except on small problems at N = 5 (64 elements: 7.1 against 8.8 us; 2535
  // elements: plain 17.4 against 19.4 us, the kernel of a CG step 43.2 against 40.0)
  const bool dot = partials != nullptr;
  const bool stage = emu_stage_fits(NP) && (h->apply_variant == 0 || (h->apply_variant < 0 && NP == 6 &&
                                                                      p.E < (dot ? 14 : 28) * (int64_t)SEM_SMS));
  const EmuForm form = emu_form(NP, p.E, dot, boxm);
  const sem_status st = stage                ? launch_b<NP, emu_stage_fits(NP), EMU_FULL>(p, boxm, dot, s)
                        : form == EMU_SCALAR ? launch_b<NP, false, EMU_SCALAR>(p, boxm, dot, s)
                        : form == EMU_SMALL  ? launch_b<NP, false, EMU_SMALL>(p, boxm, dot, s)
                                             : launch_b<NP, false, EMU_FULL>(p, boxm, dot, s);
  if (st != SEM_OK) return st;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return sem_fail(SEM_ERR_CUDA, std::string("emu apply launch: ") + cudaGetErrorString(e));
  return SEM_OK;
}

}  // namespace semu
