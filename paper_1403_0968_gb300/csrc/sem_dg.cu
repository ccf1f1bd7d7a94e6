// Discontinuous-Galerkin shallow-water volume kernel of arXiv 1403.0968 §4.3 (include/sem_dg.h).
//
// Per element and node the kernel forms the fluxes F, G of the conservative shallow-water system
// from the nodal fields, combines them with the element's affine-map factors into
// Xr = rx F + ry G and Xs = sx F + sy G, and applies the weak derivative matrices:
// rhs = Drw Xr + Dsw Xs + S.  Per element it reads 5 Np field values and 4 factors, writes 3 Np values
// and performs 12 Np^2 flops in the products (k_dg_volume has the layout and its reasons).
//
// The operators are built on the host in FP64 from the orthonormal (Dubiner) basis of the
// triangle: psi_ij = P_i(a) ((1-s)/2)^i P_j^(2i+1,0)(s) / sqrt(2 / ((2i+1)(i+j+1))) with the
// collapsed coordinate a = 2(1+r)/(1-s) - 1; the product P_i(a) ((1-s)/2)^i is evaluated by the
// Legendre three-term recurrence multiplied through by ((1-s)/2)^(k+1), which has no division and
// so no singularity at the vertex s = 1.
#include <cmath>
#include <vector>

#include "../../include/sem_dg.h"
#include "sem_internal.h"
#include "sem_tma.cuh"

__device__ int g_dg_bad;  // zero-area / clockwise triangle flag of sem_dg_geometry

namespace {

constexpr int DG_NT = 256;  // threads of a block of k_dg_nodes

__host__ __device__ constexpr int dg_np(int N) { return (N + 1) * (N + 2) / 2; }
// Row stride of the operator block in device memory, in elements of a type of `es` bytes: an odd
// number of 16-byte vectors, zero padded.
__host__ __device__ constexpr int dg_vw(int es) { return 16 / es; }
__host__ __device__ constexpr int dg_ld(int N, int es) {
  return ((dg_np(N) + dg_vw(es) - 1) / dg_vw(es)) % 2 ? (dg_np(N) + dg_vw(es) - 1) / dg_vw(es) * dg_vw(es)
                                                        : ((dg_np(N) + dg_vw(es) - 1) / dg_vw(es) + 1) * dg_vw(es);
}
__host__ __device__ constexpr int dg_xw(int N, int es) {  // X row length: Np rounded up to whole vectors
  return (dg_np(N) + dg_vw(es) - 1) / dg_vw(es) * dg_vw(es);
}
// ---------------------------------------------------------------------------------------------
// host: operators
// ---------------------------------------------------------------------------------------------

// P_k^(alpha,0)(x) and its derivative, k = 0..n (three-term recurrence and its derivative)
void jacobi_p(int n, double alpha, double x, double *P, double *dP) {
  P[0] = 1.0;
  dP[0] = 0.0;
  if (n >= 1) {
    P[1] = ((alpha + 2.0) * x + alpha) / 2.0;
    dP[1] = (alpha + 2.0) / 2.0;
  }
  for (int k = 2; k <= n; ++k) {
    const double a1 = 2.0 * k * (k + alpha) * (2.0 * k + alpha - 2.0);
    const double b = 2.0 * k + alpha - 1.0;
    const double c2 = (2.0 * k + alpha) * (2.0 * k + alpha - 2.0);
    const double d = 2.0 * (k + alpha - 1.0) * (k - 1.0) * (2.0 * k + alpha);
    P[k] = (b * (c2 * x + alpha * alpha) * P[k - 1] - d * P[k - 2]) / a1;
    dP[k] = (b * (c2 * P[k - 1] + (c2 * x + alpha * alpha) * dP[k - 1]) - d * dP[k - 2]) / a1;
  }
}

// In-place Gauss-Jordan inverse with partial pivoting (n x n, row-major); false if singular.
bool invert(std::vector<double> &A, int n) {
  std::vector<double> I(n * n, 0.0);
  for (int i = 0; i < n; ++i) I[i * n + i] = 1.0;
  for (int c = 0; c < n; ++c) {
    int p = c;
    for (int r = c + 1; r < n; ++r)
      if (std::fabs(A[r * n + c]) > std::fabs(A[p * n + c])) p = r;
    if (A[p * n + c] == 0.0) return false;
    if (p != c)
      for (int k = 0; k < n; ++k) {
        std::swap(A[p * n + k], A[c * n + k]);
        std::swap(I[p * n + k], I[c * n + k]);
      }
    const double inv = 1.0 / A[c * n + c];
    for (int k = 0; k < n; ++k) {
      A[c * n + k] *= inv;
      I[c * n + k] *= inv;
    }
    for (int r = 0; r < n; ++r) {
      if (r == c) continue;
      const double f = A[r * n + c];
      if (f == 0.0) continue;
      for (int k = 0; k < n; ++k) {
        A[r * n + k] -= f * A[c * n + k];
        I[r * n + k] -= f * I[c * n + k];
      }
    }
  }
  A.swap(I);
  return true;
}

std::vector<double> matmul(const std::vector<double> &A, const std::vector<double> &B, int n) {
  std::vector<double> C(n * n, 0.0);
  for (int i = 0; i < n; ++i)
    for (int k = 0; k < n; ++k) {
      const double a = A[i * n + k];
      for (int j = 0; j < n; ++j) C[i * n + j] += a * B[k * n + j];
    }
  return C;
}

std::vector<double> transpose(const std::vector<double> &A, int n) {
  std::vector<double> T(n * n);
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < n; ++j) T[j * n + i] = A[i * n + j];
  return T;
}

// Vandermonde matrices of the orthonormal basis at the equispaced nodes: V, d/dr, d/ds
void vandermonde(int N, std::vector<double> &V, std::vector<double> &Vr, std::vector<double> &Vs) {
  const int np = dg_np(N);
  V.assign(np * np, 0.0);
  Vr.assign(np * np, 0.0);
  Vs.assign(np * np, 0.0);
  std::vector<double> Q(N + 2), Qr(N + 2), Qs(N + 2), P(N + 1), dP(N + 1);
  int n = 0;
  for (int b = 0; b <= N; ++b)
    for (int a = 0; a + b <= N; ++a, ++n) {
      const double r = -1.0 + 2.0 * a / N, s = -1.0 + 2.0 * b / N;
      // Q_k = P_k(a) q^k, q = (1-s)/2:  (k+1) Q_{k+1} = (2k+1) (a q) Q_k - k q^2 Q_{k-1}, a q = r + (1+s)/2
      const double aq = r + 0.5 * (1.0 + s), q = 0.5 * (1.0 - s), q2 = q * q, dq2s = -q;
      Q[0] = 1.0, Qr[0] = 0.0, Qs[0] = 0.0;
      Q[1] = aq, Qr[1] = 1.0, Qs[1] = 0.5;
      for (int k = 1; k < N; ++k) {
        Q[k + 1] = ((2.0 * k + 1.0) * aq * Q[k] - k * q2 * Q[k - 1]) / (k + 1.0);
        Qr[k + 1] = ((2.0 * k + 1.0) * (Q[k] + aq * Qr[k]) - k * q2 * Qr[k - 1]) / (k + 1.0);
        Qs[k + 1] = ((2.0 * k + 1.0) * (0.5 * Q[k] + aq * Qs[k]) - k * (dq2s * Q[k - 1] + q2 * Qs[k - 1])) / (k + 1.0);
      }
      int m = 0;
      for (int i = 0; i <= N; ++i) {
        jacobi_p(N - i, 2.0 * i + 1.0, s, P.data(), dP.data());
        for (int j = 0; i + j <= N; ++j, ++m) {
          const double w = 1.0 / std::sqrt(2.0 / ((2.0 * i + 1.0) * (i + j + 1.0)));
          V[n * np + m] = w * Q[i] * P[j];
          Vr[n * np + m] = w * Qr[i] * P[j];
          Vs[n * np + m] = w * (Qs[i] * P[j] + Q[i] * dP[j]);
        }
      }
    }
}

// ---------------------------------------------------------------------------------------------
// device: volume kernel
// ---------------------------------------------------------------------------------------------

// Layout of the volume kernel for meshes that fill the chip (k_dg_nodes below for smaller ones, see
// dg_rule).  The products are a GEMM with M = Np rows, K = 2 Np and three columns (the fields) per element.  A
// lane owns one element and RI of its rows (RS lanes share an element): it walks the nodes once, with the
// six flux combinations of a node in registers (nothing of X goes through shared memory), and adds their
// products with a column of Drw and of Dsw to 3 RI sums.  The operator columns come from shared memory
// 16 bytes at a time, one load for 3 x 4 products; FP32 products run two rows to an instruction (FFMA2: the
// scalar FMA rate at half the issue slots).  A warp stages the fields of its WE elements by asynchronous
// copies, one batch ahead, and its results leave through the same buffer; warps are independent of one
// another.
//
// Rounding: the products of SG * RS nodes are summed on their own and then added to the output, so that most
// roundings happen at a fraction of its size (one addition in 8 to 16 products).  RMS error against FP64,
// FP32, of each node's pair of products added to the output / one chain of all products / these groups:
// N = 3 8.76e-8 / 9.12e-8 / 8.22e-8, 5 1.05e-7 / 1.13e-7 / 9.2e-8, 7 1.40e-7 / 1.48e-7 / 1.22e-7, 8 1.72e-7 /
// 1.82e-7 / 1.58e-7.  At N = 1 (3 nodes) groups gain nothing, and in FP32 at N = 2 they take registers: pairs there.
//
// What bounds it at N = 7, FP32: the operator loads (each returns 512 bytes to registers, four cycles of the
// SM's shared-memory path, for 12 FMA cycles per scheduler) and the FMA pipe, half busy; with the products
// left out the copies alone take 48 us of the 95 us.  212,552 triangles, k_dg_nodes / this kernel, caches warm: FP32
// N = 1..8 7.4 / 5.6, 17 / 8.6, 28 / 14, 79 / 26, 135 / 42, 109 / 67, 154 / 95, 319 / 147 us; FP64 N = 3..8 387 / 353,
// 822 / 721, 1508 / 1374, 2478 / 2224, 3977 / 3537, 6966 / 5759 us (the FP64 pipe: 4640 us at N = 8 for the products
// alone).
template <typename T, int N, int RS_>
struct DgCfg {
  static constexpr int NP = dg_np(N), VW = dg_vw(sizeof(T)), RS = RS_;
  static constexpr int WE = 32 / RS;                        // elements per warp
  static constexpr int RW = sizeof(T) == 4 ? 2 : 1;         // rows per product instruction
  static constexpr int RI = ((NP + RS - 1) / RS + RW - 1) / RW * RW;  // rows per lane
  static constexpr int RP = (RI + VW - 1) / VW * VW;        // row stride of an operator column
  static constexpr bool PAIR = N == 1 || (N == 2 && sizeof(T) == 4);  // a node's two products join the sum by themselves
  // else the products of SG * RS nodes do (a divisor of Np where there is one near)
  static constexpr int SG = PAIR                ? 1
                            : RS == 4           ? (sizeof(T) == 8 && N >= 4 ? 2 : 1)
                            : N == 2            ? 2 / RS
                            : RS == 2           ? (N == 6 ? 2 : 3)
                            : N == 5            ? 7
                                                : 5;
  static constexpr int QW = WE * 3 * NP, BW = WE * 2 * NP;  // field and bathymetry values of a batch
  static constexpr int PW = 2 * QW + BW;                    // values staged per warp (fields twice)
  static constexpr int DW = NP * RS * 2 * RP;               // operator values per block
  static constexpr int FIT = (int)((227 * 1024 / sizeof(T) - DW) / PW);
  // at most two warps per scheduler; a fifth alone would leave three schedulers with one each
  static constexpr int W = FIT >= 8 ? 8 : FIT == 5 ? 4 : FIT;  // warps per block
  static constexpr size_t SMEM = (size_t)(DW + W * PW) * sizeof(T);
  static_assert(W >= 1 && SMEM <= 227 * 1024, "shared memory of a block");
  static_assert(QW * sizeof(T) % 16 == 0 && BW * sizeof(T) % 16 == 0 && DW * sizeof(T) % 16 == 0, "16-byte regions");
};

template <typename T, int V>
struct alignas(V * sizeof(T)) DgVec {
  T v[V];
};

// a = operator rows times one flux value, a += the same, a += b (two rows to an instruction in FP32)
__device__ __forceinline__ void dg_mul(float *a, const float *d, float x) {
  const float2 r = __fmul2_rn(make_float2(d[0], d[1]), make_float2(x, x));
  a[0] = r.x, a[1] = r.y;
}
__device__ __forceinline__ void dg_fma(float *a, const float *d, float x) {
  const float2 r = __ffma2_rn(make_float2(d[0], d[1]), make_float2(x, x), make_float2(a[0], a[1]));
  a[0] = r.x, a[1] = r.y;
}
__device__ __forceinline__ void dg_add(float *a, const float *b) {
  const float2 r = __fadd2_rn(make_float2(a[0], a[1]), make_float2(b[0], b[1]));
  a[0] = r.x, a[1] = r.y;
}
__device__ __forceinline__ void dg_mul(double *a, const double *d, double x) { *a = *d * x; }
__device__ __forceinline__ void dg_fma(double *a, const double *d, double x) { *a = fma(*d, x, *a); }
__device__ __forceinline__ void dg_add(double *a, const double *b) { *a += *b; }

// 1 / h: one Newton-Raphson step on the hardware's approximation in its fused form, r + r (1 - h r) (Markstein,
// IBM J. Res. Dev. 34, 1990), within a unit in the last place of the quotient.  A division's branch would
// keep the fluxes of the next node apart from the products of this one (212,552 triangles, FP32, N = 7: 103
// against 95 us).  The approximation itself is kept where the step has no meaning: h zero, infinite or so small
// that its reciprocal overflows (the error is then NaN or infinite).
__device__ __forceinline__ float dg_reciprocal(float h) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(h));
  const float e = fmaf(-h, r, 1.f);
  return fabsf(e) < 1.f ? fmaf(r, e, r) : r;
}
__device__ __forceinline__ double dg_reciprocal(double h) { return 1.0 / h; }

// n values from global to shared by the lanes of a warp, 16 bytes at a time when src starts on a
// 16-byte boundary (wide), else one value at a time
template <typename T>
__device__ __forceinline__ void dg_fetch(T *dst, const T *src, int n, bool wide, int lane) {
  constexpr int VW = dg_vw(sizeof(T));
  int done = 0;
  if (wide) {
    const int nv = n / VW;
    for (int q = lane; q < nv; q += 32)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst + q * VW)), "l"(src + q * VW) : "memory");
    done = nv * VW;
  }
  for (int q = done + lane; q < n; q += 32)
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_addr(dst + q)), "l"(src + q), "n"((int)sizeof(T))
                 : "memory");
}

template <typename T, int N, int RS_>
__global__ void __launch_bounds__(32 * DgCfg<T, N, RS_>::W)
    k_dg_volume(int64_t E, T g, const T *__restrict__ ops, const T *__restrict__ Q, const T *__restrict__ Bxy,
                const T *__restrict__ geo, T *__restrict__ rhs, int wide) {
  using C = DgCfg<T, N, RS_>;
  constexpr int NP = C::NP, RS = C::RS, WE = C::WE, RI = C::RI, RP = C::RP, VW = C::VW, W = C::W, SG = C::SG;
  constexpr int LD = dg_ld(N, sizeof(T));
  extern __shared__ __align__(16) unsigned char dg_smem[];
  T *sD = reinterpret_cast<T *>(dg_smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  T *sB = sD + C::DW + warp * C::PW, *sQ = sB + C::BW, *sQn = sQ + C::QW;
  const int el = lane % WE, part = lane / WE, i0 = part * RI;
  // a warp's batches of WE elements: consecutive ones go to different blocks, so that a mesh with
  // fewer batches than warps spreads over the SMs
  const int64_t nbatch = (E + WE - 1) / WE, stride = (int64_t)gridDim.x * W;
  int64_t batch = (int64_t)warp * gridDim.x + blockIdx.x;
  auto fetch = [&](T *dst, const T *src, int64_t b, int per, bool w) {
    if (b < nbatch) {
      const int64_t e0 = b * WE;
      dg_fetch<T>(dst, src + e0 * per, (int)(E - e0 < WE ? E - e0 : WE) * per, w, lane);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch(sQ, Q, batch, 3 * NP, wide & 1);
  // operators as [node j][row part][Drw, Dsw][rows of the part], zero padded
  for (int q = tid; q < C::DW; q += 32 * W) {
    const int i = q % RP, m = q / RP % 2, p = q / (2 * RP) % RS, j = q / (2 * RP * RS), row = p * RI + i;
    sD[q] = (i < RI && row < NP) ? ops[m * NP * LD + row * LD + j] : T(0);
  }
  __syncthreads();
  for (; batch < nbatch; batch += stride) {
    const int64_t e0 = batch * WE;
    const int ne = (int)(E - e0 < WE ? E - e0 : WE);
    const bool live = el < ne;  // slots past the mesh work on the batch's first element and write nothing
    const int slot = live ? el : 0;
    const T *ge = geo + (e0 + slot) * 4, *be = sB + slot * 2 * NP;
    T *qe = sQ + slot * 3 * NP;
    const T rx = ge[0], ry = ge[1], sx = ge[2], sy = ge[3];
    // the batch's fields were asked for one batch ago; its bathymetry and the next batch's fields
    // arrive while the products run
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    fetch(sB, Bxy, batch, 2 * NP, wide & 2);
    fetch(sQn, Q, batch + stride, 3 * NP, wide & 1);
    T acc[3][RI] = {};
    // The RS lanes of an element take the fluxes of RS nodes, one node each, and pass them on to one
    // another; they are formed one group of nodes ahead, beside the products of the group before.
    auto flux = [&](int j, T(&x)[6]) {
      const int jc = j < NP ? j : NP - 1;
      const T h = qe[jc], hu = qe[NP + jc], hv = qe[2 * NP + jc];
      const T ih = dg_reciprocal(h), a = hu * ih, b = hv * ih, p = T(0.5) * g * h * h;
      const T F1 = hu * a + p, F2 = hu * b, G1 = hv * a, G2 = hv * b + p;
      x[0] = rx * hu + ry * hv, x[1] = rx * F1 + ry * G1, x[2] = rx * F2 + ry * G2;
      x[3] = sx * hu + sy * hv, x[4] = sx * F1 + sy * G1, x[5] = sx * F2 + sy * G2;
      if (NP % RS != 0 && j >= NP) {  // past the last node: its products add nothing
#pragma unroll
        for (int f = 0; f < 6; ++f) x[f] = T(0);
      }
    };
    T x[6], xn[6];
    flux(part, x);
#pragma unroll 1
    for (int j0 = 0; j0 < NP; j0 += SG * RS) {
      T sum[3][RI];  // this group's products
#pragma unroll
      for (int g = 0; g < SG; ++g) {
        const int js = j0 + g * RS;
        if (NP % (SG * RS) != 0 && g > 0 && js >= NP) break;
        flux(js + RS + part, xn);
#pragma unroll
        for (int k = 0; k < RS; ++k) {  // node js + (part ^ k), from the lane that owns it
          T y[6];
#pragma unroll
          for (int f = 0; f < 6; ++f) y[f] = k == 0 ? x[f] : __shfl_xor_sync(0xffffffffu, x[f], k * WE);
          const int jk = js + (part ^ k), jc = NP % RS == 0 || jk < NP ? jk : NP - 1;
          const DgVec<T, VW> *d = reinterpret_cast<const DgVec<T, VW> *>(sD + (jc * RS + part) * 2 * RP);
#pragma unroll
          for (int q = 0; q < RP / VW; ++q) {
#pragma unroll
            for (int m = 0; m < 2; ++m) {  // Drw with Xr, then Dsw with Xs
              const DgVec<T, VW> w = d[m * (RP / VW) + q];
#pragma unroll
              for (int i = 0; i < VW; i += C::RW)
                if (q * VW + i < RI) {
#pragma unroll
                  for (int f = 0; f < 3; ++f) {
                    T *t = &sum[f][q * VW + i];
                    if (m == 0 && (C::PAIR || (g == 0 && k == 0)))
                      dg_mul(t, &w.v[i], y[f]);
                    else
                      dg_fma(t, &w.v[i], y[3 * m + f]);
                    if (m == 1 && C::PAIR) {
                      if (sizeof(T) == 8 && g == 0 && k == 0 && j0 == 0)
                        for (int r = 0; r < C::RW; ++r) acc[f][q * VW + i + r] = t[r];
                      else
                        dg_add(&acc[f][q * VW + i], t);
                    }
                  }
                }
            }
          }
        }
#pragma unroll
        for (int f = 0; f < 6; ++f) x[f] = xn[f];
      }
      if constexpr (!C::PAIR) {
        if (sizeof(T) == 8 && j0 == 0) {  // (an FP64 addition less)
#pragma unroll
          for (int f = 0; f < 3; ++f)
#pragma unroll
            for (int i = 0; i < RI; ++i) acc[f][i] = sum[f][i];
        } else {
#pragma unroll
          for (int f = 0; f < 3; ++f)
#pragma unroll
            for (int i = 0; i < RI; i += C::RW) dg_add(&acc[f][i], &sum[f][i]);
        }
      }
    }
    // bathymetry source at this lane's rows, then the results take the place of the fields
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncwarp();
    // (rows in pairs where every row of pairs starts on one)
    constexpr int VE = NP % 2 == 0 && RI % 2 == 0 ? 2 : 1;
    using VR = DgVec<T, VE>;
    VR *q0 = reinterpret_cast<VR *>(qe + i0);
    const VR *b0 = reinterpret_cast<const VR *>(be + i0);
#pragma unroll
    for (int r = 0; r < RI / VE; ++r)
      if (i0 + r * VE < NP) {
        const VR h = q0[r], bx = b0[r], by = b0[NP / VE + r];
#pragma unroll
        for (int k = 0; k < VE; ++k) {
          acc[1][r * VE + k] -= g * h.v[k] * bx.v[k];
          acc[2][r * VE + k] -= g * h.v[k] * by.v[k];
        }
      }
    __syncwarp();
    if (live) {
#pragma unroll
      for (int r = 0; r < RI / VE; ++r)
        if (i0 + r * VE < NP) {
#pragma unroll
          for (int f = 0; f < 3; ++f) {
            VR o;
#pragma unroll
            for (int k = 0; k < VE; ++k) o.v[k] = acc[f][r * VE + k];
            q0[f * (NP / VE) + r] = o;
          }
        }
    }
    __syncwarp();
    T *out = rhs + e0 * 3 * NP;
    const int n = ne * 3 * NP;
    int done = 0;
    if (wide & 4) {
      using VO = DgVec<T, VW>;
      for (int q = lane; q < n / VW; q += 32) reinterpret_cast<VO *>(out)[q] = reinterpret_cast<const VO *>(sQ)[q];
      done = n / VW * VW;
    }
    for (int q = done + lane; q < n; q += 32) out[q] = sQ[q];
    __syncwarp();
    T *t = sQ;
    sQ = sQn;
    sQn = t;
  }
}

// The volume kernel for small meshes: one thread per element node.  A block takes batches of
// floor(256 / Np) groups of ET elements and stays resident over many batches; the operators (rows zero
// padded to an odd number of 16-byte vectors, so that threads on consecutive rows hit distinct banks) and
// the batch's Xr, Xs sit in shared memory and are read 16 bytes at a time (X as a broadcast).
// Elements per thread: with ET > 1 every operator vector serves ET elements (212,800 triangles: ET = 2 1.2x
// over 1 at N = 6..8, slower at N = 2; ET = 3 a further 5% at N = 7 and 8.5% at N = 8; ET = 4 slower); FP64 keeps
// 1 (its FMA pipe is the bound, and its shared memory would not fit).
__host__ __device__ constexpr int dg_et(int N, int es) { return es == 4 && N >= 7 ? 3 : es == 4 && N >= 3 ? 2 : 1; }

template <typename T, int N>
__global__ void __launch_bounds__(DG_NT) k_dg_nodes(int64_t E, T g, const T *__restrict__ ops,
                                                     const T *__restrict__ Q, const T *__restrict__ Bxy,
                                                     const T *__restrict__ geo, T *__restrict__ rhs) {
  constexpr int NP = dg_np(N), LD = dg_ld(N, sizeof(T)), XW = dg_xw(N, sizeof(T));
  constexpr int ET = dg_et(N, sizeof(T)), EG = DG_NT / NP, EB = EG * ET;  // groups, elements per batch
  constexpr int VW = dg_vw(sizeof(T)), NV = XW / VW;  // 16-byte vectors per row
  __shared__ alignas(16) T sD[2 * NP * LD];
  __shared__ alignas(16) T sX[EB][6][XW];
  const int tid = threadIdx.x;
  for (int q = tid; q < 2 * NP * LD; q += DG_NT) sD[q] = ops[q];
  // zero the padding of the X rows (it meets the zero padding of the operator rows)
  if constexpr (XW > NP) {
    for (int q = tid; q < EB * 6 * (XW - NP); q += DG_NT) {
      const int row = q / (XW - NP);
      sX[row / 6][row % 6][NP + q % (XW - NP)] = T(0);
    }
  }
  const int el = tid / NP, i = tid - el * NP;  // group (ET consecutive elements of a batch), node
  const bool grp = el < EG;
  const DgVec<T, VW> *dr = reinterpret_cast<const DgVec<T, VW> *>(sD + i * LD);
  const DgVec<T, VW> *ds = reinterpret_cast<const DgVec<T, VW> *>(sD + NP * LD + i * LD);
  const DgVec<T, VW> *x0 = reinterpret_cast<const DgVec<T, VW> *>(&sX[grp ? el * ET : 0][0][0]);
  constexpr int XS = 6 * NV;  // vectors per element in sX
  // persistent blocks: the operators are loaded once per block, batches of EB elements follow
  const int64_t nbatch = (E + EB - 1) / EB;
  for (int64_t batch = blockIdx.x; batch < nbatch; batch += gridDim.x) {
    const int64_t e0 = batch * EB + (int64_t)el * ET;
    T h[ET], bx[ET], by[ET];
#pragma unroll
    for (int t = 0; t < ET; ++t) {
      const int64_t e = e0 + t;
      h[t] = T(1), bx[t] = T(0), by[t] = T(0);
      if (grp && e < E) {
        const T *q = Q + e * 3 * NP + i;
        h[t] = q[0];
        const T hu = q[NP], hv = q[2 * NP];
        bx[t] = Bxy[e * 2 * NP + i];
        by[t] = Bxy[e * 2 * NP + NP + i];
        const T rx = geo[e * 4 + 0], ry = geo[e * 4 + 1], sx = geo[e * 4 + 2], sy = geo[e * 4 + 3];
        const T ih = T(1) / h[t], u = hu * ih, v = hv * ih, p = T(0.5) * g * h[t] * h[t];
        const T F0 = hu, F1 = hu * u + p, F2 = hu * v;
        const T G0 = hv, G1 = hv * u, G2 = hv * v + p;
        T(*X)[XW] = sX[el * ET + t];
        X[0][i] = rx * F0 + ry * G0;
        X[1][i] = rx * F1 + ry * G1;
        X[2][i] = rx * F2 + ry * G2;
        X[3][i] = sx * F0 + sy * G0;
        X[4][i] = sx * F1 + sy * G1;
        X[5][i] = sx * F2 + sy * G2;
      }
    }
    __syncthreads();
    if (grp && e0 < E) {
      // 16-byte loads: one operator vector serves three fields of ET elements; each X vector is the
      // same for every thread of the element (a broadcast)
      T a[ET][3];
#pragma unroll
      for (int t = 0; t < ET; ++t) a[t][0] = a[t][1] = a[t][2] = T(0);
#pragma unroll
      for (int jv = 0; jv < NV; ++jv) {
        const DgVec<T, VW> wr = dr[jv], ws = ds[jv];
#pragma unroll
        for (int t = 0; t < ET; ++t) {
          const DgVec<T, VW> *xt = x0 + t * XS;
          const DgVec<T, VW> r0 = xt[0 * NV + jv], r1 = xt[1 * NV + jv], r2 = xt[2 * NV + jv];
          const DgVec<T, VW> s0 = xt[3 * NV + jv], s1 = xt[4 * NV + jv], s2 = xt[5 * NV + jv];
          // a vector's products are summed on their own (N = 1: a node's), as in k_dg_volume
          T p0 = T(0), p1 = T(0), p2 = T(0);
#pragma unroll
          for (int k = 0; k < VW; ++k) {
            if (N == 1 || k == 0) {
              p0 = wr.v[k] * r0.v[k], p1 = wr.v[k] * r1.v[k], p2 = wr.v[k] * r2.v[k];
            } else {
              p0 += wr.v[k] * r0.v[k], p1 += wr.v[k] * r1.v[k], p2 += wr.v[k] * r2.v[k];
            }
            p0 += ws.v[k] * s0.v[k], p1 += ws.v[k] * s1.v[k], p2 += ws.v[k] * s2.v[k];
            if (N == 1 || k == VW - 1) {
              if (jv == 0 && (N > 1 || k == 0))
                a[t][0] = p0, a[t][1] = p1, a[t][2] = p2;
              else
                a[t][0] += p0, a[t][1] += p1, a[t][2] += p2;
            }
          }
        }
      }
#pragma unroll
      for (int t = 0; t < ET; ++t) {
        const int64_t e = e0 + t;
        if (e < E) {
          T *o = rhs + e * 3 * NP + i;
          o[0] = a[t][0];
          o[NP] = a[t][1] - g * h[t] * bx[t];
          o[2 * NP] = a[t][2] - g * h[t] * by[t];
        }
      }
    }
    __syncthreads();  // the next batch overwrites sX
  }
}

// rx, ry, sx, sy of each triangle: the inverse of [[x_r, x_s], [y_r, y_s]] with x_r = (x2 - x1)/2,
// x_s = (x3 - x1)/2 (and y alike); bad is set when the Jacobian is not positive
template <typename T>
__global__ void k_dg_geometry(int64_t E, const double *__restrict__ v, T *__restrict__ geo, int *bad) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= E) return;
  const double *p = v + e * 6;
  const double xr = 0.5 * (p[2] - p[0]), xs = 0.5 * (p[4] - p[0]);
  const double yr = 0.5 * (p[3] - p[1]), ys = 0.5 * (p[5] - p[1]);
  const double J = xr * ys - xs * yr;
  if (!(J > 0.0)) atomicOr(bad, 1);
  geo[e * 4 + 0] = (T)(ys / J);
  geo[e * 4 + 1] = (T)(-xs / J);
  geo[e * 4 + 2] = (T)(-yr / J);
  geo[e * 4 + 3] = (T)(xr / J);
}

template <typename T, int N, int RS>
sem_status launch_dg_lanes(int64_t E, double g, const void *ops, const void *Q, const void *Bxy, const void *geo,
                        void *rhs, int sms, cudaStream_t s) {
  using C = DgCfg<T, N, RS>;
  static std::atomic<unsigned long long> attr_done;
  SEM_CUDA_TRY((set_smem_limit_once(k_dg_volume<T, N, RS>, C::SMEM, attr_done)));
  // persistent grid: as many blocks as fit on the device at once (each loads the operators once)
  int per_sm = 0;
  SEM_CUDA_TRY((cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_dg_volume<T, N, RS>, 32 * C::W, C::SMEM)));
  const int64_t batches = (E + C::WE - 1) / C::WE, resident = (int64_t)sms * (per_sm > 0 ? per_sm : 1);
  const int64_t blocks = batches < resident ? batches : resident;
  auto aligned = [](const void *p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; };
  const int wide = (aligned(Q) ? 1 : 0) | (aligned(Bxy) ? 2 : 0) | (aligned(rhs) ? 4 : 0);
  k_dg_volume<T, N, RS><<<(unsigned)blocks, 32 * C::W, C::SMEM, s>>>(
      E, (T)g, static_cast<const T *>(ops), static_cast<const T *>(Q), static_cast<const T *>(Bxy),
      static_cast<const T *>(geo), static_cast<T *>(rhs), wide);
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

template <typename T, int N>
sem_status launch_dg_nodes(int64_t E, double g, const void *ops, const void *Q, const void *Bxy, const void *geo,
                           void *rhs, int sms, cudaStream_t s) {
  constexpr int EB = DG_NT / dg_np(N) * dg_et(N, sizeof(T));
  int per_sm = 0;
  SEM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_dg_nodes<T, N>, DG_NT, 0));
  const int64_t batches = (E + EB - 1) / EB, resident = (int64_t)sms * (per_sm > 0 ? per_sm : 1);
  const int64_t blocks = batches < resident ? batches : resident;
  k_dg_nodes<T, N><<<(unsigned)blocks, DG_NT, 0, s>>>(
      E, (T)g, static_cast<const T *>(ops), static_cast<const T *>(Q), static_cast<const T *>(Bxy),
      static_cast<const T *>(geo), static_cast<T *>(rhs));
  SEM_CUDA_TRY(cudaGetLastError());
  return SEM_OK;
}

// Which kernel a mesh of E triangles takes, by triangles per SM: below `a` one thread per node, below `b` `f1`
// lanes per element, from there `f2` lanes (0: one thread per node).  A warp of the lane form holds 8 to 32
// elements, so that a small mesh leaves schedulers without a warp (FP64 above all, whose pipe belongs to a
// scheduler); one thread per node spreads it.  More lanes per element lie between.  Measured with the
// caches warm, us for one thread per node | 1 / 2 / 4 lanes:
//   FP32, 3200 triangles     N = 2 2.1 | 2.6 / 2.6 / 2.6   4 3.6 | 4.0 / 3.9 / 3.4    7 6.4 | - / 8.0 / 8.3
//         8192               N = 3 3.4 | 2.9 / 3.5 / 3.7   5 8.2 | 5.6 / 5.6 / 5.6    7 9.4 | - / 8.5 / 8.6
//         33800              N = 1 2.6 | 2.7 / 2.9 / 3.2   4 13.5 | 6.0 / 6.6 / 8.0   8 53 | - / 30 / 33
//         212,552            N = 1 7.4 | 5.6 / 8.2 / 11.5  6 106 | 73 / 67 / 72       8 320 | 313 / 147 / 159
//   FP64, 800                N = 1 5.9 | 8.1 / 7.3 / 4.2   4 11.8 | 65 / 39 / 21.4    7 23 | - / 159 / 86
//         3200               N = 3 8.5 | 34 / 19 / 14.4    5 28 | - / 67 / 42         7 82 | - / 159 / 86
//         15488              N = 3 36 | 35 / 31 / 40       5 118 | - / 113 / 135      8 525 | - / 524 / 483
//         45000              N = 2 40 | 45 / 47 / 68       4 179 | 175 / 183 / 190    8 1499 | - / 1318 / 1332
struct DgRule {
  int a, f1, b, f2;
};
template <typename T>
__host__ __device__ constexpr DgRule dg_rule(int N) {
  if (sizeof(T) == 4)
    return N == 1   ? DgRule{260, 1, 0, 1}
           : N == 2 ? DgRule{85, 1, 0, 1}
           : N == 3 ? DgRule{50, 1, 0, 1}
           : N == 4 ? DgRule{0, 4, 50, 1}
           : N == 5 ? DgRule{26, 1, 0, 1}
           : N == 6 ? DgRule{40, 2, 0, 2}
           : N == 7 ? DgRule{50, 2, 0, 2}
                    : DgRule{27, 2, 0, 2};
  return N == 1   ? DgRule{0, 4, 50, 0}
         : N == 2 ? DgRule{0, 0, 0, 0}
         : N == 3 ? DgRule{145, 1, 0, 1}
         : N == 4 ? DgRule{46, 4, 115, 1}
         : N == 5 ? DgRule{145, 2, 0, 2}
                  : DgRule{25, 4, 0, 4};
}

template <typename T, int N>
sem_status launch_dg(int64_t E, double g, const void *ops, const void *Q, const void *Bxy, const void *geo,
                     void *rhs, cudaStream_t s) {
  constexpr DgRule R = dg_rule<T>(N);
  int dev = 0, sms = 0;
  SEM_CUDA_TRY(cudaGetDevice(&dev));
  SEM_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  if constexpr (R.a > 0 || R.f2 == 0) {
    if (E < (int64_t)sms * R.a || (R.f2 == 0 && E >= (int64_t)sms * R.b))
      return launch_dg_nodes<T, N>(E, g, ops, Q, Bxy, geo, rhs, sms, s);
  }
  if constexpr (R.f1 > 0 && R.b > 0) {
    if (R.f2 == 0 || E < (int64_t)sms * R.b) return launch_dg_lanes<T, N, R.f1>(E, g, ops, Q, Bxy, geo, rhs, sms, s);
  }
  if constexpr (R.f2 > 0)
    return launch_dg_lanes<T, N, R.f2>(E, g, ops, Q, Bxy, geo, rhs, sms, s);
  else
    return SEM_OK;  // not reached
}

template <typename T>
sem_status dg_dispatch(int N, int64_t E, double g, const void *ops, const void *Q, const void *Bxy, const void *geo,
                       void *rhs, cudaStream_t s) {
  switch (N) {
    case 1: return launch_dg<T, 1>(E, g, ops, Q, Bxy, geo, rhs, s);
    case 2: return launch_dg<T, 2>(E, g, ops, Q, Bxy, geo, rhs, s);
    case 3: return launch_dg<T, 3>(E, g, ops, Q, Bxy, geo, rhs, s);
    case 4: return launch_dg<T, 4>(E, g, ops, Q, Bxy, geo, rhs, s);
    case 5: return launch_dg<T, 5>(E, g, ops, Q, Bxy, geo, rhs, s);
    case 6: return launch_dg<T, 6>(E, g, ops, Q, Bxy, geo, rhs, s);
    case 7: return launch_dg<T, 7>(E, g, ops, Q, Bxy, geo, rhs, s);
    case 8: return launch_dg<T, 8>(E, g, ops, Q, Bxy, geo, rhs, s);
    default: return sem_fail(SEM_ERR_INVALID, "DG order must be 1..8");
  }
}

}  // namespace

extern "C" sem_status sem_dg_operators(int32_t N, double *Drw, double *Dsw) {
  if (N < 1 || N > SEM_DG_MAX_ORDER) return sem_fail(SEM_ERR_INVALID, "DG order must be 1..8");
  if (!Drw || !Dsw) return sem_fail(SEM_ERR_INVALID, "NULL argument");
  const int np = dg_np(N);
  std::vector<double> V, Vr, Vs;
  vandermonde(N, V, Vr, Vs);
  std::vector<double> Vinv = V;
  if (!invert(Vinv, np)) return sem_fail(SEM_ERR_INVALID, "singular Vandermonde matrix");
  const std::vector<double> Dr = matmul(Vr, Vinv, np), Ds = matmul(Vs, Vinv, np);
  const std::vector<double> A = matmul(V, transpose(V, np), np);             // Mhat^-1
  const std::vector<double> Ainv = matmul(transpose(Vinv, np), Vinv, np);    // Mhat
  const std::vector<double> Wr = matmul(matmul(A, transpose(Dr, np), np), Ainv, np);
  const std::vector<double> Ws = matmul(matmul(A, transpose(Ds, np), np), Ainv, np);
  for (int q = 0; q < np * np; ++q) {
    Drw[q] = Wr[q];
    Dsw[q] = Ws[q];
  }
  return SEM_OK;
}

extern "C" sem_status sem_dg_operator_bytes(int32_t N, sem_prec prec, size_t *bytes) {
  if (N < 1 || N > SEM_DG_MAX_ORDER) return sem_fail(SEM_ERR_INVALID, "DG order must be 1..8");
  if (prec != SEM_FP64 && prec != SEM_FP32) return sem_fail(SEM_ERR_INVALID, "DG precision must be FP64 or FP32");
  if (!bytes) return sem_fail(SEM_ERR_INVALID, "NULL argument");
  const int es = prec == SEM_FP64 ? 8 : 4;
  *bytes = (size_t)2 * dg_np(N) * dg_ld(N, es) * es;
  return SEM_OK;
}

extern "C" sem_status sem_dg_load_operators(int32_t N, sem_prec prec, void *d_ops, size_t bytes, sem_stream_t stream) {
  size_t need = 0;
  sem_status st = sem_dg_operator_bytes(N, prec, &need);
  if (st != SEM_OK) return st;
  if (!d_ops || bytes < need) return sem_fail(SEM_ERR_INVALID, "operator buffer missing or too small");
  const int np = dg_np(N), ld = dg_ld(N, prec == SEM_FP64 ? 8 : 4);
  std::vector<double> Wr(np * np), Ws(np * np);
  st = sem_dg_operators(N, Wr.data(), Ws.data());
  if (st != SEM_OK) return st;
  std::vector<double> d64(2 * np * ld, 0.0);
  for (int i = 0; i < np; ++i)
    for (int j = 0; j < np; ++j) {
      d64[i * ld + j] = Wr[i * np + j];
      d64[np * ld + i * ld + j] = Ws[i * np + j];
    }
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (prec == SEM_FP64) {
    SEM_CUDA_TRY(cudaMemcpyAsync(d_ops, d64.data(), need, cudaMemcpyHostToDevice, s));
  } else {
    std::vector<float> d32(d64.size());
    for (size_t q = 0; q < d64.size(); ++q) d32[q] = (float)d64[q];
    SEM_CUDA_TRY(cudaMemcpyAsync(d_ops, d32.data(), need, cudaMemcpyHostToDevice, s));
    SEM_CUDA_TRY(cudaStreamSynchronize(s));  // the host copy goes out of scope
    return SEM_OK;
  }
  SEM_CUDA_TRY(cudaStreamSynchronize(s));
  return SEM_OK;
}

extern "C" sem_status sem_dg_volume(sem_prec prec, int32_t N, int64_t E, double g, const void *d_ops, const void *d_Q,
                                    const void *d_Bxy, const void *d_geo, void *d_rhs, sem_stream_t stream) {
  if (!d_ops || !d_Q || !d_Bxy || !d_geo || !d_rhs) return sem_fail(SEM_ERR_INVALID, "NULL argument");
  if (E < 1) return sem_fail(SEM_ERR_INVALID, "element count must be positive");
  if (N < 1 || N > SEM_DG_MAX_ORDER) return sem_fail(SEM_ERR_INVALID, "DG order must be 1..8");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (prec == SEM_FP64) return dg_dispatch<double>(N, E, g, d_ops, d_Q, d_Bxy, d_geo, d_rhs, s);
  if (prec == SEM_FP32) return dg_dispatch<float>(N, E, g, d_ops, d_Q, d_Bxy, d_geo, d_rhs, s);
  return sem_fail(SEM_ERR_INVALID, "DG precision must be SEM_FP64 or SEM_FP32");
}

extern "C" sem_status sem_dg_geometry(sem_prec prec, int64_t E, const double *d_verts, void *d_geo,
                                      sem_stream_t stream) {
  if (!d_verts || !d_geo) return sem_fail(SEM_ERR_INVALID, "NULL argument");
  if (E < 1) return sem_fail(SEM_ERR_INVALID, "element count must be positive");
  if (prec != SEM_FP64 && prec != SEM_FP32) return sem_fail(SEM_ERR_INVALID, "DG precision must be FP64 or FP32");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  int *bad = nullptr;  // a static device word (calls on one device must not run concurrently)
  SEM_CUDA_TRY(cudaGetSymbolAddress(reinterpret_cast<void **>(&bad), g_dg_bad));
  SEM_CUDA_TRY(cudaMemsetAsync(bad, 0, sizeof(int), s));
  const unsigned blocks = (unsigned)((E + 255) / 256);
  if (prec == SEM_FP64)
    k_dg_geometry<double><<<blocks, 256, 0, s>>>(E, d_verts, static_cast<double *>(d_geo), bad);
  else
    k_dg_geometry<float><<<blocks, 256, 0, s>>>(E, d_verts, static_cast<float *>(d_geo), bad);
  SEM_CUDA_TRY(cudaGetLastError());
  int bad_h = 0;
  SEM_CUDA_TRY(cudaMemcpyAsync(&bad_h, bad, sizeof(int), cudaMemcpyDeviceToHost, s));
  SEM_CUDA_TRY(cudaStreamSynchronize(s));
  if (bad_h) return sem_fail(SEM_ERR_INVALID, "triangle with non-positive Jacobian (clockwise or degenerate)");
  return SEM_OK;
}
