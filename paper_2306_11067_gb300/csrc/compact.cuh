// FP16 storage of the V-cycle's smoother data (mixed precision, a batch
// whose columns share one lambda: the paper's chain and its right-hand-side
// batches).
//
// A V-cycle only has to be a fixed symmetric positive definite operator for
// PCG; its level operators need not be exact.  On the one-column chain the
// smoother data is most of what the cycle reads (a coarse point's stencil
// is 25 + 25 coefficients against one vector entry), so it is stored in
// FP16, each array scaled by a power of two that puts its largest value
// just below 2^13:
//
//  * finest level: the squared edge weights w_s, w_e and diag(A^T A), FP16
//    (lambda-independent, rebuilt with the weights); the cycle forms
//    lam^2 L^T W^ L + diag(ga^) from them, so the level operator keeps the
//    structure of the exact one (a weighted graph Laplacian plus a positive
//    diagonal) with every weight rounded to 11 significant bits;
//  * coarse level k: per lambda, the 24 off-diagonal coefficients of
//    K_k(lam) = lam^2 G_L^k + G_A^k, FP16 (48 bytes per point against 256
//    for the FP32 rows of both parts), and the diagonal in FP32: the row sum
//    s_p = (G_A^k 1)_p (the rows of G_L^k sum to zero) minus the sum of the
//    stored off-diagonals, so K^ 1 = G_A 1 exactly and the rounding perturbs
//    K by a zero-row-sum (Laplacian-like) term of relative size 2^-11 that
//    keeps it positive definite.
//
// The coarsest level keeps its exact FP64 factorisation.  Tested against
// the oracle's model of the same storage (oracle.multigrid, storage="fp16").
#pragma once
#include <cuda_fp16.h>

#include <cmath>

#include "kernels.cuh"

namespace lcmg {

constexpr int kCompactOff = 24;     // stored coefficients per coarse point
constexpr double kHalfTarget = 8192.0;  // scaled maxima lie in (4096, 8192]

// power of two putting max (> 0) in (kHalfTarget / 2, kHalfTarget]
inline double half_scale(double max) {
  if (!(max > 0.0)) return 1.0;
  return std::ldexp(1.0, (int)std::floor(std::log2(kHalfTarget / max)));
}

// finest level in FP16: the operator of FineOp with rounded weights
struct FineOpH {
  int nv, nh;
  const __half* __restrict__ ws;  // w_s 2^e_w
  const __half* __restrict__ we;  // w_e 2^e_w
  const __half* __restrict__ ga;  // diag(A^T A) 2^e_g
  float sw, sg;                   // 2^-e_w, 2^-e_g
  static constexpr int kRadius = 1;

  __device__ __forceinline__ float ws_(int64_t p) const { return __half2float(ws[p]) * sw; }
  __device__ __forceinline__ float we_(int64_t p) const { return __half2float(we[p]) * sw; }
  __device__ __forceinline__ float ga_(int64_t p) const { return __half2float(ga[p]) * sg; }

  template <class F>
  __device__ __forceinline__ float lap(int64_t p, int i, int j, F v) const {
    const float zp = v(p);
    float acc = 0;
    if (i + 1 < nv) acc += ws_(p) * (zp - v(p + 1));
    if (i > 0) acc += ws_(p - 1) * (zp - v(p - 1));
    if (j + 1 < nh) acc += we_(p) * (zp - v(p + nv));
    if (j > 0) acc += we_(p - nv) * (zp - v(p - nv));
    return acc;
  }
  template <class F>
  __device__ __forceinline__ float apply(int64_t p, int i, int j, float lam2, F v) const {
    return lam2 * lap(p, i, j, v) + ga_(p) * v(p);
  }
  template <class F>
  __device__ __forceinline__ float apply_off(int64_t p, int i, int j, float lam2, F v) const {
    const float zp = v(0, 0);
    float acc = 0;
    if (i + 1 < nv) acc += ws_(p) * (zp - v(1, 0));
    if (i > 0) acc += ws_(p - 1) * (zp - v(-1, 0));
    if (j + 1 < nh) acc += we_(p) * (zp - v(0, 1));
    if (j > 0) acc += we_(p - nv) * (zp - v(0, -1));
    return lam2 * acc + ga_(p) * zp;
  }
  __device__ __forceinline__ double diagL(int64_t p, int i, int j) const {
    double s = 0;
    if (i + 1 < nv) s += (double)ws_(p);
    if (i > 0) s += (double)ws_(p - 1);
    if (j + 1 < nh) s += (double)we_(p);
    if (j > 0) s += (double)we_(p - nv);
    return s;
  }
  __device__ __forceinline__ double l1(int64_t p, int i, int j, double lam2) const {
    return 2.0 * lam2 * diagL(p, i, j) + (double)ga_(p);
  }
  __device__ __forceinline__ double center(int64_t p, int i, int j, double lam2) const {
    return lam2 * diagL(p, i, j) + (double)ga_(p);
  }
};

// Coarse level in FP16: the off-diagonal coefficients of K(lam) for the
// offsets o = (di+2) + 5 (dj+2) in increasing o, o = 12 left out, scaled by
// 2^e, and per point the diagonal in the same units (the row sum of G_A
// minus the stored off-diagonals).  Two layouts, one per form of the cycle:
//
//  * one sweep (row streaming, vcoarse.cuh): the coefficients of 64 points of
//    a grid row lie together, [row j][block of 64 along i][24][64], so a warp
//    reads one coefficient of 64 points as one 128-byte line, the 24 of them
//    at fixed distances from one address;
//  * two sweeps (the tiles of vfused.cuh, one point per thread): the 24 of a
//    point lie together, three 16-byte words (kByPoint).  24 two-byte loads
//    per point made a cycle with two sweeps 5 to 13% slower: 1024 x 1024 156
//    -> 174 us, four columns of 512 x 512 164 -> 180 us on GB300.
template <bool kByPoint>
struct CoarseH16 {
  int nv, nh;
  int64_t n;
  const __half* __restrict__ rows;
  const float* __restrict__ c;     // diagonals x 2^e
  float sc;                        // 2^-e
  static constexpr int kRadius = 2;

  __host__ __device__ static int64_t blocks(int nv) { return (nv + 63) / 64; }
  // elements of `rows` (that of the blocks is at least 24 n)
  __host__ __device__ static int64_t size(int nv, int nh) { return blocks(nv) * nh * (24 * 64); }
  // blocks: the first coefficient of point (i, j); coefficient h follows at + 64 h
  __device__ __forceinline__ const __half* at(int i, int j) const {
    return rows + ((int64_t)j * blocks(nv) + (i >> 6)) * (24 * 64) + (i & 63);
  }

  // k[o] of K(lam) of point p = (i, j) for o < 25 (lam2 is already in the stored rows)
  __device__ __forceinline__ void coefs(int64_t p, int i, int j, float (&k)[28]) const {
    if constexpr (kByPoint) {
      const uint4* q = reinterpret_cast<const uint4*>(rows) + 3 * p;
      const uint4 q0 = q[0], q1 = q[1], q2 = q[2];
      const uint32_t w[12] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w, q2.x, q2.y, q2.z, q2.w};
#pragma unroll
      for (int h = 0; h < 12; ++h) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[h]));
        k[h < 6 ? 2 * h : 2 * h + 1] = f.x * sc;
        k[h < 6 ? 2 * h + 1 : 2 * h + 2] = f.y * sc;
      }
    } else {
      const __half* q = at(i, j);
#pragma unroll
      for (int h = 0; h < kCompactOff; ++h) k[h < 12 ? h : h + 1] = __half2float(q[64 * h]) * sc;
    }
    k[12] = c[p] * sc;
    k[25] = k[26] = k[27] = 0;
  }
  template <class F>
  __device__ __forceinline__ float apply_k(const float (&k)[28], int i, int j, F v) const {
    float acc = 0;
    if (i >= 2 && i + 2 < nv && j >= 2 && j + 2 < nh) {
#pragma unroll
      for (int dj = -2; dj <= 2; ++dj)
#pragma unroll
        for (int di = -2; di <= 2; ++di) acc += k[(di + 2) + 5 * (dj + 2)] * v(di, dj);
      return acc;
    }
#pragma unroll
    for (int dj = -2; dj <= 2; ++dj) {
      const int jj = j + dj;
      if (jj < 0 || jj >= nh) continue;
#pragma unroll
      for (int di = -2; di <= 2; ++di) {
        const int ii = i + di;
        if (ii < 0 || ii >= nv) continue;
        acc += k[(di + 2) + 5 * (dj + 2)] * v(di, dj);
      }
    }
    return acc;
  }
  template <class F>
  __device__ __forceinline__ float apply_off(int64_t p, int i, int j, float, F v) const {
    float k[28];
    coefs(p, i, j, k);
    return apply_k(k, i, j, v);
  }
  template <class F>
  __device__ __forceinline__ float apply(int64_t p, int i, int j, float lam2, F v) const {
    auto vo = [&](int di, int dj) { return v((int64_t)(i + di) + (int64_t)(j + dj) * nv); };
    return apply_off(p, i, j, lam2, vo);
  }
  __device__ __forceinline__ double l1(int64_t p, int i, int j, double) const {
    float k[28];
    coefs(p, i, j, k);
    double s1 = 0;
    for (int o = 0; o < kStencil; ++o) s1 += fabs((double)k[o]);
    return s1;
  }
  __device__ __forceinline__ double center(int64_t p, int i, int j, double) const {
    float k[28];
    coefs(p, i, j, k);
    return (double)k[12];
  }
};
using CoarseOpH = CoarseH16<false>;
using CoarseRowsH = CoarseH16<true>;

// dst = fp16(src * scale), rounded to nearest from FP64
static __global__ void k_half_scaled(int64_t n, const double* __restrict__ src, double scale,
                                     __half* __restrict__ dst) {
  for (int64_t p = (int64_t)blockIdx.x * kBlock + threadIdx.x; p < n; p += (int64_t)gridDim.x * kBlock)
    dst[p] = __double2half(src[p] * scale);
}

// s[p] = sum_o g[o][p] (25 x n SoA, o in increasing order), in FP32
static __global__ void k_rowsum25(int64_t n, const double* __restrict__ g, float* __restrict__ s) {
  for (int64_t p = (int64_t)blockIdx.x * kBlock + threadIdx.x; p < n; p += (int64_t)gridDim.x * kBlock) {
    double t = 0.0;
    for (int o = 0; o < kStencil; ++o) t += g[(int64_t)o * n + p];
    s[p] = (float)t;
  }
}

// *mx = max |v| over v (n values, or the 24 off-diagonal rows of a 25 x n
// SoA stencil when stencil25); non-negative doubles order like their bits
static __global__ void k_maxabs(int64_t n, const double* __restrict__ v, int stencil25,
                                unsigned long long* __restrict__ mx) {
  double m = 0.0;
  const int rows = stencil25 ? kStencil : 1;
  for (int o = 0; o < rows; ++o) {
    if (stencil25 && o == 12) continue;
    for (int64_t p = (int64_t)blockIdx.x * kBlock + threadIdx.x; p < n; p += (int64_t)gridDim.x * kBlock)
      m = fmax(m, fabs(v[(int64_t)o * n + p]));
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, off));
  if ((threadIdx.x & 31) == 0) atomicMax(mx, (unsigned long long)__double_as_longlong(m));
}

// The rows of K(lam) = lam2 G_L + G_A in FP16 (x scale, a power of two) and
// their diagonals: s the row sums of G_A.  One thread per point, so that
// every read of G_L and G_A runs along the points.
template <bool kByPoint>
static __global__ void __launch_bounds__(kBlock)
    k_compact_rows(int nv, int nh, int64_t n, const double* __restrict__ gl, const double* __restrict__ ga, double lam2,
                   double scale, const float* __restrict__ s, __half* __restrict__ rows, float* __restrict__ c) {
  const float fscale = (float)scale;
  for (int64_t p = (int64_t)blockIdx.x * kBlock + threadIdx.x; p < n; p += (int64_t)gridDim.x * kBlock) {
    const int j = (int)(p / nv), i = (int)(p - (int64_t)j * nv);
    __half* q = kByPoint ? rows + kCompactOff * p
                         : rows + ((int64_t)j * CoarseOpH::blocks(nv) + (i >> 6)) * (24 * 64) + (i & 63);
    float sum = 0.f;
#pragma unroll 8
    for (int h = 0; h < kCompactOff; ++h) {
      const int o = h < 12 ? h : h + 1;
      const double k = lam2 * gl[(int64_t)o * n + p] + ga[(int64_t)o * n + p];
      const __half v = __double2half(k * scale);
      q[(kByPoint ? 1 : 64) * h] = v;
      sum += __half2float(v);
    }
    c[p] = s[p] * fscale - sum;
  }
}

}  // namespace lcmg
