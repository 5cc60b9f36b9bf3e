// Device kernels of the multigrid-preconditioned CG solver.
//
// Operators (paper sections in brackets):
//   * K(lam) = A^T A + lam^2 L^T D^2 L, applied in two stages: y = A p (CSR
//     SpMM), then q = A^T y + lam^2 L^T W L p with W = D^2 (transposed CSR,
//     no atomics) with the dot p^T q fused  [Sec. 3.2, eq. (normal)].
//   * The V-cycle operator K_pre(lam) = lam^2 G_L + G_A with G_L^0 = L^T W L
//     (5-point, variable coefficient) and G_A^0 = diag(A^T A); coarse levels
//     are Galerkin products P^T G P with cell-centred bilinear P, which are
//     5 x 5 (25-point) stencils  [Sec. 3.1, Algorithm 1].
#pragma once
#include "common.cuh"

namespace lcmg {

// ---------------------------------------------------------------------------
// 1-D cell-centred linear interpolation weight P(a, I) from coarse cell I
// (of nc) to fine cell a (of 2 nc): 3/4 from the parent, 1/4 from the
// nearest other coarse cell; a missing neighbour's weight goes to the parent.
// ---------------------------------------------------------------------------
// (In the precision of the kernel that uses it: the weights 1, 3/4, 1/4
// are exact in any format, and an FP32 kernel then needs no FP64 work.)
template <class T = double>
__device__ __forceinline__ T pw1(int a, int I, int nc) {
  const int d = a - 2 * I;
  if (d == 0) return I == 0 ? T(1) : T(0.75);
  if (d == 1) return I == nc - 1 ? T(1) : T(0.75);
  if (d == -1 || d == 2) return T(0.25);
  return T(0);
}

// sum of v over a warp, in every lane
__device__ __forceinline__ double warp_sum64(double v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// Compensated dot product in the working precision (Ogita, Rump and Oishi,
// "Accurate sum and dot product", 2005, Algorithm Dot2): each product is
// split exactly into p + e with one FMA, the running sum is kept exact to
// rounding as s + c with TwoSum, so the result is as accurate as a dot
// product in twice the working precision.  The mixed path's FP32 kernels
// accumulate their dot products this way and convert s + c to FP64 once per
// thread: on this GPU the FP64 pipe runs at a small fraction of the FP32 one.
struct Dot2 {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float a, float b) {
    const float p = a * b;
    const float e = fmaf(a, b, -p);  // a b = p + e exactly
    const float t = s + p;
    const float z = t - s;
    c += (s - (t - z)) + (p - z) + e;  // TwoSum error of s + p, plus e
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
  __device__ __forceinline__ double warp_sum() const { return warp_sum64(value()); }
};

// A thread's dot-product accumulator: FP64 for FP64 vectors, Dot2 for FP32
template <class T>
struct DotAcc {
  double s = 0.0;
  __device__ __forceinline__ void add(double a, double b) { s += a * b; }
  __device__ __forceinline__ double value() const { return s; }
  __device__ __forceinline__ double warp_sum() const { return warp_sum64(s); }
};
template <>
struct DotAcc<float> : Dot2 {};

// ---------------------------------------------------------------------------
// Level operators
// ---------------------------------------------------------------------------
// Fine level: ws[p] = weight of edge (i,j)-(i+1,j), we[p] = weight of edge
// (i,j)-(i,j+1) (zero on the last row / column), ga = diag(A^T A).
template <class T>
struct FineOp {
  int nv, nh;
  const T* __restrict__ ws;
  const T* __restrict__ we;
  const T* __restrict__ ga;

  // (L^T W L z)_p for the value accessor v(q) of one column
  template <class F>
  __device__ __forceinline__ T lap(int64_t p, int i, int j, F v) const {
    const T zp = v(p);
    T acc = 0;
    if (i + 1 < nv) acc += ws[p] * (zp - v(p + 1));
    if (i > 0) acc += ws[p - 1] * (zp - v(p - 1));
    if (j + 1 < nh) acc += we[p] * (zp - v(p + nv));
    if (j > 0) acc += we[p - nv] * (zp - v(p - nv));
    return acc;
  }
  template <class F>
  __device__ __forceinline__ T apply(int64_t p, int i, int j, T lam2, F v) const {
    return lam2 * lap(p, i, j, v) + ga[p] * v(p);
  }
  // the same with the value accessor v(di, dj) of the neighbour at offset
  // (di, dj) (shared-memory tiles)
  static constexpr int kRadius = 1;
  template <class F>
  __device__ __forceinline__ T apply_off(int64_t p, int i, int j, T lam2, F v) const {
    const T zp = v(0, 0);
    T acc = 0;
    if (i + 1 < nv) acc += ws[p] * (zp - v(1, 0));
    if (i > 0) acc += ws[p - 1] * (zp - v(-1, 0));
    if (j + 1 < nh) acc += we[p] * (zp - v(0, 1));
    if (j > 0) acc += we[p - nv] * (zp - v(0, -1));
    return lam2 * acc + ga[p] * zp;
  }
  __device__ __forceinline__ double diagL(int64_t p, int i, int j) const {
    double s = 0;
    if (i + 1 < nv) s += (double)ws[p];
    if (i > 0) s += (double)ws[p - 1];
    if (j + 1 < nh) s += (double)we[p];
    if (j > 0) s += (double)we[p - nv];
    return s;
  }
  // sum_q |k_pq| and k_pp of lam2 G_L + G_A
  __device__ __forceinline__ double l1(int64_t p, int i, int j, double lam2) const {
    return 2.0 * lam2 * diagL(p, i, j) + (double)ga[p];
  }
  __device__ __forceinline__ double center(int64_t p, int i, int j, double lam2) const {
    return lam2 * diagL(p, i, j) + (double)ga[p];
  }
  // enumerate (neighbour, coefficient) of row p of lam2 G_L + G_A
  template <class F>
  __device__ __forceinline__ void row(int64_t p, int i, int j, double lam2, F emit) const {
    emit(p, center(p, i, j, lam2));
    if (i + 1 < nv) emit(p + 1, -lam2 * (double)ws[p]);
    if (i > 0) emit(p - 1, -lam2 * (double)ws[p - 1]);
    if (j + 1 < nh) emit(p + nv, -lam2 * (double)we[p]);
    if (j > 0) emit(p - nv, -lam2 * (double)we[p - nv]);
  }
};

// Coarse level: per point a row of kCoefStride values, the 25 coefficients
// of lam^2-part G_L at [0, 25) and of G_A at [32, 57); the coefficient of
// neighbour (i+di, j+dj) has offset o = (di+2) + 5 (dj+2).  Coefficients of
// neighbours outside the grid are zero.
constexpr int kCoefStride = 64;

template <class T>
struct CoefVec;
template <>
struct CoefVec<float> {
  using V = float4;
  static constexpr int W = 4;
};
template <>
struct CoefVec<double> {
  using V = double2;
  static constexpr int W = 2;
};

template <class T>
__device__ __forceinline__ void vstore(T* dst, const typename CoefVec<T>::V& v);
template <>
__device__ __forceinline__ void vstore<float>(float* d, const float4& v) { d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w; }
template <>
__device__ __forceinline__ void vstore<double>(double* d, const double2& v) { d[0] = v.x; d[1] = v.y; }

template <class T>
struct CoarseOp {
  int nv, nh;
  int64_t n;
  const T* __restrict__ cf;  // [n][kCoefStride]

  // k[o] = lam2 G_L[o] + G_A[o] for point p (vector loads)
  __device__ __forceinline__ void coefs(int64_t p, T lam2, T (&k)[28]) const {
    using VT = typename CoefVec<T>::V;
    constexpr int W = CoefVec<T>::W;
    const VT* row = reinterpret_cast<const VT*>(cf + p * kCoefStride);
    T gl[28], ga[28];
#pragma unroll
    for (int q = 0; q < 28 / W; ++q) {
      vstore<T>(gl + q * W, row[q]);
      vstore<T>(ga + q * W, row[32 / W + q]);
    }
#pragma unroll
    for (int o = 0; o < 28; ++o) k[o] = lam2 * gl[o] + ga[o];
  }

  template <class F>
  __device__ __forceinline__ T apply(int64_t p, int i, int j, T lam2, F v) const {
    T k[28];
    coefs(p, lam2, k);
    T acc = 0;
    if (i >= 2 && i + 2 < nv && j >= 2 && j + 2 < nh) {
#pragma unroll
      for (int dj = -2; dj <= 2; ++dj)
#pragma unroll
        for (int di = -2; di <= 2; ++di) acc += k[(di + 2) + 5 * (dj + 2)] * v(p + di + (int64_t)dj * nv);
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
        acc += k[(di + 2) + 5 * (dj + 2)] * v((int64_t)ii + (int64_t)jj * nv);
      }
    }
    return acc;
  }
  static constexpr int kRadius = 2;
  template <class F>
  __device__ __forceinline__ T apply_off(int64_t p, int i, int j, T lam2, F v) const {
    T k[28];
    coefs(p, lam2, k);
    return apply_k(k, i, j, v);
  }
  // the same with the coefficients k of the point already loaded (coefs)
  template <class F>
  __device__ __forceinline__ T apply_k(const T (&k)[28], int i, int j, F v) const {
    T acc = 0;
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
  __device__ __forceinline__ double l1(int64_t p, int i, int j, double lam2) const {
    const T* row = cf + p * kCoefStride;
    double s = 0;
    for (int o = 0; o < kStencil; ++o) s += fabs(lam2 * (double)row[o] + (double)row[32 + o]);
    return s;
  }
  __device__ __forceinline__ double center(int64_t p, int, int, double lam2) const {
    const T* row = cf + p * kCoefStride;
    return lam2 * (double)row[12] + (double)row[32 + 12];
  }
  template <class F>
  __device__ __forceinline__ void row(int64_t p, int i, int j, double lam2, F emit) const {
    const T* rw = cf + p * kCoefStride;
    for (int dj = -2; dj <= 2; ++dj) {
      const int jj = j + dj;
      if (jj < 0 || jj >= nh) continue;
      for (int di = -2; di <= 2; ++di) {
        const int ii = i + di;
        if (ii < 0 || ii >= nv) continue;
        const int o = (di + 2) + 5 * (dj + 2);
        emit((int64_t)ii + (int64_t)jj * nv, lam2 * (double)rw[o] + (double)rw[32 + o]);
      }
    }
  }
};

// SoA (25 x n per part, from the Galerkin products) -> AoS rows of the
// smoother; entries 25..31 and 57..63 are zero.
template <class T>
__global__ void k_coef_pack(int64_t n, const double* __restrict__ gl, const double* __restrict__ ga,
                            T* __restrict__ cf) {
  for (int64_t t = (int64_t)blockIdx.x * kBlock + threadIdx.x; t < n * kCoefStride;
       t += (int64_t)gridDim.x * kBlock) {
    const int64_t p = t / kCoefStride;
    const int o = (int)(t - p * kCoefStride);
    double v = 0.0;
    if (o < kStencil) v = gl[(int64_t)o * n + p];
    else if (o >= 32 && o < 32 + kStencil) v = ga[(int64_t)(o - 32) * n + p];
    cf[t] = (T)v;
  }
}

// ---------------------------------------------------------------------------
// Per-column PCG state (device) and the scalar updates that follow the dot
// products.  They run either as their own small kernels or in the last
// block of the kernel that produced the partial sums ("last block done":
// every block writes its partials, fences, takes a ticket; the block that
// takes the final ticket sums all partials in block order, so the result
// does not depend on which block finished last).
// ---------------------------------------------------------------------------
struct ColState {
  double* rz;      // r^T z of the current iterate
  double* rz2;     // the same value, written by every writer of rz; the
                   // one-column fused beta writes rz2 only and the fused
                   // alpha that follows reads rz2 and copies it to rz, so
                   // neither kernel reads a slot it writes
  double* alpha;
  double* beta;
  double* rr;      // ||r||^2 (recursive)
  double* rmax;    // largest ||r||^2 since the last reliable update
  double* tol2cc;  // tol^2 ||c||^2
  int* active;
  int* iters;
  int* status;
  int* pending;    // recursive residual reached tol: true residual needed
  int* counters;   // [0] active columns, [1] pending columns, [2] reliable-update votes
  int keep;        // 1: a column whose true residual fails the check continues
                   // from its current search direction (residual replacement);
                   // 0: it restarts with p = z
};

// The recursive residual of column col reached tol: the column waits for
// its true-residual check.  With st.keep its beta and rz advance as in a
// regular step (k_update_p then forms p = z + beta p for it), so that a
// failed check continues CG from that direction with the residual replaced.
__device__ __forceinline__ void mark_pending(const ColState& st, int col, double rzn) {
  st.pending[col] = 1;
  st.active[col] = 0;
  if (st.keep && rzn > 0.0) {
    st.beta[col] = rzn / st.rz[col];
    st.rz[col] = rzn;
    st.rz2[col] = rzn;
  } else {
    st.beta[col] = 0.0;
  }
}

// ---------------------------------------------------------------------------
// CSR SpMM over B interleaved columns.  One warp per row; the 32 lanes are
// S = 32/G nnz-groups x G column groups of CPG columns each, so a lane
// reads one (value, column) pair and CPG consecutive vector entries per
// step; the S partial sums are combined with xor shuffles.
//   MODE 0: Y[r] = (A X)[r]
//   MODE 1: Q[r] = (A^T Y)[r] + lam2 (L^T W L P)[r], dot partials of P.Q
//           (rows are pixels; X = Y of the first stage)
//   MODE 2: partials of ||(A X)[r] - b[r]||^2   (residual norm rho)
//   MODE 3: R[r] = C[r] - ((A^T Y)[r] + lam2 (L^T W L P)[r] + 0), partials
//           of R.R   (true residual of the normal equations)
// ---------------------------------------------------------------------------
struct SpmmArgs {
  int64_t rows;
  const int64_t* rp;
  const int32_t* ci;
  int B;        // leading dimension (columns) of every batched vector
  int c0;       // first column handled by this launch (blockIdx.y adds chunks)
  int nb;       // columns in [c0, c0 + nb) are handled
  int nl;       // MODE 2: lambdas per right-hand side (b column = col / nl)
  int nrhs;     // MODE 2: columns of b
  int variant;            // one-column kernel (k_spmv1): 0 = the pass's default,
                          // 1 = 32 lanes x 4, 2 = 16 lanes x 8, 3 = 8 lanes x 8;
                          // FP32 vectors only (else as 3): 4 = 8 x 8 with at
                          // least 5 blocks per SM, 5 = 8 x 8 with 6, 6 = 8 x 4
                          // with 8
  // one-column kernel: column of nonzero k of row r = rbase[r] + c16[k]
  // (null: ci), 6 instead of 8 bytes per FP32 nonzero
  const uint16_t* c16;
  const int32_t* rbase;
};

template <class V, class T, class TO, int G, int CPG, int MODE>
__global__ void __launch_bounds__(kBlock)
    k_spmm(SpmmArgs a, const V* __restrict__ va, const T* __restrict__ X, TO* __restrict__ Y,
           FineOp<T> fop, const T* __restrict__ P, const T* __restrict__ C,
           const double* __restrict__ lam2, const double* __restrict__ bvec,
           double* __restrict__ part) {
  constexpr int S = 32 / G;
  __shared__ double sdot[kBlock / 32][G * CPG];
  const int lane = threadIdx.x & 31, warp_in_block = threadIdx.x >> 5;
  const int g = lane % G, s = lane / G;
  const int64_t warp = ((int64_t)blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * kBlock) >> 5;
  const int cfirst = a.c0 + blockIdx.y * (G * CPG);
  const int cend = min(a.c0 + a.nb, cfirst + G * CPG);
  const int cbase = cfirst + g * CPG;
  double dacc[CPG];
#pragma unroll
  for (int t = 0; t < CPG; ++t) dacc[t] = 0.0;

  constexpr int U = 4;  // nonzeros per lane in flight
  for (int64_t r = warp; r < a.rows; r += nwarps) {
    const int64_t k0 = a.rp[r], k1 = a.rp[r + 1];
    T acc[CPG];
#pragma unroll
    for (int t = 0; t < CPG; ++t) acc[t] = 0;
    for (int64_t kb = k0 + s; kb < k1; kb += S * U) {
      // the matrix is streamed once per apply: load it evict-first so the
      // gathered vectors stay in L2; all loads of the step are independent
      int cu[U];
      T vu[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int64_t k = kb + (int64_t)u * S;
        const bool ok = k < k1;
        cu[u] = ok ? __ldcs(a.ci + k) : 0;
        vu[u] = ok ? (T)__ldcs(va + k) : (T)0;
      }
      T xv[U][CPG];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const T* xr = X + (int64_t)cu[u] * a.B + cbase;
#pragma unroll
        for (int t = 0; t < CPG; ++t) xv[u][t] = (cbase + t < cend) ? xr[t] : (T)0;
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int t = 0; t < CPG; ++t) acc[t] += vu[u] * xv[u][t];
    }
#pragma unroll
    for (int off = G; off < 32; off <<= 1)
#pragma unroll
      for (int t = 0; t < CPG; ++t) acc[t] += __shfl_xor_sync(0xffffffffu, acc[t], off);
    if (s == 0) {
      int i = 0, j = 0;
      if (MODE == 1 || MODE == 3) {
        j = (int)(r / fop.nv);
        i = (int)(r - (int64_t)j * fop.nv);
      }
#pragma unroll
      for (int t = 0; t < CPG; ++t) {
        const int col = cbase + t;
        if (col >= cend) continue;
        if (MODE == 0) {
          Y[r * a.B + col] = (TO)acc[t];
        } else if (MODE == 1 || MODE == 3) {
          auto pv = [&](int64_t q) { return P[q * a.B + col]; };
          const T lap = fop.lap(r, i, j, pv);
          const T qv = acc[t] + (T)lam2[col] * lap;
          if (MODE == 1) {
            Y[r * a.B + col] = (TO)qv;
            dacc[t] += to_d(P[r * a.B + col]) * to_d(qv);
          } else {
            const T rv = C[r * a.B + col] - qv;
            Y[r * a.B + col] = (TO)rv;
            dacc[t] += to_d(rv) * to_d(rv);
          }
        } else {  // MODE 2
          const double e = to_d(acc[t]) - bvec[r * a.nrhs + col / a.nl];
          dacc[t] += e * e;
        }
      }
    }
  }
  if (MODE != 0) {
    // lanes s == 0 hold the column-group sums of their warp
    if (s == 0) {
#pragma unroll
      for (int t = 0; t < CPG; ++t) sdot[warp_in_block][g * CPG + t] = dacc[t];
    }
    __syncthreads();
    const int width = cend - cfirst;
    if ((int)threadIdx.x < width) {
      double sum = 0.0;
      for (int w = 0; w < kBlock / 32; ++w) sum += sdot[w][threadIdx.x];
      part[(int64_t)blockIdx.x * a.B + cfirst + threadIdx.x] = sum;
    }
  }
}

// ---------------------------------------------------------------------------
// One column (a batch of B = 1, the paper's warm-start chain).  A row is
// handled by LPR lanes, so a warp works on 32 / LPR rows at once; each lane
// keeps U nonzeros in flight, and the row pointers of the warp's next rows
// are loaded before the current rows' gathers (PF).  Same modes as k_spmm.
// Measured on GB300 (256^2 CT, 15M nonzeros): y = A p is fastest with 32
// lanes per row and U = 4; the transposed pass, whose epilogue (L^T W L p
// and p.q) runs on one lane per row, with 8 lanes per row and U = 8.
// C16: column indices as 16-bit offsets from a per-row base (a.c16,
// a.rbase), when every row's column span is below 65,536.
// ---------------------------------------------------------------------------
// MINB: resident blocks per SM the register allocation must allow (the
// launch bound; more blocks = fewer registers per thread).
template <class T, int LPR>
constexpr int spmv1_minb() { return sizeof(T) == 4 ? (LPR == 32 ? 8 : 4) : (LPR == 32 ? 5 : 3); }

template <class V, class T, class TO, int MODE, int U, int LPR, bool PF, bool C16, int MINB>
__global__ void __launch_bounds__(kBlock, MINB)
    k_spmv1(SpmmArgs a, const V* __restrict__ va, const T* __restrict__ X, TO* __restrict__ Y,
            FineOp<T> fop, const T* __restrict__ P, const T* __restrict__ C,
            const double* __restrict__ lam2, const double* __restrict__ bvec,
            double* __restrict__ part) {
  constexpr int RPW = 32 / LPR;  // rows per warp step
  __shared__ double sdot[kBlock / 32];
  const int lane = threadIdx.x & 31;
  const int sl = lane % LPR, hw = lane / LPR;
  const int64_t warp = ((int64_t)blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * kBlock) >> 5;
  const int64_t ld = a.B;
  const int col = a.c0;
  const T l2 = (MODE == 1 || MODE == 3) ? (T)lam2[col] : (T)0;
  double dacc = 0.0;
  int64_t wr = warp;
  int64_t r = wr * RPW + hw;
  int64_t k0 = 0, k1 = 0;
  int rb = 0;
  if (r < a.rows) {
    k0 = a.rp[r];
    k1 = a.rp[r + 1];
    if (C16) rb = a.rbase[r];
  }
  // every lane of a warp runs the same number of steps (the shuffles below
  // take the whole warp); lanes past the last row compute nothing
  while (wr * RPW < a.rows) {
    const int64_t wrn = wr + nwarps;
    const int64_t rn = wrn * RPW + hw;
    int64_t k0n = 0, k1n = 0;
    int rbn = 0;
    if (PF && rn < a.rows) {
      k0n = a.rp[rn];
      k1n = a.rp[rn + 1];
      if (C16) rbn = a.rbase[rn];
    }
    T acc = 0;
    for (int64_t kb = k0 + sl; kb < k1; kb += LPR * U) {
      // the matrix is streamed once per apply: evict-first loads
      int cu[U];
      T vu[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int64_t k = kb + (int64_t)u * LPR;
        const bool ok = k < k1;
        if (C16)
          cu[u] = ok ? rb + (int)__ldcs(a.c16 + k) : 0;
        else
          cu[u] = ok ? __ldcs(a.ci + k) : 0;
        vu[u] = ok ? (T)__ldcs(va + k) : (T)0;
      }
      T xv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) xv[u] = X[(int64_t)cu[u] * ld + col];
#pragma unroll
      for (int u = 0; u < U; ++u) acc += vu[u] * xv[u];
    }
#pragma unroll
    for (int off = LPR / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (sl == 0 && r < a.rows) {
      if (MODE == 0) {
        Y[r * ld + col] = (TO)acc;
      } else if (MODE == 1 || MODE == 3) {
        const int j = (int)(r / fop.nv), i = (int)(r - (int64_t)j * fop.nv);
        auto pv = [&](int64_t q) { return P[q * ld + col]; };
        const T qv = acc + l2 * fop.lap(r, i, j, pv);
        if (MODE == 1) {
          Y[r * ld + col] = (TO)qv;
          dacc += to_d(P[r * ld + col]) * to_d(qv);
        } else {
          const T rv = C[r * ld + col] - qv;
          Y[r * ld + col] = (TO)rv;
          dacc += to_d(rv) * to_d(rv);
        }
      } else {  // MODE 2
        const double e = to_d(acc) - bvec[r * a.nrhs + col / a.nl];
        dacc += e * e;
      }
    }
    wr = wrn;
    r = rn;
    if (PF) {
      k0 = k0n;
      k1 = k1n;
      rb = rbn;
    } else if (r < a.rows) {
      k0 = a.rp[r];
      k1 = a.rp[r + 1];
      if (C16) rb = a.rbase[r];
    }
  }
  if (MODE != 0) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) dacc += __shfl_xor_sync(0xffffffffu, dacc, off);
    if (lane == 0) sdot[threadIdx.x >> 5] = dacc;
    __syncthreads();
    if (threadIdx.x == 0) {
      double sum = 0.0;
      for (int w = 0; w < kBlock / 32; ++w) sum += sdot[w];
      part[(int64_t)blockIdx.x * ld + col] = sum;
    }
  }
}

constexpr int kCsrPad = 4;  // padding elements after the last nonzero of a CSR array

// ---------------------------------------------------------------------------
// V-cycle level kernels (point x column mapping)
// ---------------------------------------------------------------------------
// dinv = 1 / sum_q |k_pq| (l1-Jacobi) or omega / k_pp (damped Jacobi)
template <class Op, class T>
__global__ void __launch_bounds__(kBlock)
    k_dinv(Op op, int64_t n, int B, const double* __restrict__ lam2, int smoother, double omega,
           T* __restrict__ dinv) {
  const ColMap cm(B);
  if (!cm.ok) return;
  for (int64_t p = cm.first(); p < n; p += cm.stride()) {
    const int j = (int)(p / op.nv), i = (int)(p - (int64_t)j * op.nv);
    const double l2 = lam2[cm.col];
    const double v = smoother == 0 ? 1.0 / op.l1(p, i, j, l2) : omega / op.center(p, i, j, l2);
    dinv[p * B + cm.col] = (T)v;
  }
}

// Pre-smoothing from a zero initial guess: one sweep gives z = dinv r; two
// sweeps give z = z1 + dinv (r - K z1) with z1 = dinv r formed on the fly.
template <class Op, class T>
__global__ void __launch_bounds__(kBlock)
    k_smooth_zero(Op op, int64_t n, int B, const T* __restrict__ lam2, const T* __restrict__ dinv,
                  const T* __restrict__ r, T* __restrict__ z, int two) {
  const ColMap cm(B);
  if (!cm.ok) return;
  const int col = cm.col;
  const T l2 = lam2[col];
  for (int64_t p = cm.first(); p < n; p += cm.stride()) {
    const T z1 = dinv[p * B + col] * r[p * B + col];
    if (!two) {
      z[p * B + col] = z1;
      continue;
    }
    const int j = (int)(p / op.nv), i = (int)(p - (int64_t)j * op.nv);
    auto v = [&](int64_t q) { return dinv[q * B + col] * r[q * B + col]; };
    const T kz = op.apply(p, i, j, l2, v);
    z[p * B + col] = z1 + dinv[p * B + col] * (r[p * B + col] - kz);
  }
}

// One Jacobi-type sweep zout = zin + dinv (r - K zin); optionally the
// partials of r . zout per column.
template <class Op, class T>
__global__ void __launch_bounds__(kBlock)
    k_smooth(Op op, int64_t n, int B, const T* __restrict__ lam2, const T* __restrict__ dinv,
             const T* __restrict__ r, const T* __restrict__ zin, T* __restrict__ zout,
             const int* __restrict__ active, double* __restrict__ part) {
  __shared__ double sm[kBlock];
  const ColMap cm(B);
  DotAcc<T> dacc;
  if (cm.ok) {
    const int col = cm.col;
    const T l2 = lam2[col];
    for (int64_t p = cm.first(); p < n; p += cm.stride()) {
      const int j = (int)(p / op.nv), i = (int)(p - (int64_t)j * op.nv);
      auto v = [&](int64_t q) { return zin[q * B + col]; };
      const T kz = op.apply(p, i, j, l2, v);
      const T rv = r[p * B + col];
      const T zn = zin[p * B + col] + dinv[p * B + col] * (rv - kz);
      zout[p * B + col] = zn;
      dacc.add(rv, zn);
    }
  }
  if (part) block_col_sum(dacc.value(), cm, sm, part + (int64_t)blockIdx.x * B);
}

// res = r - K z
template <class Op, class T>
__global__ void __launch_bounds__(kBlock)
    k_residual(Op op, int64_t n, int B, const T* __restrict__ lam2, const T* __restrict__ r,
               const T* __restrict__ z, T* __restrict__ res) {
  const ColMap cm(B);
  if (!cm.ok) return;
  const int col = cm.col;
  const T l2 = lam2[col];
  for (int64_t p = cm.first(); p < n; p += cm.stride()) {
    const int j = (int)(p / op.nv), i = (int)(p - (int64_t)j * op.nv);
    auto v = [&](int64_t q) { return z[q * B + col]; };
    res[p * B + col] = r[p * B + col] - op.apply(p, i, j, l2, v);
  }
}

// rc = P^T res_f  (R = P^T, Sec. 3.1)
template <class T>
__global__ void __launch_bounds__(kBlock)
    k_restrict(int nvc, int nhc, int B, const T* __restrict__ rf, T* __restrict__ rc) {
  const ColMap cm(B);
  if (!cm.ok) return;
  const int col = cm.col;
  const int nvf = 2 * nvc, nhf = 2 * nhc;
  const int64_t nc = (int64_t)nvc * nhc;
  for (int64_t p = cm.first(); p < nc; p += cm.stride()) {
    const int J = (int)(p / nvc), I = (int)(p - (int64_t)J * nvc);
    T acc = 0;
#pragma unroll
    for (int b = 2 * J - 1; b <= 2 * J + 2; ++b) {
      if (b < 0 || b >= nhf) continue;
      const T wb = pw1<T>(b, J, nhc);
#pragma unroll
      for (int a2 = 2 * I - 1; a2 <= 2 * I + 2; ++a2) {
        if (a2 < 0 || a2 >= nvf) continue;
        acc += wb * pw1<T>(a2, I, nvc) * rf[((int64_t)a2 + (int64_t)b * nvf) * B + col];
      }
    }
    rc[p * B + col] = acc;
  }
}

// z_f += P e_c
template <class T>
__global__ void __launch_bounds__(kBlock)
    k_prolong_add(int nvc, int nhc, int B, const T* __restrict__ ec, T* __restrict__ zf) {
  const ColMap cm(B);
  if (!cm.ok) return;
  const int col = cm.col;
  const int nvf = 2 * nvc;
  const int64_t nf = (int64_t)nvf * 2 * nhc;
  for (int64_t p = cm.first(); p < nf; p += cm.stride()) {
    const int b = (int)(p / nvf), a2 = (int)(p - (int64_t)b * nvf);
    const int I0 = a2 >> 1, J0 = b >> 1;
    const int I1 = (a2 & 1) ? I0 + 1 : I0 - 1;
    const int J1 = (b & 1) ? J0 + 1 : J0 - 1;
    T acc = 0;
    const int Is[2] = {I0, I1}, Js[2] = {J0, J1};
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int J = Js[u];
      if (J < 0 || J >= nhc) continue;
      const T wb = pw1<T>(b, J, nhc);
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const int I = Is[t];
        if (I < 0 || I >= nvc) continue;
        acc += wb * pw1<T>(a2, I, nvc) * ec[((int64_t)I + (int64_t)J * nvc) * B + col];
      }
    }
    zf[p * B + col] += acc;
  }
}

// ---------------------------------------------------------------------------
// Coarsest level: e = K_c(lam)^{-1} r with the explicit inverse (FP64).
// Block (x, col) computes rows 8x .. 8x + 7 of column col, one warp per row.
// ---------------------------------------------------------------------------
template <class T>
__global__ void __launch_bounds__(kBlock)
    k_coarse_solve(int nc, int B, const double* __restrict__ kinv, const T* __restrict__ rc,
                   T* __restrict__ ec) {
  extern __shared__ double rs[];
  const int col = blockIdx.y;
  for (int q = threadIdx.x; q < nc; q += kBlock) rs[q] = to_d(rc[(int64_t)q * B + col]);
  __syncthreads();
  const double* M = kinv + (int64_t)col * nc * nc;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  {
    const int i = blockIdx.x * (kBlock / 32) + w;
    if (i >= nc) return;
    double s = 0.0;
    for (int q = lane; q < nc; q += 32) s += M[(int64_t)i * nc + q] * rs[q];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) ec[(int64_t)i * B + col] = from_d<T>(s);
  }
}

// Assemble the dense K_c(lam) = lam^2 G_L + G_A of the coarsest level for
// every column: M[col][p][q].  M must be zeroed first.
template <class Op>
__global__ void __launch_bounds__(kBlock)
    k_dense_assemble(Op op, int64_t n, int B, const double* __restrict__ lam2,
                     double* __restrict__ M) {
  const ColMap cm(B);
  if (!cm.ok) return;
  for (int64_t p = cm.first(); p < n; p += cm.stride()) {
    const int j = (int)(p / op.nv), i = (int)(p - (int64_t)j * op.nv);
    double* row = M + ((int64_t)cm.col * n + p) * n;
    op.row(p, i, j, lam2[cm.col], [&](int64_t q, double k) { row[q] += k; });
  }
}

// Explicit inverse K^{-1} = L^{-T} L^{-1} of the coarsest-level matrices
// M = L L^T (symmetric positive definite, n x n, one per column of the
// batch).  Factorisation, X = L^{-1} and K^{-1} = X^T X advance together, 16
// columns of L per launch, in place on the lower triangle: at step k, with
// block row / column k the pivot,
//   tile (i, j), i >= j > k:  M_ij  -= L_ik L_jk^T       (trailing matrix)
//   tile (i, j), i > k >= j:  S_ij  -= L_ik X_kj         (S_ij becomes X_ij at step i)
//   tile (i, j), k >= i >= j: K_ij  += X_ki^T X_kj       (the inverse)
// where S_kk = I and the last two start from 0 at step j and at step i.  Both
// factors of every product are rows u solved against the pivot block's
// factor, u_t = (u_t - sum_{s<t} u_s L_ts) / L_tt: rows of M_ik, or columns
// of S_kj.  Every element sees the additions of the unblocked algorithm in
// its order (increasing k), so the result does not depend on the tiling.
//
// A step is two launches: k_inverse_panel solves the panel of every block row
// (one block each, which goes through the pivot block's 16 dependent pivots
// itself rather than wait for a third launch) and k_inverse_update advances
// every tile with two of the panels.
//
// What bounds it: the chain of pivots at small n (a square root of 590 cycles,
// a quotient of 575 and a multiply-add of 65 each), so little else stands in
// it: the pivot block and the panel have 256 threads each, and a column's
// threads lie in different SM quarters for the two solves; at large n the FP64
// pipe (less than two multiply-adds per clock and SM) of the updates.  A step
// reads `src` and writes `dst` (the pivot row and column are read by every
// panel).
// info[col] = the 1-based index of the first pivot that was not positive.
//
// The square root and the quotients are the correctly rounded ones of the
// library, so the values are those of the unblocked steps bit for bit.
// (One reciprocal per pivot and products round twice: a solution of the 256 x
// 256 CT system came out 1.1e-8 from the oracle's, where the quotients stay
// below 1e-8.)
//
// Measured on GB300, panel + update of a step: n = 160 17.1 + 4.1 us, n = 256
// 17.2 + 4.2, n = 567 17.2 + 8.4 (the panel 23.9 when zeros were divided too).
// One launch whose every tile solved both of its panels again took 18.7 us at
// 256 and 61 us at 567; one block per column that did all of it in global
// memory 123 ms at n = 567.
constexpr int kInvTile = 16;

// element (rr, cc) of tile (u, v), u >= v; a last partial tile is padded with
// the rows and columns of the identity
__device__ __forceinline__ double inverse_get(const double* __restrict__ S, int n, int u, int v, int rr, int cc) {
  const int i = u * kInvTile + rr, j = v * kInvTile + cc;
  if (i < n && j < n) return S[(int64_t)i * n + j];
  return i == j ? 1.0 : 0.0;
}

static __global__ void __launch_bounds__(2 * kInvTile * kInvTile)
    k_inverse_panel(int n, int k, const double* __restrict__ srcall, double* __restrict__ panall,
                    int* __restrict__ info) {
  constexpr int Q = kInvTile;
  // the pivot block (then its factor, lower triangle) and the panel
  __shared__ double A[2][Q][Q + 1];
  __shared__ double s_piv;
  __shared__ int bad;
  const int col = blockIdx.y, b = blockIdx.x;
  const double* __restrict__ S = srcall + (int64_t)col * n * n;
  // group 0: pivot block, 1: the panel of block row b; a half warp holds a
  // column, the groups' columns shifted by one warp
  const int g = threadIdx.x / (Q * Q), l = threadIdx.x % (Q * Q);
  const int c = 2 * ((l / 32 + 8 - g) % 8) + (l / 16) % 2, r = l % Q;
  auto get = [&](int u, int v, int rr, int cc) { return inverse_get(S, n, u, v, rr, cc); };
  double x;
  if (g == 0) {
    x = get(k, k, r, c);
  } else if (b > k) {  // rows of M_bk
    x = get(b, k, r, c);
  } else if (b == k) {  // the identity
    x = r == c ? 1.0 : 0.0;
  } else {  // the columns of S_kb
    x = get(k, b, c, r);
  }
  auto pivot = [&](int t, double a) {
    if (!(a > 0.0)) {
      if (!bad) bad = k * Q + t + 1;
      a = 1.0;
    }
    s_piv = sqrt(a);
  };
  if (threadIdx.x == 0) {
    bad = 0;
    pivot(0, x);
  }
  __syncthreads();
  for (int t = 0; t < Q; ++t) {
    if (c == t) {  // column t, final
      // zeros (and the pivot block's unused upper half) are kept out of the
      // division, whose path for them takes 1670 cycles instead of 730; the
      // empty asm keeps the compiler from folding the two selections away
      const double piv = s_piv;
      const bool skip = x == 0.0 || (g == 0 && r <= t);
      double num = skip ? 1.0 : x;
      asm volatile("" : "+d"(num));
      const double quot = num / piv;
      x = g == 0 && r == t ? piv : skip ? x : quot;
      A[g][r][t] = x;
    }
    __syncthreads();
    if (c > t && (g != 0 || r >= c)) {
      x -= A[g][r][t] * A[0][c][t];
      if (g == 0 && c == t + 1 && r == c) pivot(c, x);
    }
    __syncthreads();
  }
  if (b == 0 && threadIdx.x == 0 && bad && info[col] == 0) info[col] = bad;
  if (g == 1) panall[((int64_t)col * gridDim.x + b) * (Q * Q) + r * Q + c] = x;
}

// tile (bi, bj), bi >= bj, of the lower triangle: one thread per element
static __global__ void __launch_bounds__(kInvTile * kInvTile)
    k_inverse_update(int n, int nb, int k, int last, const double* __restrict__ srcall, double* __restrict__ dstall,
                     const double* __restrict__ panall) {
  constexpr int Q = kInvTile;
  __shared__ double A[2][Q][Q + 1];
  const int col = blockIdx.y;
  const double* __restrict__ S = srcall + (int64_t)col * n * n;
  double* __restrict__ O = dstall + (int64_t)col * n * n;
  int bi = (int)((sqrtf(8.f * (float)blockIdx.x + 1.f) - 1.f) * 0.5f);
  while ((bi + 1) * (bi + 2) / 2 <= (int)blockIdx.x) ++bi;
  while (bi * (bi + 1) / 2 > (int)blockIdx.x) --bi;
  const int bj = (int)blockIdx.x - bi * (bi + 1) / 2;
  const int r = threadIdx.x / Q, c = threadIdx.x % Q;
  const bool trail = bi > k;  // the tile subtracts (else it adds)
  const double* pan = panall + (int64_t)col * nb * (Q * Q) + threadIdx.x;
  double x = (trail ? bj == k : bi == k) ? 0.0 : inverse_get(S, n, bi, bj, r, c);
  const double u = pan[bi * (Q * Q)];
  A[0][r][c] = trail ? -u : u;
  A[1][r][c] = pan[bj * (Q * Q)];
  __syncthreads();
#pragma unroll
  for (int t = 0; t < Q; ++t) x = fma(A[0][r][t], A[1][c][t], x);
  const int i = bi * Q + r, j = bj * Q + c;
  if (i < n && j < n) {
    O[(int64_t)i * n + j] = x;
    if (last && bi != bj) O[(int64_t)j * n + i] = x;
  }
}

// ---------------------------------------------------------------------------
// Galerkin coarse operators G_c = P^T G_f P (Sec. 3.1).  The fine operator is either the level-0
// 5-point L^T W L (part 0), the level-0 diagonal diag(A^T A) (part 1), or a
// 25-point coarse stencil (part 2).
// ---------------------------------------------------------------------------
struct RapIn {
  int part;
  int nvf, nhf;
  int64_t nf;
  const double* ws;
  const double* we;
  const double* ga;
  const double* g25;
  __device__ __forceinline__ double coef(int di, int dj, int64_t f, int fi, int fj) const {
    if (part == 2) return g25[((di + 2) + 5 * (dj + 2)) * nf + f];
    if (part == 1) return (di == 0 && dj == 0) ? ga[f] : 0.0;
    // part 0: L^T W L
    if (di == 0 && dj == 0) {
      double s = 0;
      if (fi + 1 < nvf) s += ws[f];
      if (fi > 0) s += ws[f - 1];
      if (fj + 1 < nhf) s += we[f];
      if (fj > 0) s += we[f - nvf];
      return s;
    }
    if (dj == 0 && di == 1) return -ws[f];
    if (dj == 0 && di == -1) return -ws[f - 1];
    if (di == 0 && dj == 1) return -we[f];
    if (di == 0 && dj == -1) return -we[f - nvf];
    return 0.0;
  }
};

// P^T G P is contracted along i first, H(b, dj, I) = sum_{a, di} w(a, I)
// w(a + di, I + oi) G(di, dj; a, b) for the fine rows b of a tile of 32 x 2
// coarse points, and then along j from shared memory.  A block takes one of
// the five oi (blockIdx.y) of one of two operators on the same grid
// (blockIdx.z).
//
// What bounds it: the FP64 pipe (about 500 multiply-adds per us on the GPU,
// 19 cycles per warp instruction on an SM), so the two contractions take
// some 700 multiply-adds per coarse point where the product over all pairs of
// fine points took 1600 terms of four operations; on small levels one block's
// chain, so the oi are separate blocks.  Measured on GB300, both operators of
// a level, against one thread per (coarse point, offset): 256 x 160 coarse
// points (5-point fine operator) 322 -> 100 us, 128 x 80 274 -> 42 us, 64 x 40 152 ->
// 16 us.
constexpr int kGalTJ = 2;                           // coarse rows per tile
constexpr int kGalThreads = 32 * (2 * kGalTJ + 2);  // a warp per fine row

// The weight of fine point 2I - 1 + q in coarse point I of nc is 1/4, 3/4 or 1;
// gal_k tells which (0, 1, 2) and sW[3 a + b] holds the products of two (a
// table, so that no FP64 operation goes into weights)
__device__ __forceinline__ int gal_k(int q, int I, int nc) {
  return q == 1 ? (I == 0 ? 2 : 1) : q == 2 ? (I == nc - 1 ? 2 : 1) : 0;
}

// H of fine row b (|dj| <= R) for I: sH[dj + 2][lane]
template <int OI>
__device__ __forceinline__ void gal_row(const RapIn& in, int R, int I, int nvc, int b, const double* sW,
                                        double (*sH)[32], int lane) {
  const bool ok = I < nvc && I + OI >= 0 && I + OI < nvc && b >= 0 && b < in.nhf;
  double w[4][4];
#pragma unroll
  for (int m = 0; m < 4; ++m)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      constexpr int kShift = 2 * OI;
      if (kShift + q - m >= -2 && kShift + q - m <= 2) w[m][q] = sW[3 * gal_k(m, I, nvc) + gal_k(q, I + OI, nvc)];
    }
  for (int dj = -R; dj <= R; ++dj) {
    double h = 0.0;
    if (ok && b + dj >= 0 && b + dj < in.nhf) {
#pragma unroll
      for (int m = 0; m < 4; ++m)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          constexpr int kShift = 2 * OI;
          const int di = kShift + q - m;  // from fine point m of I to fine point q of I + OI
          if (di < -2 || di > 2) continue;
          if (in.part != 2 && ((di != 0 && dj != 0) || di < -R || di > R)) continue;
          const int a = 2 * I - 1 + m;
          if (a < 0 || a >= in.nvf || a + di < 0 || a + di >= in.nvf) continue;
          h += w[m][q] * in.coef(di, dj, (int64_t)a + (int64_t)b * in.nvf, a, b);
        }
    }
    sH[dj + 2][lane] = h;
  }
}

static __global__ void __launch_bounds__(kGalThreads)
    k_galerkin(RapIn in0, RapIn in1, int nvc, int nhc, double* __restrict__ out0, double* __restrict__ out1) {
  __shared__ double sH[2 * kGalTJ + 2][5][32];  // [fine row][dj][I]
  __shared__ double sW[9];
  if (threadIdx.x < 9) {
    const int a = threadIdx.x / 3, b = threadIdx.x % 3;
    sW[threadIdx.x] = (a == 0 ? 0.25 : a == 1 ? 0.75 : 1.0) * (b == 0 ? 0.25 : b == 1 ? 0.75 : 1.0);
  }
  __syncthreads();
  const RapIn& in = blockIdx.z == 0 ? in0 : in1;
  double* __restrict__ out = blockIdx.z == 0 ? out0 : out1;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nti = (nvc + 31) / 32, oi = (int)blockIdx.y - 2;
  const int I = (int)blockIdx.x % nti * 32 + lane, J0 = (int)blockIdx.x / nti * kGalTJ;
  const int R = in.part == 2 ? 2 : in.part == 0 ? 1 : 0;  // |dj| <= R
  const int64_t nc = (int64_t)nvc * nhc;
  const int b = 2 * J0 - 1 + w;  // along i: warp w takes fine row b
  switch (oi) {
    case -2: gal_row<-2>(in, R, I, nvc, b, sW, sH[w], lane); break;
    case -1: gal_row<-1>(in, R, I, nvc, b, sW, sH[w], lane); break;
    case 0: gal_row<0>(in, R, I, nvc, b, sW, sH[w], lane); break;
    case 1: gal_row<1>(in, R, I, nvc, b, sW, sH[w], lane); break;
    default: gal_row<2>(in, R, I, nvc, b, sW, sH[w], lane); break;
  }
  __syncthreads();
  // along j: the warps share (coarse row, oj)
  for (int task = w; task < 5 * kGalTJ; task += kGalThreads / 32) {
    const int Jl = task / 5, oj = task - 5 * Jl - 2, J = J0 + Jl;
    if (I >= nvc || J >= nhc) continue;
    double g = 0.0;
    if (I + oi >= 0 && I + oi < nvc && J + oj >= 0 && J + oj < nhc) {
#pragma unroll
      for (int m = 0; m < 4; ++m)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int dj = 2 * oj + q - m;
          if (dj < -R || dj > R) continue;
          g += sW[3 * gal_k(m, J, nhc) + gal_k(q, J + oj, nhc)] * sH[2 * Jl + m][dj + 2][lane];
        }
    }
    out[(int64_t)((oi + 2) + 5 * (oj + 2)) * nc + (int64_t)J * nvc + I] = g;
  }
}

// The same product term by term, one thread per (coarse point, offset): for
// the paper's own method (params.precond = 1), whose V(2,1) amplifies rounding
// so strongly that at small lambda FGMRES stalls near 1e-9; another order of
// these sums moved its solutions by 1e-8 there.
static __global__ void __launch_bounds__(kBlock) k_galerkin_terms(RapIn in, int nvc, int nhc, double* __restrict__ out) {
  const int64_t nc = (int64_t)nvc * nhc;
  const int R = (in.part == 2) ? 2 : 1;
  for (int64_t t = (int64_t)blockIdx.x * kBlock + threadIdx.x; t < nc * kStencil;
       t += (int64_t)gridDim.x * kBlock) {
    const int o = (int)(t / nc);
    const int64_t P = t - (int64_t)o * nc;
    const int J = (int)(P / nvc), I = (int)(P - (int64_t)J * nvc);
    const int oi = o % 5 - 2, oj = o / 5 - 2;
    const int It = I + oi, Jt = J + oj;
    double sum = 0.0;
    if (It >= 0 && It < nvc && Jt >= 0 && Jt < nhc) {
      for (int b = 2 * J - 1; b <= 2 * J + 2; ++b) {
        if (b < 0 || b >= in.nhf) continue;
        const double wb = pw1(b, J, nhc);
        for (int a = 2 * I - 1; a <= 2 * I + 2; ++a) {
          if (a < 0 || a >= in.nvf) continue;
          const double wab = wb * pw1(a, I, nvc);
          const int64_t f = (int64_t)a + (int64_t)b * in.nvf;
          for (int dj = -R; dj <= R; ++dj) {
            const int d = b + dj;
            if (d < 0 || d >= in.nhf) continue;
            const double wd = pw1(d, Jt, nhc);
            if (wd == 0.0) continue;
            for (int di = -R; di <= R; ++di) {
              const int c = a + di;
              if (c < 0 || c >= in.nvf) continue;
              if (in.part != 2 && di != 0 && dj != 0) continue;
              const double wc = pw1(c, It, nvc);
              if (wc == 0.0) continue;
              sum += wab * in.coef(di, dj, f, a, b) * wc * wd;
            }
          }
        }
      }
    }
    out[t] = sum;
  }
}

// ---------------------------------------------------------------------------
// PCG recurrences.  Per-column scalars live in device memory; a column
// whose active flag is 0 is frozen (converged, stopped, or waiting for its
// true-residual check) and left unchanged.
// ---------------------------------------------------------------------------
// x += alpha p ; r -= alpha q ; partials of r.r
template <class T, class TX>
__global__ void __launch_bounds__(kBlock)
    k_update_xr(int64_t n, int B, ColState st, const T* __restrict__ p, const T* __restrict__ q,
                TX* __restrict__ x, T* __restrict__ r, double* __restrict__ part) {
  __shared__ double sm[kBlock];
  const ColMap cm(B);
  DotAcc<T> acc;
  if (cm.ok && st.active[cm.col]) {
    const int col = cm.col;
    const double al = st.alpha[col];
    const T alT = (T)al;
    for (int64_t i = cm.first(); i < n; i += cm.stride()) {
      const int64_t e = i * B + col;
      x[e] = (TX)(x[e] + (TX)al * (TX)p[e]);
      const T rn = r[e] - alT * q[e];
      r[e] = rn;
      acc.add(rn, rn);
    }
  }
  block_col_sum(acc.value(), cm, sm, part + (int64_t)blockIdx.x * B);
}

// ---- one column: the updates with their scalars ---------------------------
// What bounds the two kernels: the vectors' bytes at large n (x, r read and
// written, p, q read; z read, p read and written), the latency of the partial sums and of
// the first loads at small n.  So the vectors move in 16-byte words, two
// words of each per thread in flight, the first two issued before the
// partial sums are taken; and the grid is at most two blocks of 512 threads
// per SM, since every block repeats the FP64 sums (the FP64 pipe runs at a
// small fraction of the FP32 one), which four warps share.  Measured on
// GB300 at 2048^2 in FP32, against scalar loads in a grid of four blocks of
// 256 threads per SM whose first warp summed alone: 33.7 -> 14.0 us and
// 21.8 -> 9.7 us (the reads, 67 and 34 MB, take 9.9 and 4.9 at the copy rate; the
// writes stay in L2; the rest is the partial sums ahead of the first store).
//
// At small n an FP64 warp instruction holds an SM for 19 cycles, so there are
// few of them: blocks of 256 threads, the block's r.r combined through shared
// memory by one warp (21 instead of 84), and the column state read before the
// sums rather than in the decision that follows them.  64 x 64 in FP64, against
// blocks of 512 and a shuffle tree per warp: 5.1 -> 4.3 and 4.9 -> 4.0 us.
constexpr int kUpdThreads = 512;
constexpr int kSumWarps = 4;  // warps that share one sum of partials

// This warp's share (warp wq of kSumWarps) of the sum of nb partials of one of
// B columns, in a fixed order, the same in every block; valid in every lane.
__device__ __forceinline__ double part_share(const double* __restrict__ part, int nb, int wq, int B = 1, int col = 0) {
  constexpr int U = 8;  // loads in flight
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  for (int base = 0; base < nb; base += 32 * kSumWarps * U) {
    double v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int b = base + (u * kSumWarps + wq) * 32 + lane;
      v[u] = b < nb ? part[(int64_t)b * B + col] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (base + u * kSumWarps * 32 < nb) s += v[u];
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  return s;
}

// 16 bytes of T
template <class T>
struct alignas(16) Pack {
  static constexpr int W = 16 / sizeof(T);
  T v[W];
};
template <class T>
__device__ __forceinline__ Pack<T> ld_pack(const T* a, int64_t i) {
  return reinterpret_cast<const Pack<T>*>(a)[i];
}
template <class T>
__device__ __forceinline__ void st_pack(T* a, int64_t i, const Pack<T>& v) {
  reinterpret_cast<Pack<T>*>(a)[i] = v;
}

// x += alpha p, r -= alpha q, partials of r.r, with alpha taken here: every
// block sums the p.q partials in the same fixed order, so all blocks compute
// the same alpha = rz / p.q (rz read from the rz2 slot) and the same
// breakdown decision; block 0 alone records the column state (iteration
// count, status, rz = rz2) and clears the counters the beta step
// accumulates.  No block reads what block 0 writes, and block 0 writes
// active = 0 only when every block has found the step void.
// (x, r, p, q are 16-byte aligned.)
template <class T>
__global__ void __launch_bounds__(kUpdThreads)
    k_update_xr_alpha(int64_t n, ColState st, int nb_pq, const double* __restrict__ pq_part,
                      const T* __restrict__ p, const T* __restrict__ q, T* __restrict__ x, T* __restrict__ r,
                      double* __restrict__ part) {
  using P = Pack<T>;
  __shared__ double s_al;
  __shared__ int s_ok;
  __shared__ double s_pq[kSumWarps];
  __shared__ double sm[kUpdThreads];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t nv = n / P::W, stride = (int64_t)gridDim.x * blockDim.x;
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  P xv[2], rv[2], pv[2], qv[2];
  auto load = [&](int64_t at) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (at + u * stride < nv) {
        pv[u] = ld_pack(p, at + u * stride);
        qv[u] = ld_pack(q, at + u * stride);
        xv[u] = ld_pack(x, at + u * stride);
        rv[u] = ld_pack(r, at + u * stride);
      }
  };
  load(i);
  const int act = st.active[0], its = st.iters[0];
  const double rzc = st.rz2[0];
  if (warp < kSumWarps) {
    const double s = part_share(pq_part, nb_pq, warp);
    if (lane == 0) s_pq[warp] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {  // the step length once per block
    const double pq = (s_pq[0] + s_pq[1]) + (s_pq[2] + s_pq[3]);
    const bool fin = isfinite(pq), ok = act && fin && pq > 0.0;
    const double al = ok ? rzc / pq : 0.0;
    s_ok = ok;
    s_al = al;
    if (blockIdx.x == 0) {
      st.rz[0] = rzc;
      st.counters[0] = 0;
      st.counters[1] = 0;
      st.counters[2] = 0;
      st.alpha[0] = al;
      if (act) {
        st.iters[0] = its + 1;
        if (!fin) {
          st.status[0] = ST_NONFINITE;
          st.active[0] = 0;
        } else if (!(pq > 0.0)) {
          st.status[0] = ST_BREAKDOWN;
          st.active[0] = 0;
        }
      }
    }
  }
  __syncthreads();
  DotAcc<T> dacc;
  if (s_ok) {
    const T al = (T)s_al;
    for (; i < nv; i += 2 * stride) {
      if (i >= 2 * stride) load(i);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        if (i + u * stride >= nv) break;
#pragma unroll
        for (int t = 0; t < P::W; ++t) {
          xv[u].v[t] += al * pv[u].v[t];
          rv[u].v[t] -= al * qv[u].v[t];
          dacc.add(rv[u].v[t], rv[u].v[t]);
        }
        st_pack(x, i + u * stride, xv[u]);
        st_pack(r, i + u * stride, rv[u]);
      }
    }
    const int64_t e = nv * P::W + threadIdx.x;  // the last n mod W elements
    if (blockIdx.x == 0 && e < n) {
      x[e] += al * p[e];
      const T rn = r[e] - al * q[e];
      r[e] = rn;
      dacc.add(rn, rn);
    }
  }
  sm[threadIdx.x] = dacc.value();
  __syncthreads();
  if (warp == 0) {
    double t = 0.0;
    for (int k = lane; k < (int)blockDim.x; k += 32) t += sm[k];
    t = warp_sum64(t);
    if (lane == 0) part[blockIdx.x] = t;
  }
}

// p = z + beta p with beta taken here (st.keep = 0): every block sums the
// r.r and r.z partials in the same fixed order and takes the same decision
// as k_scalar_col_beta (non-finite, converged -> true-residual check,
// iteration limit, breakdown, or a regular step with beta = rz_new / rz);
// only a regular step updates p.  Block 0 alone writes the column state; the
// new rz goes to the rz2 slot (the fused alpha of the next iteration reads
// it there and copies it to rz), so no block reads a value written in this
// kernel, and block 0 clears active only when every block has found no
// regular step.  (z, p are 16-byte aligned.)
template <class T>
__global__ void __launch_bounds__(kUpdThreads)
    k_update_p_beta(int64_t n, ColState st, int nb_rr, const double* __restrict__ rr_part, int nb_rz,
                    const double* __restrict__ rz_part, int maxit, double rel_trigger, const T* __restrict__ z,
                    T* __restrict__ p) {
  using P = Pack<T>;
  __shared__ double s_be;
  __shared__ int s_kind;
  __shared__ double s_sum[2 * kSumWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t nv = n / P::W, stride = (int64_t)gridDim.x * blockDim.x;
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  P zv[2], pv[2];
  auto load = [&](int64_t at) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (at + u * stride < nv) {
        zv[u] = ld_pack(z, at + u * stride);
        pv[u] = ld_pack(p, at + u * stride);
      }
  };
  load(i);
  const int act = st.active[0], its = st.iters[0], pend = st.pending[0];
  const double rz = st.rz[0], tol = st.tol2cc[0], rmax = st.rmax[0];
  if (warp < 2 * kSumWarps) {
    const double s = warp < kSumWarps ? part_share(rr_part, nb_rr, warp) : part_share(rz_part, nb_rz, warp - kSumWarps);
    if (lane == 0) s_sum[warp] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {  // the decision and beta once per block
    const double rr = (s_sum[0] + s_sum[1]) + (s_sum[2] + s_sum[3]);
    const double rzn = (s_sum[4] + s_sum[5]) + (s_sum[6] + s_sum[7]);
    int kind = -1;  // -1 inactive, 0 regular, 1 converged, 2 limit, 3 breakdown, 4 non-finite
    if (act) {
      if (!isfinite(rr) || !isfinite(rzn)) kind = 4;
      else if (rr <= tol) kind = 1;
      else if (its >= maxit) kind = 2;
      else if (!(rzn > 0.0)) kind = 3;
      else kind = 0;
    }
    const double be = kind == 0 ? rzn / rz : 0.0;
    s_kind = kind;
    s_be = be;
    if (blockIdx.x == 0) {
      if (act) {
        st.rr[0] = rr;
        if (kind == 0) {
          st.beta[0] = be;
          st.rz2[0] = rzn;
          if (rel_trigger > 0.0 && rr < rel_trigger * rmax) atomicAdd(&st.counters[2], 1);
        } else {
          st.beta[0] = 0.0;
          st.active[0] = 0;
          if (kind == 1) st.pending[0] = 1;
          if (kind == 2) st.status[0] = ST_MAXIT;
          if (kind == 3) st.status[0] = ST_BREAKDOWN;
          if (kind == 4) st.status[0] = ST_NONFINITE;
        }
      }
      if (kind == 0) atomicAdd(&st.counters[0], 1);
      if (pend || kind == 1) atomicAdd(&st.counters[1], 1);
    }
  }
  __syncthreads();
  if (s_kind != 0) return;
  const T be = (T)s_be;
  for (; i < nv; i += 2 * stride) {
    if (i >= 2 * stride) load(i);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (i + u * stride >= nv) break;
#pragma unroll
      for (int t = 0; t < P::W; ++t) pv[u].v[t] = zv[u].v[t] + be * pv[u].v[t];
      st_pack(p, i + u * stride, pv[u]);
    }
  }
  const int64_t e = nv * P::W + threadIdx.x;
  if (blockIdx.x == 0 && e < n) p[e] = z[e] + be * p[e];
}

// p = z + beta p
template <class T>
__global__ void __launch_bounds__(kBlock)
    k_update_p(int64_t n, int B, ColState st, const T* __restrict__ z, T* __restrict__ p) {
  const ColMap cm(B);
  if (!cm.ok || !(st.active[cm.col] || (st.keep && st.pending[cm.col]))) return;
  const int col = cm.col;
  const T be = (T)st.beta[col];
  for (int64_t i = cm.first(); i < n; i += cm.stride()) {
    const int64_t e = i * B + col;
    p[e] = z[e] + be * p[e];
  }
}

// restart for the flagged columns: p = z (and the caller sets rz)
template <class T>
__global__ void __launch_bounds__(kBlock)
    k_copy_cols(int64_t n, int B, const int* __restrict__ flag, const T* __restrict__ src,
                T* __restrict__ dst) {
  const ColMap cm(B);
  if (!cm.ok || (flag && !flag[cm.col])) return;
  for (int64_t i = cm.first(); i < n; i += cm.stride()) dst[i * B + cm.col] = src[i * B + cm.col];
}

// Scalar kernels run as one block of kScalarThreads threads: warp w sums
// the block partials of columns w, w + 32, ... with a fixed lane stride and
// shuffle tree (deterministic), and lane 0 applies the per-column update.
constexpr int kScalarThreads = 1024;

__device__ __forceinline__ double warp_sum_parts(const double* part, int nblk, int B, int col) {
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  for (int b = lane; b < nblk; b += 32) s += part[(int64_t)b * B + col];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  return s;
}

// serial form for callers that are one thread per column
__device__ __forceinline__ double sum_parts(const double* part, int nblk, int B, int col) {
  double s = 0.0;
  for (int b = 0; b < nblk; ++b) s += part[(int64_t)b * B + col];
  return s;
}

// One block per column sums that column's partials (a fixed order:
// deterministic), so that the FP64 additions are spread over B multiprocessors;
// four warps per sum, both sums of the beta step at once, since the adds of a
// shuffle tree cost an SM 19 cycles per warp.  Measured on GB300 against 16 warps
// and one sum after the other, 1216 partials, 4 columns: alpha 4.0 -> 2.5 us, beta
// 10.2 -> 4.3 us.
constexpr int kColThreads = 64 * kSumWarps;

// alpha = rz / p^T q ; grid = B blocks.  Also clears the counters that
// k_scalar_col_beta accumulates.
static __global__ void __launch_bounds__(kColThreads)
    k_scalar_col_alpha(int B, int nblk, const double* __restrict__ pq_part, ColState st) {
  __shared__ double s_sum[kSumWarps];
  const int col = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (col == 0 && threadIdx.x < 3) st.counters[threadIdx.x] = 0;
  const int act = st.active[col], its = st.iters[col];
  const double rz = st.rz[col];
  if (warp < kSumWarps) {
    const double s = part_share(pq_part, nblk, warp, B, col);
    if (lane == 0) s_sum[warp] = s;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  if (!act) {
    st.alpha[col] = 0.0;
    return;
  }
  const double pq = (s_sum[0] + s_sum[1]) + (s_sum[2] + s_sum[3]);
  st.iters[col] = its + 1;
  if (!isfinite(pq)) {
    st.status[col] = ST_NONFINITE;
    st.active[col] = 0;
    st.alpha[col] = 0.0;
  } else if (!(pq > 0.0)) {
    st.status[col] = ST_BREAKDOWN;
    st.active[col] = 0;
    st.alpha[col] = 0.0;
  } else {
    st.alpha[col] = rz / pq;
  }
}

// rr, recursive convergence and beta for one column per block; counters
// (cleared by k_scalar_col_alpha) accumulate with integer atomics.
static __global__ void __launch_bounds__(kColThreads)
    k_scalar_col_beta(int B, int nblk_rr, const double* __restrict__ rr_part, int nblk_rz,
                      const double* __restrict__ rz_part, ColState st, int maxit, double rel_trigger) {
  __shared__ double s_sum[2 * kSumWarps];
  const int col = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int act = st.active[col], its = st.iters[col];
  const double rz = st.rz[col], tol = st.tol2cc[col], rmax = st.rmax[col];
  const double s = warp < kSumWarps ? part_share(rr_part, nblk_rr, warp, B, col)
                                    : part_share(rz_part, nblk_rz, warp - kSumWarps, B, col);
  if (lane == 0) s_sum[warp] = s;
  __syncthreads();
  if (threadIdx.x != 0) return;
  if (act) {
    const double rr = (s_sum[0] + s_sum[1]) + (s_sum[2] + s_sum[3]);
    const double rzn = (s_sum[4] + s_sum[5]) + (s_sum[6] + s_sum[7]);
    st.rr[col] = rr;
    if (!isfinite(rr) || !isfinite(rzn)) {
      st.status[col] = ST_NONFINITE;
      st.active[col] = 0;
      st.beta[col] = 0.0;
    } else if (rr <= tol) {
      mark_pending(st, col, rzn);
    } else if (its >= maxit) {
      st.status[col] = ST_MAXIT;
      st.active[col] = 0;
      st.beta[col] = 0.0;
    } else if (!(rzn > 0.0)) {
      st.status[col] = ST_BREAKDOWN;
      st.active[col] = 0;
      st.beta[col] = 0.0;
    } else {
      st.beta[col] = rzn / rz;
      st.rz[col] = rzn;
      st.rz2[col] = rzn;
      if (rel_trigger > 0.0 && rr < rel_trigger * rmax) atomicAdd(&st.counters[2], 1);
    }
  }
  if (st.active[col]) atomicAdd(&st.counters[0], 1);
  if (st.pending[col]) atomicAdd(&st.counters[1], 1);
}

// Sum partials of a column reduction into out[col] (FP64).
static __global__ void __launch_bounds__(kScalarThreads)
    k_sum_parts(int B, int nblk, const double* __restrict__ part, double* __restrict__ out) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int col = w; col < B; col += kScalarThreads / 32) {
    const double s = warp_sum_parts(part, nblk, B, col);
    if (lane == 0) out[col] = s;
  }
}

// ---------------------------------------------------------------------------
// Element-wise helpers
// ---------------------------------------------------------------------------
// dst[p][j] = src[p][j / per] (expand per-right-hand-side data to columns)
template <class TS, class TD>
__global__ void k_expand_cols(int64_t n, int B, int per, int nsrc, const TS* __restrict__ src,
                              TD* __restrict__ dst) {
  const ColMap cm(B);
  if (!cm.ok) return;
  for (int64_t i = cm.first(); i < n; i += cm.stride())
    dst[i * B + cm.col] = (TD)src[i * nsrc + cm.col / per];
}

// convert / copy with type change
template <class TS, class TD>
__global__ void k_convert(int64_t count, const TS* __restrict__ src, TD* __restrict__ dst) {
  for (int64_t i = (int64_t)blockIdx.x * kBlock + threadIdx.x; i < count; i += (int64_t)gridDim.x * kBlock)
    dst[i] = (TD)src[i];
}

// planar [B][n] <-> interleaved [n][B]
static __global__ void k_planar_to_inter(int64_t n, int B, const double* __restrict__ src, double* __restrict__ dst) {
  const ColMap cm(B);
  if (!cm.ok) return;
  for (int64_t i = cm.first(); i < n; i += cm.stride()) dst[i * B + cm.col] = src[(int64_t)cm.col * n + i];
}
static __global__ void k_inter_to_planar(int64_t n, int B, const double* __restrict__ src, double* __restrict__ dst) {
  const ColMap cm(B);
  if (!cm.ok) return;
  for (int64_t i = cm.first(); i < n; i += cm.stride()) dst[(int64_t)cm.col * n + i] = src[i * B + cm.col];
}

// dst[i][j] = src_j[i] for planar column pointers src_j (null -> 0)
static __global__ void k_gather_cols(int64_t n, int B, const double* const* __restrict__ src,
                                     double* __restrict__ dst) {
  const ColMap cm(B);
  if (!cm.ok) return;
  const double* s = src[cm.col];
  for (int64_t i = cm.first(); i < n; i += cm.stride()) dst[i * B + cm.col] = s ? s[i] : 0.0;
}

// dst_j[i] = src[i][j] for non-null planar column pointers dst_j
static __global__ void k_scatter_cols(int64_t n, int B, const double* __restrict__ src,
                                      double* const* __restrict__ dst) {
  const ColMap cm(B);
  if (!cm.ok) return;
  double* d = dst[cm.col];
  if (!d) return;
  for (int64_t i = cm.first(); i < n; i += cm.stride()) d[i] = src[i * B + cm.col];
}

// dst[i][j] = src[i][map[j]] (src has nsrc columns)
static __global__ void k_gather_map(int64_t n, int B, int nsrc, const int* __restrict__ map,
                                    const double* __restrict__ src, double* __restrict__ dst) {
  const ColMap cm(B);
  if (!cm.ok) return;
  const int sc = map[cm.col];
  for (int64_t i = cm.first(); i < n; i += cm.stride()) dst[i * B + cm.col] = src[i * nsrc + sc];
}

static __global__ void k_negate(int64_t count, double* __restrict__ x) {
  for (int64_t i = (int64_t)blockIdx.x * kBlock + threadIdx.x; i < count; i += (int64_t)gridDim.x * kBlock)
    x[i] = -x[i];
}

// x64 += (double) xlo ; xlo = 0   (reliable update of the mixed path)
static __global__ void k_flush_x(int64_t count, float* __restrict__ xlo, double* __restrict__ x) {
  for (int64_t i = (int64_t)blockIdx.x * kBlock + threadIdx.x; i < count; i += (int64_t)gridDim.x * kBlock) {
    x[i] += (double)xlo[i];
    xlo[i] = 0.0f;
  }
}

// column sums of squares over the rows of A^T: diag(A^T A)
template <class V>
__global__ void k_diag_ata(int64_t n, const int64_t* __restrict__ rpT, const V* __restrict__ vT,
                           double* __restrict__ diag) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * kBlock) >> 5;
  for (int64_t r = warp; r < n; r += nw) {
    double s = 0.0;
    for (int64_t k = rpT[r] + lane; k < rpT[r + 1]; k += 32) {
      const double v = (double)vT[k];
      s += v * v;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) diag[r] = s;
  }
}

// edge weights d -> per-pixel squared weights ws, we
static __global__ void k_edge_to_pixel(int nv, int nh, const double* __restrict__ d, double* __restrict__ ws,
                                double* __restrict__ we) {
  const int64_t n = (int64_t)nv * nh;
  const int64_t nvert = (int64_t)nh * (nv - 1);
  for (int64_t p = (int64_t)blockIdx.x * kBlock + threadIdx.x; p < n; p += (int64_t)gridDim.x * kBlock) {
    const int j = (int)(p / nv), i = (int)(p - (int64_t)j * nv);
    double a = 0.0, b = 0.0;
    if (i + 1 < nv) {
      const double v = d[i + (int64_t)j * (nv - 1)];
      a = v * v;
    }
    if (j + 1 < nh) {
      const double v = d[nvert + i + (int64_t)j * nv];
      b = v * v;
    }
    ws[p] = a;
    we[p] = b;
  }
}

// eta^2 partials: ||D L x||^2 = sum ws (x_{p+1}-x_p)^2 + we (x_{p+nv}-x_p)^2
static __global__ void __launch_bounds__(kBlock)
    k_seminorm(int nv, int nh, int B, const double* __restrict__ ws, const double* __restrict__ we,
               const double* __restrict__ x, double* __restrict__ part) {
  __shared__ double sm[kBlock];
  const ColMap cm(B);
  const int64_t n = (int64_t)nv * nh;
  double acc = 0.0;
  if (cm.ok) {
    for (int64_t p = cm.first(); p < n; p += cm.stride()) {
      const int j = (int)(p / nv), i = (int)(p - (int64_t)j * nv);
      const double xp = x[p * B + cm.col];
      if (i + 1 < nv) {
        const double t = x[(p + 1) * B + cm.col] - xp;
        acc += ws[p] * t * t;
      }
      if (j + 1 < nh) {
        const double t = x[(p + nv) * B + cm.col] - xp;
        acc += we[p] * t * t;
      }
    }
  }
  block_col_sum(acc, cm, sm, part + (int64_t)blockIdx.x * B);
}

// weight update (eq. (g)): stage 1 writes |v_e| = |d_e (L x)_e| and block maxima
static __global__ void k_weighted_grad(int nv, int nh, const double* __restrict__ d, const double* __restrict__ x,
                                double* __restrict__ absv, double* __restrict__ bmax) {
  __shared__ double sm[kBlock];
  const int64_t nvert = (int64_t)nh * (nv - 1);
  const int64_t ne = nvert + (int64_t)(nh - 1) * nv;
  double m = 0.0;
  for (int64_t e = (int64_t)blockIdx.x * kBlock + threadIdx.x; e < ne; e += (int64_t)gridDim.x * kBlock) {
    double g;
    if (e < nvert) {
      const int64_t j = e / (nv - 1), i = e - j * (nv - 1);
      const int64_t p = i + j * nv;
      g = x[p + 1] - x[p];
    } else {
      const int64_t f = e - nvert;
      const int64_t j = f / nv, i = f - j * nv;
      const int64_t p = i + j * nv;
      g = x[p + nv] - x[p];
    }
    const double v = fabs(d[e] * g);
    absv[e] = v;
    m = fmax(m, v);
  }
  sm[threadIdx.x] = m;
  __syncthreads();
  for (int s = kBlock / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) sm[threadIdx.x] = fmax(sm[threadIdx.x], sm[threadIdx.x + s]);
    __syncthreads();
  }
  if (threadIdx.x == 0) bmax[blockIdx.x] = sm[0];
}

// stage 2: d <- max(1 - (|v|/vmax)^q, d_min) d   (unchanged if vmax == 0)
static __global__ void k_weight_apply(int64_t ne, int nblk, const double* __restrict__ bmax,
                               const double* __restrict__ absv, double q, double d_min,
                               double* __restrict__ d) {
  __shared__ double vmax;
  if (threadIdx.x == 0) {
    double m = 0.0;
    for (int b = 0; b < nblk; ++b) m = fmax(m, bmax[b]);
    vmax = m;
  }
  __syncthreads();
  if (vmax == 0.0) return;
  for (int64_t e = (int64_t)blockIdx.x * kBlock + threadIdx.x; e < ne; e += (int64_t)gridDim.x * kBlock) {
    const double g = absv[e] / vmax;
    const double gq = (q == 2.0) ? g * g : (q == 1.0 ? g : pow(g, q));
    d[e] = fmax(1.0 - gq, d_min) * d[e];
  }
}

// partials of x . y per column
template <class T>
__global__ void __launch_bounds__(kBlock)
    k_col_dot(int64_t n, int B, const T* __restrict__ x, const T* __restrict__ y, double* __restrict__ part) {
  __shared__ double sm[kBlock];
  const ColMap cm(B);
  DotAcc<T> acc;
  if (cm.ok)
    for (int64_t i = cm.first(); i < n; i += cm.stride()) acc.add(x[i * B + cm.col], y[i * B + cm.col]);
  block_col_sum(acc.value(), cm, sm, part + (int64_t)blockIdx.x * B);
}

// start of a solve: per-column state from ||c||^2 and the true residual
static __global__ void k_init_state(int B, double tol, const double* __restrict__ cc, const double* __restrict__ rr,
                             ColState st) {
  const int col = threadIdx.x;
  if (col >= B) return;
  st.tol2cc[col] = tol * tol * cc[col];
  st.iters[col] = 0;
  st.pending[col] = 0;
  st.rr[col] = rr[col];
  st.rmax[col] = rr[col];
  st.alpha[col] = 0.0;
  st.beta[col] = 0.0;
  if (!isfinite(rr[col])) {
    st.status[col] = ST_NONFINITE;
    st.active[col] = 0;
  } else if (rr[col] <= st.tol2cc[col]) {
    st.status[col] = ST_CONVERGED;
    st.active[col] = 0;
  } else {
    st.status[col] = ST_RUNNING;
    st.active[col] = 1;
  }
}

// True-residual check / reliable update.  flag[col]: 1 = restart (pending
// column whose true residual is still above tol), 2 = replace the residual
// of a running column (mixed path), 0 = leave.
static __global__ void k_true_check(int B, const double* __restrict__ rr_true, ColState st, int replace_active,
                             int* __restrict__ flag) {
  __shared__ int cnt[2];
  if (threadIdx.x < 2) cnt[threadIdx.x] = 0;
  __syncthreads();
  const int col = threadIdx.x;
  if (col < B) {
    int f = 0;
    const double rr = rr_true[col];
    if (st.pending[col]) {
      st.pending[col] = 0;
      if (rr <= st.tol2cc[col]) {
        st.status[col] = ST_CONVERGED;
      } else if (!isfinite(rr)) {
        st.status[col] = ST_NONFINITE;
      } else {
        st.active[col] = 1;
        st.rmax[col] = rr;
        st.rr[col] = rr;
        f = st.keep ? 2 : 1;  // 2: replace the residual only; 1: also restart
      }
    } else if (st.active[col] && replace_active) {
      st.rmax[col] = rr;
      st.rr[col] = rr;
      f = 2;
    }
    flag[col] = f;
    if (st.active[col]) atomicAdd(&cnt[0], 1);
    if (f == 1) atomicAdd(&cnt[1], 1);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    st.counters[0] = cnt[0];
    st.counters[1] = 0;
    st.counters[2] = 0;
    st.counters[3] = cnt[1];
  }
}

// r[:, col] = (T) r64[:, col] for flagged columns
template <class T>
__global__ void k_take_residual(int64_t n, int B, const int* __restrict__ flag, const double* __restrict__ r64,
                                T* __restrict__ r) {
  const ColMap cm(B);
  if (!cm.ok || !flag[cm.col]) return;
  for (int64_t i = cm.first(); i < n; i += cm.stride()) r[i * B + cm.col] = (T)r64[i * B + cm.col];
}

// after a restart V-cycle: rz = r.z and p = z for restarted columns
template <class T>
__global__ void k_restart_finish(int64_t n, int B, int nblk, const double* __restrict__ part,
                                 const int* __restrict__ flag, ColState st, const T* __restrict__ z,
                                 T* __restrict__ p) {
  const ColMap cm(B);
  if (!cm.ok || flag[cm.col] != 1) return;
  if (blockIdx.x == 0 && cm.k == 0) st.rz[cm.col] = st.rz2[cm.col] = sum_parts(part, nblk, B, cm.col);
  for (int64_t i = cm.first(); i < n; i += cm.stride()) p[i * B + cm.col] = z[i * B + cm.col];
}

// zero every column of a batch whose flag is set (c = 0 systems)
static __global__ void k_zero_cols(int64_t n, int B, const double* __restrict__ cc, double* __restrict__ x) {
  const ColMap cm(B);
  if (!cm.ok || cc[cm.col] != 0.0) return;
  for (int64_t i = cm.first(); i < n; i += cm.stride()) x[i * B + cm.col] = 0.0;
}

// ---------------------------------------------------------------------------
// Blur forward operator: zero-boundary correlation with a kh x kw PSF.
//   (A x)(i, j) = sum_{u,v} psf[u + rv][v + rh] x(i + u, j + v)
//   (A^T y)(i, j) = sum_{u,v} psf[u + rv][v + rh] y(i - u, j - v)
// ---------------------------------------------------------------------------
struct PsfArgs {
  int nv, nh, rv, rh;   // radii: kh = 2 rv + 1, kw = 2 rh + 1
  const double* psf;    // row-major kh x kw
};

template <class T, int TRANS>
__device__ __forceinline__ T psf_apply(const PsfArgs& a, const T* __restrict__ psf, int64_t p, int i, int j,
                                       const T* __restrict__ x, int B, int col) {
  const int kw = 2 * a.rh + 1;
  T acc = 0;
  for (int v = -a.rh; v <= a.rh; ++v) {
    const int jj = TRANS ? j - v : j + v;
    if (jj < 0 || jj >= a.nh) continue;
    for (int u = -a.rv; u <= a.rv; ++u) {
      const int ii = TRANS ? i - u : i + u;
      if (ii < 0 || ii >= a.nv) continue;
      acc += psf[(u + a.rv) * kw + (v + a.rh)] * x[((int64_t)ii + (int64_t)jj * a.nv) * B + col];
    }
  }
  return acc;
}

// y = A x (MODE 0) or partials of ||A x - b||^2 (MODE 2)
template <class T, int MODE>
__global__ void __launch_bounds__(kBlock)
    k_psf_forward(PsfArgs a, const T* __restrict__ psf, int B, const T* __restrict__ x, T* __restrict__ y,
                  const double* __restrict__ bvec, int nl, int nrhs, double* __restrict__ part) {
  __shared__ double sm[kBlock];
  const ColMap cm(B);
  const int64_t n = (int64_t)a.nv * a.nh;
  double acc = 0.0;
  if (cm.ok) {
    for (int64_t p = cm.first(); p < n; p += cm.stride()) {
      const int j = (int)(p / a.nv), i = (int)(p - (int64_t)j * a.nv);
      const T v = psf_apply<T, 0>(a, psf, p, i, j, x, B, cm.col);
      if (MODE == 0) {
        y[p * B + cm.col] = v;
      } else {
        const double e = to_d(v) - bvec[p * nrhs + cm.col / nl];
        acc += e * e;
      }
    }
  }
  if (MODE == 2) block_col_sum(acc, cm, sm, part + (int64_t)blockIdx.x * B);
}

// q = A^T y + lam2 L^T W L p with partials of p.q (MODE 1), or
// r = c - (A^T y + lam2 L^T W L p) with partials of r.r (MODE 3)
template <class T, class TO, int MODE>
__global__ void __launch_bounds__(kBlock)
    k_psf_normal(PsfArgs a, const T* __restrict__ psf, int B, const T* __restrict__ y, FineOp<T> fop,
                 const T* __restrict__ P, const T* __restrict__ C, const double* __restrict__ lam2,
                 TO* __restrict__ out, double* __restrict__ part) {
  __shared__ double sm[kBlock];
  const ColMap cm(B);
  const int64_t n = (int64_t)a.nv * a.nh;
  DotAcc<T> acc;
  if (cm.ok) {
    const int col = cm.col;
    const T l2 = (T)lam2[col];
    for (int64_t p = cm.first(); p < n; p += cm.stride()) {
      const int j = (int)(p / a.nv), i = (int)(p - (int64_t)j * a.nv);
      const T aty = psf_apply<T, 1>(a, psf, p, i, j, y, B, col);
      auto pv = [&](int64_t q) { return P[q * B + col]; };
      const T qv = aty + l2 * fop.lap(p, i, j, pv);
      if (MODE == 1) {
        out[p * B + col] = (TO)qv;
        acc.add(P[p * B + col], qv);
      } else {
        const T rv = C[p * B + col] - qv;
        out[p * B + col] = (TO)rv;
        acc.add(rv, rv);
      }
    }
  }
  block_col_sum(acc.value(), cm, sm, part + (int64_t)blockIdx.x * B);
}

// c = A^T b for the n_rhs right-hand sides (interleaved [n][nrhs])
static __global__ void k_psf_rhs(PsfArgs a, int nrhs, const double* __restrict__ b, double* __restrict__ c) {
  const ColMap cm(nrhs);
  if (!cm.ok) return;
  const int64_t n = (int64_t)a.nv * a.nh;
  for (int64_t p = cm.first(); p < n; p += cm.stride()) {
    const int j = (int)(p / a.nv), i = (int)(p - (int64_t)j * a.nv);
    c[p * nrhs + cm.col] = psf_apply<double, 1>(a, a.psf, p, i, j, b, nrhs, cm.col);
  }
}

// diag(A^T A)_p = sum of psf^2 over offsets whose row p - (u, v) is inside
static __global__ void k_psf_diag(PsfArgs a, double* __restrict__ diag) {
  const int64_t n = (int64_t)a.nv * a.nh;
  const int kw = 2 * a.rh + 1;
  for (int64_t p = (int64_t)blockIdx.x * kBlock + threadIdx.x; p < n; p += (int64_t)gridDim.x * kBlock) {
    const int j = (int)(p / a.nv), i = (int)(p - (int64_t)j * a.nv);
    double s = 0.0;
    for (int v = -a.rh; v <= a.rh; ++v) {
      const int jj = j - v;
      if (jj < 0 || jj >= a.nh) continue;
      for (int u = -a.rv; u <= a.rv; ++u) {
        const int ii = i - u;
        if (ii < 0 || ii >= a.nv) continue;
        const double w = a.psf[(u + a.rv) * kw + (v + a.rh)];
        s += w * w;
      }
    }
    diag[p] = s;
  }
}


}  // namespace lcmg
