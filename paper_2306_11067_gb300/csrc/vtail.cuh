// The small coarse levels of the V(1,1) cycle (Algorithm 1, nu = 1, FP16
// level operators) and the coarsest-level solve in one kernel.
//
// Below about a thousand points a level's two kernels are a few
// microseconds of launch and memory latency each for a few kilobytes of
// work, and a 10-level cycle has several such levels.  Here one block of
// 1024 threads per column runs them all: down the levels (z1 = D r, res = r
// - K z1, r_c = R res), the coarsest solve (the dense inverse of the
// coarsest K(lambda) applied in FP64), and up again (z0 = z1 + P e_c, z =
// z0 + D (r - K z0)), with a block barrier between the steps.  Everything
// the levels read (the FP16 coefficients, diagonals, D and the right-hand
// side of the first of them) is copied into shared memory once, with
// asynchronous copies, and every vector the steps produce stays there: only
// the correction of the first tail level is written back.  A thread takes
// two neighbouring points; z and the residual lie in arrays with two zero
// points on every side, so that no stencil tests for the level's edge.  At
// most kTailPoints points on the first tail level keep the whole tail within
// shared memory whatever the level's shape.
#pragma once
#include "compact.cuh"
#include "launch.h"
#include "vcoarse.cuh"

namespace lcmg {

constexpr int kTailThreads = 1024;
constexpr int kTailMaxLevels = 12;

// one level of the tail and where its arrays live in shared memory (byte
// offsets, multiples of 16)
struct TailLevel {
  CoarseOpH op;         // in global memory (copied in)
  const float* dinv;    // global
  const float* rhs;     // global right-hand side (first level only)
  float* z;             // global correction (first level only)
  int o_rows, o_c, o_d, o_r, o_t, o_res, o_z;
};
struct TailArgs {
  int nlev;  // levels in the tail, the last one the coarsest
  TailLevel lv[kTailMaxLevels];
  const double* kinv;  // coarsest inverse, nc x nc per column
  int nc;
};
// floats of a level's array with two points of padding on every side
__host__ __device__ constexpr int tail_padded(int nv, int nh) { return (nv + 4) * (nh + 4); }

// (K z) at the points p, p + 1 of a level, in the operator's units: rows the
// level's coefficients [24][n], zp the padded z at point p
__device__ __forceinline__ Pair tail_apply(const __half* rows, const float* c, const float* zp, int n, int p, int ld) {
  Pair s{0.f, 0.f};
#pragma unroll
  for (int dj = 0; dj < 5; ++dj) {
    float z[6];
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const float2 f = *reinterpret_cast<const float2*>(zp + (dj - 2) * ld + 2 * t - 2);
      z[2 * t] = f.x;
      z[2 * t + 1] = f.y;
    }
#pragma unroll
    for (int di = 0; di < 5; ++di) {
      const int o = di + 5 * dj;
      const float2 k = o == 12 ? make_float2(c[p], c[p + 1])
                               : __half22float2(*reinterpret_cast<const __half2*>(rows + (o < 12 ? o : o - 1) * n + p));
      s.a += k.x * z[di];
      s.b += k.y * z[di + 1];
    }
  }
  return s;
}

__global__ void __launch_bounds__(kTailThreads) k_vtail_h(TailArgs a, int B) {
  extern __shared__ __align__(16) unsigned char tail_sm[];
  const int col = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto F = [&](int off) { return reinterpret_cast<float*>(tail_sm + off); };
  // copy in: coefficients, diagonals and D of every level but the coarsest,
  // the right-hand side of the first; zero the padded arrays
  for (int k = 0; k + 1 < a.nlev; ++k) {
    const TailLevel& L = a.lv[k];
    const int nv = L.op.nv, n = nv * L.op.nh, np = n / 2;
    float* rows = F(L.o_rows);  // pairs of coefficients
    for (int e = threadIdx.x; e < kCompactOff * np; e += kTailThreads) {
      const int h = e / np, p = 2 * (e - h * np);
      const int j = p / nv, i = p - j * nv;
      cp_async_elem(rows + e, reinterpret_cast<const float*>(L.op.at(i, j) + 64 * h), L.op.c, true);
    }
    float* c = F(L.o_c);
    float* d = F(L.o_d);
    for (int p = threadIdx.x; p < n; p += kTailThreads) {
      cp_async_elem(c + p, L.op.c + p, L.op.c, true);
      cp_async_elem(d + p, L.dinv + (int64_t)p * B + col, L.dinv, true);
    }
    if (k == 0) {
      float* r = F(L.o_r);
      for (int p = threadIdx.x; p < n; p += kTailThreads) cp_async_elem(r + p, L.rhs + (int64_t)p * B + col, L.rhs, true);
    }
    float *t = F(L.o_t), *res = F(L.o_res);
    for (int p = threadIdx.x; p < tail_padded(nv, L.op.nh); p += kTailThreads) t[p] = res[p] = 0.f;
  }
  cp_async_wait_all();
  __syncthreads();
  // down
  for (int k = 0; k + 1 < a.nlev; ++k) {
    const TailLevel& L = a.lv[k];
    const int nv = L.op.nv, nh = L.op.nh, nvc = nv / 2, nhc = nh / 2, ld = nv + 4;
    const int n = nv * nh;
    const __half* rows = reinterpret_cast<const __half*>(tail_sm + L.o_rows);
    const float *c = F(L.o_c), *d = F(L.o_d), *r = F(L.o_r);
    float *t = F(L.o_t), *res = F(L.o_res);
    for (int p = threadIdx.x; p < n; p += kTailThreads) {
      const int j = p / nv, i = p - j * nv;
      t[(i + 2) + (j + 2) * ld] = d[p] * r[p];
    }
    __syncthreads();
    for (int q = threadIdx.x; q < n / 2; q += kTailThreads) {
      const int p = 2 * q, j = p / nv, i = p - j * nv, e = (i + 2) + (j + 2) * ld;
      const Pair kz = tail_apply(rows, c, t + e, n, p, ld);
      res[e] = r[p] - kz.a * L.op.sc;
      res[e + 1] = r[p + 1] - kz.b * L.op.sc;
    }
    __syncthreads();
    float* rc = F(a.lv[k + 1].o_r);
    for (int P = threadIdx.x; P < nvc * nhc; P += kTailThreads) {
      const int J = P / nvc, I = P - J * nvc;
      const float wi[4] = {0.25f, I == 0 ? 1.f : 0.75f, I == nvc - 1 ? 1.f : 0.75f, 0.25f};
      const float wj[4] = {0.25f, J == 0 ? 1.f : 0.75f, J == nhc - 1 ? 1.f : 0.75f, 0.25f};
      float acc = 0.f;
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int m = 0; m < 4; ++m) acc += wj[u] * wi[m] * res[(2 * I + 1 + m) + (2 * J + 1 + u) * ld];
      rc[P] = acc;
    }
    __syncthreads();
  }
  // coarsest: e = K_c^{-1} r_c in FP64, one row per warp (as k_coarse_solve)
  {
    const TailLevel& C = a.lv[a.nlev - 1];
    const float* rc = F(C.o_r);
    float* ec = F(C.o_z);
    const double* M = a.kinv + (int64_t)col * a.nc * a.nc;
    for (int i = warp; i < a.nc; i += kTailThreads / 32) {
      double sum = 0.0;
      for (int q = lane; q < a.nc; q += 32) sum += M[(int64_t)i * a.nc + q] * (double)rc[q];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
      if (lane == 0) ec[i] = (float)sum;
    }
    __syncthreads();
  }
  // up
  for (int k = a.nlev - 2; k >= 0; --k) {
    const TailLevel& L = a.lv[k];
    const int nv = L.op.nv, nh = L.op.nh, nvc = nv / 2, nhc = nh / 2, ld = nv + 4;
    const int n = nv * nh;
    const __half* rows = reinterpret_cast<const __half*>(tail_sm + L.o_rows);
    const float *c = F(L.o_c), *d = F(L.o_d), *r = F(L.o_r), *t = F(L.o_t);
    const float* ec = F(a.lv[k + 1].o_z);
    float *z0 = F(L.o_res), *z = F(L.o_z);
    for (int p = threadIdx.x; p < n; p += kTailThreads) {
      const int j = p / nv, i = p - j * nv, e = (i + 2) + (j + 2) * ld;
      float wi, vi, wj, vj;
      pw1_near_far(i, nv, wi, vi);
      pw1_near_far(j, nh, wj, vj);
      const int Ia = i >> 1, Ja = j >> 1;
      const int Ib = min(max((i & 1) ? Ia + 1 : Ia - 1, 0), nvc - 1);
      const int Jb = min(max((j & 1) ? Ja + 1 : Ja - 1, 0), nhc - 1);
      z0[e] = t[e] + (wj * (wi * ec[Ia + Ja * nvc] + vi * ec[Ib + Ja * nvc]) +
                      vj * (wi * ec[Ia + Jb * nvc] + vi * ec[Ib + Jb * nvc]));
    }
    __syncthreads();
    for (int q = threadIdx.x; q < n / 2; q += kTailThreads) {
      const int p = 2 * q, j = p / nv, i = p - j * nv, e = (i + 2) + (j + 2) * ld;
      const Pair kz = tail_apply(rows, c, z0 + e, n, p, ld);
      const float za = z0[e] + d[p] * (r[p] - kz.a * L.op.sc);
      const float zb = z0[e + 1] + d[p + 1] * (r[p + 1] - kz.b * L.op.sc);
      float* o = k == 0 ? L.z + (int64_t)p * B + col : z + p;
      o[0] = za;
      o[k == 0 ? B : 1] = zb;
    }
    __syncthreads();
  }
}

}  // namespace lcmg
