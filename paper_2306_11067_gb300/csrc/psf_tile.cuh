// Blur with a point-spread function that has no 1-D factors, in tiles.
//
// A block computes 32 points along i x TJ rows of one column; a thread four
// neighbouring points along i.  The samples (with a halo of the PSF's radii)
// and the coefficients lie in shared memory, both read in words of four: a
// thread keeps a window of eight samples of a row, so that 16 multiply-adds
// take two shared-memory reads, where one output per thread took two global
// reads per multiply-add.  The transposed operator is the same sum with the
// coefficients reversed along both axes.
//
// FP32 only: in FP64 the multiply-adds bound the plain form already (29 us at
// 200 x 152, 15 x 15 taps, against 39 in tiles).
//
// What bounds it: on images of a few hundred points a side the latency of
// the staging and of the 4 (2 rh + 1) (rv / 2 + 1) dependent window steps,
// so small images take tiles of 8 rows in blocks of two warps; on large ones
// the multiply-adds.  Measured on GB300 at 200 x 152, 15 x 15 taps,
// against one output per thread: A 19.8 -> 7.1 us, A^T with the epilogue 21.5 ->
// 9.0 us.
#pragma once
#include "kernels.cuh"

namespace lcmg {

constexpr int kPsfTI = 32;                 // points along i per tile
constexpr int kPsfWarps = 8;               // most warps per block
// Dynamic shared memory of a block without an opt-in: 48 KB less the kernel's
// own array (the warps' partial sums).  Larger PSFs keep one output per thread.
constexpr size_t kPsfSmem = 48 * 1024 - kPsfWarps * sizeof(double);

// epilogues, as of the banded passes
enum : int { PSF_STORE = 0, PSF_NORMAL = 1 };

__host__ __device__ constexpr int psf_padded(int taps) { return (taps + 3) / 4 * 4; }
inline size_t psf_smem(int rv, int rh, int tj) {
  const size_t ku = psf_padded(2 * rv + 1);
  return sizeof(float) * ((size_t)(tj + 2 * rh) * (kPsfTI + ku) + (size_t)(2 * rh + 1) * ku);
}

template <int TRANS, int EPI>
__global__ void __launch_bounds__(32 * kPsfWarps)
    k_psf_tile(PsfArgs a, const float* __restrict__ psf, int B, const float* __restrict__ in, float* __restrict__ out,
               FineOp<float> fop, const float* __restrict__ P, const double* __restrict__ lam2,
               double* __restrict__ part) {
  using Quad = Pack<float>;
  extern __shared__ __align__(16) float psf_raw[];
  __shared__ double sred[kPsfWarps];
  const int nv = a.nv, nh = a.nh, ku = 2 * a.rv + 1, kw = 2 * a.rh + 1, KU = psf_padded(ku), PW = kPsfTI + KU;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int tj = blockDim.x >> 3, li = threadIdx.x & 7, jl = threadIdx.x >> 3;
  const int col = blockIdx.y;
  float* sx = psf_raw;                            // sx[jj][m] = in(i0 - rv + m, j0 - rh + jj)
  float* sc = sx + (size_t)(tj + 2 * a.rh) * PW;  // sc[v][u], zero beyond the taps
  for (int e = threadIdx.x; e < kw * KU; e += blockDim.x) {
    const int v = e / KU, u = e - v * KU;
    sc[e] = u >= ku ? 0.f : TRANS ? psf[(ku - 1 - u) * kw + (kw - 1 - v)] : psf[u * kw + v];
  }
  const float l2 = EPI == PSF_NORMAL ? (float)lam2[col] : 0.f;
  Dot2 dot;
  const int nti = (nv + kPsfTI - 1) / kPsfTI, ntiles = nti * ((nh + tj - 1) / tj);
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int i0 = tile % nti * kPsfTI, j0 = tile / nti * tj;
    for (int row = w; row < tj + 2 * a.rh; row += nw) {
      const int j = j0 - a.rh + row;
      for (int m = lane; m < PW; m += 32) {
        const int i = i0 - a.rv + m;
        const bool ok = j >= 0 && j < nh && i >= 0 && i < nv;
        cp_async_elem(sx + row * PW + m, in + (ok ? ((int64_t)i + (int64_t)j * nv) * B + col : 0), in, ok);
      }
    }
    cp_async_wait_all();
    __syncthreads();
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int v = 0; v < kw; ++v) {
      const float* x = sx + (jl + v) * PW + 4 * li;
      const float* c = sc + v * KU;
      Quad w0 = *reinterpret_cast<const Quad*>(x);
      int u = 0;
      for (; u + 4 <= ku; u += 4) {
        const Quad w1 = *reinterpret_cast<const Quad*>(x + u + 4), k = *reinterpret_cast<const Quad*>(c + u);
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
          for (int t = 0; t < 4; ++t) acc[t] += k.v[e] * (t + e < 4 ? w0.v[(t + e) & 3] : w1.v[(t + e) & 3]);
        w0 = w1;
      }
      // the last one or three taps (the others of their word don't exist)
      const Quad w1 = *reinterpret_cast<const Quad*>(x + u + 4), k = *reinterpret_cast<const Quad*>(c + u);
#pragma unroll
      for (int e = 0; e < 3; ++e)
        if (u + e < ku) {
#pragma unroll
          for (int t = 0; t < 4; ++t) acc[t] += k.v[e] * (t + e < 4 ? w0.v[(t + e) & 3] : w1.v[(t + e) & 3]);
        }
    }
    const int j = j0 + jl;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int i = i0 + 4 * li + t;
      if (i >= nv || j >= nh) continue;
      const int64_t p = (int64_t)i + (int64_t)j * nv;
      if (EPI == PSF_STORE) {
        out[p * B + col] = acc[t];
      } else {
        auto pv = [&](int64_t q) { return P[q * B + col]; };
        const float kv = acc[t] + l2 * fop.lap(p, i, j, pv);
        out[p * B + col] = kv;
        dot.add(P[p * B + col], kv);
      }
    }
    __syncthreads();  // the samples are overwritten by the next tile
  }
  if (EPI != PSF_STORE) {
    const double s = dot.warp_sum();
    if (lane == 0) sred[w] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int k = 0; k < nw; ++k) t += sred[k];
      part[(int64_t)blockIdx.x * B + col] = t;
    }
  }
}

}  // namespace lcmg
