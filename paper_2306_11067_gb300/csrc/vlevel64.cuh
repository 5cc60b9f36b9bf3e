// Levels of the V(1,1) cycle (Algorithm 1, nu = 1) in FP64 for a batch whose
// columns share one lambda: the two kernels per level of vfused.cuh, with
//
//  * on the coarse levels the 25 coefficients of K_k(lambda) = lambda^2 G_L
//    + G_A formed once per lambda (k_rows64, [25][n_k]) instead of at every
//    point of every sweep: half of the multiply-adds and half of the bytes;
//  * tiles of 2 x 2, 4 x 4 or 8 x 8 coarse points, chosen per level;
//  * a point's 25 coefficients, its r and D read before the window they are
//    applied to is formed, without bounds tests (one point per thread; the
//    loads behind tests at the boundary were waited for one by one): levels of
//    32 x 32 points 5.7 + 5.6 -> 4.2 + 3.6 us;
//  * no FP64 work for the interpolation weights (products of 1, 3/4 and 1/4,
//    read from a table).
//
// What bounds them: the FP64 pipe (19 cycles per warp instruction and SM).
// A level of 32 x 32 points is 4 tiles of 8 x 8 coarse points, so 4 SMs
// worked on it; smaller tiles compute more halo points in all but spread
// them over the SMs, and the launcher takes the tile side with the fewest
// residual points on the busiest SM (tiles64).  The sums per point are
// those of vfused.cuh in the same order.
#pragma once
#include <type_traits>

#include "vfused.cuh"

namespace lcmg {

// K(lambda) of a coarse level, coefficient o of point p at kr[o n + p]
struct RowsOp64 {
  int nv, nh;
  int64_t n;
  const double* __restrict__ kr;
  static constexpr int kRadius = 2;
  // the point's coefficients (zero towards points outside the level)
  struct Row {
    double k[25];
  };
  __device__ __forceinline__ Row row_of(int64_t p) const {
    Row w;
#pragma unroll
    for (int o = 0; o < 25; ++o) w.k[o] = kr[o * n + p];
    return w;
  }
  // (the caller's v is zero outside the level, and so are the coefficients)
  template <class F>
  __device__ __forceinline__ double apply_off(int64_t p, int, int, double, F v) const {
    double acc = 0;
#pragma unroll
    for (int o = 0; o < 25; ++o) acc += kr[o * n + p] * v(o % 5 - 2, o / 5 - 2);
    return acc;
  }
  template <class F>
  __device__ __forceinline__ double apply_row(const Row& w, F v) const {
    double acc = 0;
#pragma unroll
    for (int o = 0; o < 25; ++o) acc += w.k[o] * v(o % 5 - 2, o / 5 - 2);
    return acc;
  }
};

// An operator's data of one point, read before the window it is applied to
// is formed; the other operators read theirs as they go.
struct NoRow64 {};
template <bool kPre, class Op>
__device__ __forceinline__ auto row_of64(const Op& op, int64_t p, int i, int j) {
  if constexpr (kPre && std::is_same<Op, RowsOp64>::value)
    return op.row_of(p);
  else
    return NoRow64{};
}
template <class F>
__device__ __forceinline__ double apply64(const RowsOp64& op, const RowsOp64::Row& w, int64_t, int, int, double, F v) {
  return op.apply_row(w, v);
}
template <class Op, class F>
__device__ __forceinline__ double apply64(const Op& op, const NoRow64&, int64_t p, int i, int j, double l2, F v) {
  return op.apply_off(p, i, j, l2, v);
}

// kr = lam2 G_L + G_A (count = 25 n values)
static __global__ void k_rows64(int64_t count, const double* __restrict__ gl, const double* __restrict__ ga,
                                double lam2, double* __restrict__ kr) {
  for (int64_t t = (int64_t)blockIdx.x * kBlock + threadIdx.x; t < count; t += (int64_t)gridDim.x * kBlock)
    kr[t] = lam2 * gl[t] + ga[t];
}

// products of two 1-D interpolation weights by their kinds (0: 1, 1: 3/4,
// 2: 1/4, 3: outside)
__device__ __constant__ double kW64[4][4] = {{1.0, 0.75, 0.25, 0.0},
                                             {0.75, 0.5625, 0.1875, 0.0},
                                             {0.25, 0.1875, 0.0625, 0.0},
                                             {0.0, 0.0, 0.0, 0.0}};
// kind of pw1(a, I, nc)
__device__ __forceinline__ int pw_kind(int a, int I, int nc) {
  if (a < 0 || a >= 2 * nc || I < 0 || I >= nc) return 3;
  const int d = a - 2 * I;
  if (d == 0) return I == 0 ? 0 : 1;
  if (d == 1) return I == nc - 1 ? 0 : 1;
  return (d == -1 || d == 2) ? 2 : 3;
}

// threads of a block: a warp multiple that covers the residual window
__host__ __device__ constexpr int vt64_threads(int tc) {
  return tc == 2 ? 64 : tc == 4 ? 128 : 384;
}

template <class Op, int TC>
__global__ void __launch_bounds__(vt64_threads(TC))
    k_vdown64(Op op, int B, const double* __restrict__ lam2, const double* __restrict__ dinv,
              const double* __restrict__ r, double* __restrict__ zpre, double* __restrict__ rc, int ntx, int ntiles) {
  constexpr int NT = vt64_threads(TC);
  constexpr int H = Op::kRadius;
  constexpr int WR = 2 * TC + 2;   // restriction window
  constexpr int W1 = WR + 2 * H;   // z1 window
  __shared__ double s1[W1 * W1];
  __shared__ double sres[WR * WR];
  const int col = blockIdx.y;
  const int nv = op.nv, nh = op.nh, nvc = nv / 2, nhc = nh / 2;
  const double l2 = lam2[col];
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int I0 = tile % ntx * TC, J0 = tile / ntx * TC;
    const int ri = 2 * I0 - 1, rj = 2 * J0 - 1;
    // this thread's residual point (one: NT covers the window), its data read first
    static_assert(WR * WR <= NT, "one residual point per thread");
    const int pi = ri + (int)threadIdx.x % WR, pj = rj + (int)threadIdx.x / WR;
    const bool pin = threadIdx.x < WR * WR && pi >= 0 && pi < nv && pj >= 0 && pj < nh;
    const int64_t pp = pin ? (int64_t)pi + (int64_t)pj * nv : 0;
    const auto row = row_of64<true>(op, pp, pi, pj);
    const double rp = r[pp * B + col];
    // z1 = D r
    for (int t = threadIdx.x; t < W1 * W1; t += NT) {
      const int i = ri - H + t % W1, j = rj - H + t / W1;
      double v = 0;
      if (i >= 0 && i < nv && j >= 0 && j < nh) {
        const int64_t e = ((int64_t)i + (int64_t)j * nv) * B + col;
        v = dinv[e] * r[e];
        // the pre-smoothed z of the tile's own points
        if (i >= 2 * I0 && i < 2 * (I0 + TC) && j >= 2 * J0 && j < 2 * (J0 + TC)) zpre[e] = v;
      }
      s1[t] = v;
    }
    __syncthreads();
    // res = r - K z1 on the restriction window
    if (threadIdx.x < WR * WR) {
      const int q = (pi - ri + H) + (pj - rj + H) * W1;
      auto vz = [&](int di, int dj) { return s1[q + di + dj * W1]; };
      sres[threadIdx.x] = pin ? rp - apply64(op, row, pp, pi, pj, l2, vz) : 0.0;
    }
    __syncthreads();
    // r_c = R res
    for (int t = threadIdx.x; t < TC * TC; t += NT) {
      const int I = I0 + t % TC, J = J0 + t / TC;
      if (I >= nvc || J >= nhc) continue;
      int ka[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) ka[m] = pw_kind(2 * I - 1 + m, I, nvc);
      double acc = 0;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int kb = pw_kind(2 * J - 1 + u, J, nhc);
#pragma unroll
        for (int m = 0; m < 4; ++m)  // (the window is zero outside the level)
          acc += kW64[kb][ka[m]] * sres[(2 * I - 1 + m - ri) + (2 * J - 1 + u - rj) * WR];
      }
      rc[((int64_t)I + (int64_t)J * nvc) * B + col] = acc;
    }
    __syncthreads();  // the windows are refilled by the next tile
  }
}

template <class Op, int TC>
__global__ void __launch_bounds__(vt64_threads(TC))
    k_vup64(Op op, int B, const double* __restrict__ lam2, const double* __restrict__ dinv,
            const double* __restrict__ r, const double* __restrict__ ec, const double* __restrict__ zpre,
            double* __restrict__ zout, int ntx, int ntiles, double* __restrict__ part) {
  constexpr int NT = vt64_threads(TC);
  constexpr int H = Op::kRadius;
  constexpr int WF = 2 * TC;      // the tile's own points
  constexpr int W0 = WF + 2 * H;  // z0 window
  __shared__ double s0[W0 * W0];
  __shared__ double sred[NT / 32];
  const int col = blockIdx.y;
  const int nv = op.nv, nh = op.nh, nvc = nv / 2, nhc = nh / 2;
  const double l2 = lam2[col];
  double dacc = 0.0;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int fi = tile % ntx * WF, fj = tile / ntx * WF;
    // this thread's own point (one: NT covers the tile), its data read first
    static_assert(WF * WF <= NT, "one point per thread");
    const int pi = fi + (int)threadIdx.x % WF, pj = fj + (int)threadIdx.x / WF;
    const bool pin = threadIdx.x < WF * WF && pi < nv && pj < nh;
    const int64_t pp = pin ? (int64_t)pi + (int64_t)pj * nv : 0;
    constexpr bool kPre = TC < 8;  // (8 x 8 tiles: the registers would leave one block per SM)
    const auto row = row_of64<kPre>(op, pp, pi, pj);
    const double rp = r[pp * B + col], dp = dinv[pp * B + col];
    // z0 = z + P e_c
    for (int t = threadIdx.x; t < W0 * W0; t += NT) {
      const int a2 = fi - H + t % W0, b = fj - H + t / W0;
      double v = 0;
      if (a2 >= 0 && a2 < nv && b >= 0 && b < nh) {
        const int Is[2] = {a2 >> 1, (a2 & 1) ? (a2 >> 1) + 1 : (a2 >> 1) - 1};
        const int Js[2] = {b >> 1, (b & 1) ? (b >> 1) + 1 : (b >> 1) - 1};
        const int ka[2] = {pw_kind(a2, Is[0], nvc), pw_kind(a2, Is[1], nvc)};
        const int kb[2] = {pw_kind(b, Js[0], nhc), pw_kind(b, Js[1], nhc)};
        double acc = 0;
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int w = 0; w < 2; ++w)
            if (ka[w] != 3 && kb[u] != 3) acc += kW64[kb[u]][ka[w]] * ec[((int64_t)Is[w] + (int64_t)Js[u] * nvc) * B + col];
        v = zpre[((int64_t)a2 + (int64_t)b * nv) * B + col] + acc;
      }
      s0[t] = v;
    }
    __syncthreads();
    // z = z0 + D (r - K z0) on the tile's own points
    if (pin) {
      const int q = (pi - fi + H) + (pj - fj + H) * W0;
      auto vz = [&](int di, int dj) { return s0[q + di + dj * W0]; };
      const double zn = s0[q] + dp * (rp - apply64(op, row, pp, pi, pj, l2, vz));
      zout[pp * B + col] = zn;
      dacc += rp * zn;
    }
    __syncthreads();
  }
  if (part) vblock_sum<NT>(dacc, sred, part, B, col);
}

}  // namespace lcmg
