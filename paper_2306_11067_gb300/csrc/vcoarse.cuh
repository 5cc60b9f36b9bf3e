// Coarse levels of the V(1,1) cycle (Algorithm 1, nu = 1) with FP16 level
// operators (CoarseOpH: 24 FP16 off-diagonal coefficients and an FP32
// diagonal per point), the mixed path's default for batches whose columns
// share one lambda:
//
//   k_vdown_h: res = r - K z1 with z1 = D r, r_c = R res         -> r_c
//   k_vup_h:   z0 = D r + P e_c, z = z0 + D (r - K z0)           -> z
//
// (z1 = D r is formed in both, not stored.)
//
// A warp owns 64 consecutive points along i, two per lane (a coarse column's
// own pair), and walks down a strip of rows j.  It keeps the 5 x 6 window of
// z around its two points in registers: a row enters once, its pair formed
// by the lane and the pairs of the neighbours along i taken by shuffles.  The
// edge lanes compute only what their neighbours need, so a warp produces 28
// coarse columns (down) or 60 columns of z (up).  A row's 24 coefficients are
// 24 loads of 128 bytes per warp at fixed distances, issued one row ahead.
//
// What bounds them: the latency of a row's loads (128 and 149 registers: 15
// and 12 warps per SM; the largest stalls at every size), at 1024^2 points with
// DRAM at half of its peak (48 of the 61 or so bytes per point are
// coefficients); so on the smaller levels strips are
// as short as it takes to give every SM 16 warps (a strip reads two rows more
// than it produces).  The 16 x 16 tiles staged in shared memory that they
// replace took about 860 warp instructions per 32 points (a 25-point stencil
// from shared memory at every point, halo points twice) where this takes
// some 90.  Measured on GB300 inside a 2048^2 solve, down / up, against those
// tiles: levels of 1024^2 and 512^2 points (mean) 19.9 / 20.2 -> 13.2 / 10.0 us,
// 256^2 4.2 / 4.7 -> 4.9 / 3.4 us (the coefficients from HBM); inside a 256^2
// one (levels of 128^2 to 32^2) 3.2 / 4.1 -> 2.5 / 2.7 us.
#pragma once
#include "compact.cuh"
#include "vfused.cuh"

namespace lcmg {

constexpr int kVcThreads = 128;
constexpr int kVcDownCols = 28;  // coarse columns per warp of k_vdown_h
constexpr int kVcUpCols = 30;    // coarse columns (pairs of z) per warp of k_vup_h
constexpr int kVcWarps = 16;     // warps per SM the strips aim at

// a lane's pair of points of one row
struct Pair {
  float a, b;
};
// the pair at points e, e + 1 of column col of an interleaved vector
template <bool kUnit>
__device__ __forceinline__ Pair ld_pair(const float* __restrict__ v, int64_t e, int B, int col) {
  if (kUnit) {
    const float2 f = *reinterpret_cast<const float2*>(v + e);
    return {f.x, f.y};
  }
  return {v[e * B + col], v[(e + 1) * B + col]};
}

// the coefficients of a lane's two points
struct PairRow {
  __half2 k[kCompactOff];
  Pair c;
};
__device__ __forceinline__ PairRow ld_row(const CoarseOpH& op, int i, int j) {
  PairRow q;
  const __half* b = op.at(i, j);
#pragma unroll
  for (int h = 0; h < kCompactOff; ++h) q.k[h] = *reinterpret_cast<const __half2*>(b + 64 * h);
  const float2 f = *reinterpret_cast<const float2*>(op.c + (int64_t)i + (int64_t)j * op.nv);
  q.c = {f.x, f.y};
  return q;
}

// z of rows j - 2 .. j + 2 at columns i - 2 .. i + 3 of the lane's pair (i, i + 1)
struct Window {
  float z[5][6];
  // the rows move up by one; the lane's pair of the new last row comes in
  __device__ __forceinline__ void push(const Pair& p) {
    const unsigned FULL = 0xffffffffu;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int t = 0; t < 6; ++t) z[u][t] = z[u + 1][t];
    z[4][0] = __shfl_up_sync(FULL, p.a, 1);
    z[4][1] = __shfl_up_sync(FULL, p.b, 1);
    z[4][2] = p.a;
    z[4][3] = p.b;
    z[4][4] = __shfl_down_sync(FULL, p.a, 1);
    z[4][5] = __shfl_down_sync(FULL, p.b, 1);
  }
  // (K z) at the pair of the middle row, in the operator's units
  __device__ __forceinline__ Pair apply(const PairRow& q) const {
    Pair s{0.f, 0.f};
#pragma unroll
    for (int o = 0; o < kStencil; ++o) {
      const int dj = o / 5, di = o % 5;
      const float2 k = o == 12 ? make_float2(q.c.a, q.c.b) : __half22float2(q.k[o < 12 ? o : o - 1]);
      s.a += k.x * z[dj][di];
      s.b += k.y * z[dj][di + 1];
    }
    return s;
  }
};

// pw1 of the nearer and the other coarse neighbour of fine index a on a line
// of n = 2 nc points (the other one falls outside at the ends)
__device__ __forceinline__ void pw1_near_far(int a, int n, float& wnear, float& wfar) {
  const bool edge = a == 0 || a == n - 1;
  wnear = edge ? 1.f : 0.75f;
  wfar = edge ? 0.f : 0.25f;
}

template <bool kUnit>
__global__ void __launch_bounds__(kVcThreads)
    k_vdown_h(CoarseOpH op, int B, const float* __restrict__ dinv, const float* __restrict__ r,
              float* __restrict__ rc, int nsi, int nstrips, int crows) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, col = blockIdx.y;
  const int nv = op.nv, nh = op.nh, nvc = nv / 2, nhc = nh / 2;
  const int st = blockIdx.x * (kVcThreads / 32) + (threadIdx.x >> 5);
  if (st >= nstrips) return;
  const int I = st % nsi * kVcDownCols - 2 + lane;  // z1 at every lane, res at 1..30, r_c at 2..29
  const int J0 = st / nsi * crows, J1 = min(J0 + crows, nhc);
  const bool in_i = I >= 0 && I < nvc;
  const int i = in_i ? 2 * I : 0;
  const bool out = in_i && lane >= 2 && lane < 2 + kVcDownCols;
  const float sc = op.sc;
  // restriction along i from the residuals at 2I - 1 .. 2I + 2
  const float w1 = I == 0 ? 1.f : 0.75f, w2 = I == nvc - 1 ? 1.f : 0.75f;
  // r and z1 = D r of row j (zero outside the level)
  auto load = [&](int j, Pair& rv, Pair& dv) {
    const int64_t e = (int64_t)i + (int64_t)min(max(j, 0), nh - 1) * nv;
    rv = ld_pair<kUnit>(r, e, B, col);
    dv = ld_pair<kUnit>(dinv, e, B, col);
    if (!in_i || j < 0 || j >= nh) rv.a = rv.b = 0.f;
  };
  const int b0 = 2 * J0 - 1, b1 = 2 * J1;  // residual rows
  float prev = 0.f, cur = 0.f;  // r_c of coarse rows (b - 1) / 2 and (b + 1) / 2 being summed
  Window W;
  // residual row b (z1 of rows b - 2 .. b + 2 in the window, rb its r)
  auto residual_row = [&](int b, const PairRow& kb, const Pair& rb) {
    const Pair kz = W.apply(kb);
    const bool in = in_i && b >= 0 && b < nh;
    const float ra = in ? rb.a - kz.a * sc : 0.f, rb2 = in ? rb.b - kz.b * sc : 0.f;
    const float left = __shfl_up_sync(FULL, rb2, 1), right = __shfl_down_sync(FULL, ra, 1);
    const float ti = 0.25f * left + w1 * ra + w2 * rb2 + 0.25f * right;
    const float wb = (b == 0 || b == nh - 1) ? 1.f : 0.75f;  // pw1(b, b / 2)
    const int m = b >> 1;
    if ((b & 1) == 0) {  // b = 2m: the last term of coarse row m - 1, the second of row m
      prev += 0.25f * ti;
      if (out && m - 1 >= J0) rc[((int64_t)I + (int64_t)(m - 1) * nvc) * B + col] = prev;
      prev = cur + wb * ti;
      cur = 0.f;
    } else {  // b = 2m + 1: the third term of row m, the first of row m + 1
      prev += wb * ti;
      cur += 0.25f * ti;
    }
  };
  // every first load is issued before the first shuffle
  Pair r5[5], d5[5];
#pragma unroll
  for (int u = 0; u < 5; ++u) load(b0 - 2 + u, r5[u], d5[u]);
  PairRow k = ld_row(op, i, max(b0, 0));
#pragma unroll
  for (int u = 0; u < 4; ++u) W.push({d5[u].a * r5[u].a, d5[u].b * r5[u].b});
  Pair r0 = r5[2], r1 = r5[3], rv = r5[4], dv = d5[4];  // r of rows b, b + 1 and b + 2
#pragma unroll 2
  for (int b = b0; b <= b1; ++b) {
    W.push({dv.a * rv.a, dv.b * rv.b});
    const Pair rb = r0;
    r0 = r1;
    r1 = rv;
    const PairRow kb = k;
    if (b < b1) {  // the next row's loads
      load(b + 3, rv, dv);
      k = ld_row(op, i, min(b + 1, nh - 1));
    }
    residual_row(b, kb, rb);
  }
}

// k_vdown_h on small levels: a block takes 28 coarse points of one coarse row,
// each of its four warps one of the four residual rows, so that the rows' load
// latencies don't add up.
template <bool kUnit>
__global__ void __launch_bounds__(kVcThreads)
    k_vdown_h1(CoarseOpH op, int B, const float* __restrict__ dinv, const float* __restrict__ r,
               float* __restrict__ rc, int nsi) {
  static_assert(kVcThreads == 128, "a warp per residual row");
  __shared__ float st[4][32];
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, col = blockIdx.y;
  const int nv = op.nv, nh = op.nh, nvc = nv / 2;
  const int I = (int)blockIdx.x % nsi * kVcDownCols - 2 + lane, J = (int)blockIdx.x / nsi;
  const bool in_i = I >= 0 && I < nvc;
  const int i = in_i ? 2 * I : 0, b = 2 * J - 1 + w;
  const PairRow k = ld_row(op, i, min(max(b, 0), nh - 1));
  Pair rv[5], dv[5];
#pragma unroll
  for (int u = 0; u < 5; ++u) {
    const int j = b - 2 + u;
    const int64_t e = (int64_t)i + (int64_t)min(max(j, 0), nh - 1) * nv;
    rv[u] = ld_pair<kUnit>(r, e, B, col);
    dv[u] = ld_pair<kUnit>(dinv, e, B, col);
    if (!in_i || j < 0 || j >= nh) rv[u].a = rv[u].b = 0.f;
  }
  Window W;
#pragma unroll
  for (int u = 0; u < 5; ++u) W.push({dv[u].a * rv[u].a, dv[u].b * rv[u].b});
  const Pair kz = W.apply(k);
  const bool in = in_i && b >= 0 && b < nh;
  const float ra = in ? rv[2].a - kz.a * op.sc : 0.f, rb = in ? rv[2].b - kz.b * op.sc : 0.f;
  const float left = __shfl_up_sync(FULL, rb, 1), right = __shfl_down_sync(FULL, ra, 1);
  const float ti = 0.25f * left + (I == 0 ? 1.f : 0.75f) * ra + (I == nvc - 1 ? 1.f : 0.75f) * rb + 0.25f * right;
  st[w][lane] = (w == 0 || w == 3 ? 0.25f : b == 0 || b == nh - 1 ? 1.f : 0.75f) * ti;
  __syncthreads();
  if (w == 0 && in_i && lane >= 2 && lane < 2 + kVcDownCols)
    rc[((int64_t)I + (int64_t)J * nvc) * B + col] = (st[0][lane] + st[1][lane]) + (st[2][lane] + st[3][lane]);
}

template <bool kUnit>
__global__ void __launch_bounds__(kVcThreads)
    k_vup_h(CoarseOpH op, int B, const float* __restrict__ dinv, const float* __restrict__ r,
            const float* __restrict__ ec, float* __restrict__ zout, int nsi, int nstrips, int crows) {
  const int lane = threadIdx.x & 31, col = blockIdx.y;
  const int nv = op.nv, nh = op.nh, nvc = nv / 2, nhc = nh / 2;
  const int st = blockIdx.x * (kVcThreads / 32) + (threadIdx.x >> 5);
  if (st >= nstrips) return;
  const int I = st % nsi * kVcUpCols - 1 + lane;  // z0 at every lane, z at 1..30
  const int j0 = 2 * (st / nsi * crows), j1 = min(j0 + 2 * crows, nh);
  const bool in_i = I >= 0 && I < nvc;
  const int Ic = in_i ? I : 0, i = 2 * Ic;
  const bool out = in_i && lane >= 1 && lane <= kVcUpCols;
  const float sc = op.sc;
  const int Il = max(Ic - 1, 0), Ir = min(Ic + 1, nvc - 1);
  float na, fa, nb, fb;  // weights along i of points 2I and 2I + 1
  pw1_near_far(2 * Ic, nv, na, fa);
  pw1_near_far(2 * Ic + 1, nv, nb, fb);
  // z0 = D r + P e_c of row j (zero outside the level); r and D out
  struct Raw {
    Pair r, d;
    float e[2][3];  // e_c of the nearer and the other coarse row at I - 1, I, I + 1
  };
  auto load = [&](int j) {
    Raw q;
    const int jc = min(max(j, 0), nh - 1);
    const int64_t e = (int64_t)i + (int64_t)jc * nv;
    q.r = ld_pair<kUnit>(r, e, B, col);
    q.d = ld_pair<kUnit>(dinv, e, B, col);
    const int Ja = jc >> 1, Jb = min(max((jc & 1) ? Ja + 1 : Ja - 1, 0), nhc - 1);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int64_t row = (int64_t)(u ? Jb : Ja) * nvc;
      const int S = kUnit ? 1 : B, co = kUnit ? 0 : col;
      q.e[u][0] = ec[(row + Il) * S + co];
      q.e[u][1] = ec[(row + Ic) * S + co];
      q.e[u][2] = ec[(row + Ir) * S + co];
    }
    return q;
  };
  auto z0 = [&](const Raw& q, int j) {
    float wn, wf;
    pw1_near_far(j, nh, wn, wf);
    const float c0 = wn * q.e[0][0] + wf * q.e[1][0];
    const float c1 = wn * q.e[0][1] + wf * q.e[1][1];
    const float c2 = wn * q.e[0][2] + wf * q.e[1][2];
    Pair z{q.d.a * q.r.a + (na * c1 + fa * c0), q.d.b * q.r.b + (nb * c1 + fb * c2)};
    if (!in_i || j < 0 || j >= nh) z.a = z.b = 0.f;
    return z;
  };
  Window W;
  auto smooth_row = [&](int j, const PairRow& kj, const Pair& rj, const Pair& dj) {
    const Pair kz = W.apply(kj);
    const float za = W.z[2][2] + dj.a * (rj.a - kz.a * sc), zb = W.z[2][3] + dj.b * (rj.b - kz.b * sc);
    if (out) {
      const int64_t e = (int64_t)i + (int64_t)j * nv;
      if (kUnit) {
        *reinterpret_cast<float2*>(zout + e) = make_float2(za, zb);
      } else {
        zout[e * B + col] = za;
        zout[(e + 1) * B + col] = zb;
      }
    }
  };
  // every first load is issued before the first shuffle
  Raw q5[5];
#pragma unroll
  for (int u = 0; u < 5; ++u) q5[u] = load(j0 - 2 + u);
  PairRow k = ld_row(op, i, j0);
#pragma unroll
  for (int u = 0; u < 4; ++u) W.push(z0(q5[u], j0 - 2 + u));
  Pair r0 = q5[2].r, d0 = q5[2].d, r1 = q5[3].r, d1 = q5[3].d;
  Raw q = q5[4];
#pragma unroll 2
  for (int j = j0; j < j1; ++j) {
    W.push(z0(q, j + 2));
    const Pair rj = r0, dj = d0;
    r0 = r1;
    d0 = d1;
    r1 = q.r;
    d1 = q.d;
    const PairRow kj = k;
    if (j + 1 < j1) {  // the next row's loads
      q = load(j + 3);
      k = ld_row(op, i, j + 1);
    }
    smooth_row(j, kj, rj, dj);
  }
}

}  // namespace lcmg
