// The finest level of the V(1,1) cycle (Algorithm 1, nu = 1) in two
// kernels, for the mixed path's FP32 vectors.
//
// With one sweep, pre-smoothing from a zero initial guess is z1 = D^{-1} r,
// so the pre-smoothed vector need not be stored: the down kernel forms it
// on the fly for the residual and the restriction, and the up kernel forms
// it again (the same values, the same formulas) under the prolongated
// correction.  D^{-1} (l1-Jacobi 1 / sum_q |k_pq|, or damped Jacobi
// omega / k_pp) is computed from the level's stored weights where it is
// needed, so the level reads r, its weights and the coarse correction and
// writes the coarse right-hand side and z, and nothing else:
//
//   k_vfine_down: z1 = D^{-1} r, res = r - K z1, r_c = P^T res
//   k_vfine_up:   z0 = z1 + P e_c, z = z0 + D^{-1} (r - K z0), partials r.z
//
// FP32 weights: a block owns a 64 x 32 tile of fine points (a 32 x 16 tile
// of coarse points) and keeps the windows its stencils need in shared memory
// (halo 2 for the down kernel, 1 for the up kernel); blocks stride over the
// tiles.  The sums per point are those of the generic tile kernels.  FP16
// weights: the row-streaming kernels at the end.
#pragma once
#include "compact.cuh"
#include "kernels.cuh"
#include "vcoarse.cuh"

namespace lcmg {

constexpr int kFineTI = 64;  // fine points per tile along i (contiguous)
constexpr int kFineTJ = 32;  // ... along j
constexpr int kFineThreads = 256;

// the four edge weights around point (i, j) (zero across the boundary) and
// diag(A^T A) there
struct FineW {
  float s, n, e, w, g;
};
__device__ __forceinline__ FineW fine_w(const FineOp<float>& op, int64_t p, int i, int j) {
  FineW f;
  f.s = i + 1 < op.nv ? op.ws[p] : 0.f;
  f.n = i > 0 ? op.ws[p - 1] : 0.f;
  f.e = j + 1 < op.nh ? op.we[p] : 0.f;
  f.w = j > 0 ? op.we[p - op.nv] : 0.f;
  f.g = op.ga[p];
  return f;
}

// D^{-1} at a point: l1-Jacobi 1 / (2 lam2 sum w + ga), or omega / (lam2 sum w + ga)
__device__ __forceinline__ float fine_dinv(const FineW& f, float l2, int smoother, float omega) {
  const float sw = f.s + f.n + f.e + f.w;
  return smoother == 0 ? 1.0f / (2.0f * l2 * sw + f.g) : omega / (l2 * sw + f.g);
}

// (K z)_p with z read at offsets of a shared-memory window (stride ld)
__device__ __forceinline__ float fine_kz(const FineW& f, float l2, const float* z, int q, int ld) {
  const float zp = z[q];
  const float acc = f.s * (zp - z[q + 1]) + f.n * (zp - z[q - 1]) + f.e * (zp - z[q + ld]) + f.w * (zp - z[q - ld]);
  return l2 * acc + f.g * zp;
}

__global__ void __launch_bounds__(kFineThreads)
    k_vfine_down(FineOp<float> op, int B, const float* __restrict__ lam2, int smoother, float omega,
                 const float* __restrict__ r, float* __restrict__ rc, int ntiles) {
  constexpr int ZI = kFineTI + 4, ZJ = kFineTJ + 4;  // z1 window, halo 2
  constexpr int RI = kFineTI + 2, RJ = kFineTJ + 2;  // residual window, halo 1
  __shared__ float sz[ZI * ZJ];
  __shared__ float sr[ZI * ZJ];
  __shared__ float sres[RI * RJ];
  const int col = blockIdx.y;
  const int nv = op.nv, nh = op.nh, nvc = nv / 2, nhc = nh / 2;
  const int nti = (nv + kFineTI - 1) / kFineTI;
  const float l2 = lam2[col];
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int i0 = (tile % nti) * kFineTI, j0 = (tile / nti) * kFineTJ;
    // z1 = D^{-1} r and r on the window (zero outside the grid)
    for (int t = threadIdx.x; t < ZI * ZJ; t += kFineThreads) {
      const int i = i0 - 2 + t % ZI, j = j0 - 2 + t / ZI;
      float zv = 0.f, rv = 0.f;
      if (i >= 0 && i < nv && j >= 0 && j < nh) {
        const int64_t p = (int64_t)i + (int64_t)j * nv;
        rv = r[p * B + col];
        zv = fine_dinv(fine_w(op, p, i, j), l2, smoother, omega) * rv;
      }
      sz[t] = zv;
      sr[t] = rv;
    }
    __syncthreads();
    // res = r - K z1
    for (int t = threadIdx.x; t < RI * RJ; t += kFineThreads) {
      const int li = t % RI, lj = t / RI;
      const int i = i0 - 1 + li, j = j0 - 1 + lj;
      float v = 0.f;
      if (i >= 0 && i < nv && j >= 0 && j < nh) {
        const int64_t p = (int64_t)i + (int64_t)j * nv;
        const int q = (li + 1) + (lj + 1) * ZI;
        v = sr[q] - fine_kz(fine_w(op, p, i, j), l2, sz, q, ZI);
      }
      sres[t] = v;
    }
    __syncthreads();
    // r_c = P^T res over the tile's coarse points
    for (int t = threadIdx.x; t < (kFineTI / 2) * (kFineTJ / 2); t += kFineThreads) {
      const int I = i0 / 2 + t % (kFineTI / 2), J = j0 / 2 + t / (kFineTI / 2);
      if (I >= nvc || J >= nhc) continue;
      float acc = 0.f;
#pragma unroll
      for (int b = 2 * J - 1; b <= 2 * J + 2; ++b) {
        if (b < 0 || b >= nh) continue;
        const float wb = pw1<float>(b, J, nhc);
#pragma unroll
        for (int a2 = 2 * I - 1; a2 <= 2 * I + 2; ++a2) {
          if (a2 < 0 || a2 >= nv) continue;
          acc += wb * pw1<float>(a2, I, nvc) * sres[(a2 - (i0 - 1)) + (b - (j0 - 1)) * RI];
        }
      }
      rc[((int64_t)I + (int64_t)J * nvc) * B + col] = acc;
    }
    __syncthreads();  // the windows are refilled by the next tile
  }
}

__global__ void __launch_bounds__(kFineThreads)
    k_vfine_up(FineOp<float> op, int B, const float* __restrict__ lam2, int smoother, float omega,
               const float* __restrict__ r, const float* __restrict__ ec, float* __restrict__ zout, int ntiles,
               double* __restrict__ part) {
  constexpr int WI = kFineTI + 2, WJ = kFineTJ + 2;          // z0 window, halo 1
  constexpr int CI = kFineTI / 2 + 2, CJ = kFineTJ / 2 + 2;  // coarse window
  __shared__ float sc[CI * CJ];
  __shared__ float s0[WI * WJ];
  __shared__ double sred[kFineThreads / 32];
  const int col = blockIdx.y;
  const int nv = op.nv, nh = op.nh, nvc = nv / 2, nhc = nh / 2;
  const int nti = (nv + kFineTI - 1) / kFineTI;
  const float l2 = lam2[col];
  Dot2 dot;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int i0 = (tile % nti) * kFineTI, j0 = (tile / nti) * kFineTJ;
    const int I0 = i0 / 2 - 1, J0 = j0 / 2 - 1;
    for (int t = threadIdx.x; t < CI * CJ; t += kFineThreads) {
      const int I = I0 + t % CI, J = J0 + t / CI;
      sc[t] = (I >= 0 && I < nvc && J >= 0 && J < nhc) ? ec[((int64_t)I + (int64_t)J * nvc) * B + col] : 0.f;
    }
    __syncthreads();
    // z0 = D^{-1} r + P e_c on the window
    for (int t = threadIdx.x; t < WI * WJ; t += kFineThreads) {
      const int a2 = i0 - 1 + t % WI, b = j0 - 1 + t / WI;
      float v = 0.f;
      if (a2 >= 0 && a2 < nv && b >= 0 && b < nh) {
        const int64_t p = (int64_t)a2 + (int64_t)b * nv;
        const float z1 = fine_dinv(fine_w(op, p, a2, b), l2, smoother, omega) * r[p * B + col];
        const int Ia = a2 >> 1, Ja = b >> 1;
        const int Ib = (a2 & 1) ? Ia + 1 : Ia - 1;
        const int Jb = (b & 1) ? Ja + 1 : Ja - 1;
        const int Is[2] = {Ia, Ib}, Js[2] = {Ja, Jb};
        float acc = 0.f;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int J = Js[u];
          if (J < 0 || J >= nhc) continue;
          const float wb = pw1<float>(b, J, nhc);
#pragma unroll
          for (int w = 0; w < 2; ++w) {
            const int I = Is[w];
            if (I < 0 || I >= nvc) continue;
            acc += wb * pw1<float>(a2, I, nvc) * sc[(I - I0) + (J - J0) * CI];
          }
        }
        v = z1 + acc;
      }
      s0[t] = v;
    }
    __syncthreads();
    // z = z0 + D^{-1} (r - K z0) on the tile's points
    for (int t = threadIdx.x; t < kFineTI * kFineTJ; t += kFineThreads) {
      const int li = t % kFineTI, lj = t / kFineTI;
      const int i = i0 + li, j = j0 + lj;
      if (i >= nv || j >= nh) continue;
      const int64_t p = (int64_t)i + (int64_t)j * nv;
      const FineW f = fine_w(op, p, i, j);
      const int q = (li + 1) + (lj + 1) * WI;
      const float rv = r[p * B + col];
      const float zn = s0[q] + fine_dinv(f, l2, smoother, omega) * (rv - fine_kz(f, l2, s0, q, WI));
      zout[p * B + col] = zn;
      dot.add(rv, zn);
    }
    __syncthreads();
  }
  if (part) {
    double dacc = dot.value();
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) dacc += __shfl_xor_sync(0xffffffffu, dacc, off);
    if ((threadIdx.x & 31) == 0) sred[threadIdx.x >> 5] = dacc;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int k = 0; k < kFineThreads / 32; ++k) s += sred[k];
      part[(int64_t)blockIdx.x * B + col] = s;
    }
  }
}


// ---------------------------------------------------------------------------
// Row-streaming forms of the two kernels for the FP16 weights.  A warp owns
// 64 consecutive points along i, two per lane (a coarse column's own pair),
// and walks down a strip of rows j: the neighbours along j are values the
// lane computed one row earlier or one row ahead (kept in registers), those
// along i are the lane's other point or the neighbouring lanes' (shuffles).
// The edge lanes compute only what their neighbours need (the halo), so a
// warp produces 60 points of z (k_vfine_up_s) or 30 coarse points of r_c
// (k_vfine_down_s) per row.  No shared memory, no barrier; a row's loads are
// issued one row ahead of their use, from addresses clamped into the arrays.
// The weights are zero on the last row and column and outside the grid, so
// no step tests for the edge.
//
// What bounds them: the latency of a row's loads, of which a lane has one row
// (10 bytes a point, and e_c) ahead of its use, in 22 (down, 80 registers) or 15
// (up, 126) warps per SM.  At 2048^2 points the largest stalls are those loads'
// (4.9 and 2.5 warps per issue), 55% of the issue slots are taken and DRAM runs
// at 26 and 22% of its peak: 42 and 46 MB, 6.2 and 6.8 us at the copy rate.
// With one point per lane it was the instructions (165 per warp and row of
// 30 points).  Measured on GB300 against
// that form, down / up: 2048^2 27.4 / 34.9 -> 18.5 / 24.1 us, 512^2 in four
// columns 12.6 / 13.4 -> 8.0 / 10.4 us, 256^2 3.9 / 3.9 -> 3.5 / 3.8 us.  With as
// many strips as 16 / 8, 24 / 16 and 32 / 32 warps per SM: 23.2 / 25.4, 18.3 /
// 24.2, 25.7 / 26.2 us at 2048^2.
//
// Each point's formulas are those of k_vfine_up / k_vfine_down, with three
// changes of rounding: D^{-1} = 1 / (2 lam^2 sum w + g) (or omega / (lam^2
// sum w + g)) is taken with the fast division (__fdividef, within 2 ulp),
// the same value in both kernels, so the cycle stays one fixed symmetric
// operator; r_c = P^T res is summed per fine row along i first, then along
// j; and P e_c along j first.
// ---------------------------------------------------------------------------
constexpr int kStripRows = 32;    // most fine rows of z per k_vfine_up_s strip
constexpr int kStripCoarse = 16;  // most coarse rows of r_c per k_vfine_down_s strip
constexpr int kFineCols = 30;     // coarse columns (pairs) per warp
constexpr int kFineDownWarps = 24;  // warps per SM the strips aim at (those resident)
constexpr int kFineUpWarps = 16;

// the stored data of a lane's pair in one row: FP16 w_s, w_e, diag(A^T A),
// w_s of the point before the pair (lane 0 alone reads it, the others have
// it from their neighbour), r
struct FineRaw {
  __half2 s, e, g;
  __half n;
  Pair r;
};
// what a lane carries from one row to the next
struct FinePair {
  Pair z;       // z1 = D^{-1} r (down) or z0 = z1 + P e_c (up)
  Pair r, d;    // r and D^{-1}
  float2 s, e;  // w_s, w_e (in stored units)
  float n;      // w_s of the point before the pair
  float2 w;     // w_e of the row before
  float2 g;     // diag(A^T A)
};

template <bool kUnit>
struct FineStream {
  FineOpH op;
  const float* __restrict__ r;
  int B, col, smoother;
  float l2s, sg, omega;  // lam^2 in the units of the stored weights
  int lane, i;           // the lane's pair (i, i + 1), clamped into the row
  bool in_i;

  __device__ __forceinline__ FineRaw load(int j) const {
    FineRaw q;
    const int64_t e = (int64_t)i + (int64_t)min(max(j, 0), op.nh - 1) * op.nv;
    q.s = *reinterpret_cast<const __half2*>(op.ws + e);
    q.e = *reinterpret_cast<const __half2*>(op.we + e);
    q.g = *reinterpret_cast<const __half2*>(op.ga + e);
    q.n = __half(0);
    if (lane == 0 && i > 0) q.n = op.ws[e - 1];
    q.r = ld_pair<kUnit>(r, e, B, col);
    return q;
  }
  // w_e of row j (zero outside the grid)
  __device__ __forceinline__ float2 edge(int j) const {
    if (!in_i || j < 0 || j >= op.nh) return make_float2(0.f, 0.f);
    return __half22float2(*reinterpret_cast<const __half2*>(op.we + (int64_t)i + (int64_t)j * op.nv));
  }
  // weights, D^{-1} and z1 of row j (all zero outside the grid); w = edge(j - 1)
  __device__ __forceinline__ FinePair row(const FineRaw& q, int j, const float2 w) const {
    FinePair f;
    const bool in = in_i && j >= 0 && j < op.nh;
    const float2 zero = make_float2(0.f, 0.f);
    f.s = in ? __half22float2(q.s) : zero;
    f.e = in ? __half22float2(q.e) : zero;
    f.g = in ? __half22float2(q.g) : zero;
    f.g.x *= sg;
    f.g.y *= sg;
    f.w = w;
    f.n = __shfl_up_sync(0xffffffffu, f.s.y, 1);
    if (lane == 0) f.n = in ? __half2float(q.n) : 0.f;
    f.r.a = in ? q.r.a : 0.f;
    f.r.b = in ? q.r.b : 0.f;
    const float sa = f.s.x + f.n + f.e.x + f.w.x, sb = f.s.y + f.s.x + f.e.y + f.w.y;
    if (smoother == 0) {
      f.d.a = __fdividef(1.0f, 2.0f * l2s * sa + f.g.x);
      f.d.b = __fdividef(1.0f, 2.0f * l2s * sb + f.g.y);
    } else {
      f.d.a = __fdividef(omega, l2s * sa + f.g.x);
      f.d.b = __fdividef(omega, l2s * sb + f.g.y);
    }
    if (!in) f.d.a = f.d.b = 0.f;
    f.z.a = f.d.a * f.r.a;
    f.z.b = f.d.b * f.r.b;
    return f;
  }
  // (K z) at the pair of row f, zm and zp the pairs of the rows before and after
  __device__ __forceinline__ Pair kz(const FinePair& f, const Pair& zm, const Pair& zp) const {
    const float zl = __shfl_up_sync(0xffffffffu, f.z.b, 1), zr = __shfl_down_sync(0xffffffffu, f.z.a, 1);
    const float a = f.s.x * (f.z.a - f.z.b) + f.n * (f.z.a - zl) + f.e.x * (f.z.a - zp.a) + f.w.x * (f.z.a - zm.a);
    const float b = f.s.y * (f.z.b - zr) + f.s.x * (f.z.b - f.z.a) + f.e.y * (f.z.b - zp.b) + f.w.y * (f.z.b - zm.b);
    return {l2s * a + f.g.x * f.z.a, l2s * b + f.g.y * f.z.b};
  }
};

template <bool kUnit>
__global__ void __launch_bounds__(kFineThreads, 2)
    k_vfine_up_s(FineOpH op, int B, const float* __restrict__ lam2, int smoother, float omega,
                 const float* __restrict__ r, const float* __restrict__ ec, float* __restrict__ zout, int nsi,
                 int nstrips, int rows, double* __restrict__ part) {
  __shared__ double sred[kFineThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int col = blockIdx.y;
  const int nv = op.nv, nh = op.nh, nvc = nv / 2, nhc = nh / 2;
  Dot2 dot;
  for (int st = blockIdx.x * (blockDim.x >> 5) + warp; st < nstrips; st += gridDim.x * (blockDim.x >> 5)) {
    const int I = st % nsi * kFineCols - 1 + lane;
    const int j0 = st / nsi * rows, j1 = min(j0 + rows, nh);
    const bool in_i = I >= 0 && I < nvc;
    const int Ic = in_i ? I : 0;
    const FineStream<kUnit> F{op, r, B, col, smoother, lam2[col] * op.sw, op.sg, omega, lane, 2 * Ic, in_i};
    const bool out = in_i && lane >= 1 && lane <= kFineCols;
    // interpolation along i (fixed for the lane): columns I, I - 1 and I + 1
    const int Il = max(Ic - 1, 0), Ir = min(Ic + 1, nvc - 1);
    float na, fa, nb, fb;
    pw1_near_far(2 * Ic, nv, na, fa);
    pw1_near_far(2 * Ic + 1, nv, nb, fb);
    struct Corr {
      float e[2][3];  // e_c of the nearer and the other coarse row at I - 1, I, I + 1
    };
    auto load_c = [&](int j) {
      Corr q;
      const int jc = min(max(j, 0), nh - 1);
      const int Ja = jc >> 1, Jb = min(max((jc & 1) ? Ja + 1 : Ja - 1, 0), nhc - 1);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int64_t e = (int64_t)(u ? Jb : Ja) * nvc;
        const int S = kUnit ? 1 : B, co = kUnit ? 0 : col;
        q.e[u][0] = ec[(e + Il) * S + co];
        q.e[u][1] = ec[(e + Ic) * S + co];
        q.e[u][2] = ec[(e + Ir) * S + co];
      }
      return q;
    };
    // z0 = D^{-1} r + P e_c at row j (zero outside the grid)
    auto row = [&](const FineRaw& q, const Corr& c, int j, const float2 w) {
      FinePair f = F.row(q, j, w);
      float wn, wf;
      pw1_near_far(j, nh, wn, wf);
      if (!in_i || j < 0 || j >= nh) wn = wf = 0.f;
      const float c0 = wn * c.e[0][0] + wf * c.e[1][0];
      const float c1 = wn * c.e[0][1] + wf * c.e[1][1];
      const float c2 = wn * c.e[0][2] + wf * c.e[1][2];
      f.z.a += na * c1 + fa * c0;
      f.z.b += nb * c1 + fb * c2;
      return f;
    };
    // every first load is issued before the first shuffle
    const FineRaw qa = F.load(j0 - 1), qb = F.load(j0);
    const Corr ca = load_c(j0 - 1), cb = load_c(j0);
    const float2 ea = F.edge(j0 - 2);
    FineRaw qn = F.load(j0 + 1);
    Corr cn = load_c(j0 + 1);
    FinePair fm = row(qa, ca, j0 - 1, ea);
    FinePair fc = row(qb, cb, j0, fm.e);
#pragma unroll 3
    for (int j = j0; j < j1; ++j) {
      const FineRaw qj = qn;
      const Corr cj = cn;
      qn = F.load(j + 2);  // the loads of the row after next
      cn = load_c(j + 2);
      const FinePair fp = row(qj, cj, j + 1, fc.e);
      const Pair kz = F.kz(fc, fm.z, fp.z);
      const float za = fc.z.a + fc.d.a * (fc.r.a - kz.a), zb = fc.z.b + fc.d.b * (fc.r.b - kz.b);
      if (out) {
        const int64_t e = (int64_t)(2 * I) + (int64_t)j * nv;
        if (kUnit) {
          *reinterpret_cast<float2*>(zout + e) = make_float2(za, zb);
        } else {
          zout[e * B + col] = za;
          zout[(e + 1) * B + col] = zb;
        }
        dot.add(fc.r.a, za);
        dot.add(fc.r.b, zb);
      }
      fm = fc;
      fc = fp;
    }
  }
  if (part) {
    const double dacc = dot.warp_sum();
    if (lane == 0) sred[warp] = dacc;
    __syncthreads();
    if (threadIdx.x == 0) {
      double sum = 0.0;
      for (int k = 0; k < (int)blockDim.x >> 5; ++k) sum += sred[k];
      part[(int64_t)blockIdx.x * B + col] = sum;
    }
  }
}

template <bool kUnit>
__global__ void __launch_bounds__(kFineThreads, 3)
    k_vfine_down_s(FineOpH op, int B, const float* __restrict__ lam2, int smoother, float omega,
                   const float* __restrict__ r, float* __restrict__ rc, int nsi, int nstrips, int crows) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int col = blockIdx.y;
  const int nh = op.nh, nvc = op.nv / 2, nhc = nh / 2;
  for (int st = blockIdx.x * (blockDim.x >> 5) + warp; st < nstrips; st += gridDim.x * (blockDim.x >> 5)) {
    const int I = st % nsi * kFineCols - 1 + lane;  // z1 at every lane, r_c at lanes 1..30
    const int J0 = st / nsi * crows, J1 = min(J0 + crows, nhc);
    const bool in_i = I >= 0 && I < nvc;
    const FineStream<kUnit> F{op, r, B, col, smoother, lam2[col] * op.sw, op.sg, omega, lane, in_i ? 2 * I : 0, in_i};
    const bool out = in_i && lane >= 1 && lane <= kFineCols;
    // restriction along i from the residuals at 2I - 1 .. 2I + 2
    const float w1 = I == 0 ? 1.f : 0.75f, w2 = I == nvc - 1 ? 1.f : 0.75f;
    const int b0 = 2 * J0 - 1, b1 = 2 * J1;  // residual rows
    // every first load is issued before the first shuffle
    const FineRaw q0 = F.load(b0 - 1), q1 = F.load(b0);
    const float2 ea = F.edge(b0 - 2);
    FineRaw qn = F.load(b0 + 1);
    FinePair fm = F.row(q0, b0 - 1, ea);
    FinePair fc = F.row(q1, b0, fm.e);
    float prev = 0.f, cur = 0.f;  // r_c of coarse rows (b - 1) / 2 and (b + 1) / 2 being summed
#pragma unroll 3
    for (int b = b0; b <= b1; ++b) {
      const FineRaw qb = qn;
      qn = F.load(b + 2);  // the loads of the row after next
      const FinePair fp = F.row(qb, b + 1, fc.e);
      const Pair kz = F.kz(fc, fm.z, fp.z);
      // res = r - K z1 (zero outside the grid: every term is)
      const float ra = fc.r.a - kz.a, rb = fc.r.b - kz.b;
      const float left = __shfl_up_sync(FULL, rb, 1), right = __shfl_down_sync(FULL, ra, 1);
      const float ti = 0.25f * left + w1 * ra + w2 * rb + 0.25f * right;  // sum over a of pw1(a, I) res(a, b)
      const float wb = (b == 0 || b == nh - 1) ? 1.f : 0.75f;             // pw1(b, b / 2)
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
      fm = fc;
      fc = fp;
    }
  }
}

}  // namespace lcmg
