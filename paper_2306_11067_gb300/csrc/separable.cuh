// Separable blur operator.
//
// A blur whose point-spread function is an outer product fv fh^T (a
// Gaussian, or the anisotropic blur of the deblurring example, Sec. 4) is
// the Kronecker product A = A_h (x) A_v of two 1-D zero-boundary Toeplitz
// correlations: A_v acts along the image columns (index i, contiguous in
// memory) and A_h along the rows (index j, stride n_v).  Hence
//
//     A^T A = (A_h^T A_h) (x) (A_v^T A_v) = T_h (x) T_v,
//
// where each T is a symmetric banded matrix of half-bandwidth 2r whose
// interior rows are the autocorrelation t_k = sum_u f_u f_{u+k} and whose
// first and last r rows lose the products that the zero boundary cuts off.
// The normal operator's data term is then two banded 1-D passes of 4r + 1
// taps each (122 multiply-adds per pixel at r = 15, against 2 (2r+1)^2 =
// 1922 for the direct 2-D form), and A, A^T are passes of 2r + 1 taps.
//
// Four kernels apply one such pass, out(o) = sum_k c_k in(o - H + k) with
// other coefficients for the boundary rows, to every line of the image along
// the contiguous axis (DIR 0) or the strided axis (DIR 1): k_band_direct (one
// output per thread; FP64, and small FP32 images), k_band_line (DIR 0) and
// k_band_rows (DIR 1) for one column of a large FP32 image, and k_band
// (either axis) for large batches of several columns in FP32 and of many (14
// or more) in FP64.  DIR 1 is the
// second pass of the normal operator and fuses its epilogue: the lam^2 L^T W
// L p term, the store and the per-block partial sums of p.q (or of the true
// residual, or of ||A x - b||^2).
#pragma once
#include "kernels.cuh"

namespace lcmg {

constexpr int kBandMaxH = 32;                              // taps <= 65
constexpr int kBandMaxR = kBandMaxH / 2;                   // boundary rows at an end of a line
constexpr int kBandChunk = 8;                              // taps per register chunk (k_band)
constexpr int kBandMaxTaps = 72;                           // 65 rounded up to the chunk
constexpr int kBandSeg = 128;                              // k_band: outputs per line per tile
constexpr int kBandLines = 32;                             // ... lines per tile (one per lane)
constexpr int kBandThreads = 256;
constexpr int kBandR = kBandSeg / (kBandThreads / 32);     // ... outputs per thread (16)

// One banded 1-D pass: out(o) = sum_{k=0}^{2H} c[k] in(o - H + k) with in
// zero outside the line, plus, for the nlo first and the nhi last outputs
// of the line, sum_k d[row][k] in(o - H + k) (row = o for the first ones,
// nlo + o - (len - nhi) for the last ones).
template <class T>
struct Band {
  int H;
  int nch;             // chunks of kBandChunk taps: ceil((2H + 1) / 8)
  int nlo, nhi;
  const T* d;          // (nlo + nhi) x (2H + 1) corrections, or null
  const T* e;          // the whole coefficient rows c + d of those outputs and, last, the
                       // interior row c: (nlo + nhi + 1) x (2H + 1), or null
  T c[kBandMaxTaps];   // zero beyond 2H
};

// epilogues of a pass (DIR 1 only, except BAND_STORE)
enum : int {
  BAND_STORE = 0,    // out = v
  BAND_NORMAL = 1,   // q = v + lam2 L^T W L P; out = q; partials of P.q
  BAND_RESID2 = 2,   // partials of (v - b)^2 (no store)
  BAND_TRUERES = 3   // r = C - (v + lam2 L^T W L P); out = r; partials of r.r
};

// ---- one column of a large FP32 image ----------------------------------------
// Both kernels move 16-byte words (lines of a multiple of 4 points) and have
// the tap count TAPS >= 2H + 1 fixed at compile time (the coefficients beyond
// 2H are zero): a sample is read once per thread and multiplied into each of
// the 16 outputs it touches.
//
// What bounds them: the instructions; 61 of the 75 or so (DIR 0) and 95 or so
// (DIR 1 with its epilogue) per output of the 61-tap pass are its
// multiply-adds.  k_band copies its tiles element by element and takes nine
// global loads per output in the epilogue.  Measured on GB300 against it at
// 2048^2, 61 taps, inside a solve: DIR 0 26.8 -> 18.0 us, DIR 1 44.7 -> 38.4 us;
// deblur chain at 2048^2 (three lambda) 521 -> 494 ms.

// Filter along the contiguous axis.  A warp takes 512 consecutive outputs of
// a line, 16 per lane; it stages its 512 + TAPS - 1 samples in shared memory
// from the 16-byte boundary below the first, 16 to a 20-float group so that
// the 16-byte reads of a quarter warp fall into different banks.  The first
// nlo and last nhi outputs of a line take their corrections from two lanes
// each (half of the taps), added through shared memory.
constexpr int kLineR = 16;                // outputs per lane
constexpr int kLineSeg = 32 * kLineR;     // outputs per warp
constexpr int kLineWarps = 8;
// samples staged: the outputs' windows, the shift to the 16-byte boundary
__host__ __device__ constexpr int line_samples(int taps) { return (kLineSeg + taps - 1 + 3 + 15) / 16 * 16; }
__host__ __device__ constexpr int line_pad(int m) { return m / 16 * 20 + m % 16; }

template <int TAPS>
__global__ void __launch_bounds__(32 * kLineWarps)
    k_band_line(int nv, int nh, const __grid_constant__ Band<float> bd, const float* __restrict__ in,
                float* __restrict__ out) {
  constexpr int N = line_samples(TAPS);
  __shared__ __align__(16) float sm_all[kLineWarps][line_pad(N) + kBandMaxH];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float* sm = sm_all[w];
  float* corr = sm + line_pad(N);  // corrections of up to kBandMaxH / 2 boundary outputs
  const int nseg = (nv + kLineSeg - 1) / kLineSeg, H = bd.H, taps = 2 * H + 1;
  // the window of output o starts at sample o - H: stage from the multiple of 4 below
  const int shift = (4 - (H & 3)) & 3;
  const int64_t ntask = (int64_t)nseg * nh;  // segment fastest
  for (int64_t task = (int64_t)blockIdx.x * kLineWarps + w; task < ntask; task += (int64_t)gridDim.x * kLineWarps) {
    const int64_t ln = task / nseg, line = ln * nv;
    const int seg0 = (int)(task - ln * nseg) * kLineSeg;
    const int a0 = seg0 - H - shift;  // first staged sample
    const float* __restrict__ x = in + line;
#pragma unroll
    for (int u = 0; u < (N / 4 + 31) / 32; ++u) {
      const int m = 4 * (u * 32 + lane), a = a0 + m;
      if (m < N) {
        const bool ok = a >= 0 && a < nv;  // (nv and a are multiples of 4)
        *reinterpret_cast<float4*>(sm + line_pad(m)) =
            ok ? *reinterpret_cast<const float4*>(x + a) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    __syncwarp();
    float acc[kLineR];
#pragma unroll
    for (int t = 0; t < kLineR; ++t) acc[t] = 0.f;
    auto filter = [&](auto sh) {
      constexpr int SH = decltype(sh)::value;
#pragma unroll
      for (int m4 = 0; m4 < (kLineR + TAPS - 1 + SH + 3) / 4; ++m4) {
        const float4 f = *reinterpret_cast<const float4*>(sm + (lane + m4 / 4) * 20 + (m4 & 3) * 4);
        const float v[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
          for (int t = 0; t < kLineR; ++t) {
            const int k = 4 * m4 + e - SH - t;
            if (k >= 0 && k < TAPS) acc[t] += bd.c[k] * v[e];
          }
      }
    };
    // H = 2r is even (A^T A), so the shift is 0 or 2
    if (shift == 0)
      filter(std::integral_constant<int, 0>{});
    else
      filter(std::integral_constant<int, 2>{});
    // boundary outputs of this segment: the head rows [seg0, ...) and the tail
    if (bd.d != nullptr && (seg0 < bd.nlo || seg0 + kLineSeg > nv - bd.nhi)) {
      const int o1 = min(seg0 + kLineSeg, nv);
#pragma unroll 1
      for (int side = 0; side < 2; ++side) {
        const int ob = side == 0 ? seg0 : max(seg0, max(nv - bd.nhi, bd.nlo));
        const int oe = side == 0 ? min(o1, bd.nlo) : o1;
        if (ob >= oe) continue;  // (uniform over the warp)
        const int o = ob + (lane >> 1);  // at most 16 rows a side
        float s = 0.f;
        if (o < oe) {
          const float* __restrict__ dr = bd.d + (int64_t)(o < bd.nlo ? o : bd.nlo + o - (nv - bd.nhi)) * taps;
          const int half = (taps + 1) / 2, k0 = (lane & 1) * half, k1 = min(taps, k0 + half);
          for (int k = k0; k < k1; ++k) s += dr[k] * sm[line_pad(o - seg0 + shift + k)];
        }
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        if ((lane & 1) == 0) corr[lane >> 1] = s;
        __syncwarp();
#pragma unroll
        for (int t = 0; t < kLineR; ++t) {
          const int oo = seg0 + lane * kLineR + t;
          if (oo >= ob && oo < oe) acc[t] += corr[oo - ob];
        }
        __syncwarp();
      }
    }
    const int o = seg0 + lane * kLineR;
    float* __restrict__ y = out + line + o;
#pragma unroll
    for (int u = 0; u < kLineR / 4; ++u)
      if (o + 4 * u < nv)
        *reinterpret_cast<float4*>(y + 4 * u) = make_float4(acc[4 * u], acc[4 * u + 1], acc[4 * u + 2], acc[4 * u + 3]);
    __syncwarp();  // the samples are overwritten by the next task
  }
}

// Filter along the strided axis, with the normal operator's epilogue
// q = v + lam2 L^T W L P and the partials of P.q.  A block takes a tile of
// 32 consecutive points along i and 128 rows j, a thread 16 rows of one
// column.  Everything the tile reads (128 + TAPS - 1 rows of samples, P with
// a halo of one, the weights) is copied to shared memory with asynchronous
// copies, the samples first, so that the filter runs while the rest arrives
// (39.7 -> 38.4 us at 2048^2, 61 taps); three blocks per SM overlap.  The weights are zero on the last row and column, so nothing
// in the epilogue tests for the image's edge.
constexpr int kRowR = 16;
constexpr int kRowWarps = 8;
constexpr int kRowTile = kRowR * kRowWarps;  // rows per tile
__host__ __device__ constexpr int rows_samples(int taps) { return kRowTile + taps - 1; }
// floats: samples, P (rows j - 1 .. j + 128), w_s, w_e (rows j - 1 ..), and the
// columns i - 1 and i + 32 of P and i - 1 of w_s
__host__ __device__ constexpr int rows_floats(int taps) {
  return 32 * (rows_samples(taps) + (kRowTile + 2) + kRowTile + (kRowTile + 1)) + 3 * kRowTile;
}

template <int TAPS>
__global__ void __launch_bounds__(32 * kRowWarps)
    k_band_rows(int nv, int nh, const __grid_constant__ Band<float> bd, const float* __restrict__ in,
                float* __restrict__ out, FineOp<float> fop, const float* __restrict__ P,
                const double* __restrict__ lam2, double* __restrict__ part) {
  extern __shared__ __align__(16) float rows_sm[];
  __shared__ double sred[kRowWarps];
  constexpr int NS = rows_samples(TAPS);
  float* su = rows_sm;                 // su[m][lane] = in(j0 - H + m)
  float* sp = su + 32 * NS;            // sp[m][lane] = P(j0 - 1 + m)
  float* sws = sp + 32 * (kRowTile + 2);
  float* swe = sws + 32 * kRowTile;    // swe[m][lane] = w_e(j0 - 1 + m)
  float* spl = swe + 32 * (kRowTile + 1);
  float* spr = spl + kRowTile;
  float* swl = spr + kRowTile;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int H = bd.H, taps = 2 * H + 1;
  const float l2 = (float)lam2[0];
  const int nib = (nv + 31) / 32, njb = (nh + kRowTile - 1) / kRowTile;
  Dot2 dot;
  for (int tile = blockIdx.x; tile < nib * njb; tile += gridDim.x) {
    const int i0 = tile % nib * 32, j0 = tile / nib * kRowTile;
    // `rows` rows from row jf of a vector, 32 points wide, zero outside
    auto stage = [&](float* dst, const float* __restrict__ v, int jf, int rows) {
      for (int e = threadIdx.x; e < 8 * rows; e += 32 * kRowWarps) {
        const int m = e >> 3, i = i0 + 4 * (e & 7), j = jf + m;
        const bool ok = i < nv && j >= 0 && j < nh;  // (nv is a multiple of 4)
        cp_async16(dst + 4 * e, v + (ok ? (int64_t)i + (int64_t)j * nv : 0), v, ok);
      }
    };
    stage(su, in, j0 - H, NS);
    cp_async_commit();  // the samples first: the filter runs while the epilogue's data arrive
    stage(sp, P, j0 - 1, kRowTile + 2);
    stage(sws, fop.ws, j0, kRowTile);
    stage(swe, fop.we, j0 - 1, kRowTile + 1);
    if (threadIdx.x < kRowTile) {
      const int j = j0 + threadIdx.x;
      const int64_t p = (int64_t)i0 + (int64_t)j * nv;
      const bool left = i0 > 0 && j < nh, right = i0 + 32 < nv && j < nh;
      cp_async_elem(spl + threadIdx.x, P + (left ? p - 1 : 0), P, left);
      cp_async_elem(spr + threadIdx.x, P + (right ? p + 32 : 0), P, right);
      cp_async_elem(swl + threadIdx.x, fop.ws + (left ? p - 1 : 0), fop.ws, left);
    }
    cp_async_commit();
    cp_async_wait_group<1>();
    __syncthreads();
    const int o0 = w * kRowR, i = i0 + lane;
    float acc[kRowR];
#pragma unroll
    for (int t = 0; t < kRowR; ++t) acc[t] = 0.f;
    const float* x = su + o0 * 32 + lane;
#pragma unroll
    for (int m = 0; m < kRowR + TAPS - 1; ++m) {
      const float v = x[32 * m];
#pragma unroll
      for (int t = 0; t < kRowR; ++t)
        if (m - t >= 0 && m - t < TAPS) acc[t] += bd.c[m - t] * v;
    }
    const int jb = j0 + o0;
    // The rows near the ends of the lines add sum_k d[row][k] in(o - H + k):
    // every warp takes some of them (left to the warps that own them they
    // hold the other six at the barrier), on the
    // samples' own rows once every warp has read them
    if (bd.d != nullptr && (j0 < bd.nlo || j0 + kRowTile > nh - bd.nhi)) {  // uniform over the block
      const int o1 = min(j0 + kRowTile, nh);
      const int nhead = max(0, min(o1, bd.nlo) - j0);             // head rows [j0, j0 + nhead)
      const int tbeg = max(j0, max(nh - bd.nhi, bd.nlo));         // tail rows [tbeg, o1)
      const int nrows = nhead + max(0, o1 - tbeg);                // at most 2 kBandMaxR
      float sum[kBandMaxR / 4];
#pragma unroll
      for (int q = 0; q < kBandMaxR / 4; ++q) {
        const int rr = w + kRowWarps * q;
        sum[q] = 0.f;
        if (rr >= nrows) continue;
        const int o = rr < nhead ? j0 + rr : tbeg + (rr - nhead);
        const float* __restrict__ dr = bd.d + (int64_t)(o < bd.nlo ? o : bd.nlo + o - (nh - bd.nhi)) * taps;
        const float* xs = su + (o - j0) * 32 + lane;
#pragma unroll 8
        for (int k = 0; k < taps; ++k) sum[q] += dr[k] * xs[32 * k];
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < kBandMaxR / 4; ++q)
        if (w + kRowWarps * q < nrows) su[(w + kRowWarps * q) * 32 + lane] = sum[q];
      __syncthreads();
#pragma unroll
      for (int t = 0; t < kRowR; ++t) {
        const int o = jb + t;
        if (o < o1 && (o < j0 + nhead || o >= tbeg))
          acc[t] += su[(o < j0 + nhead ? o - j0 : nhead + o - tbeg) * 32 + lane];
      }
    }
    cp_async_wait_group<0>();
    __syncthreads();
    // q = acc + lam2 L^T W L P
    const bool ok = i < nv;
    float* __restrict__ y = out + (int64_t)i + (int64_t)jb * nv;
    const float* pc = sp + (o0 + 1) * 32 + lane;
    float pm = pc[-32], pz = pc[0], wm = swe[o0 * 32 + lane];
#pragma unroll
    for (int t = 0; t < kRowR; ++t) {
      const int row = o0 + t;
      const float pn = pc[32 * (t + 1)];
      const float pl = lane > 0 ? pc[32 * t - 1] : spl[row], pr = lane < 31 ? pc[32 * t + 1] : spr[row];
      const float ws = sws[row * 32 + lane], wl = lane > 0 ? sws[row * 32 + lane - 1] : swl[row];
      const float we = swe[(row + 1) * 32 + lane];
      const float lap = ws * (pz - pr) + wl * (pz - pl) + we * (pz - pn) + wm * (pz - pm);
      const float q = acc[t] + l2 * lap;
      if (ok && j0 + row < nh) {
        y[(int64_t)t * nv] = q;
        dot.add(pz, q);
      }
      pm = pz;
      pz = pn;
      wm = we;
    }
    __syncthreads();  // the tile is refilled
  }
  const double dacc = dot.warp_sum();
  if (lane == 0) sred[w] = dacc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int k = 0; k < kRowWarps; ++k) s += sred[k];
    part[blockIdx.x] = s;
  }
}

// ---- large FP32 batches of several columns, lines that are not a multiple of 4,
// ---- and wide FP64 batches
// A block filters tiles of 32 lines x 128 outputs of one column, staged in shared
// memory.  At 512 x 512, 4 columns, 37 taps it takes 9.6 + 13.5 us; forms of the
// two kernels above that read single interleaved elements took 12.6 + 16.8.
template <class T>
__host__ __device__ constexpr int band_smem_line(int nch) { return kBandSeg + kBandChunk * nch; }

// shared memory of one block: the staged input tile (line stride LEN + 1)
// and the output tile (line stride kBandSeg + 1)
template <class T>
__host__ __device__ constexpr size_t band_smem_bytes(int nch) {
  return (size_t)kBandLines * ((band_smem_line<T>(nch) + 1) + (kBandSeg + 1)) * sizeof(T);
}

template <class T, class TO, int DIR, int EPI, int TAPS>
__global__ void __launch_bounds__(kBandThreads)
    k_band(int nv, int nh, int B, Band<T> bd, const T* __restrict__ in, TO* __restrict__ out, FineOp<T> fop,
           const T* __restrict__ P, const T* __restrict__ C, const double* __restrict__ lam2,
           const double* __restrict__ bvec, double* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char band_raw[];
  T* sm = reinterpret_cast<T*>(band_raw);
  __shared__ double sred[kBandThreads / 32];
  const int col = blockIdx.y;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int len = DIR == 0 ? nv : nh;       // samples along the filter
  const int nlines = DIR == 0 ? nh : nv;
  const int LEN = band_smem_line<T>(bd.nch);
  const int LS = LEN + 1;                   // DIR 0 line stride (odd: no bank conflicts)
  const int nseg = (len + kBandSeg - 1) / kBandSeg;
  const int ntiles = nseg * ((nlines + kBandLines - 1) / kBandLines);
  const int H = bd.H;
  const T l2 = (EPI == BAND_NORMAL || EPI == BAND_TRUERES) ? (T)lam2[col] : (T)0;
  // tile-local index of (line, sample m)
  auto sidx = [&](int line, int m) { return DIR == 0 ? line * LS + m : m * kBandLines + line; };
  auto gpt = [&](int along, int line) -> int64_t {
    return DIR == 0 ? (int64_t)along + (int64_t)line * nv : (int64_t)line + (int64_t)along * nv;
  };
  DotAcc<T> dot;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int seg0 = (tile % nseg) * kBandSeg;
    const int line0 = (tile / nseg) * kBandLines;
    // stage in(seg0 - H + m) for m in [0, LEN) of the tile's lines (zero
    // outside) with asynchronous copies, consecutive threads along the
    // contiguous axis; every copy of the tile is in flight before the wait
    if (DIR == 0) {
      for (int line = w; line < kBandLines; line += kBandThreads / 32) {
        const int ln = line0 + line;
        for (int m = lane; m < LEN; m += 32) {
          const int a = seg0 - H + m;
          const bool ok = a >= 0 && a < len && ln < nlines;
          cp_async_elem(sm + sidx(line, m), in + (ok ? gpt(a, ln) * B + col : 0), in, ok);
        }
      }
    } else {
      for (int e = threadIdx.x; e < kBandLines * LEN; e += kBandThreads) {
        const int ln = line0 + (e & (kBandLines - 1)), m = e / kBandLines;
        const int a = seg0 - H + m;
        const bool ok = a >= 0 && a < len && ln < nlines;
        cp_async_elem(sm + sidx(e & (kBandLines - 1), m), in + (ok ? gpt(a, ln) * B + col : 0), in, ok);
      }
    }
    cp_async_wait_all();
    __syncthreads();
    const int o0 = w * kBandR;  // first output of this thread (tile-local)
    T acc[kBandR];
#pragma unroll
    for (int t = 0; t < kBandR; ++t) acc[t] = 0;
    if constexpr (TAPS > 0) {
      // acc[t] += c[k] in(o0 + t + k): sample m = t + k feeds outputs t with
      // 0 <= m - t < TAPS; every tap term in increasing k, as in the chunked form
      const T* line = sm + sidx(lane, o0);
      constexpr int stride = DIR == 0 ? 1 : kBandLines;
#pragma unroll
      for (int m = 0; m < kBandR + TAPS - 1; ++m) {
        const T v = line[m * stride];
#pragma unroll
        for (int t = 0; t < kBandR; ++t)
          if (m - t >= 0 && m - t < TAPS) acc[t] += bd.c[m - t] * v;
      }
    } else {
      for (int q = 0; q < bd.nch; ++q) {
        T cc[kBandChunk];
#pragma unroll
        for (int k = 0; k < kBandChunk; ++k) cc[k] = bd.c[q * kBandChunk + k];
        T win[kBandR + kBandChunk - 1];
#pragma unroll
        for (int m = 0; m < kBandR + kBandChunk - 1; ++m) win[m] = sm[sidx(lane, o0 + q * kBandChunk + m)];
#pragma unroll
        for (int t = 0; t < kBandR; ++t)
#pragma unroll
          for (int k = 0; k < kBandChunk; ++k) acc[t] += cc[k] * win[t + k];
      }
    }
    // The rows near the ends of the line whose coefficients differ (zero
    // boundary) add sum_k d[row][k] in(o - H + k).  Only the tiles at the
    // ends of a line hold such rows; there every thread of the block takes
    // a share of the (row, line) sums, on the output tile in shared memory
    // (the owners of the first and last outputs alone would hold the block
    // at the barrier for the whole of these sums).
    constexpr int OS = kBandSeg + 1;
    T* so = sm + kBandLines * LS;
    const bool corr = bd.d != nullptr && (seg0 < bd.nlo || seg0 + kBandSeg > len - bd.nhi);  // block-uniform
    if (DIR == 0 || corr) {
#pragma unroll
      for (int t = 0; t < kBandR; ++t) so[lane * OS + o0 + t] = acc[t];
    }
    if (corr) {
      __syncthreads();
      const int taps = 2 * H + 1;
      const int ohi = min(seg0 + kBandSeg, len);
      const int hend = min(ohi, bd.nlo);                             // head rows [seg0, hend)
      const int tbeg = max(seg0, max(len - bd.nhi, bd.nlo));         // tail rows [tbeg, ohi)
      const int nhead = max(0, hend - seg0), nrows = nhead + max(0, ohi - tbeg);
      for (int e = threadIdx.x; e < nrows * kBandLines; e += kBandThreads) {
        const int line = e & (kBandLines - 1), rr = e / kBandLines;
        const int o = rr < nhead ? seg0 + rr : tbeg + (rr - nhead);
        const int row = o < bd.nlo ? o : bd.nlo + o - (len - bd.nhi);
        const T* dr = bd.d + (int64_t)row * taps;
        const int ol = o - seg0;
        T sum = 0;
        for (int k = 0; k < taps; ++k) sum += dr[k] * sm[sidx(line, ol + k)];
        so[line * OS + ol] += sum;
      }
    }
    if constexpr (DIR == 0) {
      // through shared memory, so that the stores run along the contiguous axis
      __syncthreads();
      for (int t = threadIdx.x; t < kBandLines * kBandSeg; t += kBandThreads) {
        const int line = t / kBandSeg, m = t - line * kBandSeg;
        const int a = seg0 + m, ln = line0 + line;
        if (a < len && ln < nlines) out[gpt(a, ln) * B + col] = (TO)so[line * OS + m];
      }
    } else {
      if (corr) {
        __syncthreads();
#pragma unroll
        for (int t = 0; t < kBandR; ++t) acc[t] = so[lane * OS + o0 + t];
      }
      const int i = line0 + lane;
      if (i < nv) {
#pragma unroll
        for (int t = 0; t < kBandR; ++t) {
          const int j = seg0 + o0 + t;
          if (j >= nh) break;
          const int64_t p = (int64_t)i + (int64_t)j * nv;
          if (EPI == BAND_STORE) {
            out[p * B + col] = (TO)acc[t];
          } else if (EPI == BAND_RESID2) {
            const double e = to_d(acc[t]) - bvec[p * B + col];
            dot.add(e, e);
          } else {
            auto pv = [&](int64_t qq) { return P[qq * B + col]; };
            const T kv = acc[t] + l2 * fop.lap(p, i, j, pv);
            if (EPI == BAND_NORMAL) {
              out[p * B + col] = (TO)kv;
              dot.add(P[p * B + col], kv);
            } else {
              const T rv = C[p * B + col] - kv;
              out[p * B + col] = (TO)rv;
              dot.add(rv, rv);
            }
          }
        }
      }
    }
    __syncthreads();  // the tile buffer is reloaded by the next tile
  }
  if (EPI != BAND_STORE) {
    double dacc = dot.value();
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) dacc += __shfl_xor_sync(0xffffffffu, dacc, off);
    if (lane == 0) sred[w] = dacc;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int k = 0; k < kBandThreads / 32; ++k) s += sred[k];
      part[(int64_t)blockIdx.x * B + col] = s;
    }
  }
}

// ---- FP64, and small FP32 images ---------------------------------------------
// The same pass with one output per thread and no staging: a thread reads
// its 2H + 1 samples through L1 (consecutive lanes consecutive points along
// the contiguous axis, so every tap of a warp is one or two lines).  Rows
// near the ends of the line take their whole coefficient row from bd.e, in
// one sum; a warp that holds both kinds of rows reads the table for all of
// its lanes (the last row of the table is the interior one).
//
// In FP64 the multiply-adds bound it, not the loads: the pipe takes 19
// cycles per warp instruction, in which L1 serves several taps; and on small
// images one output per thread uses the whole GPU.  Measured on GB300, both
// passes of A^T A in FP64, against tiles of 32 lines x 128 outputs staged in
// shared memory (2 blocks at 64 x 64): 64 x 64, 37 taps 55 + 64 -> 4.5 +
// 9.6 us; 240 x 176, 29 and 25 taps 44 + 56 -> 4.5 + 9.3 us; 1024 x 1024, 61
// taps 164 + 190 -> 128 + 161 us (the multiply-adds alone take 120 each).
// The loads of U taps are issued together (16 on small images, where a warp
// or two per SM sub-partition leave the pass to their latency; 8 on large
// ones, for the registers): 64 x 64, 37 taps 4.6 + 8.9 -> 4.4 + 5.5 us; 1024 x
// 1024, 61 taps 128 + 161 -> 128 + 150 us.
template <class T, class TO, int DIR, int EPI, int U>  // U taps in flight
__global__ void __launch_bounds__(kBandThreads)
    k_band_direct(int nv, int nh, int B, const __grid_constant__ Band<T> bd, const T* __restrict__ in,
                  TO* __restrict__ out, FineOp<T> fop, const T* __restrict__ P, const T* __restrict__ C,
                  const double* __restrict__ lam2, const double* __restrict__ bvec, double* __restrict__ part) {
  __shared__ double sred[kBandThreads / 32];
  const int col = blockIdx.y;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int H = bd.H, taps = 2 * H + 1;
  const int len = DIR == 0 ? nv : nh;
  const int64_t n = (int64_t)nv * nh;
  const int64_t step = (DIR == 0 ? 1 : (int64_t)nv) * B;  // elements between taps
  const T l2 = (EPI == BAND_NORMAL || EPI == BAND_TRUERES) ? (T)lam2[col] : (T)0;
  DotAcc<T> dot;
  // every lane of a warp runs the same number of steps (the vote below)
  for (int64_t p0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; p0 < n; p0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = p0 + lane;
    const bool ok = p < n;
    const int j = (n >> 31) == 0 ? (int)((unsigned)p / (unsigned)nv) : (int)(p / nv);
    const int i = (int)(p - (int64_t)j * nv);
    const int o = DIR == 0 ? i : j;
    const T* __restrict__ x = in + ok * (p * B + col);
    // taps inside the line: k0 <= k < k1
    const int k0 = ok ? max(0, H - o) : 0, k1 = ok ? min(taps, len + H - o) : 0;
    const bool edge = ok && bd.e != nullptr && (o < bd.nlo || o >= len - bd.nhi);
    T acc = 0;
    // U taps at a time: their loads, then their multiply-adds
    if (!__any_sync(0xffffffffu, edge || !ok || k0 > 0 || k1 < taps)) {
      const T* xk = x - H * step;
      int kb = 0;
      for (; kb + U <= taps; kb += U) {
        T xv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) xv[u] = xk[(kb + u) * step];
#pragma unroll
        for (int u = 0; u < U; ++u) acc += bd.c[kb + u] * xv[u];
      }
      for (; kb < taps; ++kb) acc += bd.c[kb] * xk[kb * step];
    } else if (!__any_sync(0xffffffffu, edge)) {
      for (int kb = 0; kb < taps; kb += U) {
        T xv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int k = kb + u;
          xv[u] = k >= k0 && k < k1 ? x[(k - H) * step] : (T)0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) acc += bd.c[kb + u < kBandMaxTaps ? kb + u : 0] * xv[u];
      }
    } else {
      const int row = !edge ? bd.nlo + bd.nhi : (o < bd.nlo ? o : bd.nlo + o - (len - bd.nhi));
      const T* __restrict__ e = bd.e + (int64_t)row * taps;
      for (int kb = 0; kb < taps; kb += U) {
        T xv[U], cv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int k = kb + u;
          const bool in = k >= k0 && k < k1;
          xv[u] = in ? x[(k - H) * step] : (T)0;
          cv[u] = in ? e[k] : (T)0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) acc += cv[u] * xv[u];
      }
    }
    if (!ok) continue;
    if (EPI == BAND_STORE) {
      out[p * B + col] = (TO)acc;
    } else if (EPI == BAND_RESID2) {
      const double e = to_d(acc) - bvec[p * B + col];
      dot.add(e, e);
    } else {
      auto pv = [&](int64_t qq) { return P[qq * B + col]; };
      const T kv = acc + l2 * fop.lap(p, i, j, pv);
      if (EPI == BAND_NORMAL) {
        out[p * B + col] = (TO)kv;
        dot.add(P[p * B + col], kv);
      } else {
        const T rv = C[p * B + col] - kv;
        out[p * B + col] = (TO)rv;
        dot.add(rv, rv);
      }
    }
  }
  if (EPI != BAND_STORE) {
    const double dacc = dot.warp_sum();
    if (lane == 0) sred[w] = dacc;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int k = 0; k < (int)blockDim.x / 32; ++k) s += sred[k];
      part[(int64_t)blockIdx.x * B + col] = s;
    }
  }
}

// diag(A^T A)_p = T_v[i][i] T_h[j][j]
static __global__ void k_sep_diag(int nv, int nh, const double* __restrict__ dv, const double* __restrict__ dh,
                                  double* __restrict__ diag) {
  const int64_t n = (int64_t)nv * nh;
  for (int64_t p = (int64_t)blockIdx.x * kBlock + threadIdx.x; p < n; p += (int64_t)gridDim.x * kBlock) {
    const int j = (int)(p / nv), i = (int)(p - (int64_t)j * nv);
    diag[p] = dv[i] * dh[j];
  }
}

}  // namespace lcmg
