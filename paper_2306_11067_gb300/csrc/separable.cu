// Host side of the separable blur operator: the coefficient sets of the
// banded 1-D passes (built in FP64 from the 1-D PSF factors) and the
// launchers of its kernels.
#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <type_traits>
#include <utility>

#include "launch.h"
#include "psf_tile.cuh"
#include "separable.cuh"

namespace lcmg {

// 1-D correlation A (len x len) with taps f[0..2r]: A[l][l+u] = f[u + r]
// for |u| <= r and 0 <= l + u < len.  The pass for A (transpose false)
// is the correlation itself; for A^T it is the correlation with the
// flipped taps (A^T[i][i-u] = f[u + r]).
SepPass sep_pass_corr(const std::vector<double>& f, bool transpose) {
  const int r = (int)f.size() / 2;
  SepPass p;
  p.H = r;
  p.c.assign(2 * r + 1, 0.0);
  for (int k = 0; k <= 2 * r; ++k) p.c[k] = transpose ? f[2 * r - k] : f[k];
  return p;
}

// T = A^T A of the 1-D correlation above: symmetric, half-bandwidth 2r,
//   T[i][i+k] = sum_{l = 0}^{len-1} f[i - l + r] f[i + k - l + r]
// (terms with |i - l| > r or |i + k - l| > r are zero).  Interior rows hold
// the autocorrelation t_k = sum_u f[u + r] f[u + k + r]; the rows i < r and
// i > len - 1 - r lose the terms with l outside [0, len) and carry the
// difference T[i][i+k] - t_k as their correction row.
SepPass sep_pass_ata(const std::vector<double>& f, int len) {
  const int r = (int)f.size() / 2;
  const int H = 2 * r, taps = 2 * H + 1;
  SepPass p;
  p.H = H;
  p.c.assign(taps, 0.0);
  for (int k = -H; k <= H; ++k) {
    double t = 0.0;
    for (int u = -r; u <= r; ++u)
      if (u + k >= -r && u + k <= r) t += f[u + r] * f[u + k + r];
    p.c[k + H] = t;
  }
  p.nlo = std::min(r, len);
  p.nhi = std::min(r, len - p.nlo);
  p.e.assign((size_t)(p.nlo + p.nhi + 1) * taps, 0.0);
  auto exact_row = [&](int i, std::vector<double>& row, double* whole) {
    for (int k = -H; k <= H; ++k) {
      double s = 0.0;
      if (i + k >= 0 && i + k < len)
        for (int l = std::max(0, std::max(i, i + k) - r); l <= std::min(len - 1, std::min(i, i + k) + r); ++l)
          s += f[i - l + r] * f[i + k - l + r];
      // the interior coefficient applies to in(i + k) only where it exists
      const double interior = (i + k >= 0 && i + k < len) ? p.c[k + H] : 0.0;
      row[k + H] = s - interior;
      whole[k + H] = s;
    }
  };
  p.d.assign((size_t)(p.nlo + p.nhi) * taps, 0.0);
  std::vector<double> row(taps);
  for (int i = 0; i < p.nlo; ++i) {
    exact_row(i, row, p.e.data() + (size_t)i * taps);
    std::copy(row.begin(), row.end(), p.d.begin() + (size_t)i * taps);
  }
  for (int q = 0; q < p.nhi; ++q) {
    exact_row(len - p.nhi + q, row, p.e.data() + (size_t)(p.nlo + q) * taps);
    std::copy(row.begin(), row.end(), p.d.begin() + (size_t)(p.nlo + q) * taps);
  }
  std::copy(p.c.begin(), p.c.end(), p.e.end() - taps);
  return p;
}

// diagonal of T (len values)
std::vector<double> sep_diag(const SepPass& p, int len) {
  const int taps = 2 * p.H + 1;
  std::vector<double> dg(len, p.c[p.H]);
  for (int i = 0; i < p.nlo; ++i) dg[i] += p.d[(size_t)i * taps + p.H];
  for (int q = 0; q < p.nhi; ++q) dg[len - p.nhi + q] += p.d[(size_t)(p.nlo + q) * taps + p.H];
  return dg;
}

template <class T>
Band<T> make_band(const SepPass& p, const T* d_dev) {
  if (p.H < 0 || p.H > kBandMaxH) throw ArgError("band half-width out of range");
  Band<T> b{};
  b.H = p.H;
  b.nch = (2 * p.H + 1 + kBandChunk - 1) / kBandChunk;
  for (int k = 0; k < kBandMaxTaps; ++k) b.c[k] = (k < (int)p.c.size()) ? (T)p.c[k] : (T)0;
  b.nlo = p.d.empty() ? 0 : p.nlo;
  b.nhi = p.d.empty() ? 0 : p.nhi;
  b.d = p.d.empty() ? nullptr : d_dev;
  b.e = p.d.empty() ? nullptr : d_dev + p.d.size();
  return b;
}

// blocks of a banded pass resident at once on the current device
template <class K>
static int band_resident(K kern, size_t smem, int threads = kBandThreads) {
  static std::mutex mu;
  static std::map<std::pair<std::pair<const void*, int>, std::pair<int, size_t>>, int> cache;
  int dev = 0;
  LCMG_CUDA(cudaGetDevice(&dev));
  const auto key = std::make_pair(std::make_pair(reinterpret_cast<const void*>(kern), threads), std::make_pair(dev, smem));
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find(key);
  if (it != cache.end()) return it->second;
  int nb = 0, sms = 0;
  LCMG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, threads, smem));
  LCMG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  if (nb < 1) throw CudaError("banded pass does not fit on an SM");
  cache[key] = nb * sms;
  return nb * sms;
}

static int clamp_blocks(int64_t want, int64_t most) { return (int)std::max<int64_t>(1, std::min(want, most)); }

template <class T, class TO, int DIR, int EPI, int TAPS>
static int band_tiles(int nv, int nh, int B, const Band<T>& bd, const T* in, TO* out, const FineOp<T>& fop, const T* P,
                   const T* C, const double* lam2, const double* bvec, double* part, int max_blocks, cudaStream_t s) {
  auto k = k_band<T, TO, DIR, EPI, TAPS>;
  const size_t smem = band_smem_bytes<T>(bd.nch);
  const int len = DIR == 0 ? nv : nh, lines = DIR == 0 ? nh : nv;
  const int64_t tiles = (int64_t)((len + kBandSeg - 1) / kBandSeg) * ((lines + kBandLines - 1) / kBandLines);
  const int blocks = clamp_blocks(tiles, std::min(max_blocks, band_resident(k, smem)));
  klaunch(k, dim3((unsigned)blocks, (unsigned)B), dim3(kBandThreads), smem, s, nv, nh, B, bd, in, out, fop, P, C,
          lam2, bvec, part);
  LCMG_LAUNCHED();
  return blocks;
}

// the tap counts of the A^T A passes of radii 4, 9 and 15 compiled in (the
// passes of an iteration); the others run in chunks of 8 taps
template <class T, int DIR, int EPI>
constexpr bool kBandCompiled = EPI != BAND_RESID2 && !(std::is_same<T, double>::value && DIR == 1 && EPI == BAND_STORE);
template <class T, class TO, int DIR, int EPI, class... A>
static int band_tiles_any(int nv, int nh, int B, const Band<T>& bd, A... args) {
  if constexpr (kBandCompiled<T, DIR, EPI>) {
    switch (2 * bd.H + 1) {
      case 17: return band_tiles<T, TO, DIR, EPI, 17>(nv, nh, B, bd, args...);
      case 37: return band_tiles<T, TO, DIR, EPI, 37>(nv, nh, B, bd, args...);
      case 61: return band_tiles<T, TO, DIR, EPI, 61>(nv, nh, B, bd, args...);
      default: break;
    }
  }
  return band_tiles<T, TO, DIR, EPI, 0>(nv, nh, B, bd, args...);
}

// k_band_line and k_band_rows: the tap count rounded up to a compiled one
template <class F>
static int by_taps(int taps, F&& f) {
  if (taps <= 17) return f(std::integral_constant<int, 17>{});
  if (taps <= 25) return f(std::integral_constant<int, 25>{});
  if (taps <= 37) return f(std::integral_constant<int, 37>{});
  if (taps <= 49) return f(std::integral_constant<int, 49>{});
  if (taps <= 61) return f(std::integral_constant<int, 61>{});
  return f(std::integral_constant<int, 65>{});
}

static int band_line(int nv, int nh, const Band<float>& bd, const float* in, float* out, int max_blocks,
                     cudaStream_t s) {
  return by_taps(2 * bd.H + 1, [&](auto taps) {
    constexpr int TAPS = decltype(taps)::value;
    const int64_t tasks = (int64_t)((nv + kLineSeg - 1) / kLineSeg) * nh;
    const int blocks = clamp_blocks((tasks + kLineWarps - 1) / kLineWarps, max_blocks);
    klaunch(k_band_line<TAPS>, dim3((unsigned)blocks), dim3(32 * kLineWarps), 0, s, nv, nh, bd, in, out);
    LCMG_LAUNCHED();
    return blocks;
  });
}
static int band_rows(int nv, int nh, const Band<float>& bd, const float* in, float* out,
                     const FineOp<float>& fop, const float* P, const double* lam2, double* part, int max_blocks,
                     cudaStream_t s) {
  return by_taps(2 * bd.H + 1, [&](auto taps) {
    constexpr int TAPS = decltype(taps)::value;
    const int64_t tiles = (int64_t)((nv + 31) / 32) * ((nh + kRowTile - 1) / kRowTile);
    const int blocks = clamp_blocks(tiles, max_blocks);
    klaunch(k_band_rows<TAPS>, dim3((unsigned)blocks), dim3(32 * kRowWarps), sizeof(float) * rows_floats(TAPS), s, nv,
            nh, bd, in, out, fop, P, lam2, part);
    LCMG_LAUNCHED();
    return blocks;
  });
}

// opt k_band and k_band_rows into their shared memory on the current device
// (outside stream capture)
template <class T, int DIR, int EPI, int TAPS>
static void band_optin() {
  const int bytes = (int)band_smem_bytes<T>((2 * kBandMaxH + 1 + kBandChunk - 1) / kBandChunk);
  LCMG_CUDA(cudaFuncSetAttribute(k_band<T, T, DIR, EPI, TAPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
}
template <class T, int DIR, int EPI>
static void band_optin_taps() {
  band_optin<T, DIR, EPI, 0>();
  if constexpr (kBandCompiled<T, DIR, EPI>) {
    band_optin<T, DIR, EPI, 17>();
    band_optin<T, DIR, EPI, 37>();
    band_optin<T, DIR, EPI, 61>();
  }
}
void prepare_band() {
  for (int taps : {17, 25, 37, 49, 61, 65})
    by_taps(taps, [&](auto t) {
      constexpr int TAPS = decltype(t)::value;
      LCMG_CUDA(cudaFuncSetAttribute(k_band_rows<TAPS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(float) * rows_floats(TAPS)));
      return 0;
    });
  band_optin_taps<float, 0, BAND_STORE>();
  band_optin_taps<float, 1, BAND_NORMAL>();
  band_optin_taps<double, 0, BAND_STORE>();
  band_optin_taps<double, 1, BAND_STORE>();
  band_optin_taps<double, 1, BAND_NORMAL>();
  band_optin_taps<double, 1, BAND_RESID2>();
  band_optin_taps<double, 1, BAND_TRUERES>();
}

template <class T, class TO, int DIR, int EPI>
static int band_direct(int nv, int nh, int B, const Band<T>& bd, const T* in, TO* out, const FineOp<T>& fop,
                       const T* P, const T* C, const double* lam2, const double* bvec, double* part, int max_blocks,
                       cudaStream_t s) {
  const int64_t n = (int64_t)nv * nh;
  // small images in blocks of two warps, so that they spread over more SMs,
  // with more taps in flight per warp
  const int threads = n <= 64 * 1024 ? 64 : kBandThreads;
  constexpr int kSmallU = 16, kLargeU = sizeof(T) == 8 ? 8 : 16;
  auto k = threads == 64 ? k_band_direct<T, TO, DIR, EPI, kSmallU> : k_band_direct<T, TO, DIR, EPI, kLargeU>;
  const int blocks = clamp_blocks((n + threads - 1) / threads, std::min(max_blocks, band_resident(k, 0, threads)));
  klaunch(k, dim3((unsigned)blocks, (unsigned)B), dim3(threads), 0, s, nv, nh, B, bd, in, out, fop, P, C, lam2, bvec,
          part);
  LCMG_LAUNCHED();
  return blocks;
}

// FP32 passes of at most this many points (x columns) run with one output per
// thread: the other kernels give a thread 16, so that below it part of the GPU
// has none.  Measured on GB300, both passes of A^T A, one column: 384 x 384,
// 61 taps 20.6 us against 22.6 in k_band_line + k_band_rows, 448 x 448 24.6
// against 22.6, 512 x 512 28.8 against 24.6; 37 taps 16.5 / 19.7, 21.4 / 20.5,
// 22.6 / 20.5.
constexpr int64_t kBandDirectMax = 440 * 440;
constexpr int64_t kBandDirectMaxTiles = 256 * 256;  // ... where the alternative is k_band

// Many columns in FP64: interleaved columns put the samples of neighbouring
// points 8 B bytes apart, and one output per thread fetches a 32-byte sector
// for each of them at every tap, where the tiles of k_band (32 x 128 outputs)
// fetch it once.  Along the contiguous axis that costs most where the distance
// is a multiple of the 128-byte line; along the strided one more with every
// column.  The tiles in turn leave part of the GPU idle where they are ragged
// or don't make the same number for every SM: `used` is the share of their
// outputs that count.  Measured on GB300 in an iteration, one output per
// thread / tiles, along i and along j: 256 x 256, 37 taps, 16 columns 145 / 116
// and 162 / 145 us, 32 columns 277 / 212 and 311 / 264, 24 columns 141 / 165
// and 223 / 206; 512 x 512, 61 taps, 16 columns 857 / 567 and 924 / 652, 8
// columns 255 / 319 and 308 / 364; 128 x 128, 37 taps, 16 columns 47 / 67 and
// 49 / 84; 320 x 320, 61 taps, 16 columns (used 0.66) 340 / 330 and 366 / 371.
static bool band64_in_tiles(int dir, int nv, int nh, int B) {
  const int len = dir == 0 ? nv : nh, lines = dir == 0 ? nh : nv, sms = sm_count();
  const int64_t tiles = (int64_t)((len + kBandSeg - 1) / kBandSeg) * ((lines + kBandLines - 1) / kBandLines) * B;
  const double used = (double)nv * nh * B / ((double)((tiles + sms - 1) / sms * sms) * (kBandSeg * kBandLines));
  return used >= 0.75 && (dir == 0 ? B % 16 == 0 : B * used >= 11.5);
}

template <class T, class TO, int DIR, int EPI>
int launch_band(int nv, int nh, int B, const Band<T>& bd, const T* in, TO* out, const FineOp<T>& fop, const T* P,
                const T* C, const double* lam2, const double* bvec, double* part, int max_blocks, cudaStream_t s) {
  if constexpr (std::is_same<T, float>::value) {
    static_assert((DIR == 0 && EPI == BAND_STORE) || (DIR == 1 && EPI == BAND_NORMAL), "the FP32 passes of A^T A");
    const int64_t work = (int64_t)nv * nh * B;
    if (B == 1 && nv % 4 == 0) {  // 16-byte words (every vector of a solve starts on such a boundary)
      if (work > kBandDirectMax) {
        if constexpr (DIR == 0)
          return band_line(nv, nh, bd, in, out, max_blocks, s);
        else
          return band_rows(nv, nh, bd, in, out, fop, P, lam2, part, max_blocks, s);
      }
    } else if (work > kBandDirectMaxTiles) {
      return band_tiles_any<T, TO, DIR, EPI>(nv, nh, B, bd, in, out, fop, P, C, lam2, bvec, part, max_blocks, s);
    }
  } else if (band64_in_tiles(DIR, nv, nh, B)) {
    return band_tiles_any<T, TO, DIR, EPI>(nv, nh, B, bd, in, out, fop, P, C, lam2, bvec, part, max_blocks, s);
  }
  return band_direct<T, TO, DIR, EPI>(nv, nh, B, bd, in, out, fop, P, C, lam2, bvec, part, max_blocks, s);
}

// Tiles of 8 rows in blocks of 64 threads while tiles of 32 would give an SM
// less than two, else of 32 rows (the halo of 2 rh rows is staged per tile); one output per thread
// where the PSF's tile does not fit in kPsfSmem (radii above 24 or so).
template <int TRANS, int EPI>
int launch_psf(const PsfArgs& a, const float* psf, int B, const float* in, float* out, const FineOp<float>& fop,
               const float* P, const double* lam2, double* part, int max_blocks, cudaStream_t s) {
  const int nti = (a.nv + kPsfTI - 1) / kPsfTI;
  auto tiles = [&](int tj) { return (int64_t)nti * ((a.nh + tj - 1) / tj); };
  const int tj = tiles(32) * B < 2 * sm_count() || psf_smem(a.rv, a.rh, 32) > kPsfSmem ? 8 : 32;
  const size_t smem = psf_smem(a.rv, a.rh, tj);
  if (smem <= kPsfSmem) {
    const int blocks = clamp_blocks(tiles(tj), max_blocks);
    klaunch(k_psf_tile<TRANS, EPI>, dim3((unsigned)blocks, (unsigned)B), dim3(8 * tj), smem, s, a, psf, B, in, out, fop, P,
            lam2, part);
    LCMG_LAUNCHED();
    return blocks;
  }
  const int g = grid_for((int64_t)a.nv * a.nh, B, max_blocks);
  if constexpr (EPI == PSF_STORE)
    klaunch(k_psf_forward<float, 0>, dim3(g), dim3(kBlock), 0, s, a, psf, B, in, out, nullptr, 1, 1, nullptr);
  else
    klaunch(k_psf_normal<float, float, 1>, dim3(g), dim3(kBlock), 0, s, a, psf, B, in, fop, P, nullptr, lam2, out, part);
  LCMG_LAUNCHED();
  return g;
}

void launch_sep_diag(int nv, int nh, const double* dv, const double* dh, double* diag, int max_blocks,
                     cudaStream_t s) {
  const int64_t n = (int64_t)nv * nh;
  const int g = (int)std::max<int64_t>(1, std::min<int64_t>((n + kBlock - 1) / kBlock, max_blocks));
  klaunch(k_sep_diag, dim3(g), dim3(kBlock), 0, s, nv, nh, dv, dh, diag);
  LCMG_LAUNCHED();
}

template Band<float> make_band<float>(const SepPass&, const float*);
template Band<double> make_band<double>(const SepPass&, const double*);
#define LCMG_BAND_INST(T, TO, DIR, EPI)                                                                          \
  template int launch_band<T, TO, DIR, EPI>(int, int, int, const Band<T>&, const T*, TO*, const FineOp<T>&,    \
                                            const T*, const T*, const double*, const double*, double*, int,     \
                                            cudaStream_t);
LCMG_BAND_INST(float, float, 0, BAND_STORE)
LCMG_BAND_INST(float, float, 1, BAND_NORMAL)
LCMG_BAND_INST(double, double, 0, BAND_STORE)
LCMG_BAND_INST(double, double, 1, BAND_STORE)
LCMG_BAND_INST(double, double, 1, BAND_NORMAL)
LCMG_BAND_INST(double, double, 1, BAND_RESID2)
LCMG_BAND_INST(double, double, 1, BAND_TRUERES)
#undef LCMG_BAND_INST

template int launch_psf<0, PSF_STORE>(const PsfArgs&, const float*, int, const float*, float*, const FineOp<float>&,
                                      const float*, const double*, double*, int, cudaStream_t);
template int launch_psf<1, PSF_NORMAL>(const PsfArgs&, const float*, int, const float*, float*, const FineOp<float>&,
                                       const float*, const double*, double*, int, cudaStream_t);

}  // namespace lcmg
