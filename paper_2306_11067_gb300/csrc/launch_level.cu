// Launchers of the V-cycle level kernels, the coarsest-level dense setup,
// the Galerkin products and the PCG vector updates.
#include <algorithm>
#include <map>
#include <mutex>
#include <type_traits>
#include <utility>

#include "launch.h"
#include "vcoarse.cuh"
#include "vtail.cuh"
#include "vfine.cuh"
#include "vfused.cuh"
#include "vlevel64.cuh"

namespace lcmg {

template <class T>
void launch_dinv(const LevelView<T>& L, int B, const double* lam2, int smoother, double omega,
                 T* dinv, int max_blocks, cudaStream_t s) {
  const int g = grid_for(L.n, B, max_blocks);
  if constexpr (std::is_same<T, float>::value) {
    if (L.h16) {
      if (L.fine)
        klaunch(k_dinv<FineOpH, float>, dim3(g), dim3(kBlock), 0, s, L.fh, L.n, B, lam2, smoother, omega, dinv);
      else
        L.ch.rows ? klaunch(k_dinv<CoarseOpH, float>, dim3(g), dim3(kBlock), 0, s, L.ch, L.n, B, lam2, smoother, omega, dinv)
                  : klaunch(k_dinv<CoarseRowsH, float>, dim3(g), dim3(kBlock), 0, s, L.cr, L.n, B, lam2, smoother, omega, dinv);
      LCMG_LAUNCHED();
      return;
    }
  }
  if (L.fine)
    klaunch(k_dinv<FineOp<T>, T>, dim3(g), dim3(kBlock), 0, s, L.fine_op(), L.n, B, lam2, smoother, omega, dinv);
  else
    klaunch(k_dinv<CoarseOp<T>, T>, dim3(g), dim3(kBlock), 0, s, L.coarse_op(), L.n, B, lam2, smoother, omega, dinv);
  LCMG_LAUNCHED();
}

template <class T>
void launch_smooth_zero(const LevelView<T>& L, int B, const T* lam2, const T* dinv, const T* r,
                        T* z, int two, int max_blocks, cudaStream_t s) {
  const int g = grid_for(L.n, B, max_blocks);
  if (L.fine)
    klaunch(k_smooth_zero<FineOp<T>, T>, dim3(g), dim3(kBlock), 0, s, L.fine_op(), L.n, B, lam2, dinv, r, z, two);
  else
    klaunch(k_smooth_zero<CoarseOp<T>, T>, dim3(g), dim3(kBlock), 0, s, L.coarse_op(), L.n, B, lam2, dinv, r, z, two);
  LCMG_LAUNCHED();
}

template <class T>
int launch_smooth(const LevelView<T>& L, int B, const T* lam2, const T* dinv, const T* r,
                  const T* zin, T* zout, const int* active, double* part, int max_blocks,
                  cudaStream_t s) {
  const int g = grid_for(L.n, B, max_blocks);
  if (L.fine)
    klaunch(k_smooth<FineOp<T>, T>, dim3(g), dim3(kBlock), 0, s, L.fine_op(), L.n, B, lam2, dinv, r, zin, zout, active, part);
  else
    klaunch(k_smooth<CoarseOp<T>, T>, dim3(g), dim3(kBlock), 0, s, L.coarse_op(), L.n, B, lam2, dinv, r, zin, zout, active, part);
  LCMG_LAUNCHED();
  return g;
}

template <class T>
void launch_residual(const LevelView<T>& L, int B, const T* lam2, const T* r, const T* z, T* res,
                     int max_blocks, cudaStream_t s) {
  const int g = grid_for(L.n, B, max_blocks);
  if (L.fine)
    klaunch(k_residual<FineOp<T>, T>, dim3(g), dim3(kBlock), 0, s, L.fine_op(), L.n, B, lam2, r, z, res);
  else
    klaunch(k_residual<CoarseOp<T>, T>, dim3(g), dim3(kBlock), 0, s, L.coarse_op(), L.n, B, lam2, r, z, res);
  LCMG_LAUNCHED();
}

int sm_count() {
  static const int count = [] {
    int dev = 0, sms = 0;
    LCMG_CUDA(cudaGetDevice(&dev));
    LCMG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    return sms;
  }();
  return count;
}

// Grid of a tile kernel: every tile once, at most the blocks resident at
// once on the device and at most kMaxTileBlocks (rows of the partial sums).
template <class K>
static int tile_grid(K kern, int threads, int ntiles) {
  static std::mutex mu;
  static std::map<std::pair<const void*, int>, int> cache;
  int dev = 0;
  LCMG_CUDA(cudaGetDevice(&dev));
  const auto key = std::make_pair(reinterpret_cast<const void*>(kern), dev);
  int wave;
  {
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache.find(key);
    if (it == cache.end()) {
      int nb = 0;
      LCMG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, threads, 0));
      it = cache.emplace(key, std::max(1, nb) * sm_count()).first;
    }
    wave = it->second;
  }
  return std::max(1, std::min(std::min(ntiles, wave), kMaxTileBlocks));
}

template <class Op, class T, int NU>
static int vdown_one(const Op& op, int B, const T* lam2, const T* dinv, const T* r, T* zpre, T* rc, int ntx,
                     int ntiles, cudaStream_t s) {
  auto k = k_vdown<Op, T, NU>;
  const int g = tile_grid(k, vtile_threads<Op, T, NU>(), ntiles);
  klaunch(k, dim3((unsigned)g, (unsigned)B), dim3(vtile_threads<Op, T, NU>()), 0, s, op, B, lam2, dinv, r, zpre, rc,
          ntx, ntiles);
  return g;
}

template <class Op, class T, int NU>
static int vup_one(const Op& op, int B, const T* lam2, const T* dinv, const T* r, const T* ec, const T* zpre,
                   T* zout, double* part, int ntx, int ntiles, cudaStream_t s) {
  auto k = k_vup<Op, T, NU>;
  const int g = tile_grid(k, vtile_threads<Op, T, NU>(), ntiles);
  klaunch(k, dim3((unsigned)g, (unsigned)B), dim3(vtile_threads<Op, T, NU>()), 0, s, op, B, lam2, dinv, r, ec, zpre,
          zout, ntx, ntiles, part);
  return g;
}

// FP64 with one sweep (vlevel64.cuh): f(integral_constant<tile side>, tiles
// along i, tiles) with the side that leaves the fewest residual points on
// the busiest SM.  A level of 512^2 points takes 8 x 8 coarse points (7
// tiles of 18^2 on an SM), one of 32^2 takes 2 x 2 (64 tiles of 6^2 against 4 of
// 18^2).  Measured on GB300 against 8 x 8 tiles with both parts of K read at
// every point (down + up): 64 x 64 problem, its 32 x 32 level 11.5 + 9.7 ->
// 5.7 + 5.6 us; 240 x 176, mean of three coarse levels 11.6 + 9.8 -> 5.8 +
// 5.9 us; 1024 x 1024, mean of five 26.6 + 21.2 -> 14 + 10 us.
template <class F>
static int tiles64(int nvc, int nhc, int B, F&& f) {
  const int sms = sm_count();
  auto nt = [](int n, int tc) { return (n + tc - 1) / tc; };
  int best = 8;
  int64_t least = INT64_MAX;
  for (int tc : {8, 4, 2}) {
    const int64_t tiles = (int64_t)nt(nvc, tc) * nt(nhc, tc) * B;
    const int64_t cost = (tiles + sms - 1) / sms * (2 * tc + 2) * (2 * tc + 2);
    if (cost < least) {
      least = cost;
      best = tc;
    }
  }
  const int ntx = nt(nvc, best), n = ntx * nt(nhc, best);
  if (best == 8) return f(std::integral_constant<int, 8>{}, ntx, n);
  if (best == 4) return f(std::integral_constant<int, 4>{}, ntx, n);
  return f(std::integral_constant<int, 2>{}, ntx, n);
}
template <class Op>
static int vdown64(const Op& op, int B, const double* lam2, const double* dinv, const double* r, double* zpre,
                   double* rc, cudaStream_t s) {
  return tiles64(op.nv / 2, op.nh / 2, B, [&](auto tc, int ntx, int nt) {
    constexpr int TC = decltype(tc)::value;
    auto k = k_vdown64<Op, TC>;
    const int g = tile_grid(k, vt64_threads(TC), nt);
    klaunch(k, dim3((unsigned)g, (unsigned)B), dim3(vt64_threads(TC)), 0, s, op, B, lam2, dinv, r, zpre, rc, ntx, nt);
    return g;
  });
}
template <class Op>
static int vup64(const Op& op, int B, const double* lam2, const double* dinv, const double* r, const double* ec,
                 const double* zpre, double* zout, double* part, cudaStream_t s) {
  return tiles64(op.nv / 2, op.nh / 2, B, [&](auto tc, int ntx, int nt) {
    constexpr int TC = decltype(tc)::value;
    auto k = k_vup64<Op, TC>;
    const int g = tile_grid(k, vt64_threads(TC), nt);
    klaunch(k, dim3((unsigned)g, (unsigned)B), dim3(vt64_threads(TC)), 0, s, op, B, lam2, dinv, r, ec, zpre, zout,
            ntx, nt, part);
    return g;
  });
}

void launch_rows64(int64_t n, const double* gl, const double* ga, double lam2, double* kr, int max_blocks,
                   cudaStream_t s) {
  const int64_t count = kStencil * n;
  const int g = (int)std::max<int64_t>(1, std::min<int64_t>((count + kBlock - 1) / kBlock, max_blocks));
  klaunch(k_rows64, dim3(g), dim3(kBlock), 0, s, count, gl, ga, lam2, kr);
  LCMG_LAUNCHED();
}

// FP16 coarse levels with one sweep (vcoarse.cuh): coarse rows per strip, so
// that the strips make kVcWarps warps per SM (of at most 16 rows; a strip
// reads two residual rows more than it produces).  Measured on GB300 at
// 1024^2 points with 8, 16 and 24 warps: down 23.7, 18.4, 22.1 us.
static int coarse_strip(int nsi, int nhc, int B) {
  const int64_t per_col = std::max<int64_t>(1, ((int64_t)sm_count() * kVcWarps) / ((int64_t)nsi * B));
  return std::max(1, std::min(16, (int)((nhc + per_col - 1) / per_col)));
}
template <class K, class... A>
static int strips_h(K k, int nsi, int crows, const CoarseOpH& op, int B, cudaStream_t s, A... args) {
  const int nst = nsi * ((op.nh / 2 + crows - 1) / crows), wpb = kVcThreads / 32;
  const int g = (nst + wpb - 1) / wpb;
  klaunch(k, dim3((unsigned)g, (unsigned)B), dim3(kVcThreads), 0, s, op, B, args..., nsi, nst, crows);
  return g;
}
static int vdown_h(const CoarseOpH& op, int B, const float* dinv, const float* r, float* rc, cudaStream_t s) {
  const int nsi = (op.nv / 2 + kVcDownCols - 1) / kVcDownCols, g = nsi * (op.nh / 2);
  const int crows = coarse_strip(nsi, op.nh / 2, B);
  if (crows == 1) {  // levels of 256^2 points (columns included) and below
    klaunch(B == 1 ? k_vdown_h1<true> : k_vdown_h1<false>, dim3((unsigned)g, (unsigned)B), dim3(kVcThreads), 0, s, op,
            B, dinv, r, rc, nsi);
    return g;
  }
  return strips_h(B == 1 ? k_vdown_h<true> : k_vdown_h<false>, nsi, crows, op, B, s, dinv, r, rc);
}
static int vup_h(const CoarseOpH& op, int B, const float* dinv, const float* r, const float* ec, float* zout,
                 cudaStream_t s) {
  const int nsi = (op.nv / 2 + kVcUpCols - 1) / kVcUpCols;
  return strips_h(B == 1 ? k_vup_h<true> : k_vup_h<false>, nsi, coarse_strip(nsi, op.nh / 2, B), op, B, s, dinv, r, ec,
                  zout);
}

template <class T>
int launch_vdown(const LevelView<T>& L, int B, const T* lam2, const T* dinv, const T* r, T* zpre, T* rc,
                 int nu, cudaStream_t s) {
  const int ntx = (L.nv / 2 + kVTile - 1) / kVTile, nty = (L.nh / 2 + kVTile - 1) / kVTile;
  const int nt = ntx * nty;
  int g;
  if constexpr (std::is_same<T, float>::value) {
    if (L.h16) {
      if (L.fine)
        g = nu == 1 ? vdown_one<FineOpH, float, 1>(L.fh, B, lam2, dinv, r, zpre, rc, ntx, nt, s)
                    : vdown_one<FineOpH, float, 2>(L.fh, B, lam2, dinv, r, zpre, rc, ntx, nt, s);
      else
        g = nu == 1 ? vdown_h(L.ch, B, dinv, r, rc, s)
                    : vdown_one<CoarseRowsH, float, 2>(L.cr, B, lam2, dinv, r, zpre, rc, ntx, nt, s);
      LCMG_LAUNCHED();
      return g;
    }
  }
  if constexpr (std::is_same<T, double>::value) {
    if (nu == 1) {
      g = L.fine ? vdown64(L.fine_op(), B, lam2, dinv, r, zpre, rc, s)
          : L.kr ? vdown64(RowsOp64{L.nv, L.nh, L.n, L.kr}, B, lam2, dinv, r, zpre, rc, s)
                 : vdown64(L.coarse_op(), B, lam2, dinv, r, zpre, rc, s);
      LCMG_LAUNCHED();
      return g;
    }
    g = L.fine ? vdown_one<FineOp<T>, T, 2>(L.fine_op(), B, lam2, dinv, r, zpre, rc, ntx, nt, s)
               : vdown_one<CoarseOp<T>, T, 2>(L.coarse_op(), B, lam2, dinv, r, zpre, rc, ntx, nt, s);
  } else if (L.fine)
    g = nu == 1 ? vdown_one<FineOp<T>, T, 1>(L.fine_op(), B, lam2, dinv, r, zpre, rc, ntx, nt, s)
                : vdown_one<FineOp<T>, T, 2>(L.fine_op(), B, lam2, dinv, r, zpre, rc, ntx, nt, s);
  else
    g = nu == 1 ? vdown_one<CoarseOp<T>, T, 1>(L.coarse_op(), B, lam2, dinv, r, zpre, rc, ntx, nt, s)
                : vdown_one<CoarseOp<T>, T, 2>(L.coarse_op(), B, lam2, dinv, r, zpre, rc, ntx, nt, s);
  LCMG_LAUNCHED();
  return g;
}

template <class T>
int launch_vup(const LevelView<T>& L, int B, const T* lam2, const T* dinv, const T* r, const T* ec,
               const T* zpre, T* zout, double* part, int nu, cudaStream_t s) {
  const int ntx = (L.nv / 2 + kVTile - 1) / kVTile, nty = (L.nh / 2 + kVTile - 1) / kVTile;
  const int nt = ntx * nty;
  int g;
  if constexpr (std::is_same<T, float>::value) {
    if (L.h16) {
      if (L.fine)
        g = nu == 1 ? vup_one<FineOpH, float, 1>(L.fh, B, lam2, dinv, r, ec, zpre, zout, part, ntx, nt, s)
                    : vup_one<FineOpH, float, 2>(L.fh, B, lam2, dinv, r, ec, zpre, zout, part, ntx, nt, s);
      else
        g = nu == 1 ? vup_h(L.ch, B, dinv, r, ec, zout, s)
                    : vup_one<CoarseRowsH, float, 2>(L.cr, B, lam2, dinv, r, ec, zpre, zout, part, ntx, nt, s);
      LCMG_LAUNCHED();
      return g;
    }
  }
  if constexpr (std::is_same<T, double>::value) {
    if (nu == 1) {
      g = L.fine ? vup64(L.fine_op(), B, lam2, dinv, r, ec, zpre, zout, part, s)
          : L.kr ? vup64(RowsOp64{L.nv, L.nh, L.n, L.kr}, B, lam2, dinv, r, ec, zpre, zout, part, s)
                 : vup64(L.coarse_op(), B, lam2, dinv, r, ec, zpre, zout, part, s);
      LCMG_LAUNCHED();
      return g;
    }
    g = L.fine ? vup_one<FineOp<T>, T, 2>(L.fine_op(), B, lam2, dinv, r, ec, zpre, zout, part, ntx, nt, s)
               : vup_one<CoarseOp<T>, T, 2>(L.coarse_op(), B, lam2, dinv, r, ec, zpre, zout, part, ntx, nt, s);
  } else if (L.fine)
    g = nu == 1 ? vup_one<FineOp<T>, T, 1>(L.fine_op(), B, lam2, dinv, r, ec, zpre, zout, part, ntx, nt, s)
                : vup_one<FineOp<T>, T, 2>(L.fine_op(), B, lam2, dinv, r, ec, zpre, zout, part, ntx, nt, s);
  else
    g = nu == 1 ? vup_one<CoarseOp<T>, T, 1>(L.coarse_op(), B, lam2, dinv, r, ec, zpre, zout, part, ntx, nt, s)
                : vup_one<CoarseOp<T>, T, 2>(L.coarse_op(), B, lam2, dinv, r, ec, zpre, zout, part, ntx, nt, s);
  LCMG_LAUNCHED();
  return g;
}

bool vtail_fits(int nlev) { return nlev >= 2 && nlev <= kTailMaxLevels; }

void launch_vtail(const TailLevelIn* levels, int nlev, const double* kinv, int nc, int B, cudaStream_t s) {
  if (!vtail_fits(nlev)) throw ArgError("tail of the V-cycle: level count out of range");
  TailArgs a{};
  a.nlev = nlev;
  int off = 0;
  auto take = [&](int bytes) {
    const int o = off;
    off += (bytes + 15) / 16 * 16;
    return o;
  };
  for (int k = 0; k < nlev; ++k) {
    const TailLevelIn& in = levels[k];
    const int n = in.op.nv * in.op.nh;
    TailLevel& L = a.lv[k];
    L.op = in.op;
    L.dinv = in.dinv;
    L.rhs = in.rhs;
    L.z = in.z;
    const bool coarsest = k == nlev - 1;
    L.o_rows = coarsest ? 0 : take(48 * n);
    L.o_c = coarsest ? 0 : take(4 * n);
    L.o_d = coarsest ? 0 : take(4 * n);
    L.o_r = take(4 * n);
    const int np = tail_padded(in.op.nv, in.op.nh);
    L.o_t = coarsest ? 0 : take(4 * np);
    L.o_res = coarsest ? 0 : take(4 * np);
    L.o_z = take(4 * n);
  }
  a.kinv = kinv;
  a.nc = nc;
  static int optin_dev = -1;
  int dev = 0;
  LCMG_CUDA(cudaGetDevice(&dev));
  if (optin_dev != dev) {
    int maxsm = 0;
    LCMG_CUDA(cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    LCMG_CUDA(cudaFuncSetAttribute(k_vtail_h, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsm));
    optin_dev = dev;
  }
  klaunch(k_vtail_h, dim3(1, (unsigned)B), dim3(kTailThreads), (size_t)off, s, a, B);
  LCMG_LAUNCHED();
}

// Blocks and threads of the fused one-column updates: one 16-byte word per
// thread, at most two blocks per SM (every block re-sums the partials of the
// dot products it needs in FP64); blocks of 256 threads while they fit on as
// many SMs, so that a short vector's FP64 work is spread
static dim3 fused_update_grid(int64_t words, int max_blocks, int* threads) {
  const int sms = sm_count();
  *threads = words <= (int64_t)sms * (kUpdThreads / 2) ? kUpdThreads / 2 : kUpdThreads;
  const int64_t want = (words + *threads - 1) / *threads;
  return dim3((unsigned)std::max<int64_t>(1, std::min(want, (int64_t)std::min(2 * sms, max_blocks))));
}

// Rows per strip of the row-streaming kernels: at most `most`, and few
// enough that the strips make `warps` warps per SM (one warp walks a strip in
// sequence, so on a small grid long strips leave most of the GPU idle), but at
// least `least` (the strip's halo rows are computed twice).
static int strip_rows(int nsi, int B, int len, int warps, int most, int least) {
  const int64_t want = (int64_t)sm_count() * warps;
  const int64_t per_col = std::max<int64_t>(1, want / ((int64_t)nsi * B));  // strips wanted along the rows
  const int rows = (int)((len + per_col - 1) / per_col);
  return std::max(least, std::min(most, rows));
}
// blocks of 8 warps, or of 2 while the strips are few (so that they spread over the SMs)
static int strip_threads(int nst, int B) { return (int64_t)nst * B <= 8 * sm_count() ? 64 : kFineThreads; }

int launch_vfine_down(const LevelView<float>& L, int B, const float* lam2, int smoother, double omega,
                      const float* r, float* rc, cudaStream_t s) {
  int g;
  if (L.h16) {  // row streaming
    const int nsi = (L.nv / 2 + kFineCols - 1) / kFineCols;
    const int crows = strip_rows(nsi, B, L.nh / 2, kFineDownWarps, kStripCoarse, 1);
    const int nst = nsi * ((L.nh / 2 + crows - 1) / crows);
    auto k = B == 1 ? k_vfine_down_s<true> : k_vfine_down_s<false>;
    const int threads = strip_threads(nst, B);
    g = std::min((nst + threads / 32 - 1) / (threads / 32), kMaxTileBlocks);
    klaunch(k, dim3((unsigned)g, (unsigned)B), dim3(threads), 0, s, L.fh, B, lam2, smoother, (float)omega, r, rc, nsi,
            nst, crows);
  } else {
    const int nt = ((L.nv + kFineTI - 1) / kFineTI) * ((L.nh + kFineTJ - 1) / kFineTJ);
    g = tile_grid(k_vfine_down, kFineThreads, nt);
    klaunch(k_vfine_down, dim3((unsigned)g, (unsigned)B), dim3(kFineThreads), 0, s, L.fine_op(), B, lam2, smoother,
            (float)omega, r, rc, nt);
  }
  LCMG_LAUNCHED();
  return g;
}

int launch_vfine_up(const LevelView<float>& L, int B, const float* lam2, int smoother, double omega,
                    const float* r, const float* ec, float* zout, double* part, cudaStream_t s) {
  int g;
  if (L.h16) {  // row streaming
    const int nsi = (L.nv / 2 + kFineCols - 1) / kFineCols;
    const int rows = strip_rows(nsi, B, L.nh, kFineUpWarps, kStripRows, 2);
    const int nst = nsi * ((L.nh + rows - 1) / rows);
    auto k = B == 1 ? k_vfine_up_s<true> : k_vfine_up_s<false>;
    const int threads = strip_threads(nst, B);
    g = std::min((nst + threads / 32 - 1) / (threads / 32), kMaxTileBlocks);
    klaunch(k, dim3((unsigned)g, (unsigned)B), dim3(threads), 0, s, L.fh, B, lam2, smoother, (float)omega, r, ec, zout,
            nsi, nst, rows, part);
  } else {
    const int nt = ((L.nv + kFineTI - 1) / kFineTI) * ((L.nh + kFineTJ - 1) / kFineTJ);
    g = tile_grid(k_vfine_up, kFineThreads, nt);
    klaunch(k_vfine_up, dim3((unsigned)g, (unsigned)B), dim3(kFineThreads), 0, s, L.fine_op(), B, lam2, smoother,
            (float)omega, r, ec, zout, nt, part);
  }
  LCMG_LAUNCHED();
  return g;
}

template <class T>
void launch_restrict(int nvc, int nhc, int B, const T* rf, T* rc, int max_blocks, cudaStream_t s) {
  const int g = grid_for((int64_t)nvc * nhc, B, max_blocks);
  klaunch(k_restrict<T>, dim3(g), dim3(kBlock), 0, s, nvc, nhc, B, rf, rc);
  LCMG_LAUNCHED();
}

template <class T>
void launch_prolong_add(int nvc, int nhc, int B, const T* ec, T* zf, int max_blocks, cudaStream_t s) {
  const int g = grid_for((int64_t)4 * nvc * nhc, B, max_blocks);
  klaunch(k_prolong_add<T>, dim3(g), dim3(kBlock), 0, s, nvc, nhc, B, ec, zf);
  LCMG_LAUNCHED();
}

template <class T>
void launch_coarse_solve(int nc, int B, const double* kinv, const T* rc, T* ec, cudaStream_t s) {
  const size_t smem = sizeof(double) * (size_t)nc;
  dim3 grid((unsigned)((nc + kBlock / 32 - 1) / (kBlock / 32)), (unsigned)B);
  klaunch(k_coarse_solve<T>, dim3(grid), dim3(kBlock), smem, s, nc, B, kinv, rc, ec);
  LCMG_LAUNCHED();
}

void launch_dense_setup(const LevelView<double>& L, int B, const double* lam2, double* M, double* W,
                        double* K, int* info, int max_blocks, cudaStream_t s) {
  const int64_t nc = L.n;
  LCMG_CUDA(cudaMemsetAsync(M, 0, sizeof(double) * (size_t)B * nc * nc, s));
  const int g = grid_for(nc, B, max_blocks);
  if (L.fine)
    klaunch(k_dense_assemble<FineOp<double>>, dim3(g), dim3(kBlock), 0, s, L.fine_op(), nc, B, lam2, M);
  else
    klaunch(k_dense_assemble<CoarseOp<double>>, dim3(g), dim3(kBlock), 0, s, L.coarse_op(), nc, B, lam2, M);
  LCMG_LAUNCHED();
  launch_dense_inverse((int)nc, B, M, W, K, info, s);
}

int64_t dense_inverse_scratch(int64_t n) {
  return n * n + (n + kInvTile - 1) / kInvTile * (kInvTile * kInvTile);
}

void launch_dense_inverse(int n, int B, const double* M, double* W, double* K, int* info, cudaStream_t s) {
  LCMG_CUDA(cudaMemsetAsync(info, 0, sizeof(int) * B, s));
  const int nb = (n + kInvTile - 1) / kInvTile, threads = kInvTile * kInvTile;
  double* pan = W + (int64_t)B * n * n;
  const double* src = M;
  for (int k = 0; k < nb; ++k) {  // the last step writes K
    double* dst = (nb - 1 - k) % 2 == 0 ? K : W;
    klaunch(k_inverse_panel, dim3((unsigned)nb, (unsigned)B), dim3(2 * threads), 0, s, n, k, src, pan, info);
    LCMG_LAUNCHED();
    klaunch(k_inverse_update, dim3((unsigned)(nb * (nb + 1) / 2), (unsigned)B), dim3(threads), 0, s, n, nb, k,
            k == nb - 1 ? 1 : 0, src, dst, (const double*)pan);
    LCMG_LAUNCHED();
    src = dst;
  }
}

void launch_galerkin(const RapIn& in0, const RapIn& in1, int nvc, int nhc, double* out0, double* out1, bool terms,
                     int max_blocks, cudaStream_t s) {
  if (terms) {
    const int64_t work = (int64_t)nvc * nhc * kStencil;
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((work + kBlock - 1) / kBlock, max_blocks));
    klaunch(k_galerkin_terms, dim3(g), dim3(kBlock), 0, s, in0, nvc, nhc, out0);
    LCMG_LAUNCHED();
    klaunch(k_galerkin_terms, dim3(g), dim3(kBlock), 0, s, in1, nvc, nhc, out1);
    LCMG_LAUNCHED();
    return;
  }
  const unsigned tiles = (unsigned)((nvc + 31) / 32) * (unsigned)((nhc + kGalTJ - 1) / kGalTJ);
  klaunch(k_galerkin, dim3(tiles, 5, 2), dim3(kGalThreads), 0, s, in0, in1, nvc, nhc, out0, out1);
  LCMG_LAUNCHED();
}

template <class T, class TX>
int launch_update_xr(int64_t n, int B, const ColState& st, const T* p, const T* q, TX* x, T* r,
                     double* part, int max_blocks, cudaStream_t s) {
  const int g = grid_for(n, B, max_blocks);
  klaunch(k_update_xr<T, TX>, dim3(g), dim3(kBlock), 0, s, n, B, st, p, q, x, r, part);
  LCMG_LAUNCHED();
  return g;
}

template <class T>
int launch_update_xr_alpha(int64_t n, const ColState& st, int nb_pq, const double* pq_part, const T* p,
                           const T* q, T* x, T* r, double* part, int max_blocks, cudaStream_t s) {
  int threads;
  const dim3 g = fused_update_grid(n / Pack<T>::W, max_blocks, &threads);
  klaunch(k_update_xr_alpha<T>, g, dim3(threads), 0, s, n, st, nb_pq, pq_part, p, q, x, r, part);
  LCMG_LAUNCHED();
  return (int)g.x;
}

template <class T>
void launch_update_p_beta(int64_t n, const ColState& st, int nb_rr, const double* rr_part, int nb_rz,
                          const double* rz_part, int maxit, double rel_trigger, const T* z, T* p, int max_blocks,
                          cudaStream_t s) {
  int threads;
  const dim3 g = fused_update_grid(n / Pack<T>::W, max_blocks, &threads);
  klaunch(k_update_p_beta<T>, g, dim3(threads), 0, s, n, st, nb_rr, rr_part, nb_rz, rz_part, maxit, rel_trigger,
          z, p);
  LCMG_LAUNCHED();
}

template <class T>
void launch_update_p(int64_t n, int B, const ColState& st, const T* z, T* p, int max_blocks,
                     cudaStream_t s) {
  const int g = grid_for(n, B, max_blocks);
  klaunch(k_update_p<T>, dim3(g), dim3(kBlock), 0, s, n, B, st, z, p);
  LCMG_LAUNCHED();
}

template <class T>
void launch_copy_cols(int64_t n, int B, const int* flag, const T* src, T* dst, int max_blocks,
                      cudaStream_t s) {
  const int g = grid_for(n, B, max_blocks);
  klaunch(k_copy_cols<T>, dim3(g), dim3(kBlock), 0, s, n, B, flag, src, dst);
  LCMG_LAUNCHED();
}

#define LCMG_INST_T(T)                                                                          \
  template void launch_dinv<T>(const LevelView<T>&, int, const double*, int, double, T*, int,   \
                               cudaStream_t);                                                   \
  template void launch_smooth_zero<T>(const LevelView<T>&, int, const T*, const T*, const T*,   \
                                      T*, int, int, cudaStream_t);                              \
  template int launch_smooth<T>(const LevelView<T>&, int, const T*, const T*, const T*,         \
                                const T*, T*, const int*, double*, int, cudaStream_t);          \
  template void launch_residual<T>(const LevelView<T>&, int, const T*, const T*, const T*, T*,  \
                                   int, cudaStream_t);                                          \
  template void launch_restrict<T>(int, int, int, const T*, T*, int, cudaStream_t);             \
  template int launch_vdown<T>(const LevelView<T>&, int, const T*, const T*, const T*, T*, T*,    \
                               int, cudaStream_t);                                                \
  template int launch_vup<T>(const LevelView<T>&, int, const T*, const T*, const T*, const T*,    \
                             const T*, T*, double*, int, cudaStream_t);                           \
  template void launch_prolong_add<T>(int, int, int, const T*, T*, int, cudaStream_t);          \
  template void launch_coarse_solve<T>(int, int, const double*, const T*, T*, cudaStream_t);    \
  template void launch_update_p<T>(int64_t, int, const ColState&, const T*, T*, int,            \
                                   cudaStream_t);                                               \
  template void launch_copy_cols<T>(int64_t, int, const int*, const T*, T*, int, cudaStream_t);       \
  template void launch_update_p_beta<T>(int64_t, const ColState&, int, const double*, int, const double*, int, \
                                        double, const T*, T*, int, cudaStream_t);
LCMG_INST_T(float)
LCMG_INST_T(double)
#undef LCMG_INST_T
template int launch_update_xr<double, double>(int64_t, int, const ColState&, const double*,
                                              const double*, double*, double*, double*, int,
                                              cudaStream_t);
template int launch_update_xr<float, float>(int64_t, int, const ColState&, const float*,
                                            const float*, float*, float*, double*, int,
                                            cudaStream_t);
template int launch_update_xr_alpha<double>(int64_t, const ColState&, int, const double*, const double*,
                                            const double*, double*, double*, double*, int, cudaStream_t);
template int launch_update_xr_alpha<float>(int64_t, const ColState&, int, const double*, const float*, const float*,
                                           float*, float*, double*, int, cudaStream_t);

}  // namespace lcmg
