// Host rules of the single-lattice step launch: the kernel variant a context
// resolves to, and the warp-strip geometry of one wave.  Plain C++ without
// CUDA, so that the CPU tests compile and exercise it on its own.
#pragma once

#include <algorithm>

#include "lbm.h"

namespace lbm {

// Shortest band of the automatic geometry: each band reloads the two rows
// around it, so on lattices above 256^2 cells bands stay at least this tall
// even below one full wave.
constexpr int kMinBandRows = 4;

// Shortest automatic band of an nx x ny lattice.  A small lattice's step is
// one short wave (replayed from a graph in runs of steps), whose length is
// the rows each warp walks through, so there the shortest bands win
// (measured, improved scheme, one column per lane: 64^2 and 128^2 2.69 us
// per step with 1-row bands against 4.1-4.2 with 4-row ones; 256^2 3.83 us
// with 2-row bands against 4.36 with 1 or 4; from 512^2 on the 4-row rule
// is as fast or faster).
inline int min_band_rows(int nx, int ny) {
  const long long cells = (long long)nx * ny;
  return cells <= 128LL * 128 ? 1 : (cells <= 256LL * 256 ? 2 : kMinBandRows);
}

// Variant for an nx x ny lattice of `precision` on a GPU of `sm_count` SMs,
// given the requested one; `step` is false for the observe (moments)
// launches, which the staged kernel does not provide.
//  * STAGED only where the bulk copies' 16-byte rule holds (FP32, nx a
//    multiple of 4, at least 64);
//  * PAIR (two columns per lane) needs even nx; AUTO takes it except in FP64,
//    where its doubled register state spills, and on lattices too small to
//    give its 64-column strips (bands of kMinBandRows rows) a quarter of the
//    resident warps, where twice the strips beat the cheaper cells (measured:
//    256^2 1.33x faster with one column per lane, 512^2 equal, 768^2 and up
//    faster with two);
//  * otherwise REGISTER (one column per lane).
inline int resolve_variant(int requested, int precision, int nx, int ny, int sm_count,
                           bool step) {
  const long long pair_items =
      (long long)((nx + 63) / 64) * ((ny + kMinBandRows - 1) / kMinBandRows);
  const bool small = pair_items * 4 < (long long)sm_count * 20;
  const bool pair_ok = nx % 2 == 0;
  const bool staged_ok = step && precision == LBM_FP32 && nx >= 64 && nx % 4 == 0;
  if (requested == LBM_VARIANT_STAGED && staged_ok) return LBM_VARIANT_STAGED;
  if (((requested == LBM_VARIANT_AUTO && precision != LBM_FP64 && !small) ||
       requested == LBM_VARIANT_PAIR) &&
      pair_ok)
    return LBM_VARIANT_PAIR;
  return LBM_VARIANT_REGISTER;
}

struct StripGeometry {
  int n_strips;   // column strips: 32 columns wide, 64 for PAIR
  int band_rows;  // rows per band
  int n_bands;    // bands of rows
  int grid;       // CTAs of warps_per_cta warps, one warp per strip x band
};

// Strips of 32 columns (64 for PAIR) and as many row bands as fill the
// `resident_warps` warp slots once (one wave: every warp of a band runs at the
// same time as its neighbours), at least min_band_rows rows each; a positive
// band_rows_override fixes the band height instead.
inline StripGeometry strip_geometry(int nx, int ny, int variant, long long resident_warps,
                                    int warps_per_cta, int band_rows_override) {
  StripGeometry g;
  const int strip_w = variant == LBM_VARIANT_PAIR ? 64 : 32;
  g.n_strips = (nx + strip_w - 1) / strip_w;
  if (band_rows_override > 0) {
    g.band_rows = std::min(band_rows_override, ny);
  } else {
    long long n_bands = std::max<long long>(1, resident_warps / g.n_strips);
    n_bands = std::min<long long>(n_bands, std::max(1, ny / min_band_rows(nx, ny)));
    g.band_rows = int((ny + n_bands - 1) / n_bands);
  }
  g.n_bands = (ny + g.band_rows - 1) / g.band_rows;
  const long long warps = (long long)g.n_strips * g.n_bands;
  g.grid = int((warps + warps_per_cta - 1) / warps_per_cta);
  return g;
}

// Bands of the FP64 one-column kernel.  The FP64 pipe bounds it whatever the
// number of warps (one warp per scheduler already saturates it), so the launch
// takes as long as the SM with most work: with w = 1, 2 or 3 warps per
// scheduler, w (80 rows + 41 (rows + 2)) FP64 instructions, the second term
// being the density and psi of a band's rows and of the two around it.  Few
// tall bands win (512^2: 14 rows, 1 warp) until they no longer divide the
// lattice evenly (8192^2: 7 bands of 1171 rows, 3 warps).
inline StripGeometry fp64_geometry(int nx, int ny, int sm_count, int warps_per_cta) {
  StripGeometry g;
  g.n_strips = (nx + 31) / 32;
  double best = 0.0;
  for (int w = 1; w <= 3; ++w) {
    const long long bands = std::min<long long>(
        ny, std::max<long long>(1, (long long)sm_count * warps_per_cta * w / g.n_strips));
    const int rows = int((ny + bands - 1) / bands);
    const double t = w * (80.0 * rows + 41.0 * (rows + 2));
    if (w == 1 || t < best) {
      best = t;
      g.band_rows = rows;
    }
  }
  g.n_bands = (ny + g.band_rows - 1) / g.band_rows;
  g.grid = int(((long long)g.n_strips * g.n_bands + warps_per_cta - 1) / warps_per_cta);
  return g;
}

// ---------------------------------------------------------------------------
// two steps per launch (lbm_two_step.cuh)
// ---------------------------------------------------------------------------
constexpr int kTwoStepCols = 56;   // columns of a strip
constexpr int kTwoStepWarps = 12;  // resident warps per SM
constexpr int kTwoStepFewWarps = 8;  // of launches that have no use for more

// Whether steps of a whole nx x ny lattice may go two per launch: FP32, or
// 16-bit storage with even nx (its columns are copied in pairs), AUTO variant
// and band height (a requested kernel or height runs as requested), a lattice
// large enough to gain, 32-bit byte offsets within a plane, and a covolume for
// which every density inside the domain of psi (b rho / 4 < 1) has a normal
// reciprocal.  Not 1 or 3 columns: the one-by-one copies of a row then all read
// the same few addresses, which takes longer than the rest of the march (us per
// step, one step per launch / two: 1 x 32000 17.4 / 51.9, 3 x 10666 8.6 / 10.6, 3
// x 133333 60 / 76; 5 x 6400 6.9 / 6.0, 7 x 57142 28.5 / 25.8; even widths gain
// from 2 on).
constexpr long long kTwoStepMinCells = 176LL * 176;
constexpr long long kTwoStepMaxCells = 1LL << 30;
inline bool two_step_applies(int requested, int precision, int nx, int ny,
                             int band_rows_override, double b) {
  const long long cells = (long long)nx * ny;
  const bool dev = precision == LBM_BF16DEV || precision == LBM_FP16DEV;
  return requested == LBM_VARIANT_AUTO && band_rows_override == 0 &&
         (precision == LBM_FP32 || (dev && nx % 2 == 0)) && nx != 1 && nx != 3 &&
         cells >= kTwoStepMinCells &&
         cells <= kTwoStepMaxCells && b > 1e-12 && b < 1e12;
}

// Strips of 56 columns and the band height that ends first.  A band of n rows
// costs about n + 4 iterations; with 4, 8 or 12 warps per SM (1, 2 or 3 per
// scheduler; numbers between leave one scheduler with more than the others
// and end no earlier) an iteration takes 0.58, 0.89 and 1.285 us (improved
// scheme, the first two in the kernel for few CTAs), so short bands of many
// warps pay only while the rows dominate.  us per step with 4 / 8 / 12 warps,
// one kernel: 512^2 4.78 / 4.99 / 5.37, 768^2 7.30 / 6.79 / 7.30, 1024^2 11.1 /
// 9.87 / 10.5, 2048^2 38.9 / 31.3 / 30.5; now 512^2 4.32, 768^2 6.35, 1024^2 9.29,
// 2048^2 29.9.
inline StripGeometry two_step_geometry(int nx, int ny, int sm_count) {
  StripGeometry g;
  g.n_strips = (nx + kTwoStepCols - 1) / kTwoStepCols;
  const double cost[3] = {0.58, 0.89, 1.285};
  double best = 0.0;
  g.band_rows = ny;
  for (int k = 0; k < 3; ++k) {
    const long long resident = (long long)sm_count * kTwoStepWarps * (k + 1) / 3;
    const long long bands = std::min<long long>(std::max<long long>(1, resident / g.n_strips), ny);
    const int rows = int((ny + bands - 1) / bands);
    const double t = (rows + 4) * cost[k];
    if (k == 0 || t < best) {
      best = t;
      g.band_rows = rows;
    }
  }
  g.n_bands = (ny + g.band_rows - 1) / g.band_rows;
  g.grid = g.n_strips * g.n_bands;
  return g;
}

// ---------------------------------------------------------------------------
// several steps per launch on tiles (lbm_tile_steps.cuh)
// ---------------------------------------------------------------------------
constexpr int kTileMinSteps = 2, kTileMaxSteps = 4;  // steps per launch
constexpr int kTileMaxWarps = 24;                    // two rows each

struct TileGeometry {
  int n_cols;   // tiles side by side
  int rows;     // rows a tile owns; 0: the lattice does not take tiles
  int grid;     // tiles
  int threads;  // per CTA
  int steps;    // steps of a launch
};

// Tiles for a lattice that they cover in one wave, one CTA per SM: as many
// rows of tiles as there are SMs for, at most 48 lattice rows each with the
// halo of two cells per step.  Up to there tiles are the fastest at every size,
// and a second wave only ties with two-step launches.  (With fewer, taller tiles
// the kernel's first version took 18 % longer at 128^2.)  Fewer steps leave more
// columns and rows to a tile, so a lattice takes the most steps that fit, us per
// step with 4 / 3 / 2 and, last, on strips (one step per launch below 176^2, two
// from there): 64^2 1.06 / 1.17 / 1.42 / 2.57, 128^2 1.22 / 1.38 / 1.54 / 2.63,
// 200^2 1.68 / 1.72 / 1.93 / 2.54, 256^2 2.07 / 2.06 / 2.12 / 2.76, 300^2 - / 2.32 /
// 2.57 / 2.86, 360^2 - / - / 2.95 / 3.34.  (Five steps gain 3 % at 16^2 and 1 % at
// 64^2 and lose from 96^2 on.)  The same requirements on
// variant, storage, band height and covolume as two_step_applies.
inline TileGeometry tile_geometry(int requested, int precision, int nx, int ny,
                                  int band_rows_override, double b, int sm_count) {
  const TileGeometry none{0, 0, 0, 0, 0};
  if (requested != LBM_VARIANT_AUTO || band_rows_override != 0 || precision != LBM_FP32 ||
      !(b > 1e-12 && b < 1e12))
    return none;
  for (int steps = kTileMaxSteps; steps >= kTileMinSteps; --steps) {
    const int halo = 2 * steps, cols = (nx - 1) / (32 - 2 * halo) + 1;
    if (cols > sm_count) continue;
    const int tile_rows = std::min(ny, sm_count / cols), rows = (ny - 1) / tile_rows + 1;
    if (rows + 2 * halo > 2 * kTileMaxWarps) continue;
    return TileGeometry{cols, rows, cols * ((ny - 1) / rows + 1),
                        32 * ((rows + 2 * halo + 1) / 2), steps};
  }
  return none;
}

}  // namespace lbm
