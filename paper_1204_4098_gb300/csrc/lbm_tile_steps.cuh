// Two to four time steps per launch for small lattices (FP32 storage).
//
// A lattice of up to ~370^2 cells is spread thinly over the GPU: its step is
// a chain of latencies (launch, load, one or two rows of arithmetic, store)
// that leaves nearly every issue slot empty, and no band height shortens it.
// Here a CTA takes a tile of a few rows and 16 columns together with the 8
// cells around it that four steps reach (two per step: the pull and the psi
// stencil), and runs the steps in shared memory between one load and one
// store.  Neighbouring CTAs compute the overlap again -- about twice the work
// of the lattice -- on SMs that would otherwise wait; nothing is exchanged
// between them.  A lattice too large for tiles of four steps takes three or
// two, with 20 or 24 columns (tile_geometry).
//
// A warp owns two rows of the tile, a lane one column: every population pulled
// is one conflict-free shared load, the two rows are one packed pair of the
// two-cell arithmetic, and the populations stay in registers from the pull to
// the collision, so that one buffer serves all steps: all pulls of a step
// come before the barrier that publishes psi, all writes after it.  The cells
// that a step can still compute shrink by two on every side; warps whose rows
// are outside only pass the barriers.  Every per-cell expression is the one of
// the one-step kernels, so the populations are the same bits.  Divisions and
// range checks as in lbm_two_step.cuh; a tile in which a check fails is run
// again with the full forms.
//
// Measured, us per step in step graphs (improved scheme), best other kernel ->
// this: 32^2 2.54 -> 1.03, 64^2 2.57 -> 1.06, 128^2 2.63 -> 1.22, 200^2 2.54 ->
// 1.68, 256^2 2.76 -> 2.07 with four steps, 300^2 2.86 -> 2.32 with three, 360^2
// 3.34 -> 2.95 with two.  A launch takes about 1.8 us + 0.24 us and 0.03 us per
// active row for every step + 0.03 us per row loaded: at 64^2 a third of its 4.3
// us is the launch itself, the rest mostly one warp's serial row of arithmetic.
// Tried without gain: one row per warp, programmatic dependent launch (64^2:
// 1.34), five steps (64^2 1.09, 96^2 1.10 -> 1.19).
#pragma once

#include "lbm_geometry.h"
#include "lbm_two_step.cuh"

namespace lbm {

// (kTileMaxWarps: lbm_geometry.h)
constexpr int kTilePlanes = kQ + 1;  // populations and psi
// floats between the planes in shared memory: those of the tallest tile, so
// that every address of a cell is one of a few registers plus a constant (64^2
// 1.10 -> 1.07 us per step, 200^2 1.71 -> 1.68, MRT 1.87 -> 1.80, against planes
// of H rows)
constexpr int kTilePlane = 2 * 32 * kTileMaxWarps;

// psi of a pair whose elements may be out of use (kNormal: ok says whether
// the used ones hold, see psi_normal).
__device__ __forceinline__ F2 psi_normal_masked(F2 rho, const Phys<float>& P, bool use_x,
                                                bool use_y, bool& ok) {
  F2 eta, om, arg;
  psi_radicand<true>(rho, P, eta, om, arg);
  const bool okx = min3_nan(rho.x(), om.x(), arg.x()) >= kNormalMin && arg.x() <= 1e30f;
  const bool oky = min3_nan(rho.y(), om.y(), arg.y()) >= kNormalMin && arg.y() <= 1e30f;
  ok = (okx || !use_x) && (oky || !use_y);
  return F2(mul_rn(arg.x(), rsqrt_normal(arg.x())), mul_rn(arg.y(), rsqrt_normal(arg.y())));
}

// The tile whose first owned cell is (x0, y0), `rows` owned rows; f: shared
// memory, kQ planes of populations and one of psi of H x 32 floats each,
// kTilePlane apart, H = 2 warps >= rows + 2 halo; 1 <= steps <= halo / 2.
// Returns (to every thread of the CTA) whether every check held.
template <int SCHEME, bool kNormal>
__device__ __forceinline__ bool run_tile(const StripArgs<StoreF32>& A, int steps, int halo,
                                         int x0, int y0, int rows, float* f) {
  constexpr bool kNeedPsi = SCHEME != kNoForce;
  const unsigned FULL = 0xffffffffu;
  const int nx = A.nx, ny = A.ny;
  const int x = threadIdx.x & 31, r = 2 * (threadIdx.x >> 5);  // this lane's column, first row
  const int H = 2 * (blockDim.x >> 5);
  constexpr int plane = kTilePlane;
  float* const psi = f + kQ * plane;
  // load: rows y0 - halo .. , the 32 columns from x0 - halo, wrapped
  {
    int c = (x0 - halo + x) % nx;
    c = c < 0 ? c + nx : c;
    int ya = (y0 - halo + r) % ny;
    ya = ya < 0 ? ya + ny : ya;
    const int yb = ya + 1 == ny ? 0 : ya + 1;
#pragma unroll
    for (int a = 0; a < kQ; ++a) {
      const float* const src = A.src + a * A.plane + c;
      cp_async<4>(&f[a * plane + r * 32 + x], src + size_t(ya) * nx);
      cp_async<4>(&f[a * plane + (r + 1) * 32 + x], src + size_t(yb) * nx);
    }
    cp_async_commit();
    cp_async_wait<0>();
  }
  __syncthreads();
  // offsets of the rows before, at and after (clamped: the values are unused)
  const int rm = max(r - 1, 0) * 32, rz = r * 32, rp = (r + 1) * 32, rq = min(r + 2, H - 1) * 32;
  const int xl = max(x - 1, 0), xr = min(x + 1, 31);
  bool bad = false, fine = true;
#pragma unroll 1
  for (int s = 1; s <= steps; ++s) {
    // pulled populations and psi: rows 2 s - 1 .. H - 2 s, columns likewise
    const bool active = r >= 2 * s - 2 && r <= H - 2 * s;  // warp-uniform
    const bool use_x = x >= 2 * s - 1 && x <= 32 - 2 * s;
    const bool use_a = use_x && r >= 2 * s - 1, use_b = use_x && r + 1 <= H - 2 * s;
    F2 P[kQ], rho = F2(0.f), c = F2(0.f);
    if (active) {
#pragma unroll
      for (int a = 0; a < kQ; ++a) {
        const float* const p = f + a * plane + (ex_of(a) == 0 ? x : (ex_of(a) == 1 ? xl : xr));
        P[a] = ey_of(a) == 0 ? F2(p[rz], p[rp]) : (ey_of(a) == 1 ? F2(p[rm], p[rz])
                                                                 : F2(p[rp], p[rq]));
      }
      rho = P[0];
#pragma unroll
      for (int a = 1; a < kQ; ++a) rho = add_rn(rho, P[a]);
      if constexpr (kNeedPsi) {
        if constexpr (kNormal) {
          bool ok;
          c = psi_normal_masked(rho, A.P, use_a, use_b, ok);
          fine = fine && ok;
        } else {
          bool fa = false, fb = false;
          c = F2(psi_of_rho(rho.x(), A.P, fa), psi_of_rho(rho.y(), A.P, fb));
          bad |= (fa && use_a) || (fb && use_b);
        }
        psi[rz + x] = c.x();
        psi[rp + x] = c.y();
      } else if constexpr (kNormal) {
        const bool oka = rho.x() >= kNormalMin && rho.x() <= 1.f / kNormalMin;
        const bool okb = rho.y() >= kNormalMin && rho.y() <= 1.f / kNormalMin;
        fine = fine && (oka || !use_a) && (okb || !use_b);
      }
    }
    __syncthreads();
    // collision: rows 2 s .. H - 1 - 2 s
    if (r >= 2 * s && r <= H - 2 - 2 * s) {
      F2 Fx = F2(0.f), Fy = F2(0.f);
      if constexpr (kNeedPsi) {
        // psi of the own rows (r, r + 1) by shuffle, of rows r - 1 and r + 2
        // from shared memory; differences and sums of the x neighbours per row
        const F2 W = F2(__shfl_up_sync(FULL, c.x(), 1), __shfl_up_sync(FULL, c.y(), 1));
        const F2 E = F2(__shfl_down_sync(FULL, c.x(), 1), __shfl_down_sync(FULL, c.y(), 1));
        const F2 Wo = F2(psi[rm + xl], psi[rq + xl]), Eo = F2(psi[rm + xr], psi[rq + xr]);
        const F2 co = F2(psi[rm + x], psi[rq + x]);
        const F2 d = sub_rn(E, W), u = add_rn(E, W), dx = sub_rn(Eo, Wo), ux = add_rn(Eo, Wo);
        const F2 third = F2(1.f / 3.f), twelfth = F2(1.f / 12.f);
        // (row before, row after) of each: before = (r - 1, r), after = (r + 1, r + 2)
        const F2 sx = fma_rn(third, d, mul_rn(twelfth, add_rn(F2(d.y(), dx.y()), F2(dx.x(), d.x()))));
        const F2 sy =
            fma_rn(third, sub_rn(F2(c.y(), co.y()), F2(co.x(), c.x())),
                   mul_rn(twelfth, sub_rn(F2(u.y(), ux.y()), F2(ux.x(), u.x()))));
        const F2 gpsi = mul_rn(F2(A.P.minus_G), c);
        Fx = mul_rn(gpsi, sx);
        Fy = mul_rn(gpsi, sy);
      }
      collide<SCHEME, kNormal>(P, rho, Fx, Fy, c, A.P);
      if (s < steps) {
#pragma unroll
        for (int a = 0; a < kQ; ++a) {
          f[a * plane + rz + x] = P[a].x();
          f[a * plane + rp + x] = P[a].y();
        }
      } else {
        const int xg = x0 - halo + x, ya = y0 - halo + r;
        // (after fewer than halo / 2 steps the halo holds results too: the
        // owned cells only)
        const bool own = x >= halo && x < 32 - halo && xg < nx && r >= halo;
        const bool sa = own && r < halo + rows && ya < ny;
        const bool sb = own && r + 1 < halo + rows && ya + 1 < ny;
        float* const dst = A.dst + size_t(ya) * nx + xg;
#pragma unroll
        for (int a = 0; a < kQ; ++a) {
          if (sa) dst[a * A.plane] = P[a].x();
          if (sb) dst[a * A.plane + nx] = P[a].y();
        }
      }
    }
    if (s < steps) __syncthreads();
  }
  if constexpr (!kNormal) {
    if (bad) atomicOr(A.status, kStatusDiverged);
    return true;
  }
  return !__syncthreads_or(!fine);
}

template <int SCHEME>
__device__ __noinline__ void run_tile_general(const StripArgs<StoreF32>& A, int steps, int halo,
                                              int x0, int y0, int rows, float* f) {
  run_tile<SCHEME, false>(A, steps, halo, x0, y0, rows, f);
}

// CTA b: tile (b % A.n_strips, b / A.n_strips) of A.band_rows rows.
template <int SCHEME>
__global__ void __launch_bounds__(32 * kTileMaxWarps, 1)
tile_steps_kernel(const __grid_constant__ StripArgs<StoreF32> A, int steps, int halo) {
  extern __shared__ __align__(16) float tile[];
  const int x0 = int(blockIdx.x % A.n_strips) * (32 - 2 * halo);
  const int y0 = int(blockIdx.x / A.n_strips) * A.band_rows;
  if (!run_tile<SCHEME, true>(A, steps, halo, x0, y0, A.band_rows, tile))
    run_tile_general<SCHEME>(A, steps, halo, x0, y0, A.band_rows, tile);
}

}  // namespace lbm
