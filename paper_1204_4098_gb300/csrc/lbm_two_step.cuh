// Two time steps in one pass over the lattice (FP32 and 16-bit storage).
//
// The one-step kernels move 72 B per cell update and run at 0.93 of the copy
// bandwidth on large lattices: they cannot get faster without moving less.
// Here a warp marches down a band of rows as they do, but carries every row
// through two steps before it is stored: the step-1 populations of the last
// three rows stay on chip (registers, and two rows of the warp's shared
// memory), so a launch reads and writes each population once per TWO steps
// (36 B per cell update).  Every per-cell expression is the one of the
// one-step kernels, so the populations are the same bits.
//
// Columns.  A row's step-2 result needs step-1 results one column further
// out for the pull and one more for psi, and those need the same again: a
// warp loads 64 columns (two per lane) and owns the inner 56.  Nothing is
// exchanged between warps, and the halo columns are ordinary columns of the
// march (the one-step kernel's extra halo loads, shuffles and psi evaluation,
// ~10 % of its instructions, have no counterpart); 8 of 64 columns are
// computed twice.  At the wrong side of the strip's edge, lanes compute
// values that nothing uses: of columns -4 .. 59 (0 .. 55 owned), step 1 needs
// psi of -3 .. 58 and step 2 of -1 .. 56, one column of each outermost lane
// (psi_row).  Rows likewise: a band of n rows pulls n + 6; the
// first iterations run only the part of the work that their rows are for (the
// whole work in all n + 7: 1024^2 10.9 us per step instead of 9.9).
//
// Balance.  With the traffic halved the kernel is bound by its instructions,
// first by the latency of dependent ones (three warps per scheduler).  Step 2
// therefore works one row behind, on the row that the previous iteration
// completed, so that the two steps of an iteration do not depend on each
// other and the loop has no branch the scheduler could not move them across.
// Divisions and roots take the bare hardware instructions; their operands are
// checked as part of the domain check (psi_normal), and a band in which a
// check fails is run again with the full forms (strip_run_two<kNormal =
// false>), which also report divergence.  One warp per CTA: strip, band and
// row are then block-uniform and their address arithmetic leaves the lanes
// (4096^2: 114.1 us per step against 116.8 with four warps per CTA).
//
// Measured on the way (improved scheme, 4096^2, us per step; one-step kernel
// 197.5): first version 141; unrolled by two 134; bare divisions and roots
// 128; no branches 123; step 2 one row behind 118; one warp per CTA 114; the
// arriving row read first and predicated copies 111.9 (150k MLUPS, DRAM at
// 0.78 of the measured copy bandwidth, FMA pipes 60 % busy, 12 warps per SM).
// 13 to 16 warps per SM (128 registers, spilling) 119-122; rows of step 1 kept
// in registers 141 (spills).  Small launches, whose SMs get 4 or 8 warps, are
// latency bound and take a kernel with 255 registers and more overlap
// (two_form): 512^2 4.65 -> 4.32, 1024^2 9.75 -> 9.29.
//
// 16-bit storage gains from the instructions that two separate steps repeat
// (the row copies, the halo's psi) and from the bare divisions: it was bound
// by issue, not by memory (BF16, us per step, one-step -> two-step: 4096^2 186 ->
// 129, 2048^2 51.1 -> 34.4, 1024^2 16.6 -> 10.7, 512^2 7.4 -> 5.1, 256^2 4.2 ->
// 3.4; FP16 the same).
#pragma once

#include "lbm_geometry.h"
#include "lbm_kernels.cuh"

namespace lbm {

constexpr int kTwoHalo = 4;              // columns loaded on each side of a strip
constexpr int kTwoCols = kTwoStepCols;   // columns a strip owns
static_assert(kTwoCols + 2 * kTwoHalo == 64, "a warp loads two columns per lane");
constexpr int kTwoStages = 3;                // rows in shared memory: one read, two in flight
constexpr int kTwoThreads = 32;              // one warp per CTA
// CTAs per SM: 12 (168 registers at most), or for launches that bring no more
// than 8 to an SM, 8 (255 registers)
constexpr int kTwoManyCtas = kTwoStepWarps, kTwoFewCtas = kTwoStepFewWarps;

// Shared memory of a warp, lane-major.  A fetched row: the 9 planes' pairs, for
// deviation storage also the density pair of the row after the pulled one (the
// two before it stay in registers).  q: step 2's last two pulled rows.
template <class S>
struct TwoRow {
  typename Vec2<typename S::T>::type d[kQ][32];
  float2 rr[S::kDev ? 32 : 1];
};
template <class S>
struct TwoSmem {
  TwoRow<S> row[kTwoStages];
  float2 q[2][kQ][32];
};

// psi of a row: the x neighbours only enter the force (Eq. 3) as their
// difference and sum, formed once per row.
struct PsiRow {
  F2 c, d, s;  // psi, psi(x + 1) - psi(x - 1), psi(x + 1) + psi(x - 1)
};

// Smallest of three with NaN kept (one instruction).
__device__ __forceinline__ float min3_nan(float a, float b, float c) {
  float r;
  asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// psi of a pair, and whether it holds as it stands: every operand of the
// reciprocals and the root (and of the reciprocals in collide, which take rho
// and psi^2) is normal and the density is inside the domain of psi.  The pair
// must be evaluated again with psi_of_rho and the full divisions where not.
constexpr float kNormalMin = 0x1p-100f;
__device__ __forceinline__ F2 psi_normal(F2 rho, const Phys<float>& P, bool& ok) {
  F2 eta, om, arg;
  psi_radicand<true>(rho, P, eta, om, arg);
  const float lo = min3_nan(min3_nan(rho.x(), om.x(), arg.x()), min3_nan(rho.y(), om.y(), arg.y()),
                            1.f);
  ok = lo >= kNormalMin && max_nan(arg.x(), arg.y()) <= 1e30f;
  return F2(mul_rn(arg.x(), rsqrt_normal(arg.x())), mul_rn(arg.y(), rsqrt_normal(arg.y())));
}

// Forms of the march, the order and the branches the compiler gets to schedule
// an iteration in; the values are the same.  kEarlyRow: the row that arrives is
// taken from shared memory before step 2's work, not after it; kStoreIf,
// kFetchIf: the stores and the row copies are predicated instead of branched
// around, so that step 2 and step 1 share a block of instructions.  More
// overlap takes registers, so what pays differs, us per step with neither / the
// form taken (as measured when the form was chosen): even nx, 12 CTAs per SM: 512^2 4.65 / 4.49, 1024^2 9.71 / 9.61,
// 4096^2 113.1 / 112.3, MRT 2048^2 32.6 / 31.6; 8 CTAs per SM: 512^2 4.62 / 4.27,
// 1024^2 9.72 / 9.38, BF16 1024^2 10.90 / 10.71; odd nx: 1023x1025 11.31 / 10.97
// with 8.  All three with 12 CTAs spill (4096^2 114.0).
enum TwoForm { kEarlyRow = 1, kStoreIf = 2, kFetchIf = 4 };
__host__ __device__ constexpr int two_form(bool dev, int scheme, bool odd, int ctas) {
  if (ctas == kTwoFewCtas)
    return dev ? kEarlyRow | kStoreIf | kFetchIf
               : (scheme == kMRT ? kEarlyRow | kFetchIf : kEarlyRow | kStoreIf);
  return odd ? kStoreIf : kEarlyRow | kFetchIf;
}

__device__ __forceinline__ void store_if(bool p, void* at, float v) {
  asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n @q st.global.f32 [%0], %1;\n}" ::"l"(at),
               "f"(v), "r"(unsigned(p)));
}
__device__ __forceinline__ void store_if(bool p, void* at, float2 v) {
  asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %3, 0;\n @q st.global.v2.f32 [%0], {%1, %2};\n}" ::"l"(at),
               "f"(v.x), "f"(v.y), "r"(unsigned(p)));
}
template <class V>
__device__ __forceinline__ void store_if(bool p, void* at, V v) {  // 32 bits
  static_assert(sizeof(V) == 4, "");
  unsigned u;
  __builtin_memcpy(&u, &v, 4);
  asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n @q st.global.b32 [%0], %1;\n}" ::"l"(at),
               "r"(u), "r"(unsigned(p)));
}
// (no bytes are read where `p` does not hold; the destination gets zeros)
template <int N>
__device__ __forceinline__ void cp_async_if(bool p, void* smem, const void* g) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(
                   unsigned(__cvta_generic_to_shared(smem))),
               "l"(g), "n"(N), "r"(p ? N : 0));
}

// Row layouts.
//  kFlatEven  even nx = pitch: a lane's two columns are one aligned pair;
//  kFlatOdd   odd nx = pitch: columns copied and stored one by one;
//  kAnyWidth  any nx, even pitch >= nx (the batch engine's rows): columns copied
//             one by one, stored as pairs (of an odd nx the last pair's second
//             column is nx, in the padding: it gets column 0's value);
//  kRing      even nx <= 64 = pitch: the warp holds whole rows, its shuffles
//             wrap around them, and no column is computed twice.  Up to 32
//             columns each half-warp takes a band of its own.
enum TwoLayout { kFlatEven, kFlatOdd, kAnyWidth, kRing };

// Two steps of one strip x band item.  kNormal: returns false as soon as a
// value fails psi_normal's check; the item then has to be run again with
// kNormal = false.  Deviation storage (kFlatEven only) rounds the populations
// between the two steps to what the one-step kernel would store and read
// back, in registers.
template <class S, int SCHEME, int LAYOUT, bool kNormal, int FORM>
__device__ __forceinline__ bool strip_run_two(const StripArgs<S>& A, int strip, int band, int lane,
                                              TwoSmem<S>& sm) {
  using T = typename S::T;
  using V = typename Vec2<T>::type;
  static_assert(std::is_same<typename S::C, float>::value && (!S::kDev || LAYOUT == kFlatEven),
                "FP32 arithmetic; 16-bit columns are copied in aligned pairs");
  constexpr unsigned kBytes = sizeof(T);
  TwoRow<S>* const st = sm.row;
  constexpr bool kNeedPsi = SCHEME != kNoForce;
  const unsigned FULL = 0xffffffffu;
  const int nx = A.nx, ny = A.ny;
  const unsigned pitch = LAYOUT == kAnyWidth ? unsigned(A.pitch) : unsigned(nx);
  int y0, y1, n_rows;  // rows of this lane's band; pulled rows of the march
  int xo, ca, cb;      // left column of this lane; its loaded columns (wrapped)
  int from_l = 0, from_r = 0;  // kRing: lanes holding the columns beside
  // whether columns of the lane are collided in step 1 / 2, and whether psi of
  // its left (_l) and right (_r) column is used there
  bool valid1, valid2;
  bool psi1_l, psi1_r, psi2_l, psi2_r;
  bool store_a, store_b;
  if constexpr (LAYOUT == kRing) {
    const int width = nx / 2;                   // lanes of a row
    const int half = nx <= 32 ? lane >> 4 : 0;  // which of the warp's bands
    const int base = half << 4, l = lane - base;
    const bool in_row = l < width;
    const int b = nx <= 32 ? 2 * band + half : band;
    y0 = A.y_begin + b * A.band_rows;
    y1 = min(y0 + A.band_rows, A.y_end);
    n_rows = A.band_rows + 6;
    xo = ca = in_row ? 2 * l : 0;
    cb = ca + 1;
    from_l = l == 0 ? base + width - 1 : lane - 1;
    from_r = l == width - 1 ? base : lane + 1;
    valid1 = valid2 = in_row;
    psi1_l = psi1_r = psi2_l = psi2_r = in_row;
    store_a = store_b = in_row;
    if (y0 >= y1) {  // a half-warp without a band: marches along, stores nothing
      y0 = A.y_begin;
      y1 = y0;
    }
  } else {
    y0 = A.y_begin + band * A.band_rows;
    y1 = min(y0 + A.band_rows, A.y_end);
    n_rows = y1 - y0 + 6;  // pulled rows y0 - 3 .. y1 + 2
    xo = strip * kTwoCols - kTwoHalo + 2 * lane;
    // (even nx: the wrapped pair stays adjacent and aligned)
    ca = ((xo % nx) + nx) % nx;
    cb = ca + 1 == nx ? 0 : ca + 1;
    valid1 = lane >= 1 && lane < 31;
    valid2 = lane >= 2 && lane < 30;
    psi1_l = lane != 0;
    psi1_r = lane != 31;
    psi2_l = lane >= 2 && lane < 31;
    psi2_r = lane >= 1 && lane < 30;
    store_a = valid2 && xo < nx;
    store_b = valid2 && xo + 1 < nx;
  }
  bool bad = false;  // a density outside the domain of psi
  bool fine = true;  // kNormal: every check held so far

  // Rows are fetched in sequence.  om, oz, op: byte offsets of the lane's
  // pair in the rows before, at and after the pulled row (a plane has at most
  // 2^30 elements, so 32 bits hold them).
  auto wrap_row = [ny](int y) { return ((y % ny) + ny) % ny; };
  int nrow = wrap_row(y0 - 2);  // the row after the next pulled one
  unsigned om = (unsigned(wrap_row(y0 - 4)) * pitch + unsigned(ca)) * kBytes;
  unsigned oz = (unsigned(wrap_row(y0 - 3)) * pitch + unsigned(ca)) * kBytes;
  auto copy = [](bool p, void* to, const char* from, auto bytes) {
    if constexpr ((FORM & kFetchIf) != 0) cp_async_if<bytes()>(p, to, from);
    else cp_async<bytes()>(to, from);
  };
  auto fetch = [&](TwoRow<S>& R, bool p) {
    const unsigned op = (unsigned(nrow) * pitch + unsigned(ca)) * kBytes;
    auto source = [&](int a) {
      const unsigned o = ey_of(a) == 0 ? oz : (ey_of(a) == 1 ? om : op);
      return reinterpret_cast<const char*>(A.src + a * A.plane) + o;
    };
#pragma unroll
    for (int a = 0; a < kQ; ++a) {
      if constexpr (LAYOUT == kFlatOdd || LAYOUT == kAnyWidth) {
        copy(p, &R.d[a][lane].x, source(a), std::integral_constant<int, 4>());
        copy(p, &R.d[a][lane].y, source(a) + 4 * (cb - ca), std::integral_constant<int, 4>());
      } else {
        copy(p, &R.d[a][lane], source(a), std::integral_constant<int, int(sizeof(V))>());
      }
    }
    if constexpr (S::kDev)
      copy(p, &R.rr[lane], reinterpret_cast<const char*>(A.rho_src) + 2u * op,
           std::integral_constant<int, 8>());
    cp_async_commit();
    om = oz;
    oz = op;
    nrow = nrow + 1 == ny ? 0 : nrow + 1;
  };
  // pull in x of plane a's values v at the lane's two columns
  auto left = [&](float v) {
    return LAYOUT == kRing ? __shfl_sync(FULL, v, from_l) : __shfl_up_sync(FULL, v, 1);
  };
  auto right = [&](float v) {
    return LAYOUT == kRing ? __shfl_sync(FULL, v, from_r) : __shfl_down_sync(FULL, v, 1);
  };
  auto pull_x = [&](int a, F2 v) {
    const int ex = ex_of(a);
    if (ex == 0) return v;
    if (ex == 1) return F2(left(v.y()), v.x());
    return F2(v.y(), right(v.x()));
  };
  // deviation storage: density pairs of the two rows before the next R.rr
  F2 ring0 = F2(0.f), ring1 = F2(0.f);
  if constexpr (S::kDev) {
    const char* const r = reinterpret_cast<const char*>(A.rho_src);
    ring0 = F2(__ldg(reinterpret_cast<const float2*>(r + 2u * om)));
    ring1 = F2(__ldg(reinterpret_cast<const float2*>(r + 2u * oz)));
  }
  auto assemble = [&](const TwoRow<S>& R, F2 (&P)[kQ]) {
    if constexpr (S::kDev) {
      const F2 rr[3] = {ring0, ring1, F2(R.rr[lane])};  // source rows r - 1, r, r + 1
#pragma unroll
      for (int a = 0; a < kQ; ++a)
        P[a] = pull_x(a, S::decode2(mul_rn(F2(w_of<float>(a)), rr[1 - ey_of(a)]), R.d[a][lane]));
      ring0 = rr[1];
      ring1 = rr[2];
    } else {
#pragma unroll
      for (int a = 0; a < kQ; ++a) P[a] = pull_x(a, F2(R.d[a][lane]));
    }
  };
  // deviation storage: the 16-bit deviations of post-collision populations f
  // of density r, and the density that absorbs their rounding
  auto encode = [&](const F2 (&f)[kQ], F2 r, V (&v)[kQ]) {
    F2 res = r;
    if constexpr (S::kDev) {
#pragma unroll
      for (int a = 0; a < kQ; ++a) {
        const F2 d = fma_rn(F2(-w_of<float>(a)), r, f[a]);
        v[a] = S::from_c2(d.x(), d.y());
        res = S::sub_from(res, v[a]);
      }
    }
    return res;
  };
  auto rho_of = [](const F2 (&P)[kQ]) {
    F2 r = P[0];
#pragma unroll
    for (int a = 1; a < kQ; ++a) r = add_rn(r, P[a]);
    return r;
  };
  // psi of a row; use_l, use_r: whether that of the lane's left and right column
  // is used (`some`: either).  Where one is, kNormal checks both: the other, of
  // a density that lacks its share from beyond the strip, can only have the item
  // run again, and masking it costs more (us per step, this / masked: 1024^2 9.29
  // / 9.73, 4096^2 111.9 / 113.9, BF16 129.4 / 133.3).  The full form reports
  // divergence, of the columns in use only.
  auto psi_row = [&](F2 r, bool some, bool use_l, bool use_r) {
    PsiRow p;
    if constexpr (kNormal) {
      bool ok;
      p.c = psi_normal(r, A.P, ok);
      // (the same value; us per step, && / &: BF16 4096^2 131.1 / 129.4, 1501 x 997
      // 13.85 / 13.99, 48 odd slabs 39.48 / 39.62)
      if constexpr (LAYOUT == kFlatOdd || LAYOUT == kAnyWidth) fine = fine && (ok || !some);
      else fine = fine & (ok | !some);
    } else {
      bool fl = false, fr = false;
      p.c = F2(psi_of_rho(r.x(), A.P, fl), psi_of_rho(r.y(), A.P, fr));
      bad |= (fl && use_l) || (fr && use_r);
    }
    const F2 W = F2(left(p.c.y()), p.c.x());
    const F2 E = F2(p.c.y(), right(p.c.x()));
    p.d = sub_rn(E, W);
    p.s = add_rn(E, W);
    return p;
  };
  // without psi only the reciprocal of the density has to be normal
  auto rho_check = [&](F2 r, bool valid) {
    if constexpr (kNormal && !kNeedPsi)
      fine = fine && ((min3_nan(r.x(), r.y(), 1.f) >= kNormalMin &&
                       max_nan(r.x(), r.y()) <= 1.f / kNormalMin) || !valid);
  };
  auto force = [&](const PsiRow& m, const PsiRow& z, const PsiRow& p, F2& Fx, F2& Fy) {
    const F2 third = F2(1.f / 3.f), twelfth = F2(1.f / 12.f);
    const F2 sx = fma_rn(third, z.d, mul_rn(twelfth, add_rn(p.d, m.d)));
    const F2 sy = fma_rn(third, sub_rn(p.c, m.c), mul_rn(twelfth, sub_rn(p.s, m.s)));
    const F2 gpsi = mul_rn(F2(A.P.minus_G), z.c);
    Fx = mul_rn(gpsi, sx);
    Fy = mul_rn(gpsi, sy);
  };
  const F2 zero = F2(0.f);
  const PsiRow none{zero, zero, zero};

  constexpr int D = kTwoStages - 1;  // rows in flight
#pragma unroll
  for (int k = 0; k < D; ++k) fetch(st[k], true);  // n_rows >= 7

  // In iteration k the pulled row r = y0 - 3 + k arrives.  Step 1 has its
  // pulled row r - 1 (P0, rho0) and the psi of rows r - 2 (m1) and r - 1 (z1).
  F2 P0[kQ], rho0 = zero;
  PsiRow m1 = none, z1 = none;
  // Step-1 populations already pulled in x: e_y = 0 of row r - 2 (d0: a = 0,
  // 1, 3), e_y = 1 of rows r - 2 and r - 3 (dn, dnn: a = 2, 5, 6).
  F2 d0[3], dn[3], dnn[3];
  // Step 2, one row behind: densities of its pulled rows r - 4 (qrhoA) and
  // r - 3 (qrhoB), psi of rows r - 5 (m2) and r - 4 (z2).
  F2 qrhoA = zero, qrhoB = zero;
  PsiRow m2 = none, z2 = none;
#pragma unroll
  for (int a = 0; a < kQ; ++a) P0[a] = zero;
#pragma unroll
  for (int k = 0; k < 3; ++k) d0[k] = dn[k] = dnn[k] = zero;

  unsigned out = (unsigned(y0) * pitch + unsigned(xo)) * kBytes;
  int sg = 0, sf = D % kTwoStages;  // stages of row r and of row r + D
  bool go = true;
  // Step 2 of iteration k: psi of its pulled row r - 3 ...
  PsiRow p2 = none;
  auto step2_psi = [&]() {
    if constexpr (kNeedPsi) p2 = psi_row(qrhoB, LAYOUT == kRing ? valid2 : valid1, psi2_l, psi2_r);
    else rho_check(qrhoB, valid2);
  };
  // ... and its output row r - 4
  auto step2_row = [&](int k) {
    F2 Gx = zero, Gy = zero, Q0[kQ];
    if constexpr (kNeedPsi) force(m2, z2, p2, Gx, Gy);
#pragma unroll
    for (int a = 0; a < kQ; ++a) Q0[a] = F2(sm.q[k & 1][a][lane]);
    collide<SCHEME, kNormal>(Q0, qrhoA, Gx, Gy, z2.c, A.P);
    const bool store = store_a && (LAYOUT != kRing || k - 7 < y1 - y0);
    auto put = [&](auto to) {
      V v[kQ];
      const F2 res = encode(Q0, qrhoA, v);
      if constexpr (S::kDev) to(store, reinterpret_cast<char*>(A.rho_dst) + 2u * out, res.v);
#pragma unroll
      for (int a = 0; a < kQ; ++a) {
        char* const at = reinterpret_cast<char*>(A.dst + a * A.plane) + out;
        if constexpr (S::kDev) {
          to(store, at, v[a]);
        } else if constexpr (LAYOUT == kFlatOdd) {
          to(store, at, Q0[a].x());
          to(store && store_b, at + kBytes, Q0[a].y());
        } else {
          to(store, at, Q0[a].v);
        }
      }
    };
    if constexpr ((FORM & kStoreIf) != 0) {
      put([](bool p, void* at, auto v) { store_if(p, at, v); });
    } else if (store) {
      put([](bool p, void* at, auto v) {
        if (p) *reinterpret_cast<decltype(v)*>(at) = v;
      });
    }
    out += pitch * kBytes;
  };
  // Step 1 of iteration k: row r arrives ...
  F2 P1[kQ];
  auto arrive = [&](int k) {
    cp_async_wait<D - 1>();
    assemble(st[sg], P1);
    sg = sg == kTwoStages - 1 ? 0 : sg + 1;
    // (into the stage read in iteration k - 1; an empty group keeps the count)
    if constexpr ((FORM & kFetchIf) != 0) fetch(st[sf], k + D < n_rows);
    else if (k + D < n_rows) fetch(st[sf], true);
    else cp_async_commit();
    sf = sf == kTwoStages - 1 ? 0 : sf + 1;
  };
  // ... and (`full`) row r - 1 is advanced, which completes step 2's pulled row
  // r - 2.
  auto step1 = [&](int k, bool full) {
    const F2 rho1 = rho_of(P1);
    PsiRow p1 = none;
    if constexpr (kNeedPsi) p1 = psi_row(rho1, LAYOUT != kRing || valid1, psi1_l, psi1_r);
    else rho_check(rho1, valid1);
    m2 = z2;
    z2 = p2;
    if (full) {
      F2 Fx = zero, Fy = zero;
      if constexpr (kNeedPsi) force(m1, z1, p1, Fx, Fy);
      collide<SCHEME, kNormal>(P0, rho0, Fx, Fy, z1.c, A.P);  // row r - 1
      if constexpr (S::kDev) {
        V v[kQ];
        const F2 res = encode(P0, rho0, v);
#pragma unroll
        for (int a = 0; a < kQ; ++a)
          P0[a] = S::decode2(mul_rn(F2(w_of<float>(a)), res), v[a]);
      }
      // step 2's pulled row r - 2 is complete
      F2 Q1[kQ];
      Q1[0] = d0[0];
      Q1[1] = d0[1];
      Q1[3] = d0[2];
      Q1[2] = dnn[0];
      Q1[5] = dnn[1];
      Q1[6] = dnn[2];
      Q1[4] = P0[4];
      Q1[7] = pull_x(7, P0[7]);
      Q1[8] = pull_x(8, P0[8]);
#pragma unroll
      for (int j = 0; j < 3; ++j) dnn[j] = dn[j];
      dn[0] = P0[2];
      dn[1] = pull_x(5, P0[5]);
      dn[2] = pull_x(6, P0[6]);
      d0[0] = P0[0];
      d0[1] = pull_x(1, P0[1]);
      d0[2] = pull_x(3, P0[3]);
      qrhoA = qrhoB;
      qrhoB = rho_of(Q1);
#pragma unroll
      for (int a = 0; a < kQ; ++a) sm.q[k & 1][a][lane] = Q1[a].v;
    }
    m1 = z1;
    z1 = p1;
    rho0 = rho1;
#pragma unroll
    for (int a = 0; a < kQ; ++a) P0[a] = P1[a];
    if constexpr (kNormal) go = __all_sync(FULL, fine);
  };
  // The first iterations do what their rows are for: psi of step 1 from row
  // y0 - 3, its collision from row y0 - 2, psi of step 2 from row y0 - 1.
#pragma unroll 1
  for (int k = 0; k < 7 && go; ++k) {
    arrive(k);
    if (k >= 5) step2_psi();
    step1(k, k >= 2);
  }
#pragma unroll 2
  for (int k = 7; k < n_rows && go; ++k) {
    if constexpr ((FORM & kEarlyRow) != 0) arrive(k);
    step2_psi();
    step2_row(k);
    if constexpr ((FORM & kEarlyRow) == 0) arrive(k);
    step1(k, true);
  }
  if (go) {
    step2_psi();
    step2_row(n_rows);
    if constexpr (kNormal) go = __all_sync(FULL, fine);
  }
  cp_async_wait<0>();
  if constexpr (!kNormal)
    if (__any_sync(FULL, bad) && lane == 0) atomicOr(A.status, kStatusDiverged);
  return go;
}

// The item again with the full divisions and domain checks (rare).
template <class S, int SCHEME, int LAYOUT>
__device__ __noinline__ void strip_run_two_general(const StripArgs<S>& A, int strip, int band,
                                                   int lane, TwoSmem<S>& sm) {
  strip_run_two<S, SCHEME, LAYOUT, false, 0>(A, strip, band, lane, sm);
}

template <class S, int SCHEME, int LAYOUT, int CTAS>
__global__ void __launch_bounds__(kTwoThreads, CTAS)
two_step_kernel(const __grid_constant__ StripArgs<S> A) {
  __shared__ TwoSmem<S> sm;
  constexpr int kForm = two_form(S::kDev, SCHEME, LAYOUT == kFlatOdd, CTAS);
  const int lane = threadIdx.x;
  const int strip = blockIdx.x % A.n_strips;  // strips of kTwoCols columns
  const int band = blockIdx.x / A.n_strips;
  if (!strip_run_two<S, SCHEME, LAYOUT, true, kForm>(A, strip, band, lane, sm))
    strip_run_two_general<S, SCHEME, LAYOUT>(A, strip, band, lane, sm);
}

}  // namespace lbm
