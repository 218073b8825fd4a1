// Fused ENO-AO sweep kernel: one launch performs, for one axis and one
// Runge-Kutta stage, every step of the spatial operator of Shen's ENO-AO
// scheme (arXiv 2108.12742) and, on the last axis, the Runge-Kutta combine.
//
// Per tile (TA lines x TS cells along the swept axis, plus a halo of G cells
// on each side, G = 4 for ENO-AO5 and 5 for ENO-AO7):
//   phase 1  per pair of neighbouring cells: state difference dU (FP64),
//            flux difference dF in difference form, Lax-Friedrichs split
//            differences df+- = (dF +- alpha dU)/2 (Sec. 2, Eq. LF_Flux_Split);
//            per cell: Roe-average ingredients (sqrt rho, velocity, H).
//   phase 2a per face: one bound per field and sign shows most faces to take
//            the top candidate everywhere and gives them their correction;
//            the others go to the tile's face list (prove_top).
//   phase 2  per listed face x_{j+1/2}: Roe average and eigenvectors (Sec. 4),
//            projection of the window differences onto each characteristic
//            field, indicators IS = MIN(delta_L, delta_R) as undivided
//            differences (Eq. New_Smoothness_Indicator, Tables 4-5), stencil
//            choice by the principle of Sec. 3.2 (ties to the higher
//            priority as in Appendix A), the chosen Table-1 value written as
//            f_j + sum_i b_i (f_{i+1} - f_i), the mirrored choice for f^-, and
//            the back-projection C_{j+1/2} = R (corr^+ + corr^-).
//   phase 3  per cell: L(u)_j = -(df+_{j-1} + df-_j + C_{j+1/2} - C_{j-1/2})/dx,
//            which equals -(F_{j+1/2} - F_{j-1/2})/dx of Eq. (1DWENOFD) because
//            F_{j+1/2} = f+_j + f-_{j+1} + C_{j+1/2}; then either store L(u)
//            for the next axis or add the earlier axes and apply the
//            third-order TVD Runge-Kutta combine in FP64, checking the new
//            state and accumulating the next step's alpha.
//
// Writing every quantity as a difference keeps FP32 rounding relative to the
// local variation |df| instead of |f|; the state and the combine stay FP64.
#pragma once

#include <cuda_runtime.h>

#include <cfloat>
#include <cstdint>

#include "enoao_internal.h"
#include "state_speed.cuh"
#include "tma.cuh"

namespace enoao {

template <int ORDER>
struct Geo {
  static constexpr int G = ORDER / 2 + 2;       // halo cells per side
  static constexpr int NC = ORDER == 7 ? 9 : 6; // candidates
  static constexpr int LO = ORDER == 7 ? 0 : 1; // used window differences d[LO..HI]
  static constexpr int HI = ORDER == 7 ? 7 : 6;
};

// Chosen value minus the centre value, f^ - f_j = sum_i B[c][i] d[i], for the
// nine candidates in priority order, with d[i] = f_{j+i-3} - f_{j+i-4}
// (Table 1 rewritten in first differences).
__constant__ double kB64[9][8] = {
    {0, 0, 0, 0, 0, 0, 0, 0},
    {0, 0, 0, 0, 1.0 / 2, 0, 0, 0},
    {0, 0, 0, 1.0 / 6, 1.0 / 3, 0, 0, 0},
    {0, 0, -1.0 / 12, 1.0 / 3, 1.0 / 4, 0, 0, 0},
    {0, 0, 0, 1.0 / 12, 1.0 / 2, -1.0 / 12, 0, 0},
    {0, 0, -1.0 / 30, 11.0 / 60, 2.0 / 5, -1.0 / 20, 0, 0},
    {0, 1.0 / 60, -1.0 / 10, 17.0 / 60, 1.0 / 3, -1.0 / 30, 0, 0},
    {0, 0, -1.0 / 60, 7.0 / 60, 1.0 / 2, -7.0 / 60, 1.0 / 60, 0},
    {0, 1.0 / 140, -11.0 / 210, 79.0 / 420, 3.0 / 7, -17.0 / 210, 1.0 / 105, 0},
};
__constant__ float kB32[9][8] = {
    {0, 0, 0, 0, 0, 0, 0, 0},
    {0, 0, 0, 0, 1.0f / 2, 0, 0, 0},
    {0, 0, 0, 1.0f / 6, 1.0f / 3, 0, 0, 0},
    {0, 0, -1.0f / 12, 1.0f / 3, 1.0f / 4, 0, 0, 0},
    {0, 0, 0, 1.0f / 12, 1.0f / 2, -1.0f / 12, 0, 0},
    {0, 0, -1.0f / 30, 11.0f / 60, 2.0f / 5, -1.0f / 20, 0, 0},
    {0, 1.0f / 60, -1.0f / 10, 17.0f / 60, 1.0f / 3, -1.0f / 30, 0, 0},
    {0, 0, -1.0f / 60, 7.0f / 60, 1.0f / 2, -7.0f / 60, 1.0f / 60, 0},
    {0, 1.0f / 140, -11.0f / 210, 79.0f / 420, 3.0f / 7, -17.0f / 210, 1.0f / 105, 0},
};

template <typename R>
__device__ __forceinline__ R bcoef(int c, int i);
template <>
__device__ __forceinline__ double bcoef<double>(int c, int i) { return kB64[c][i]; }
template <>
__device__ __forceinline__ float bcoef<float>(int c, int i) { return kB32[c][i]; }

// Coefficient i of the top candidate (S_{j-2}^{j+2} of ENO-AO5, S_{j-3}^{j+3}
// of ENO-AO7), the same values as its row of kB32 / kB64, as immediates.
template <int ORDER, typename R>
__device__ __forceinline__ R bcoef_top(int i) {
  if constexpr (ORDER == 5) {
    constexpr R b[8] = {R(0), R(0), R(-1) / R(30), R(11) / R(60), R(2) / R(5), R(-1) / R(20), R(0),
                        R(0)};
    return b[i];
  } else {
    constexpr R b[8] = {R(0),         R(1) / R(140), R(-11) / R(210), R(79) / R(420),
                        R(3) / R(7), R(-17) / R(210), R(1) / R(105),  R(0)};
    return b[i];
  }
}

// Square root in the bulk precision (an unqualified sqrt on a float can
// resolve to the double routine, which runs on the slow FP64 unit).
__device__ __forceinline__ double bsqrt(double a) { return sqrt(a); }
__device__ __forceinline__ float bsqrt(float a) { return sqrtf(a); }
// Reciprocal and quotient in the bulk precision.  FP64 keeps correctly
// rounded division (parity with the FP64 oracle); the FP32 bulk path uses the
// fast hardware reciprocal (error of a few ulp, far inside the FP32-bulk
// tolerance) -- correctly rounded FP32 division is a long routine.
__device__ __forceinline__ double brcp(double a) { return 1.0 / a; }
__device__ __forceinline__ float brcp(float a) { return __fdividef(1.0f, a); }
__device__ __forceinline__ double bdiv(double a, double b) { return a / b; }
__device__ __forceinline__ float bdiv(float a, float b) { return __fdividef(a, b); }
// A product that is rounded before whatever is added to it, in every kernel.
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
// a b + c d with the first product fused.  Sums of products are written out
// with fma, dot2 and mul_rn from the state to the choice: which product the
// compiler fuses by itself changes from one kernel to the next, and every
// kernel must give the same bits -- the re-decision passes most of all, which
// re-derive the FP32 pick of a near-tie from its window.
template <typename T>
__device__ __forceinline__ T dot2(T a, T b, T c, T d) {
  return fma(a, b, mul_rn(c, d));
}
// Absolute value (a sign-bit operation, no floating-point instruction).
__device__ __forceinline__ double rabs(double a) { return fabs(a); }
__device__ __forceinline__ float rabs(float a) { return fabsf(a); }
// Order key of a non-negative value: for doubles the bit pattern read as an
// integer orders exactly like the value (NaN above everything), so indicator
// comparisons and minima run on the integer units instead of the FP64 unit,
// which is 1/64 of the FP32 rate on this part.
__device__ __forceinline__ long long okey(double a) { return __double_as_longlong(a); }
__device__ __forceinline__ float okey(float a) { return a; }
template <typename R>
__device__ __forceinline__ R rmin(R a, R b) { return okey(a) < okey(b) ? a : b; }

// Narrowing of a phase-1 input (an FP64 state component or the difference of
// two) to FP32 in six integer operations: the exponent word is clamped at the
// smallest normal FP32 exponent (so zero needs no branch), half an FP32 ulp
// is added at mantissa bit 28 with the carry running into the exponent, and
// the word is shifted into place with the exponent rebased from 1023 to 127.
// Round to nearest for every magnitude in [2^-126, 2^128) (an exact tie
// rounds away from zero); zero keeps its sign; a magnitude below 2^-126 gives
// one below 2^-126.  Magnitudes of 2^128 and more are out of range: a state
// that large fails the state check of its step, which narrows with f32_rn.
// The hardware conversion issues to the FP64 unit and is slower here.
__device__ __forceinline__ float f32_near(double x) {
  const unsigned lo = __double2loint(x), hi = __double2hiint(x);
  const unsigned hc = max(hi & 0x7FFFFFFFu, 896u << 20);
  const unsigned long long w =
      ((static_cast<unsigned long long>(hc - (896u << 20)) << 32) | lo) + 0x10000000ull;
  return __uint_as_float(static_cast<unsigned>(w >> 29) | (hi & 0x80000000u));
}

// FP64 value in the bulk precision, and a bulk value widened to FP64.
template <typename R>
__device__ __forceinline__ R to_bulk(double x);
template <>
__device__ __forceinline__ double to_bulk<double>(double x) { return x; }
template <>
__device__ __forceinline__ float to_bulk<float>(double x) { return f32_near(x); }
__device__ __forceinline__ double to_f64(double x) { return x; }
__device__ __forceinline__ double to_f64(float x) { return f64_of(x); }
// A constant of the sweep in the bulk precision: the FP64 argument, or its
// FP32 copy set on the host (SweepArgs, set_derived_constants).
template <typename R>
__device__ __forceinline__ R bconst(double d, float f);
template <>
__device__ __forceinline__ double bconst<double>(double d, float) { return d; }
template <>
__device__ __forceinline__ float bconst<float>(double, float f) { return f; }

// ENO-AO choice on one window of first differences d[LO..HI] (d[i] between
// offsets i-4 and i-3 of the centre cell).  Returns f^ - f_centre.  When
// CHECK is set, 'marginal' reports a decision that rounding of size tol_abs
// or a relative gap tie_rel could have changed.
// Rounding bound of the FP32 bulk indicators.  e[i] = sum_c |L_c| |df_c| is the
// magnitude of the terms whose FP32 sum gave d[i], so d[i] carries an error of
// at most feps * e[i] (feps = (NV + 8) eps32 covers the projection sum and the
// flux difference behind it).  An undivided difference of d sums its inputs
// with binomial weights, so the same Pascal sums of e bound its error; IS_c,
// the smaller of two such differences, is off by at most the larger bound.
template <int ORDER, typename R, bool CHECK>
__device__ __forceinline__ R eno_select(const R (&d)[8], R delta, R tie_rel, const R (&e)[8],
                                        R feps, int& pick_out, bool& marginal) {
  using GE = Geo<ORDER>;
  constexpr int LO = GE::LO, HI = GE::HI, NC = GE::NC;
  // Principle 1 first for the top candidate (highest priority): at or below
  // delta it is the pick whatever the other indicators are -- the smooth
  // case, most windows -- and only its indicator, its rounding bound and its
  // Table-1 value (compile-time coefficients) are needed.  Its two undivided
  // differences of order 5 (7) are formed directly with their binomial
  // weights; the difference table of the other candidates is built only when
  // the top one is above delta.
  const auto kdelta = okey(delta);
  R IS_top;
  if constexpr (ORDER == 7) {
    auto b6 = [&](int o) {  // sum_k (-1)^k C(6,k) d[o+k]
      R t = d[o] + d[o + 6];
      t = fma(R(-6), d[o + 1] + d[o + 5], t);
      t = fma(R(15), d[o + 2] + d[o + 4], t);
      return fma(R(-20), d[o + 3], t);
    };
    IS_top = rmin(rabs(b6(0)), rabs(b6(1)));
  } else {
    auto b4 = [&](int o) {  // sum_k (-1)^k C(4,k) d[o+k]
      R t = d[o] + d[o + 4];
      t = fma(R(-4), d[o + 1] + d[o + 3], t);
      return fma(R(6), d[o + 2], t);
    };
    IS_top = rmin(rabs(b4(1)), rabs(b4(2)));
  }
  int pick;
  R corr = R(0);
  if (okey(IS_top) <= kdelta) {
    pick = NC - 1;
    // its nonzero coefficients: d[2..5] (ENO-AO5), d[1..6] (ENO-AO7)
#pragma unroll
    for (int i = ORDER == 5 ? 2 : 1; i <= (ORDER == 5 ? 5 : 6); ++i)
      corr = fma(bcoef_top<ORDER, R>(i), d[i], corr);
    if constexpr (CHECK) {
      // its bound: the Pascal sums of e over its two differences, written out
      R qa, qb;
      if constexpr (ORDER == 7) {
        qa = e[0] + e[6] + R(6) * (e[1] + e[5]) + R(15) * (e[2] + e[4]) + R(20) * e[3];
        qb = e[1] + e[7] + R(6) * (e[2] + e[6]) + R(15) * (e[3] + e[5]) + R(20) * e[4];
      } else {
        qa = e[1] + e[5] + R(4) * (e[2] + e[4]) + R(6) * e[3];
        qb = e[2] + e[6] + R(4) * (e[3] + e[5]) + R(6) * e[4];
      }
      marginal = rabs(IS_top - delta) <= tie_rel * delta + feps * fmaxf(qa, qb);
    }
  } else {
    R s2[8], s3[8], s4[8], s5[8], s6[8];
#pragma unroll
    for (int i = LO; i < HI; ++i) s2[i] = d[i + 1] - d[i];
#pragma unroll
    for (int i = LO; i < HI - 1; ++i) s3[i] = s2[i + 1] - s2[i];
#pragma unroll
    for (int i = LO; i < HI - 2; ++i) s4[i] = s3[i + 1] - s3[i];
#pragma unroll
    for (int i = LO; i < HI - 3; ++i) s5[i] = s4[i + 1] - s4[i];
    if constexpr (ORDER == 7) {
#pragma unroll
      for (int i = 0; i < 3; ++i) s6[i] = s5[i + 1] - s5[i];
    }
    R IS[9];
    // min(a/2, b/2) = min(a, b)/2 exactly (scaling by a power of two)
    IS[0] = R(0.5) * rmin(rabs(d[3]) + rabs(d[2]), rabs(d[4]) + rabs(d[5]));
    IS[1] = rmin(rabs(s2[3]), rabs(s2[4]));
    IS[2] = rmin(rabs(s3[2]), rabs(s3[3]));
    IS[3] = rmin(rabs(s4[1]), rabs(s4[2]));
    IS[4] = rmin(rabs(s4[2]), rabs(s4[3]));
    if constexpr (ORDER == 7) {
      IS[5] = rmin(rabs(s5[1]), rabs(s5[2]));
      IS[6] = rmin(rabs(s6[0]), rabs(s6[1]));
      IS[7] = rmin(rabs(s6[1]), rabs(s6[2]));
    }
    IS[NC - 1] = IS_top;
    // Principle 1 over the others (the top is above delta here).
    pick = -1;
#pragma unroll
    for (int c = 0; c < NC - 1; ++c)
      if (okey(IS[c]) <= kdelta) pick = c;
    const bool thr = pick >= 0;
    // Principle 2: otherwise the smallest IS, equal values to the higher priority.
    R best = IS[0];
    if (!thr) {
      pick = 0;
#pragma unroll
      for (int c = 1; c < NC; ++c)
        if (okey(IS[c]) <= okey(best)) {
          best = IS[c];
          pick = c;
        }
    }
    if constexpr (CHECK) {
      const R rel = tie_rel * delta;
      bool m = false;
      // per-candidate bounds: Pascal sums of e over each indicator's differences
      R q2[8], q3[8], q4[8], q5[8], q6[8], q7[8];
#pragma unroll
      for (int i = LO; i < HI; ++i) q2[i] = e[i] + e[i + 1];
#pragma unroll
      for (int i = LO; i < HI - 1; ++i) q3[i] = q2[i] + q2[i + 1];
#pragma unroll
      for (int i = LO; i < HI - 2; ++i) q4[i] = q3[i] + q3[i + 1];
#pragma unroll
      for (int i = LO; i < HI - 3; ++i) q5[i] = q4[i] + q4[i + 1];
      R tol[9];
      tol[0] = feps * R(0.5) * fmaxf(e[3] + e[2], e[4] + e[5]);
      tol[1] = feps * fmaxf(q2[3], q2[4]);
      tol[2] = feps * fmaxf(q3[2], q3[3]);
      tol[3] = feps * fmaxf(q4[1], q4[2]);
      tol[4] = feps * fmaxf(q4[2], q4[3]);
      tol[5] = feps * fmaxf(q5[1], q5[2]);
      if constexpr (ORDER == 7) {
#pragma unroll
        for (int i = 0; i < 3; ++i) q6[i] = q5[i] + q5[i + 1];
#pragma unroll
        for (int i = 0; i < 2; ++i) q7[i] = q6[i] + q6[i + 1];
        tol[6] = feps * fmaxf(q6[0], q6[1]);
        tol[7] = feps * fmaxf(q6[1], q6[2]);
        tol[8] = feps * fmaxf(q7[0], q7[1]);
      }
      if (thr) {
#pragma unroll
        for (int c = 0; c < NC; ++c) m |= (c >= pick) && (rabs(IS[c] - delta) <= rel + tol[c]);
      } else {
        R tp = tol[0];
#pragma unroll
        for (int c = 1; c < NC; ++c)
          if (c == pick) tp = tol[c];
        m = (best - delta) <= rel + tp;
        const R relA = tie_rel * best + tp;
        // Candidates 3 and 4 (and 6 and 7 of ENO-AO7) take the minimum over
        // two differences of which they share the middle one, b: with
        // IS_lo = min(a, b) and IS_hi = min(b, c), IS_lo wins exactly when
        // a < b and a < c, so the margin of the pair is max(a - b, a - c), not
        // IS_lo - IS_hi (which is zero whenever b is the smaller of both).
        R gap[9];
#pragma unroll
        for (int c = 0; c < NC; ++c) gap[c] = IS[c] - best;
        if (pick == 4) {
          const R a = rabs(s4[1]), b = rabs(s4[2]), c = rabs(s4[3]);
          gap[3] = fmaxf(a - b, a - c);
        }
        if constexpr (ORDER == 7) {
          if (pick == 7) {
            const R a = rabs(s6[0]), b = rabs(s6[1]), c = rabs(s6[2]);
            gap[6] = fmaxf(a - b, a - c);
          }
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) m |= (c != pick) && (gap[c] <= relA + tol[c]);
      }
      marginal = m;
    }
#pragma unroll
    for (int i = LO; i <= HI; ++i) corr = fma(bcoef<R>(pick, i), d[i], corr);
  }
  pick_out = pick;
  return corr;
}

// The FP64 choice on a window of FP64 differences: the indicators, their
// comparisons and the bounds of both in FP32 (from the differences rounded
// once, so an indicator is off by a few FP32 roundings of the magnitudes it
// sums: 8 eps covers the deepest table), and the choice again in FP64 where
// those bounds leave it open -- the same choice as FP64 throughout.  The value
// is FP64.  The FP64 unit, 1/64 of the FP32 rate, is left with the 6 to 8
// operations of the value instead of some 50 of tables and comparisons (scalar
// ENO-AO7 fluxes of 4096 x 2048 cells 1.86 -> 1.02 ms, a 97 x 80 x 63 Euler step,
// hardly any of whose faces are proven, 9.1 -> 6.7 ms).
template <int ORDER>
__device__ __forceinline__ double choose64(const double (&d)[8], double delta, float delta_f,
                                           int& pick) {
  using GE = Geo<ORDER>;
  float d32[8], mag[8], sum = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    d32[i] = f32_rn(d[i]);
    mag[i] = fabsf(d32[i]);
    sum += mag[i];
  }
  bool open;
  eno_select<ORDER, float, true>(d32, delta_f, 1e-5f, mag, 8.0f * FLT_EPSILON, pick, open);
  if (open || !(sum < INFINITY) || !(delta_f >= 1e-30f)) {
    const double none[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    return eno_select<ORDER, double, false>(d, delta, 0.0, none, 0.0, pick, open);
  }
  double corr = 0.0;
#pragma unroll
  for (int i = GE::LO; i <= GE::HI; ++i) corr = fma(bcoef<double>(pick, i), d[i], corr);
  return corr;
}

// Conserved component stored at position c of the permuted state for a sweep
// along axis dir (momentum along dir first, tangential momenta cyclic).
template <int NV>
__device__ __forceinline__ int perm_comp(int c, int dir) {
  if (NV == 1 || c == 0 || c == NV - 1) return c;
  constexpr int ND = NV > 2 ? NV - 2 : 1;
  return 1 + (dir + c - 1) % ND;
}

// Conserved component k of a state held in permuted order, by selects (an
// index computed from the runtime axis would put the array in local memory).
template <int NV, typename T>
__device__ __forceinline__ T comp_of(const T (&up)[NV], int k, int dir) {
  if constexpr (NV < 3) {
    return up[k];
  } else {
    if (k == 0 || k == NV - 1) return up[k];
    T r = up[1];
#pragma unroll
    for (int c = 2; c < NV - 1; ++c) r = perm_comp<NV>(c, dir) == k ? up[c] : r;
    return r;
  }
}

template <int NV, typename T>
__device__ __forceinline__ T inv_density(const T (&q)[NV]) {
  return NV > 1 ? brcp(q[0]) : T(0);
}

// Flux difference F(qb) - F(qa) along the sweep axis, written in differences
// so that rounding scales with |dq| (Euler: F = [m, m u + p, m_t u, (E+p) u]).
// ia, ib: 1 / density of the two cells (inv_density), which neighbouring
// pairs share.
template <int NV, typename T>
__device__ __forceinline__ void flux_diff(const T (&qa)[NV], const T (&qb)[NV], const T (&dq)[NV],
                                          T gm1, T adv, T ia, T ib, T (&dF)[NV]) {
  if constexpr (NV == 1) {
    dF[0] = adv * dq[0];
  } else {
    constexpr int NT = NV - 3;  // tangential components
    const T u = qa[1] * ia;
    T vt[NT > 0 ? NT : 1], dvt[NT > 0 ? NT : 1];
    const T du = fma(-u, dq[0], dq[1]) * ib;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      vt[t] = qa[2 + t] * ia;
      dvt[t] = fma(-vt[t], dq[0], dq[2 + t]) * ib;
    }
    T v2, dke2;  // |v|^2, and v . dv + |dv|^2 / 2
    if constexpr (NT == 0) {
      v2 = mul_rn(u, u);
      dke2 = fma(u, du, T(0.5) * mul_rn(du, du));
    } else {
      v2 = dot2(u, u, vt[0], vt[0]);
      T vdv = dot2(u, du, vt[0], dvt[0]);
      T dv2 = dot2(du, du, dvt[0], dvt[0]);
#pragma unroll
      for (int t = 1; t < NT; ++t) {
        v2 = fma(vt[t], vt[t], v2);
        vdv = fma(vt[t], dvt[t], vdv);
        dv2 = fma(dvt[t], dvt[t], dv2);
      }
      dke2 = fma(T(0.5), dv2, vdv);
    }
    const T dke = dot2(T(0.5) * dq[0], v2, qb[0], dke2);
    const T ea = fma(T(-0.5) * qa[0], v2, qa[NV - 1]);  // internal energy
    const T de = dq[NV - 1] - dke;
    const T ub = u + du;
    dF[0] = dq[1];
    dF[1] = fma(gm1, de, dot2(dq[1], ub, qa[1], du));
#pragma unroll
    for (int t = 0; t < NT; ++t) dF[2 + t] = dot2(dq[2 + t], ub, qa[2 + t], du);
    dF[NV - 1] = dot2(fma(gm1, de, dq[NV - 1]), ub, fma(gm1, ea, qa[NV - 1]), du);
  }
}

// Physical flux of a permuted state (used only for interface-flux output).
template <int NV>
__device__ __forceinline__ void phys_flux(const double (&q)[NV], double gm1, double adv,
                                          double (&F)[NV]) {
  if constexpr (NV == 1) {
    F[0] = adv * q[0];
  } else {
    double ke = 0.0;
#pragma unroll
    for (int i = 1; i < NV - 1; ++i) ke += q[i] * q[i];
    ke = 0.5 * ke / q[0];
    const double p = gm1 * (q[NV - 1] - ke);
    const double un = q[1] / q[0];
    F[0] = q[1];
    F[1] = q[1] * un + p;
#pragma unroll
    for (int i = 2; i < NV - 1; ++i) F[i] = q[i] * un;
    F[NV - 1] = (q[NV - 1] + p) * un;
  }
}

// Roe-average ingredients of one cell: sqrt(rho), velocity, total enthalpy.
template <int NV, typename T>
__device__ __forceinline__ void roe_prims(const T (&q)[NV], T gm1, T ir, T (&pr)[NV]) {
  if constexpr (NV > 1) {
    T ke = T(0);
#pragma unroll
    for (int i = 1; i < NV - 1; ++i) {
      pr[i] = q[i] * ir;
      ke = fma(q[i], pr[i], ke);
    }
    pr[0] = bsqrt(q[0]);
    pr[NV - 1] = fma(gm1, fma(T(-0.5), ke, q[NV - 1]), q[NV - 1]) * ir;  // (E + p) / rho
  }
}

// Eigen-system of the Euler flux Jacobian at the Roe state of a face.
template <int NV, typename T>
struct Eigen {
  T u, vt[NV > 3 ? NV - 3 : 1], H, c, ic, b1, b2, q2;
};

template <int NV, typename T>
__device__ __forceinline__ void roe_eigen(const T (&pl)[NV], const T (&prr)[NV], T gm1,
                                          Eigen<NV, T>& E) {
  constexpr int NT = NV - 3;
  const T inv = brcp(pl[0] + prr[0]);
  const T wl = pl[0] * inv, wr = prr[0] * inv;
  E.u = dot2(wl, pl[1], wr, prr[1]);
#pragma unroll
  for (int t = 0; t < NT; ++t) E.vt[t] = dot2(wl, pl[2 + t], wr, prr[2 + t]);
  T q2;
  if constexpr (NT < 2) {
    q2 = mul_rn(E.u, E.u);
    if constexpr (NT == 1) q2 = fma(E.vt[0], E.vt[0], q2);
  } else {
    q2 = fma(E.vt[1], E.vt[1], dot2(E.u, E.u, E.vt[0], E.vt[0]));
  }
  E.H = dot2(wl, pl[NV - 1], wr, prr[NV - 1]);
  E.q2 = q2;
  const T c2 = gm1 * fma(T(-0.5), q2, E.H);
  E.c = bsqrt(c2);
  E.ic = brcp(E.c);
  E.b1 = bdiv(gm1, c2);
  E.b2 = mul_rn(T(0.5) * q2, E.b1);
}

// The constant c ? 1 : 0 (and c ? 1 : -1) by an integer select: a
// floating-point select of constants can become a conversion instruction,
// which issues to the FP64 unit.
template <typename T>
__device__ __forceinline__ T one_if(bool c) {
  if constexpr (sizeof(T) == 4) return __int_as_float(c ? 0x3f800000 : 0);
  return c ? T(1) : T(0);
}
template <typename T>
__device__ __forceinline__ T sign_if(bool c) {
  if constexpr (sizeof(T) == 4) return __int_as_float(c ? 0x3f800000 : (int)0xbf800000u);
  return c ? T(1) : T(-1);
}

// Row v of L = R^{-1}; fields ordered (u-c, entropy, shear..., u+c).
template <int NV, typename T>
__device__ __forceinline__ void left_row(const Eigen<NV, T>& E, int v, T (&L)[NV]) {
  constexpr int NT = NV - 3;
  if (v == 0 || v == NV - 1) {
    const T s = sign_if<T>(v == 0);
    L[0] = T(0.5) * fma(s * E.u, E.ic, E.b2);
    L[1] = T(0.5) * fma(-E.b1, E.u, -(s * E.ic));
#pragma unroll
    for (int t = 0; t < NT; ++t) L[2 + t] = T(-0.5) * E.b1 * E.vt[t];
    L[NV - 1] = T(0.5) * E.b1;
  } else if (v == 1) {
    L[0] = T(1) - E.b2;
    L[1] = E.b1 * E.u;
#pragma unroll
    for (int t = 0; t < NT; ++t) L[2 + t] = E.b1 * E.vt[t];
    L[NV - 1] = -E.b1;
  } else {
    // shear field v: selects instead of indexing by v, so that L, E stay
    // in registers when the caller loops over v without unrolling
    T w = E.vt[0];
#pragma unroll
    for (int t = 1; t < NT; ++t) w = v - 2 == t ? E.vt[t] : w;
#pragma unroll
    for (int i = 1; i < NV; ++i) L[i] = one_if<T>(i == v);
    L[0] = -w;
  }
}

// Component v (a shear field, 2 <= v <= NV - 2) of a permuted vector, by
// selects so that the vector stays in registers.
template <int NV, typename T>
__device__ __forceinline__ T shear_comp(const T (&x)[NV], int v) {
  static_assert(NV >= 4, "shear fields exist for NV >= 4");
  T r = x[2];
#pragma unroll
  for (int c = 3; c < NV - 1; ++c) r = v == c ? x[c] : r;
  return r;
}

// Column v of R.
template <int NV, typename T>
__device__ __forceinline__ void right_col(const Eigen<NV, T>& E, int v, T (&Rc)[NV]) {
  constexpr int NT = NV - 3;
  if (v == 0 || v == NV - 1) {
    const T s = sign_if<T>(v != 0);
    Rc[0] = T(1);
    Rc[1] = E.u + s * E.c;
#pragma unroll
    for (int t = 0; t < NT; ++t) Rc[2 + t] = E.vt[t];
    Rc[NV - 1] = fma(s * E.u, E.c, E.H);
  } else if (v == 1) {
    Rc[0] = T(1);
    Rc[1] = E.u;
#pragma unroll
    for (int t = 0; t < NT; ++t) Rc[2 + t] = E.vt[t];
    Rc[NV - 1] = T(0.5) * E.q2;
  } else {
    T w = E.vt[0];
#pragma unroll
    for (int t = 1; t < NT; ++t) w = v - 2 == t ? E.vt[t] : w;
#pragma unroll
    for (int i = 0; i < NV - 1; ++i) Rc[i] = one_if<T>(i == v);
    Rc[NV - 1] = w;
  }
}

// Ghost-cell map along the swept axis; s lies within one halo width of
// [0, n) (n is at least the halo width), so the periodic wrap is one add or
// subtract -- no integer division, whose 64-bit form runs on the FP64 unit.
// A sub-domain's split axis (kBcHalo) keeps its ghost layers in the arrays,
// next to the interior: positions outside [0, n) are read where they are.
__device__ __forceinline__ long long bc_map(long long s, long long n, int bc) {
  if (bc == 0) return s < 0 ? s + n : (s >= n ? s - n : s);
  if (bc == kBcHalo) return s;
  return s < 0 ? 0 : (s >= n ? n - 1 : s);
}

// Geometry of one tile: cell(a, s) = base + (a0 + a) * stride_a + s * stride_d.
struct TileGeo {
  long long s0, a0, base, stride_a, stride_d, na, nd;
  long long b;                             // index along the remaining axis (dir != 0)
  long long fbase, fstride_a, fstride_d;  // same for the face array (nd + 1 faces)
  int nts;                                 // valid cells of the tile along dir
};

__device__ __forceinline__ TileGeo tile_geo(const SweepArgs& A, long long tile) {
  TileGeo g;
  // tile counts fit 32 bits (checked on the host): 32-bit division only
  const unsigned t32 = (unsigned)tile, tsn = (unsigned)A.tiles_s, tan = (unsigned)A.tiles_a;
  const unsigned rest32 = t32 / tsn;
  const long long ts_i = t32 - rest32 * tsn;
  const long long b = rest32 / tan;
  const long long ta_i = rest32 - (unsigned)b * tan;
  const long long n0 = A.n[0], n1 = A.n[1], n2 = A.n[2];
  g.s0 = ts_i * A.ts;
  g.a0 = ta_i * A.ta;
  g.b = b;
  if (A.dir == 0) {
    g.nd = n0; g.na = n1 * n2;
    g.base = 0; g.stride_a = n0; g.stride_d = 1;
    g.fbase = 0; g.fstride_a = n0 + 1; g.fstride_d = 1;
  } else if (A.dir == 1) {
    g.nd = n1; g.na = n0;
    g.base = b * n1 * n0; g.stride_a = 1; g.stride_d = n0;
    g.fbase = b * (n1 + 1) * n0; g.fstride_a = 1; g.fstride_d = n0;
  } else {
    g.nd = n2; g.na = n0;
    g.base = b * n0; g.stride_a = 1; g.stride_d = n0 * n1;
    g.fbase = b * n0; g.fstride_a = 1; g.fstride_d = n0 * n1;
  }
  g.base += A.org;  // sub-domains: the interior starts after the low ghost layers
  const long long left = g.nd - g.s0;
  g.nts = (int)(left < A.ts ? left : A.ts);
  return g;
}

// Cell index within a component.  The Euler systems index with 32 bits (2^32
// cells of three or more FP64 components in three state arrays do not fit the
// device's memory), so that an access is one multiply-add onto a component's
// uniform base; scalar arrays can be longer.
template <int NV>
struct CellIndex {
  using type = unsigned;
};
template <>
struct CellIndex<1> {
  using type = unsigned long long;
};
template <int NV>
using cell_t = typename CellIndex<NV>::type;

// Loads the input state of one cell in sweep order.  COHERENT loads go
// through L2 (the batched kernel reads states it wrote itself); otherwise the
// read-only path is used (a sweep never writes the array it stencils from).
template <int NV, bool COHERENT = false>
__device__ __forceinline__ void load_state(const SweepArgs& A, cell_t<NV> cell, double (&q)[NV]) {
#pragma unroll
  for (int c = 0; c < NV; ++c) {
    const double* p = A.comp.u_in[c] + cell;
    q[c] = COHERENT ? __ldcg(p) : __ldg(p);
  }
}

// Lane group of W lanes (a power of two, at least the 2G window cells) that
// re-decides one choice in FP64 together: lane r holds window cell r, forms
// difference r with its neighbour's state, and the projected window is then
// gathered by shuffles; every lane of the group returns the same pick.  Groups
// of the same warp work on different choices at the same time, so the FP64
// unit (1/64 of the FP32 rate) runs on full warps instead of single lanes.
template <int NV, int ORDER, bool COHERENT, int W>
__device__ __forceinline__ int redo_group(const SweepArgs& A, const TileGeo& g, int a,
                                          long long sj, int v, int sgn, double alpha, int r) {
  constexpr int G = Geo<ORDER>::G;
  static_assert(W >= 2 * G, "a lane per window cell");
  const unsigned FULL = 0xffffffffu;
  const double gm1 = A.gm1;
  const long long line = g.base + (g.a0 + a) * g.stride_a;
  const int rr = r < 2 * G ? r : 2 * G - 1;
  double q[NV];
  load_state<NV, COHERENT>(A, line + bc_map(sj - G + 1 + rr, g.nd, A.bc) * g.stride_d, q);
  double L[NV];
  if constexpr (NV > 1) {
    double ql[NV], qr[NV], pl[NV], prr[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) {
      ql[c] = __shfl_sync(FULL, q[c], G - 1, W);
      qr[c] = __shfl_sync(FULL, q[c], G, W);
    }
    roe_prims<NV, double>(ql, gm1, inv_density<NV>(ql), pl);
    roe_prims<NV, double>(qr, gm1, inv_density<NV>(qr), prr);
    Eigen<NV, double> E;
    roe_eigen<NV, double>(pl, prr, gm1, E);
    left_row<NV, double>(E, v, L);
  } else {
    L[0] = 1.0;
  }
  double qn[NV];
#pragma unroll
  for (int c = 0; c < NV; ++c) qn[c] = __shfl_down_sync(FULL, q[c], 1, W);
  double w = 0.0;
  {
    double dq[NV], dF[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) dq[c] = qn[c] - q[c];
    const double ia = inv_density<NV>(q), ib = __shfl_down_sync(FULL, ia, 1, W);
    flux_diff<NV, double>(q, qn, dq, gm1, A.adv_speed, ia, ib, dF);
    const double sa = sgn == 0 ? alpha : -alpha;
#pragma unroll
    for (int c = 0; c < NV; ++c) w = fma(L[c], 0.5 * fma(sa, dq[c], dF[c]), w);
  }
  // window difference k (between cells k and k+1) sits in group lane k
  double d[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) d[i] = 0.0;
#pragma unroll
  for (int i = Geo<ORDER>::LO; i <= Geo<ORDER>::HI; ++i) {
    const int k = sgn == 0 ? i - 4 + G - 1 : 4 - i + G - 1;
    const double wk = __shfl_sync(FULL, w, k, W);
    d[i] = sgn == 0 ? wk : -wk;
  }
  int pick;
  bool m;
  const double nomx[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  eno_select<ORDER, double, false>(d, A.delta, 0.0, nomx, 0.0, pick, m);
  return pick;
}

// The same FP64 re-decision by one thread alone: it walks the window cell by
// cell (two states live at a time).  Used when a warp has many flagged
// choices at once, so that all lanes work on their own choices in parallel
// instead of the warp serving them a few at a time.
template <int NV, int ORDER, bool COHERENT>
__device__ __forceinline__ int redo_lane(const SweepArgs& A, const TileGeo& g, int a, long long sj,
                                         int v, int sgn, double alpha) {
  using GE = Geo<ORDER>;
  constexpr int G = GE::G;
  const double gm1 = A.gm1;
  const long long line = g.base + (g.a0 + a) * g.stride_a;
  // window cell r (0..2G-1) is cell sj - G + 1 + r of the line; the face lies
  // between cells G-1 and G
  auto load_cell = [&](int r, double (&q)[NV]) {
    load_state<NV, COHERENT>(A, line + bc_map(sj - G + 1 + r, g.nd, A.bc) * g.stride_d, q);
  };
  double L[NV];
  if constexpr (NV > 1) {
    double ql[NV], qr[NV], pl[NV], prr[NV];
    load_cell(G - 1, ql);
    load_cell(G, qr);
    roe_prims<NV, double>(ql, gm1, inv_density<NV>(ql), pl);
    roe_prims<NV, double>(qr, gm1, inv_density<NV>(qr), prr);
    Eigen<NV, double> E;
    roe_eigen<NV, double>(pl, prr, gm1, E);
    left_row<NV, double>(E, v, L);
  } else {
    L[0] = 1.0;
  }
  const double sa = sgn == 0 ? alpha : -alpha;
  // d[i] is difference k = i + G - 5 (sign 0) or G + 3 - i (sign 1, negated),
  // between window cells k and k+1; consecutive i share one cell
  double d[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) d[i] = 0.0;
  double qlo[NV], qhi[NV];
  {
    const int k0 = sgn == 0 ? GE::LO + G - 5 : G + 3 - GE::LO;
    load_cell(k0, qlo);
    load_cell(k0 + 1, qhi);
  }
  double ilo = inv_density<NV>(qlo), ihi = inv_density<NV>(qhi);
#pragma unroll
  for (int i = GE::LO; i <= GE::HI; ++i) {
    double dq[NV], dF[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) dq[c] = qhi[c] - qlo[c];
    flux_diff<NV, double>(qlo, qhi, dq, gm1, A.adv_speed, ilo, ihi, dF);
    double w = 0.0;
#pragma unroll
    for (int c = 0; c < NV; ++c) w = fma(L[c], 0.5 * fma(sa, dq[c], dF[c]), w);
    d[i] = sgn == 0 ? w : -w;
    if (i < GE::HI) {
      const int k = sgn == 0 ? i + G - 5 : G + 3 - i;
      if (sgn == 0) {
#pragma unroll
        for (int c = 0; c < NV; ++c) qlo[c] = qhi[c];
        load_cell(k + 2, qhi);
        ilo = ihi;
        ihi = inv_density<NV>(qhi);
      } else {
#pragma unroll
        for (int c = 0; c < NV; ++c) qhi[c] = qlo[c];
        load_cell(k - 1, qlo);
        ihi = ilo;
        ilo = inv_density<NV>(qlo);
      }
    }
  }
  int pick;
  bool m;
  const double nomx[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  eno_select<ORDER, double, false>(d, A.delta, 0.0, nomx, 0.0, pick, m);
  return pick;
}

// Position of the n-th (0-based) set bit of x, or -1.
__device__ __forceinline__ int nth_set_bit(unsigned x, int n) {
  for (int i = 0; i < n && x; ++i) x &= x - 1;
  return x ? __ffs(x) - 1 : -1;
}

// Runs body(a, e) over the items of a TA x cnt tile.  x sweeps (sfast):
// each thread keeps one line a and strides along e (lanes along the line);
// y/z sweeps: each thread keeps one line a (lanes across lines, i.e. along x)
// and strides along e.  TA is a power of two dividing the block size, so the
// mapping is shifts and masks -- no per-item integer division.
template <typename F>
__device__ __forceinline__ void for_items(int lgTA, int cnt, bool sfast, F&& body) {
  const int bd = blockDim.x, tid = threadIdx.x;
  if (sfast) {
    const int lgTpl = __ffs(bd) - 1 - lgTA;  // threads per line = bd / TA
    const int a = tid >> lgTpl, tpl = 1 << lgTpl;
    for (int e = tid & (tpl - 1); e < cnt; e += tpl) body(a, e);
  } else {
    const int a = tid & ((1 << lgTA) - 1);
    const int step = bd >> lgTA;
    for (int e = tid >> lgTA; e < cnt; e += step) body(a, e);
  }
}

// The mapping of for_items as values: this thread's line a, its first item
// e0 and the stride between its items.
__device__ __forceinline__ void item_start(int lgTA, bool sfast, int& a, int& e0, int& step) {
  const int bd = blockDim.x, tid = threadIdx.x;
  if (sfast) {
    const int lgTpl = __ffs(bd) - 1 - lgTA;
    a = tid >> lgTpl;
    step = 1 << lgTpl;
    e0 = tid & (step - 1);
  } else {
    a = tid & ((1 << lgTA) - 1);
    step = bd >> lgTA;
    e0 = tid >> lgTA;
  }
}

// Whether a sweep variant proves most faces to take the top candidate before
// any projection (phase 2a below): all with one splitting constant.
template <bool FIELD>
constexpr bool kProve = !FIELD;

// Per-cell vectors in shared memory.  FP32 vectors of the Euler equations are
// one float4 per cell, so a cell moves in one 128-bit access: the 1D system
// has a fourth value to spare (kSpare: phase 1 keeps a bound of the proof
// there), the 3D system keeps its fifth in a plane behind the float4s.  FP64,
// scalar and per-field 1D and 3D sweeps keep one plane per component.
template <int NV, typename R, bool FIELD>
struct CellVec {
  static constexpr bool kAoS = sizeof(R) == 4 && (NV == 4 || (NV >= 3 && !FIELD));
  static constexpr bool kSpare = kAoS && NV == 3;
  static constexpr int kSlots = kSpare ? 4 : NV;  // values of R per cell
  __device__ __forceinline__ static void load(const R* base, int cells, int i, R (&v)[NV]) {
    if constexpr (kAoS) {
      const float4 t = reinterpret_cast<const float4*>(base)[i];
      v[0] = t.x, v[1] = t.y, v[2] = t.z;
      if constexpr (NV >= 4) v[3] = t.w;
      if constexpr (NV == 5) v[4] = base[4 * cells + i];
    } else {
#pragma unroll
      for (int c = 0; c < NV; ++c) v[c] = base[c * cells + i];
    }
  }
  __device__ __forceinline__ static void store(R* base, int cells, int i, const R (&v)[NV]) {
    if constexpr (kSpare) {  // the fourth value stays
      reinterpret_cast<float2*>(base)[2 * i] = make_float2(v[0], v[1]);
      base[4 * i + 2] = v[2];
    } else if constexpr (kAoS) {
      reinterpret_cast<float4*>(base)[i] = make_float4(v[0], v[1], v[2], v[3]);
      if constexpr (NV == 5) base[4 * cells + i] = v[4];
    } else {
#pragma unroll
      for (int c = 0; c < NV; ++c) base[c * cells + i] = v[c];
    }
  }
  // with the spare fourth value of the 1D system
  __device__ __forceinline__ static void store4(R* base, int i, const R (&v)[NV], R w) {
    reinterpret_cast<float4*>(base)[i] = make_float4(v[0], v[1], v[2], w);
  }
};

// Lax-Friedrichs split differences of one pair of neighbouring cells in the
// bulk precision (phase 1): dq = qb - qa rounded once from FP64, the flux
// difference in difference form, and (dF +- alpha dq)/2 written as
// dF/2 +- (alpha/2) dq (the same bits: halving is exact).
// Returns sum_c max(|fp_c|, |fm_c|) = sum_c |dF_c|/2 + alpha |dq_c|/2, the
// magnitude that bounds the FP32 rounding of both (unused results cost nothing).
template <int NV, typename R>
__device__ __forceinline__ R split_diff(const double (&qa64)[NV], const double (&qb64)[NV],
                                        const R (&qa)[NV], const R (&qb)[NV], R gm1, R adv,
                                        R halpha, R ia, R ib, R (&fp)[NV], R (&fm)[NV]) {
  R dq[NV], dF[NV], m = R(0);
#pragma unroll
  for (int c = 0; c < NV; ++c) dq[c] = to_bulk<R>(qb64[c] - qa64[c]);
  flux_diff<NV, R>(qa, qb, dq, gm1, adv, ia, ib, dF);
#pragma unroll
  for (int c = 0; c < NV; ++c) {
    const R hdF = R(0.5) * dF[c];
    fp[c] = fma(halpha, dq[c], hdF);
    fm[c] = fma(-halpha, dq[c], hdF);
    m = fma(halpha, rabs(dq[c]), m + rabs(hdF));
  }
  return m;
}

// The same pair of cells for per-field splitting: dF/2 and dq/2 (exact
// halvings), to be split per characteristic field after the projection.
template <int NV, typename R>
__device__ __forceinline__ void split_parts(const double (&qa64)[NV], const double (&qb64)[NV],
                                            const R (&qa)[NV], const R (&qb)[NV], R gm1, R adv,
                                            R ia, R ib, R (&hdF)[NV], R (&hdq)[NV]) {
  R dq[NV], dF[NV];
#pragma unroll
  for (int c = 0; c < NV; ++c) dq[c] = to_bulk<R>(qb64[c] - qa64[c]);
  flux_diff<NV, R>(qa, qb, dq, gm1, adv, ia, ib, dF);
#pragma unroll
  for (int c = 0; c < NV; ++c) {
    hdF[c] = R(0.5) * dF[c];
    hdq[c] = R(0.5) * dq[c];
  }
}

// Per-field splitting constant of characteristic field v (u-c, entropy,
// shear..., u+c) along axis dir: max |u_d - c|, max |u_d|, max |u_d + c|.
template <int NV>
__device__ __forceinline__ double field_alpha(const StepState* st, int dir, int v) {
  return st->alpha_f[dir][v == 0 ? 0 : (v == NV - 1 ? 2 : 1)];
}

// FP32 bulk: the state is checked, and the next step's alpha taken, on each
// step's final state; the kinetic energy, sound speed and |u| + c are FP32,
// the energy difference E - ke stays FP64.  The alpha of a later stage of the
// same step (per-stage alpha) is taken in FP64 like the FP64 path's: the
// stage's stencil choices must not depend on FP32 rounding of the splitting
// constant.  unew is the combined state of cell in conserved order.
template <int NV>
__device__ __forceinline__ void bulk_state_check(const SweepArgs& A, long long cell,
                                                 const double (&unew)[NV], int mode,
                                                 double (&amax)[3]) {
  StepState* st = A.st;
  if constexpr (NV > 1) {
    if (A.stage < 2 && (mode & kModeAlpha)) {
      double s[3];
      if (!speeds64<NV, false>(unew, A.gamma, s)) {
        atomicOr(&st->err, kErrNonPhys);
        atomicMin(&st->err_cell, cell);
      } else {
#pragma unroll
        for (int d = 0; d < NV - 2; ++d) amax[d] = fmax(amax[d], s[d]);
      }
      return;
    }
  }
  if (A.stage == 2) {
    if constexpr (NV > 1) {
      double s[3];
      if (!speeds32<NV, false>(unew, A.gamma, s)) {
        atomicOr(&st->err, kErrNonPhys);
        atomicMin(&st->err_cell, cell);
      } else if (mode & kModeAlpha) {
#pragma unroll
        for (int d = 0; d < NV - 2; ++d)
          if (okey(s[d]) > okey(amax[d])) amax[d] = s[d];  // non-negative: bits order like values
      }
    } else if (!isfinite(unew[0])) {
      atomicOr(&st->err, kErrNonPhys);
      atomicMin(&st->err_cell, cell);
    }
  }
}

// Per-field variant (last stage only): the state check, and per axis the
// maxima of |u_d - c|, |u_d| and |u_d + c| in amax[3 d + 0..2], in FP32 like
// the one-alpha path's |u_d| + c.
template <int NV>
__device__ __forceinline__ void bulk_state_check(const SweepArgs& A, long long cell,
                                                 const double (&unew)[NV], int mode,
                                                 double (&amax)[9]) {
  StepState* st = A.st;
  if (A.stage != 2) return;
  if constexpr (NV > 1) {
    double s[9];
    if (!speeds32<NV, true>(unew, A.gamma, s)) {
      atomicOr(&st->err, kErrNonPhys);
      atomicMin(&st->err_cell, cell);
    } else if (mode & kModeAlpha) {
#pragma unroll
      for (int k = 0; k < 3 * (NV - 2); ++k)
        if (okey(s[k]) > okey(amax[k])) amax[k] = s[k];
    }
  }
}

// The axis class and the mode bits that a sweep kernel of a given shape
// (enoao_internal.h) knows at compile time; kShapeAny takes both from its
// arguments.
template <int SHAPE>
__device__ __forceinline__ bool shape_x(const SweepArgs& A) {
  if constexpr (SHAPE == kShapeXStore || SHAPE == kShapeXCombine) return true;
  if constexpr (SHAPE == kShapeYStore || SHAPE == kShapeYCombine) return false;
  return A.dir == 0;
}
template <int SHAPE>
__device__ __forceinline__ int shape_mode(const SweepArgs& A) {
  if constexpr (SHAPE == kShapeXStore) return kModeRhsStore;
  if constexpr (SHAPE == kShapeXCombine) return kModeCombine | (A.mode & kModeAlpha);
  if constexpr (SHAPE == kShapeYStore) return kModeRhsStore | kModeRhsAdd;
  if constexpr (SHAPE == kShapeYCombine) return kModeCombine | kModeRhsAdd | (A.mode & kModeAlpha);
  if constexpr (SHAPE == kShapeFlux) return kModeFlux;
  return A.mode;
}

// FP64 path: whether FP32 bounds show a new state to be physical and, when the
// next alpha is being taken, its |u_d| + c to be no more than the maxima so
// far (some 33 FP64 operations per cell of a combining sweep otherwise, of about
// 190; 2048^2 step 8.60 -> 8.08 ms).  The margins (1e-5 and 1e-6 of the summed magnitudes) cover the FP32
// rounding of every operation; NaN, infinities and values beyond FP32's range
// are never shown.
template <int NV, int KA>
__device__ __forceinline__ bool state_is_plain(const double (&u)[NV], float gm1, bool alpha,
                                               const double (&amax)[KA]) {
  const float rho = f32_rn(u[0]), E = f32_rn(u[NV - 1]);
  float m[NV], m2 = 0.0f;
#pragma unroll
  for (int c = 1; c < NV - 1; ++c) {
    m[c] = f32_rn(u[c]);
    m2 = fmaf(m[c], m[c], m2);
  }
  const float ir = __fdividef(1.0f, rho), ke = 0.5f * m2 * ir;
  const float ei = E - ke, sum = E + ke;
  bool ok = rho > 1e-30f && sum < 1e30f && ei > 1e-5f * sum;
  if (alpha) {
    const float c = sqrtf((1.0f + gm1) * gm1 * fmaf(1e-6f, sum, ei) * ir);
#pragma unroll
    for (int d = 0; d < NV - 2; ++d) {
      const float s = fmaf(fabsf(m[1 + d]), ir, c);
      ok = ok && s * 1.00001f <= f32_rn(amax[d]);
    }
  }
  return ok;
}

// Number of alpha maxima a sweep accumulates: |u_d| + c per axis, or with
// per-field constants |u_d - c|, |u_d|, |u_d + c| per axis.
template <bool FIELD>
constexpr int kAmax = FIELD ? 9 : 3;

// Entry of a tile's face list: line, face and the near-tie flags of the face's
// choices (bit field * 2 + sign).
__device__ __forceinline__ unsigned face_entry(int a, int f) {
  return (unsigned)a << 26 | (unsigned)f << 10;
}
__device__ __forceinline__ int entry_line(unsigned e) { return (int)(e >> 26); }
__device__ __forceinline__ int entry_face(unsigned e) { return (int)(e >> 10 & 0xffffu); }
__device__ __forceinline__ unsigned entry_flags(unsigned e) { return e & 0x3ffu; }

// The shared-memory planes of a tile, sizes as sweep_smem_bytes: per extended
// cell the split differences df+ and df-, the face correction C, the Roe
// ingredients, in FP32 bulk with kProve the magnitude of the pair's split
// differences, and one word for the face list (faces not proven, or with
// flagged choices).  The 1D system keeps the magnitude with df+ and two of its three
// Roe ingredients with df- and C (the spare values).  Shared by the tile's
// phases and the out-of-line re-decision.
template <int NV, int ORDER, typename R, bool FIELD>
struct TileView {
  using GE = Geo<ORDER>;
  using CV = CellVec<NV, R, FIELD>;
  static constexpr bool FP32 = sizeof(R) == 4;
  static constexpr bool MAG = FP32 && kProve<FIELD> && NV != 3;
  R* dfp;
  R* dfm;
  R* Cf;
  R* prim;         // 1D FP32: the third ingredient only
  float* mag;      // MAG
  unsigned* list;
  int cells, SE;
  __device__ __forceinline__ TileView(unsigned char* smem_raw, int ta, int se)
      : cells(tile_cells(ta, se)), SE(se) {
    dfp = reinterpret_cast<R*>(smem_raw);
    dfm = dfp + CV::kSlots * cells;
    Cf = dfm + CV::kSlots * cells;
    prim = Cf + CV::kSlots * cells;
    R* p = prim + (NV == 1 ? 0 : (CV::kSpare ? 1 : NV)) * cells;
    mag = reinterpret_cast<float*>(p);
    if constexpr (MAG) p += cells;
    list = reinterpret_cast<unsigned*>(p);
  }
  // Roe ingredients of the cell at slot i
  __device__ __forceinline__ void load_prims(int i, R (&pr)[NV]) const {
    if constexpr (CV::kSpare) {
      pr[0] = dfm[4 * i + 3];
      pr[1] = Cf[4 * i + 3];
      pr[2] = prim[i];
    } else {
      CV::load(prim, cells, i, pr);
    }
  }
  __device__ __forceinline__ int sidx(int a, int e) const { return a * SE + e; }
  // Projected window of face j (extended cells) onto the field with left
  // eigenvector row L: sign 0 is the f^+ window centred on cell j, sign 1 the
  // mirrored f^- window centred on cell j+1 (d[i] = -(L df^-) at j+4-i).
  __device__ __forceinline__ void window(int a, int j, int sgn, const R (&L)[NV], R (&d)[8]) const {
    const R* src = sgn == 0 ? dfp : dfm;
#pragma unroll
    for (int i = 0; i < 8; ++i) d[i] = R(0);
#pragma unroll
    for (int i = GE::LO; i <= GE::HI; ++i) {
      const int e = sidx(a, sgn == 0 ? j - 4 + i : j + 4 - i);
      R x[NV];
      CV::load(src, cells, e, x);
      R acc = R(0);
#pragma unroll
      for (int c = 0; c < NV; ++c) acc = fma(L[c], x[c], acc);
      d[i] = sgn == 0 ? acc : -acc;
    }
  }
  // the same window with the magnitudes sum_c |L_c| |df_c| of its terms
  __device__ __forceinline__ void window_mag(int a, int j, int sgn, const R (&L)[NV], R (&d)[8],
                                             R (&m)[8]) const {
    const R* src = sgn == 0 ? dfp : dfm;
#pragma unroll
    for (int i = 0; i < 8; ++i) d[i] = m[i] = R(0);
#pragma unroll
    for (int i = GE::LO; i <= GE::HI; ++i) {
      const int e = sidx(a, sgn == 0 ? j - 4 + i : j + 4 - i);
      R x[NV];
      CV::load(src, cells, e, x);
      R acc = R(0), mag = R(0);
#pragma unroll
      for (int c = 0; c < NV; ++c) {
        acc = fma(L[c], x[c], acc);
        mag = fma(rabs(L[c]), rabs(x[c]), mag);
      }
      d[i] = sgn == 0 ? acc : -acc;
      m[i] = mag;
    }
  }
  // The same for shear field v, whose left row is e_v - w e_0 (w its
  // tangential Roe velocity): one multiply-add per difference instead of NV.
  __device__ __forceinline__ void window_shear(int a, int j, int sgn, int v, R w, R (&d)[8],
                                               R (&m)[8]) const {
    if constexpr (NV >= 4) {
      const R* src = sgn == 0 ? dfp : dfm;
#pragma unroll
      for (int i = 0; i < 8; ++i) d[i] = m[i] = R(0);
#pragma unroll
      for (int i = GE::LO; i <= GE::HI; ++i) {
        const int e = sidx(a, sgn == 0 ? j - 4 + i : j + 4 - i);
        R x[NV];
        CV::load(src, cells, e, x);
        const R xv = shear_comp<NV>(x, v);
        const R acc = fma(-w, x[0], xv);
        d[i] = sgn == 0 ? acc : -acc;
        if constexpr (FP32) m[i] = fma(rabs(w), rabs(x[0]), rabs(xv));
      }
    }
  }
  // Per-field windows: dfp / dfm hold dF/2 and dq/2; field v splits after the
  // projection, d = L dF/2 +- alpha_v L dq/2 (sign 0: +, sign 1: mirrored -),
  // with magnitude sum |L||dF/2| + alpha_v sum |L||dq/2| for the near-tie bound.
  __device__ __forceinline__ void window_field(int a, int j, int sgn, int v, const R (&L)[NV], R w,
                                               R av, R (&d)[8], R (&m)[8]) const {
    const bool shear = NV >= 4 && v >= 2 && v <= NV - 2;
    const R sa = sgn == 0 ? av : -av;
#pragma unroll
    for (int i = 0; i < 8; ++i) d[i] = m[i] = R(0);
#pragma unroll
    for (int i = GE::LO; i <= GE::HI; ++i) {
      const int e = sidx(a, sgn == 0 ? j - 4 + i : j + 4 - i);
      R xF[NV], xq[NV];
      CV::load(dfp, cells, e, xF);
      CV::load(dfm, cells, e, xq);
      R aF = R(0), aq = R(0), mF = R(0), mq = R(0);
      if constexpr (NV >= 4) {
        if (shear) {
          const R fv = shear_comp<NV>(xF, v), qv = shear_comp<NV>(xq, v);
          aF = fma(-w, xF[0], fv);
          aq = fma(-w, xq[0], qv);
          if constexpr (FP32) {
            mF = rabs(fv) + rabs(w) * rabs(xF[0]);
            mq = rabs(qv) + rabs(w) * rabs(xq[0]);
          }
        }
      }
      if (!shear) {
#pragma unroll
        for (int c = 0; c < NV; ++c) {
          aF = fma(L[c], xF[c], aF);
          aq = fma(L[c], xq[c], aq);
          if constexpr (FP32) {
            mF += rabs(L[c]) * rabs(xF[c]);
            mq += rabs(L[c]) * rabs(xq[c]);
          }
        }
      }
      const R acc = fma(sa, aq, aF);
      d[i] = sgn == 0 ? acc : -acc;
      m[i] = fma(av, mq, mF);
    }
  }
  // Projected window of field v (the same arithmetic in phase 2 and in the
  // phase-2b check of a flagged choice, which must reproduce its pick).
  __device__ __forceinline__ void field_window(int a, int j, int sgn, int v, const R (&L)[NV], R w,
                                               R av, R (&d)[8], R (&mag)[8]) const {
    const bool shear = NV >= 4 && v >= 2 && v <= NV - 2;
    if constexpr (FIELD) {
      window_field(a, j, sgn, v, L, w, av, d, mag);
      return;
    }
    (void)av;
    if (shear) {
      window_shear(a, j, sgn, v, w, d, mag);
    } else if constexpr (FP32) {
      window_mag(a, j, sgn, L, d, mag);
    } else {
      window(a, j, sgn, L, d);
#pragma unroll
      for (int i = 0; i < 8; ++i) mag[i] = R(0);
    }
  }
};

// Roe average and eigenvectors of the face at slot i (between cells i and i+1).
template <int NV, int ORDER, typename R, bool FIELD>
__device__ __forceinline__ void face_eigen(const TileView<NV, ORDER, R, FIELD>& tv, int i, R gm1,
                                           Eigen<NV, R>& E) {
  R pl[NV], prr[NV];
  tv.load_prims(i, pl);
  tv.load_prims(i + 1, prr);
  roe_eigen<NV, R>(pl, prr, gm1, E);
}

// Phase 2a on one face (between cells j and j+1 of its line; x is its slot):
// proves that every characteristic field takes the top candidate for both
// signs, and if so gives the correction C they make, with the operations (and
// the bits) of choose_face but without its indicators, selection and bounds.
//
// The top candidate's indicator is at most |L_v . D|, D the undivided
// difference of df+- over the window's five (ENO-AO7: seven) middle pairs; D
// carries an FP32 error of at most feps times the Pascal sum P of the pairs'
// magnitudes, so |L_v . D| one of at most K feps P, K the largest entry of the
// left rows.  When |L_v . D| + K feps P is below delta by more than the
// near-tie margin, principle 1 of Sec. 3.2 picks the top candidate without a
// near-tie.  One difference decides a field instead of two per candidate and
// their bounds; the faces of resolved flow end here (98 to 99.5 % of 2D data
// at 2048^2 and more), the others go to the tile's face list.  The sweeps are
// bound by issue slots: 1,440 instructions per face and cell before, 815 (x)
// and 1,060 (y) with it; 4096^2 ENO-AO5 sweeps 0.81 -> 0.52 ms (x, 2 x 120
// tiles) and 1.00 -> 0.69 ms (y, 16 x 15), 512^3 ENO-AO7 stage 54 -> 28 ms.
// (Without the projection, as the FP64 path does it, they took 0.41 and 0.60
// ms; but R (L s) and s differ by FP32 rounding, which later stages' near-ties
// turn into other choices.)
// FRONTS: return as soon as the first sign's differences fail.  For the listing
// sweeps, whose flows leave most faces of a tile unproven (2D Riemann
// configuration 1, 800^2, late: ENO-AO5 701 -> 691, ENO-AO7 1175 -> 1145 us a step with
// the ENO-AO7 registers below); on resolved flow the branch costs a little (4096^2
// ENO-AO5 step 4.47 -> 4.53 ms), so the others do without.
template <int NV, int ORDER, bool FIELD, bool FRONTS>
__device__ __forceinline__ bool prove_top(const TileView<NV, ORDER, float, FIELD>& tv, int x,
                                          float gm1, float limit, float (&C)[NV]) {
  using CV = CellVec<NV, float, FIELD>;
  constexpr int H = ORDER == 7 ? 3 : 2;  // pairs j-H .. j+H
  constexpr float feps = (NV + 8) * FLT_EPSILON;
  constexpr float bw[4] = {1.0f, ORDER == 7 ? -6.0f : -4.0f, ORDER == 7 ? 15.0f : 6.0f, -20.0f};
  // window entries i whose Table-1 coefficients are nonzero
  constexpr int B0 = ORDER == 5 ? 2 : 1, B1 = ORDER == 5 ? 5 : 6;
  constexpr int ND = NV == 1 ? 1 : 3;       // dense rows: u-c, entropy, u+c
  constexpr int NS = NV > 3 ? NV - 3 : 0;   // shear fields
  float L[ND][NV], vt[NS > 0 ? NS : 1], K = 1.0f;
  Eigen<NV, float> E;
  if constexpr (NV > 1) {
    face_eigen<NV, ORDER, float, FIELD>(tv, x, gm1, E);
    left_row<NV, float>(E, 0, L[0]);
    left_row<NV, float>(E, 1, L[1]);
    left_row<NV, float>(E, NV - 1, L[2]);
#pragma unroll
    for (int t = 0; t < NS; ++t) {
      vt[t] = E.vt[t];
      K = fmaxf(K, fabsf(vt[t]));
    }
    // (the acoustic rows' later entries are halves of the entropy row's)
    K = fmaxf(K, fmaxf(fmaxf(fabsf(L[0][0]), fabsf(L[2][0])), fmaxf(fabsf(L[0][1]), fabsf(L[2][1]))));
#pragma unroll
    for (int c = 0; c < NV; ++c) K = fmaxf(K, fabsf(L[1][c]));
  } else {
    L[0][0] = 1.0f;
  }
  float m[2 * H + 1];
  float cv[ND], cs[NS > 0 ? NS : 1];  // values of the dense and the shear fields
  bool ok = true;
  float most = 0.0f;  // the largest |L_v . D|
#pragma unroll
  for (int sgn = 0; sgn < 2; ++sgn) {
    const float* src = sgn == 0 ? tv.dfp : tv.dfm;
    float D[NV], corr[ND], corrs[NS > 0 ? NS : 1];
#pragma unroll
    for (int c = 0; c < NV; ++c) D[c] = 0.0f;
#pragma unroll
    for (int v = 0; v < ND; ++v) corr[v] = 0.0f;
#pragma unroll
    for (int t = 0; t < NS; ++t) corrs[t] = 0.0f;
    // pair j + k: window entry 4 + k of f^+ (sign 0), 4 - k of f^- (sign 1,
    // negated); in the order of the entries
#pragma unroll
    for (int i = 4 - H; i <= 4 + H; ++i) {
      const int k = sgn == 0 ? i - 4 : 4 - i;
      float p[NV];
      if constexpr (CV::kSpare) {
        const float4 t = reinterpret_cast<const float4*>(src)[x + k];
        p[0] = t.x, p[1] = t.y, p[2] = t.z;
        if (sgn == 0) m[k + H] = t.w;
      } else {
        CV::load(src, tv.cells, x + k, p);
        if (sgn == 0) m[k + H] = tv.mag[x + k];
      }
      const float w = bw[k <= 0 ? k + H : H - k];
#pragma unroll
      for (int c = 0; c < NV; ++c) D[c] = fmaf(w, p[c], D[c]);
      if (i >= B0 && i <= B1) {
        const float b = bcoef_top<ORDER, float>(i);
#pragma unroll
        for (int v = 0; v < ND; ++v) {
          float acc = 0.0f;
#pragma unroll
          for (int c = 0; c < NV; ++c) acc = fmaf(L[v][c], p[c], acc);
          corr[v] = fmaf(b, sgn == 0 ? acc : -acc, corr[v]);
        }
#pragma unroll
        for (int t = 0; t < NS; ++t) {
          const float acc = fmaf(-vt[t], p[0], p[2 + t]);
          corrs[t] = fmaf(b, sgn == 0 ? acc : -acc, corrs[t]);
        }
      }
    }
#pragma unroll
    for (int v = 0; v < ND; ++v) {
      float d = 0.0f;
#pragma unroll
      for (int c = 0; c < NV; ++c) d = fmaf(L[v][c], D[c], d);
      most = fmaxf(most, fabsf(d));
      ok = ok && d == d;  // fmaxf drops a NaN
      cv[v] = sgn == 0 ? corr[v] : cv[v] + corr[v];
    }
#pragma unroll
    for (int t = 0; t < NS; ++t) {
      const float d = fmaf(-vt[t], D[0], D[2 + t]);
      most = fmaxf(most, fabsf(d));
      cs[t] = sgn == 0 ? corrs[t] : cs[t] + corrs[t];
    }
    if (FRONTS && sgn == 0 && !(ok && most <= limit)) return false;
  }
  float P;
  if constexpr (ORDER == 7)
    P = fmaf(20.0f, m[3], fmaf(15.0f, m[2] + m[4], fmaf(6.0f, m[1] + m[5], m[0] + m[6])));
  else
    P = fmaf(6.0f, m[2], fmaf(4.0f, m[1] + m[3], m[0] + m[4]));
  if constexpr (NV == 1) {
    C[0] = cv[0];
  } else {
    // the fields in order: u-c, entropy, shear..., u+c
#pragma unroll
    for (int c = 0; c < NV; ++c) C[c] = 0.0f;
    float Rc[NV];
    right_col<NV, float>(E, 0, Rc);
#pragma unroll
    for (int c = 0; c < NV; ++c) C[c] = fmaf(Rc[c], cv[0], C[c]);
    right_col<NV, float>(E, 1, Rc);
#pragma unroll
    for (int c = 0; c < NV; ++c) C[c] = fmaf(Rc[c], cv[1], C[c]);
#pragma unroll
    for (int t = 0; t < NS; ++t) {
      C[2 + t] += cs[t];
      C[NV - 1] = fmaf(vt[t], cs[t], C[NV - 1]);
    }
    right_col<NV, float>(E, NV - 1, Rc);
#pragma unroll
    for (int c = 0; c < NV; ++c) C[c] = fmaf(Rc[c], cv[ND - 1], C[c]);
  }
  return ok && fmaf(K * feps, P, most) <= limit;  // false for NaN
}

// The same for the FP64 path: the proof in FP32 from the FP64 differences and
// ingredients (narrowed on the integer units: the FP64 unit, 1/64 of the FP32
// rate, bounds this path, and its issue slots are nine tenths idle), the
// correction in FP64.  The proof only decides; what it cannot decide with its
// margin goes through the FP64 indicators.  The margin, in units of eps = 2^-23:
// D is off by at most (NV + 8) P (narrowing, and sums of five or seven weighted
// terms), P the Pascal sum of |df|.  The left rows are off through c^2 = (gamma-1)
// (H - |v|^2/2), whose terms are each off by a few roundings of H -- H by 1.5
// (narrowing, weights, sum), |v|^2/2 by 5 (|u_l|, |u_r| <= sqrt(2 H), so also where
// their average cancels) -- that is by 6.5 h relative, h = (gamma-1) H / c^2 >= 1 (E.H
// E.b1); 8 h covers that and the entries' own products.  A row times D is then off
// by at most K (NV + 8 + 8 h) P, K the largest term of the rows' entries.  With every
// field on the top candidate R L = I, so the values need no projection: C is
// a sum of FP64 differences, 8 NV (ENO-AO7: 12 NV) operations instead of 500.
// 2048^2 ENO-AO5 sweeps: x 4.15 -> 1.13 ms, y 4.38 -> 1.20 ms (with choose64
// and the neighbours' shared 1 / density).
template <int NV, int ORDER, bool FIELD, bool FRONTS>
__device__ __forceinline__ bool prove_top(const TileView<NV, ORDER, double, FIELD>& tv, int x,
                                          float gm1, float limit, double (&C)[NV]) {
  using CV = CellVec<NV, double, FIELD>;
  constexpr int H = ORDER == 7 ? 3 : 2;  // pairs j-H .. j+H
  constexpr float bw[4] = {1.0f, ORDER == 7 ? -6.0f : -4.0f, ORDER == 7 ? 15.0f : 6.0f, -20.0f};
  constexpr int B0 = ORDER == 5 ? 2 : 1, B1 = ORDER == 5 ? 5 : 6;
  constexpr int ND = NV == 1 ? 1 : 3, NS = NV > 3 ? NV - 3 : 0;
  float L[ND][NV], vt[NS > 0 ? NS : 1], K = 1.0f, feps = (NV + 16) * FLT_EPSILON;
  if constexpr (NV > 1) {
    double p64[NV];
    float pl[NV], prr[NV];
    tv.load_prims(x, p64);
#pragma unroll
    for (int c = 0; c < NV; ++c) pl[c] = f32_rn(p64[c]);
    tv.load_prims(x + 1, p64);
#pragma unroll
    for (int c = 0; c < NV; ++c) prr[c] = f32_rn(p64[c]);
    Eigen<NV, float> E;
    roe_eigen<NV, float>(pl, prr, gm1, E);
    left_row<NV, float>(E, 0, L[0]);
    left_row<NV, float>(E, 1, L[1]);
    left_row<NV, float>(E, NV - 1, L[2]);
#pragma unroll
    for (int t = 0; t < NS; ++t) {
      vt[t] = E.vt[t];
      K = fmaxf(K, fabsf(vt[t]));
    }
    // bounds on the entries from the terms they are sums of (a left row's
    // rounding is relative to those)
    const float q = sqrtf(E.q2);
    K = fmaxf(K, fmaxf(fmaxf(1.0f + E.b2, 0.5f * fmaf(q, E.ic, E.b2)),
                       fmaxf(0.5f * fmaf(E.b1, q, E.ic), E.b1 * fmaxf(q, 1.0f))));
    feps = (NV + 8 + 8.0f * E.H * E.b1) * FLT_EPSILON;
  } else {
    L[0][0] = 1.0f;
  }
  bool ok = true;
#pragma unroll 1
  for (int sgn = 0; sgn < 2; ++sgn) {
    const double* src = sgn == 0 ? tv.dfp : tv.dfm;
    float D[NV], P = 0.0f;
#pragma unroll
    for (int c = 0; c < NV; ++c) D[c] = 0.0f;
#pragma unroll
    for (int k = -H; k <= H; ++k) {
      double p[NV];
      CV::load(src, tv.cells, x + k, p);
      const float w = bw[k <= 0 ? k + H : H - k];
#pragma unroll
      for (int c = 0; c < NV; ++c) {
        const float pc = f32_rn(p[c]);
        D[c] = fmaf(w, pc, D[c]);
        P = fmaf(fabsf(w), fabsf(pc), P);
      }
    }
    float d = 0.0f;
#pragma unroll
    for (int v = 0; v < ND; ++v) {
      float t = 0.0f;
#pragma unroll
      for (int c = 0; c < NV; ++c) t = fmaf(L[v][c], D[c], t);
      d = fmaxf(d, fabsf(t));
      ok = ok && t == t;  // fmaxf drops a NaN
    }
#pragma unroll
    for (int t = 0; t < NS; ++t) d = fmaxf(d, fabsf(fmaf(-vt[t], D[0], D[2 + t])));
    ok = ok && fmaf(K * feps, P, d) <= limit;  // false for NaN
  }
  if (!ok) return false;
#pragma unroll
  for (int sgn = 0; sgn < 2; ++sgn) {
    const double* src = sgn == 0 ? tv.dfp : tv.dfm;
    double corr[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) corr[c] = 0.0;
#pragma unroll
    for (int i = B0; i <= B1; ++i) {
      double p[NV];
      CV::load(src, tv.cells, x + (sgn == 0 ? i - 4 : 4 - i), p);
      const double b = bcoef_top<ORDER, double>(i);
#pragma unroll
      for (int c = 0; c < NV; ++c) corr[c] = fma(b, sgn == 0 ? p[c] : -p[c], corr[c]);
    }
#pragma unroll
    for (int c = 0; c < NV; ++c) C[c] = sgn == 0 ? corr[c] : C[c] + corr[c];
  }
  return true;
}

// The raw state of a tile staged in shared memory by TMA: conserved
// component c of line a at extended cell e is p[c rc + a ra + (e + xoff) re]
// (the layout of the copied box; xoff is the alignment slack of x boxes).
struct RawTile {
  const double* p = nullptr;
  int rc = 0, ra = 0, re = 0, xoff = 0;
};
struct NoHook {
  __device__ __forceinline__ void operator()() const {}
};

// What every tile of a stage's sweep shares: the splitting constant of the
// swept axis, the step size, and what follows from them in the bulk precision
// (made once, by one thread, and kept in shared memory: made per tile they
// cost every thread conversions on the FP64 unit).
template <typename R>
struct TileConst {
  double alpha_d, dt;
  R alpha;
  float dt32, wdt32;    // FP32 bulk combine: dt and the stage's weight of dt L
  float limit;          // bound of prove_top
  R inv_dx;
};
// With per-field constants also those of u-c, of entropy and shear, of u+c (a
// struct of its own: the longer one cost batches 0.5 %).
template <typename R>
struct FieldConst : TileConst<R> {
  R af[3];
};
template <bool FIELD, typename R>
struct SweepConst {
  using type = TileConst<R>;
};
template <typename R>
struct SweepConst<true, R> {
  using type = FieldConst<R>;
};
template <int ORDER, typename R>
__device__ __forceinline__ void tile_const(const SweepArgs& A, double alpha_d, double dt,
                                           TileConst<R>& k) {
  k.alpha_d = alpha_d;
  k.dt = dt;
  k.alpha = (R)alpha_d;
  k.inv_dx = bconst<R>(A.inv_dx, A.inv_dx_f);
  k.dt32 = f32_rn(dt);
  k.wdt32 = f32_rn((A.stage == 0 ? 1.0 : (A.stage == 1 ? 0.25 : 2.0 / 3.0)) * dt);
  // below delta by more than the near-tie margin (and the bound's own
  // rounding); FP64 has no near-ties and takes a margin of its own.  A delta
  // near the end of FP32's range, where narrowed differences vanish, proves
  // nothing.
  k.limit = !(A.delta_f >= 1e-30f) ? -1.0f : A.delta_f - fmaf(sizeof(R) == 4 ? A.tie_rel_f : 1e-3f, A.delta_f, 1e-3f * A.delta_f);
}

// Whether the tile is the one that writes face f (the face between two tiles
// belongs to the one on its right, the last face to the last).
__device__ __forceinline__ bool owns_face(const SweepArgs& A, const TileGeo& g, int f) {
  const long long gface = g.s0 + f;  // face index between cells gface-1 and gface
  return (gface <= g.nd) && (f < A.ts || gface == g.nd);
}
// Index of face f of line a in the face arrays.
__device__ __forceinline__ long long face_index(const TileGeo& g, int a, int f) {
  return g.fbase + (g.a0 + a) * g.fstride_a + (g.s0 + f) * g.fstride_d;
}

// Phase 2 of one face: its correction C by projection and selection of every
// field and sign; returns the choices that are near-ties (FP32 bulk).
template <int NV, int ORDER, typename R, bool COHERENT, bool FIELD, int SHAPE>
__device__ __forceinline__ unsigned choose_face(const SweepArgs& A, const TileGeo& g,
                                                const TileView<NV, ORDER, R, FIELD>& tv,
                                                const TileConst<R>& K, const int a, const int f) {
  using CV = CellVec<NV, R, FIELD>;
  constexpr int G = Geo<ORDER>::G;
  constexpr bool FP32 = sizeof(R) == 4;
  const int cells = tv.cells, mode = shape_mode<SHAPE>(A);
  R* const dfm = tv.dfm;
  R* const Cf = tv.Cf;
  auto sidx = [&](int aa, int e) { return tv.sidx(aa, e); };
  const R gm1 = bconst<R>(A.gm1, A.gm1_f);
  const R delta = bconst<R>(A.delta, A.delta_f);
  const R tie_rel = bconst<R>(A.tie_rel, A.tie_rel_f);
  // splitting constant of field v: alpha, or per field max |u_d - c|, |u_d|, |u_d + c|
  auto afield = [&](int v) {
    if constexpr (FIELD)
      return static_cast<const FieldConst<R>&>(K).af[v == 0 ? 0 : (v == NV - 1 ? 2 : 1)];
    return K.alpha;
  };
  const int j = G - 1 + f;  // face j+1/2 in extended cells
  Eigen<NV, R> E;
  if constexpr (NV > 1) face_eigen<NV, ORDER, R, FIELD>(tv, sidx(a, j), gm1, E);
  const bool own = owns_face(A, g, f);
  R C[NV];
#pragma unroll
  for (int c = 0; c < NV; ++c) C[c] = R(0);
  unsigned fix = 0;
#pragma unroll 1
  for (int v = 0; v < NV; ++v) {
    // shear fields (2D/3D Euler) have a sparse left row e_v - w e_0
    const bool shear = NV >= 4 && v >= 2 && v <= NV - 2;
    R L[NV], w = R(0);
    if constexpr (NV > 1) {
      left_row<NV, R>(E, v, L);
      if constexpr (NV >= 4) w = -L[0];
    } else {
      L[0] = R(1);
    }
    // f^+ then mirrored f^- window, one live at a time
    R cv = R(0);
    const R av = afield(v);
    if constexpr (FIELD) {
      // the face's centre part: - alpha_v L dq/2 of the face's own pair
      R xq[NV];
      CV::load(dfm, cells, sidx(a, j), xq);
      R aq = R(0);
      if constexpr (NV >= 4) {
        if (shear) aq = shear_comp<NV>(xq, v) - w * xq[0];
      }
      if (!shear) {
#pragma unroll
        for (int c = 0; c < NV; ++c) aq += L[c] * xq[c];
      }
      cv = -av * aq;
    }
#pragma unroll
    for (int sgn = 0; sgn < 2; ++sgn) {
      R d[8], mag[8];
      tv.field_window(a, j, sgn, v, L, w, av, d, mag);
      int pick;
      bool marg = false;
      R corr;
      if constexpr (FP32)
        corr = eno_select<ORDER, R, true>(d, delta, tie_rel, mag, R(NV + 8) * R(FLT_EPSILON), pick,
                                          marg);
      else
        corr = choose64<ORDER>(d, delta, A.delta_f, pick);
      if constexpr (FP32) {
        if (marg) fix |= 1u << (v * 2 + sgn);  // re-decided in FP64 (phase 2b or the pass)
      }
      if ((mode & kModeFlux) && A.idx_out && own)
        A.idx_out[(v * 2 + sgn) * A.nfaces + face_index(g, a, f)] = (int8_t)pick;
      cv += corr;
    }
    if constexpr (NV >= 4) {
      if (shear) {
        // column v of R is e_v + w e_{NV-1}
#pragma unroll
        for (int c = 2; c < NV - 1; ++c) C[c] += c == v ? cv : R(0);
        C[NV - 1] = fma(w, cv, C[NV - 1]);
        continue;
      }
    }
    if constexpr (NV > 1) {
      R Rc[NV];
      right_col<NV, R>(E, v, Rc);
#pragma unroll
      for (int c = 0; c < NV; ++c) C[c] = fma(Rc[c], cv, C[c]);
    } else {
      C[0] += cv;
    }
  }
  CV::store(Cf, cells, sidx(a, j), C);
  return fix;
}

// Lanes that share a face of a short list: one per field and sign.
template <int NV>
constexpr int kFaceLanes = NV == 1 ? 2 : (NV <= 4 ? 8 : 16);

// choose_face of a face whose choices are spread over the kFaceLanes lanes of
// an aligned group, lane r taking field r / 2, sign r % 2 (the operations of
// choose_face, so the same bits): a tile's list is mostly a few faces, which
// one per thread would leave to a few lanes, each with ten dependent
// selections (FP64 1D sweep of 2000 cells 31 -> 19 us).  Lists longer than one
// round of groups go one face per lane, where no lane idles and the face's
// eigenvectors are formed once.  Every lane of the warp calls it; valid is the same over a group.
template <int NV, int ORDER, typename R, bool COHERENT, int SHAPE>
__device__ __forceinline__ unsigned choose_face_group(const SweepArgs& A, const TileGeo& g,
                                                      const TileView<NV, ORDER, R, false>& tv,
                                                      const int a, const int f, const bool valid) {
  using CV = CellVec<NV, R, false>;
  using GE = Geo<ORDER>;
  constexpr int G = GE::G, W = kFaceLanes<NV>;
  constexpr bool FP32 = sizeof(R) == 4;
  const unsigned FULL = 0xffffffffu;
  const int r = threadIdx.x & (W - 1);
  const int v = r >> 1 < NV ? r >> 1 : 0, sgn = r & 1;
  const R gm1 = bconst<R>(A.gm1, A.gm1_f);
  const int j = G - 1 + f, x = tv.sidx(a, j);
  Eigen<NV, R> E;
  const bool shear = NV >= 4 && v >= 2 && v <= NV - 2;
  R L[NV], w = R(0);
  if constexpr (NV > 1) {
    face_eigen<NV, ORDER, R, false>(tv, x, gm1, E);
    left_row<NV, R>(E, v, L);
    if constexpr (NV >= 4) w = -L[0];
  } else {
    L[0] = R(1);
  }
  R d[8], mag[8];
  const R* src = sgn == 0 ? tv.dfp : tv.dfm;
#pragma unroll
  for (int i = 0; i < 8; ++i) d[i] = mag[i] = R(0);
#pragma unroll
  for (int i = GE::LO; i <= GE::HI; ++i) {
    R q[NV], acc = R(0), m = R(0);
    CV::load(src, tv.cells, x + (sgn == 0 ? i - 4 : 4 - i), q);
    if constexpr (NV >= 4) {
      if (shear) {
        const R qv = shear_comp<NV>(q, v);
        acc = fma(-w, q[0], qv);
        if constexpr (FP32) m = fma(rabs(w), rabs(q[0]), rabs(qv));
      }
    }
    if (!shear) {
#pragma unroll
      for (int c = 0; c < NV; ++c) {
        acc = fma(L[c], q[c], acc);
        if constexpr (FP32) m = fma(rabs(L[c]), rabs(q[c]), m);
      }
    }
    d[i] = sgn == 0 ? acc : -acc;
    mag[i] = m;
  }
  int pick;
  bool marg = false;
  R corr;
  if constexpr (FP32)
    corr = eno_select<ORDER, R, true>(d, A.delta_f, A.tie_rel_f, mag, R(NV + 8) * R(FLT_EPSILON),
                                      pick, marg);
  else
    corr = choose64<ORDER>(d, A.delta, A.delta_f, pick);
  const bool mine = valid && r < 2 * NV;
  if ((shape_mode<SHAPE>(A) & kModeFlux) && A.idx_out && mine && owns_face(A, g, f))
    A.idx_out[r * A.nfaces + face_index(g, a, f)] = (int8_t)pick;
  const R cv = corr + __shfl_xor_sync(FULL, corr, 1);  // f^+ and f^- of the field
  R C[NV];
#pragma unroll
  for (int c = 0; c < NV; ++c) C[c] = R(0);
#pragma unroll
  for (int k = 0; k < NV; ++k) {  // the fields in order
    const R ck = __shfl_sync(FULL, cv, 2 * k, W);
    if constexpr (NV == 1) {
      C[0] += ck;
    } else if (k >= 2 && k <= NV - 2) {
      C[k] += ck;
      C[NV - 1] = fma(E.vt[k >= 2 ? k - 2 : 0], ck, C[NV - 1]);
    } else {
      R Rc[NV];
      right_col<NV, R>(E, k, Rc);
#pragma unroll
      for (int c = 0; c < NV; ++c) C[c] = fma(Rc[c], ck, C[c]);
    }
  }
  if (valid && r == 0) CV::store(tv.Cf, tv.cells, x, C);
  if constexpr (FP32) {
    const unsigned all = __ballot_sync(FULL, marg && r < 2 * NV);
    return all >> (threadIdx.x & 31 & ~(W - 1)) & ((1u << (2 * NV)) - 1u);
  }
  return 0u;
}

// Phase 2 of the faces on the tile's list (kProve), one per thread, or by
// groups of lanes when the list is short enough for one round of them; their
// near-ties go into the list's entries.  Returns whether this
// thread met one.
template <int NV, int ORDER, typename R, bool COHERENT, int SHAPE>
__device__ __forceinline__ bool listed_faces(const SweepArgs& A, const TileGeo& g,
                                             unsigned char* smem_raw, const TileConst<R>& K,
                                             int n) {
  const TileView<NV, ORDER, R, false> tv(smem_raw, A.ta, A.se);
  bool any = false;
  constexpr int W = kFaceLanes<NV>;
  if (n * W <= (int)blockDim.x) {  // a group of lanes per face, one round
    const int i = threadIdx.x / W;
    if ((int)(threadIdx.x & ~31u) < n * W) {  // warps with a face
      const bool valid = i < n;
      const unsigned entry = tv.list[valid ? i : 0];
      const unsigned fix = choose_face_group<NV, ORDER, R, COHERENT, SHAPE>(
          A, g, tv, entry_line(entry), entry_face(entry), valid);
      if (fix && valid) {
        if ((threadIdx.x & (W - 1)) == 0) tv.list[i] = entry | fix;
        any = true;
      }
    }
    return any;
  }
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const unsigned entry = tv.list[i];
    const unsigned fix = choose_face<NV, ORDER, R, COHERENT, false, SHAPE>(
        A, g, tv, K, entry_line(entry), entry_face(entry));
    if (fix) {
      tv.list[i] = entry | fix;
      any = true;
    }
  }
  return any;
}
// The same out of line: most tiles have no such face, and the projection and
// selection code then neither sets the register budget of the other phases nor
// stands between them in the instruction cache.
template <int NV, int ORDER, bool COHERENT, int SHAPE>
__device__ __noinline__ bool listed_faces_call(const SweepArgs& A, const TileGeo& g,
                                               unsigned char* smem_raw, const TileConst<float>& K,
                                               int n) {
  return listed_faces<NV, ORDER, float, COHERENT, SHAPE>(A, g, smem_raw, K, n);
}

// Phase 2 of a tile without the proof: every face, one per thread; returns whether
// this thread met a near-tie.
template <int NV, int ORDER, typename R, bool COHERENT, bool FIELD, int SHAPE>
__device__ __forceinline__ bool all_faces(const SweepArgs& A, const TileGeo& g,
                                            unsigned char* smem_raw, const TileConst<R>& K,
                                            int lgTA, bool sfast, int* nlist) {
  const TileView<NV, ORDER, R, FIELD> tv(smem_raw, A.ta, A.se);
  bool any = false;
  for_items(lgTA, g.nts + 1, sfast, [&](const int a, const int f) {
    if (g.a0 + a >= g.na) return;
    const unsigned fix = choose_face<NV, ORDER, R, COHERENT, FIELD, SHAPE>(A, g, tv, K, a, f);
    if constexpr (sizeof(R) == 4) {
      if (fix) {
        tv.list[atomicAdd(nlist, 1)] = face_entry(a, f) | fix;
        any = true;
      }
    }
  });
  return any;
}
// The same out of line (per-field constants, FP32, 2D): its two projections per window cell otherwise
// spill in the other phases too (1024^2 ENO-AO7 x and y sweeps 133 -> 129 and
// 139 -> 136 us).  3D (96^3 ENO-AO5 stage 615 -> 657 us) and FP64, which has the
// registers (1.60 -> 1.68 ms), stay inline.
template <int NV, int ORDER, bool COHERENT, int SHAPE>
__device__ __noinline__ bool field_faces_call(const SweepArgs& A, const TileGeo& g,
                                              unsigned char* smem_raw, const TileConst<float>& K,
                                              int lgTA, bool sfast, int* nlist) {
  return all_faces<NV, ORDER, float, COHERENT, true, SHAPE>(A, g, smem_raw, K, lgTA, sfast, nlist);
}

// Phase 2b of a tile (FP32 bulk, near-ties re-decided in the sweep): the
// flagged choices are re-decided from the FP64 state by lane groups of the
// warp (redo_group), or lane by lane when a warp has many (redo_lane), then
// each face applies the changes of its chosen values to its correction C in a
// fixed field/sign order.  Out of line: only tiles with flagged choices call
// it, and its FP64 code does not raise the register footprint of the common
// path.  Ends with a block barrier.
template <int NV, int ORDER, bool COHERENT, bool FIELD, int SHAPE>
__device__ __forceinline__ void redecide_tile(const SweepArgs& A, const TileGeo& g,
                                              unsigned char* smem_raw, int nlist, double alpha_d,
                                              unsigned long long& nfall) {
  using R = float;
  using GE = Geo<ORDER>;
  using CV = CellVec<NV, R, FIELD>;
  constexpr int G = GE::G;
  StepState* st = A.st;
  const TileView<NV, ORDER, R, FIELD> tv(smem_raw, A.ta, A.se);
  R* Cf = tv.Cf;
  const int cells = tv.cells;
  auto sidx = [&](int a, int e) { return tv.sidx(a, e); };
  const int mode = shape_mode<SHAPE>(A);
  const R gm1 = bconst<R>(A.gm1, A.gm1_f);
  const R delta = bconst<R>(A.delta, A.delta_f);
  const R tie_rel = bconst<R>(A.tie_rel, A.tie_rel_f);
  const R alpha = (R)alpha_d;
  R alo = alpha, amid = alpha, ahi = alpha;
  if constexpr (FIELD) {
    alo = (R)st->alpha_f[A.dir][0];
    amid = (R)st->alpha_f[A.dir][1];
    ahi = (R)st->alpha_f[A.dir][2];
  }
  auto afield = [&](int v) { return v == 0 ? alo : (v == NV - 1 ? ahi : amid); };
  auto alpha64 = [&](int v) {
    if constexpr (FIELD) return field_alpha<NV>(st, A.dir, v);
    return alpha_d;
  };
  auto field_window = [&](int a, int j, int sgn, int v, const R (&L)[NV], R w, R av, R (&d)[8],
                          R (&mag)[8]) { tv.field_window(a, j, sgn, v, L, w, av, d, mag); };
  constexpr int W = 2 * G <= 8 ? 8 : 16;  // lanes per re-decision group
  constexpr int NG = 32 / W;
  constexpr int kFewRounds = ORDER == 7 ? 3 : 2;  // rounds of redo_group that cost a lone one
  const unsigned FULL = 0xffffffffu;
  const int bd = blockDim.x, tid = threadIdx.x, lane = tid & 31;
  // The flagged entries to the front of the list (one warp, in place: an
  // entry never moves behind one not yet read), so that the choices of a
  // warp's faces below fill its lanes.
  __shared__ int s_nflag, s_nchoice;
  if (tid < 32) {
    int n = 0;
    unsigned nc = 0;
    for (int base = 0; base < nlist; base += 32) {
      const unsigned e = base + lane < nlist ? tv.list[base + lane] : 0u;
      const unsigned m = __ballot_sync(FULL, entry_flags(e) != 0u);
      if (entry_flags(e)) tv.list[n + __popc(m & ((1u << lane) - 1u))] = e;
      n += __popc(m);
      nc += __popc(entry_flags(e));
      __syncwarp();
    }
    nc = __reduce_add_sync(FULL, nc);
    if (lane == 0) s_nflag = n, s_nchoice = (int)nc;
  }
  __syncthreads();
  // The warps that share them: a round of 32 choices each (redo_lane), or, of a
  // few choices, a round of NG (redo_group), which costs little more in all and
  // ends sooner.  In 32 faces a warp, whatever their choices, the first warps
  // took all and each scheduler's FP64 pipe but theirs stood idle: tiles along a
  // front then set the length of a sweep (1024^2 quadrant jumps, per-field
  // ENO-AO7 y sweep 309 -> 179 us, one-alpha ENO-AO5 stage 186 -> 152 us; composite
  // wave ENO-AO7 N = 400 33.3 -> 28.3 us a step).  Where a launch has no more tiles
  // than SMs nothing else would use the pipes: as many warps as there are
  // rounds of NG.  In a batch the blocks' other problems do: no more rounds in
  // all than one warp would take (1024 uneven problems, ENO-AO5: 1.00 ms a step
  // either way, 1.09 split as sweeps are).  By faces alone, without the choices'
  // number, sweeps with a choice or two a tile took longer than in one warp
  // (512^2 noise, ENO-AO5 stage 157 -> 163 us).
  const int nflag = s_nflag, nchoice = s_nchoice;
  const bool dense = A.redo_split == kSplitDense;
  const int few = A.redo_split == kSplitAll ? nchoice : (dense ? kFewRounds : 3) * NG;
  const int rounds = nchoice <= few ? (nchoice + NG - 1) / NG
                     : dense ? max(nchoice / 32, (nflag + 31) / 32) : (nchoice + 31) / 32;
  const int nw = min(bd >> 5, rounds);
  const int share = min(32, (nflag + nw - 1) / nw);  // faces of a warp at a time
  const int wid = tid >> 5;
  for (int base = wid < nw ? wid * share : nflag; base < nflag; base += nw * share) {
    const unsigned entry = lane < share && base + lane < nflag ? tv.list[base + lane] : 0u;
    const int al = entry_line(entry), f = entry_face(entry);
    const int j = G - 1 + f;
    unsigned fix = entry_flags(entry);
    // The warp's T choices in rounds (with each face's lane serving its own
    // flags, a warp took up to ten rounds for a few choices each: 256^3
    // ENO-AO7 x sweep 1.8 -> 1.0 ms, 800^2 0.23 -> 0.16 ms).  Many left: one per lane (redo_lane),
    // 32 in a round -- an instruction of the FP64 unit costs the same
    // whatever its active lanes.  A few left: NG per round, each by W lanes
    // together (redo_group), which takes about 2/5 (ENO-AO5) or 1/3 of the
    // instructions of a lone re-decision.  Every round clears at least one
    // choice, so the default bound (64 NV rounds) is never reached; a
    // smaller bound (a test knob) can be: then the error word says so and
    // the choices left keep their FP32 pick.
    const int m = __popc(fix);
    int pre = m;  // inclusive, then exclusive prefix sum over the lanes
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(FULL, pre, o);
      if (lane >= o) pre += t;
    }
    const int T = __shfl_sync(FULL, pre, 31);
    pre -= m;
    unsigned long long picks = 0ull;
    int done = 0;
    for (int pass = 0; done < T; ++pass) {
      if (pass >= A.redo_passes) {
        if (lane == 0) atomicOr(&st->err, kErrTimeout);
        break;
      }
      const bool lone = T - done > kFewRounds * NG;
      const int per = lone ? 32 : NG;
      // this lane's (its group's) choice of the round: number ci, of the
      // face of lane jl
      const int ci = done + (lone ? lane : lane / W);
      int jl = 0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {  // the last lane whose first choice is <= ci
        const int pq = __shfl_sync(FULL, pre, jl + o);
        if (pq <= ci) jl += o;
      }
      const unsigned mj = __shfl_sync(FULL, fix, jl);
      const int prej = __shfl_sync(FULL, pre, jl);
      const int aj = __shfl_sync(FULL, al, jl), fj = __shfl_sync(FULL, f, jl);
      const bool valid = ci < T;
      const int kb = valid ? nth_set_bit(mj, ci - prej) : 0;
      // (a group without a choice works on the face of the last one, unused)
      const int k = kb < 0 ? 0 : kb;
      int pick = 0;
      if (lone) {
        if (valid)
          pick = redo_lane<NV, ORDER, COHERENT>(A, g, aj, g.s0 + fj - 1, k >> 1, k & 1,
                                                alpha64(k >> 1));
      } else {
        pick = redo_group<NV, ORDER, COHERENT, W>(A, g, aj, g.s0 + fj - 1, k >> 1, k & 1,
                                                  alpha64(k >> 1), lane & (W - 1));
      }
      __syncwarp();
      // each face's lane collects its choices of the round
      unsigned todo = fix;
      int most = __reduce_max_sync(FULL, (unsigned)m);
      for (int t = 0; t < most; ++t) {
        const int c = pre + t - done;
        const int src = c >= 0 && c < per ? (lone ? c : c * W) : 0;
        const int got = __shfl_sync(FULL, pick, src);
        const int kk = todo ? __ffs(todo) - 1 : 0;
        todo &= todo - 1;
        if (t < m && c >= 0 && c < per) {
          picks |= (unsigned long long)got << (4 * kk);
          ++nfall;
        }
      }
      done += per;
    }
    // choices left by a pass bound keep their FP32 pick
    const int have = done - pre < 0 ? 0 : (done - pre < m ? done - pre : m);
    for (int t = m; t > have; --t) fix &= ~(1u << (31 - __clz(fix)));
    if (!fix) continue;
    // apply the changed choices of this face
    Eigen<NV, R> E;
    if constexpr (NV > 1) {
      face_eigen<NV, ORDER, R, FIELD>(tv, sidx(al, j), gm1, E);
    }
    const bool own = owns_face(A, g, f);
    R dC[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) dC[c] = R(0);
#pragma unroll 1
    for (int k = 0; k < 2 * NV; ++k) {
      if (!(fix & (1u << k))) continue;
      const int v = k >> 1, sgn = k & 1;
      const int pick = (int)((picks >> (4 * k)) & 15ull);
      const bool shear = NV >= 4 && v >= 2 && v <= NV - 2;
      R L[NV], w = R(0);
      if constexpr (NV > 1) {
        left_row<NV, R>(E, v, L);
        if constexpr (NV >= 4) w = -L[0];
      } else {
        L[0] = R(1);
      }
      R d[8], mag[8];
      field_window(al, j, sgn, v, L, w, afield(v), d, mag);
      int pick_old;
      bool m;
      const R nomx[8] = {R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0)};
      const R corr_old = eno_select<ORDER, R, false>(d, delta, tie_rel, nomx, R(0), pick_old, m);
      if (pick != pick_old) {
        R corr = R(0);
#pragma unroll
        for (int i = GE::LO; i <= GE::HI; ++i) corr = fma(bcoef<R>(pick, i), d[i], corr);
        const R dv = corr - corr_old;
        if (shear) {
#pragma unroll
          for (int c = 2; c < NV - 1; ++c) dC[c] += c == v ? dv : R(0);
          dC[NV - 1] = fma(w, dv, dC[NV - 1]);
        } else if constexpr (NV > 1) {
          R Rc[NV];
          right_col<NV, R>(E, v, Rc);
#pragma unroll
          for (int c = 0; c < NV; ++c) dC[c] = fma(Rc[c], dv, dC[c]);
        } else {
          dC[0] += dv;
        }
      }
      if ((mode & kModeFlux) && A.idx_out && own)
        A.idx_out[(v * 2 + sgn) * A.nfaces + face_index(g, al, f)] = (int8_t)pick;
    }
    const int sj = sidx(al, j);
    R Cv[NV];
    CV::load(Cf, cells, sj, Cv);
#pragma unroll
    for (int c = 0; c < NV; ++c) Cv[c] += dC[c];
    CV::store(Cf, cells, sj, Cv);
  }
  __syncthreads();
}

// The same, not inlined (only one copy of the code, called by the tiles that
// have flags): where the FP64 re-decision code would otherwise set the
// register budget of the whole tile.
template <int NV, int ORDER, bool COHERENT, bool FIELD, int SHAPE>
__device__ __noinline__ void redecide_tile_call(const SweepArgs& A, const TileGeo& g,
                                                unsigned char* smem_raw, int nlist, double alpha_d,
                                                unsigned long long& nfall) {
  redecide_tile<NV, ORDER, COHERENT, FIELD, SHAPE>(A, g, smem_raw, nlist, alpha_d, nfall);
}

// One tile of a sweep (phases 1-3 above).  amax accumulates |u_d| + c of
// combined states (last stage), nfall counts FP64 re-decisions.  FIELD: each
// characteristic field splits with its own constant (st->alpha_f): phase 1
// keeps dF/2 and dq/2, the split follows the projection, and the face's
// centre part 1/2 R diag(alpha) L dq moves into its correction C.
// TMA: phase 1 reads the tile's raw state from rt instead of global memory.
// PROOF: prove faces first, where the sweep can (kProve).
// hook() runs before the tile's last barrier, with TMA once every thread is
// past phase 1 (the raw buffer is then free for the next tile's copy).
template <int NV, int ORDER, typename R, bool COHERENT = false, bool DEFER = false,
          bool FIELD = false, bool TMA = false, int SHAPE = kShapeAny, typename Hook = NoHook,
          bool PROOF = true>
__device__ __forceinline__ void sweep_tile(const SweepArgs& A, const TileGeo& g,
                                           unsigned char* smem_raw, const TileConst<R>& K,
                                           double (&amax)[kAmax<FIELD>],
                                           unsigned long long& nfall, const RawTile& rt = RawTile{},
                                           Hook hook = Hook{}) {
  static_assert(!FIELD || NV >= 3, "per-field constants are for the Euler equations");
  using GE = Geo<ORDER>;
  constexpr int G = GE::G;
  constexpr bool FP32 = sizeof(R) == 4;
  constexpr bool PROVE = kProve<FIELD> && PROOF;
  // the code of faces not proven and of near-ties out of line
  constexpr bool CALL = FP32 && !FIELD && SHAPE != kShapeAny;
  StepState* st = A.st;
  const int TA = A.ta;
  // row pitch A.se (>= A.ts + 2G), chosen on the host for conflict-free banks
  const TileView<NV, ORDER, R, FIELD> tv(smem_raw, TA, A.se);
  const int cells = tv.cells;
  R* const dfp = tv.dfp;
  R* const dfm = tv.dfm;
  R* const Cf = tv.Cf;
  R* const prim = tv.prim;
  // faces on the tile's list (those not proven in phase 2a; per field, those
  // with flagged choices)
  __shared__ int s_nlist;
  if ((FP32 || PROVE) && threadIdx.x == 0) s_nlist = 0;

  const int dir = A.dir;
  const bool sfast = shape_x<SHAPE>(A);
  const double alpha_d = K.alpha_d, dt = K.dt;
  const R alpha = K.alpha;
  const R halpha = R(0.5) * alpha;
  const R gm1 = bconst<R>(A.gm1, A.gm1_f);
  const R adv = bconst<R>(A.adv_speed, A.adv_f);
  const int mode = shape_mode<SHAPE>(A);
  const R inv_dx_r = K.inv_dx;
  // FP32 bulk combine: dt and the stage's weight of dt L in FP32
  const float dt32 = K.dt32, wdt32 = K.wdt32;
  const float inc_w = A.stage == 1 ? -0.75f : -f32_rn(1.0 / 12.0);  // weight of the carried increment
  // Shared-memory rows of SE cells per line for every axis: unit stride
  // along the swept axis (window offsets are immediates); SE is odd, so the
  // y/z sweeps, whose lanes run across lines, hit distinct banks.
  auto sidx = [&](int a, int e) { return tv.sidx(a, e); };
  using CV = CellVec<NV, R, FIELD>;
  const int lgTA = __ffs(TA) - 1;  // TA is a power of two (checked on the host)
  const int nts = g.nts;
  const int sext = nts + 2 * G;  // extended cells in use
  // extended cell e of line a is cell ext0 + a sa + e sd, except ghosts of a
  // tile at the end of its lines
  const bool edge = A.bc != kBcHalo && (g.s0 < G || g.s0 + nts + G > g.nd);
  const cell_t<NV> sa = g.stride_a, sd = g.stride_d;
  const cell_t<NV> ext0 = g.base + g.a0 * g.stride_a + (g.s0 - G) * g.stride_d;

  // ---------------- phase 1: split differences and Roe ingredients
  {
    const int cnt = sext;
    // the tile's raw state: staged by TMA, or straight from global memory
    auto cell_state = [&](int a, int ee, double (&q)[NV]) {
      if constexpr (TMA) {
        const double* p = rt.p + a * rt.ra + (ee + rt.xoff) * rt.re;
#pragma unroll
        for (int c = 0; c < NV; ++c) q[c] = p[perm_comp<NV>(c, dir) * rt.rc];
      } else {
        cell_t<NV> cell = ext0 + (cell_t<NV>)a * sa + (cell_t<NV>)ee * sd;
        if (edge)
          cell = g.base + (g.a0 + a) * g.stride_a + bc_map(g.s0 - G + ee, g.nd, A.bc) * g.stride_d;
        load_state<NV, COHERENT>(A, cell, q);
      }
    };
    // cell e's Roe ingredients, and the split differences of the pair (e, e+1)
    auto prim_out = [&](int a, int e, const R (&qa)[NV], R ir) {
      if constexpr (NV > 1) {
        if (e >= G - 1 && e <= G + nts) {
          R pr[NV];
          roe_prims<NV, R>(qa, gm1, ir, pr);
          if constexpr (CV::kSpare) {
            dfm[4 * sidx(a, e) + 3] = pr[0];
            Cf[4 * sidx(a, e) + 3] = pr[1];
            prim[sidx(a, e)] = pr[2];
          } else {
            CV::store(prim, cells, sidx(a, e), pr);
          }
        }
      }
    };
    auto pair_out = [&](int a, int e, const double (&qa64)[NV], const R (&qa)[NV],
                        const double (&qb64)[NV], const R (&qb)[NV], R ia, R ib) {
      R fp[NV], fm[NV], m = R(0);
      if constexpr (FIELD)
        split_parts<NV, R>(qa64, qb64, qa, qb, gm1, adv, ia, ib, fp, fm);  // dF/2, dq/2
      else
        m = split_diff<NV, R>(qa64, qb64, qa, qb, gm1, adv, halpha, ia, ib, fp, fm);
      if constexpr (CV::kSpare) {
        CV::store4(dfp, sidx(a, e), fp, m);
        CV::store(dfm, cells, sidx(a, e), fm);  // its spare value: a Roe ingredient
      } else {
        CV::store(dfp, cells, sidx(a, e), fp);
        CV::store(dfm, cells, sidx(a, e), fm);
        if constexpr (PROVE && tv.MAG) tv.mag[sidx(a, e)] = m;
      }
    };
    if (sfast) {
      // x sweeps: lanes along the line (coalesced), one pair per item
      for_items(lgTA, cnt, sfast, [&](const int a, const int e) {
        if (g.a0 + a >= g.na) return;
        double qa64[NV];
        cell_state(a, e, qa64);
        R qa[NV];
#pragma unroll
        for (int c = 0; c < NV; ++c) qa[c] = to_bulk<R>(qa64[c]);
        const R ia = inv_density<NV>(qa);
        prim_out(a, e, qa, ia);
        if (e + 1 < cnt) {
          double qb64[NV];
          cell_state(a, e + 1, qb64);
          R qb[NV];
#pragma unroll
          for (int c = 0; c < NV; ++c) qb[c] = to_bulk<R>(qb64[c]);
          pair_out(a, e, qa64, qa, qb64, qb, ia, inv_density<NV>(qb));
        }
      });
    } else {
      // y/z sweeps: lanes across lines, so a thread can take a run of
      // consecutive cells of its line without losing coalescing; each cell
      // is then loaded and narrowed once (the right cell of one pair is the
      // left cell of the next), the run's last pair reaching one cell on
      int a, j0, step;
      item_start(lgTA, false, a, j0, step);
      const int run = (cnt + step - 1) >> (__ffs(step) - 1);  // step is a power of two
      int e = j0 * run;
      const int e_end = min(e + run, cnt);
      if (g.a0 + a < g.na && e < e_end) {
        double q64[NV];
        cell_state(a, e, q64);
        R q[NV];
#pragma unroll
        for (int c = 0; c < NV; ++c) q[c] = to_bulk<R>(q64[c]);
        R ir = inv_density<NV>(q);
        for (;; ++e) {
          prim_out(a, e, q, ir);
          if (e + 1 >= cnt) break;
          double n64[NV];
          cell_state(a, e + 1, n64);
          R n[NV];
#pragma unroll
          for (int c = 0; c < NV; ++c) n[c] = to_bulk<R>(n64[c]);
          const R in = inv_density<NV>(n);
          pair_out(a, e, q64, q, n64, n, ir, in);
          if (e + 1 >= e_end) break;
          ir = in;
#pragma unroll
          for (int c = 0; c < NV; ++c) {
            q64[c] = n64[c];
            q[c] = n[c];
          }
        }
      }
    }
  }
  __syncthreads();
  if constexpr (TMA) hook();

  // ---------------- phase 2a: prove the smooth faces, list the others
  const int nfaces_tile = nts + 1;
  bool any_fix = false;  // FP32 bulk: this thread flagged a near-tie
  if constexpr (PROVE) {
    for_items(lgTA, nfaces_tile, sfast, [&](const int a, const int f) {
      if (g.a0 + a >= g.na) return;
      const int x = sidx(a, G - 1 + f);
      R C[NV];
      if (prove_top<NV, ORDER, FIELD, DEFER>(tv, x, A.gm1_f, K.limit, C)) {
        CV::store(Cf, cells, x, C);
        if ((mode & kModeFlux) && A.idx_out && owns_face(A, g, f)) {
          const long long fc = face_index(g, a, f);
          for (int k = 0; k < 2 * NV; ++k) A.idx_out[k * A.nfaces + fc] = (int8_t)(GE::NC - 1);
        }
      } else {
        tv.list[atomicAdd(&s_nlist, 1)] = face_entry(a, f);
      }
    });
    __syncthreads();
  }

  // ---------------- phase 2: per face choice and back-projection
  {
    if constexpr (PROVE) {
      if (s_nlist > 0) {
        if constexpr (CALL)
          any_fix = listed_faces_call<NV, ORDER, COHERENT, SHAPE>(A, g, smem_raw, K, s_nlist);
        else
          any_fix = listed_faces<NV, ORDER, R, COHERENT, SHAPE>(A, g, smem_raw, K, s_nlist);
      }
    } else if constexpr (FIELD && FP32 && NV == 4) {
      any_fix = field_faces_call<NV, ORDER, COHERENT, SHAPE>(A, g, smem_raw, K, lgTA, sfast,
                                                             &s_nlist);
    } else {
      any_fix = all_faces<NV, ORDER, R, COHERENT, FIELD, SHAPE>(A, g, smem_raw, K, lgTA, sfast,
                                                                &s_nlist);
    }
  }

  // ---------------- phase 2b (FP32 bulk): the faces with flagged choices
  if constexpr (!FP32) {
    if (!PROVE || s_nlist > 0) __syncthreads();
  } else if (PROVE && s_nlist == 0) {
    // every face proven: C is complete since the barrier of phase 2a
  } else if constexpr (DEFER) {
    // list the faces that this tile owns for the grid-wide pass, which
    // corrects both cells of each, whichever tiles they lie in, so results do
    // not depend on tiles.  Nothing here changes Cf: phase 3 uses the FP32
    // choices.
    __syncthreads();
    const int n = s_nlist;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const unsigned entry = tv.list[i], fix = entry_flags(entry);
      if (!fix || !owns_face(A, g, entry_face(entry))) continue;
      const unsigned slot = atomicAdd(&st->redo_n, 1u);
      if (slot < A.redo_cap) {
        const long long fc = face_index(g, entry_line(entry), entry_face(entry));
        A.redo[slot] = ((unsigned long long)fc << 16) | fix;
      } else {
        atomicOr(&st->err, kErrRedoFull);
      }
    }
  } else {
    // FP64 re-decision of the tile's near-ties; only tiles with flagged
    // choices run it.
    if (__syncthreads_or(any_fix)) {
      if constexpr (CALL)
        redecide_tile_call<NV, ORDER, COHERENT, FIELD, SHAPE>(A, g, smem_raw, s_nlist, alpha_d, nfall);
      else
        redecide_tile<NV, ORDER, COHERENT, FIELD, SHAPE>(A, g, smem_raw, s_nlist, alpha_d, nfall);
    }
  }

  // ---------------- phase 3: flux difference and Runge-Kutta combine
  if (mode & kModeFlux) {
    const int cnt = nts + 1;
    const long long nf = A.nfaces;
    for_items(lgTA, cnt, sfast, [&](const int a, const int f) {
      if (g.a0 + a >= g.na) return;
      if (!owns_face(A, g, f)) return;
      const long long gface = g.s0 + f;
      const int j = G - 1 + f;
      const long long la = g.base + (g.a0 + a) * g.stride_a;
      double ql[NV], qr[NV], Fl[NV], Fr[NV];
      load_state<NV, COHERENT>(A, la + bc_map(gface - 1, g.nd, A.bc) * g.stride_d, ql);
      load_state<NV, COHERENT>(A, la + bc_map(gface, g.nd, A.bc) * g.stride_d, qr);
      phys_flux<NV>(ql, A.gm1, A.adv_speed, Fl);
      phys_flux<NV>(qr, A.gm1, A.adv_speed, Fr);
      const long long fc = face_index(g, a, f);
      R Cv[NV];
      CV::load(Cf, cells, sidx(a, j), Cv);
#pragma unroll
      for (int c = 0; c < NV; ++c) {
        if constexpr (FIELD) {
          // F^ = (F_l + F_r)/2 + C, the split's centre part being inside C
          A.fhat[perm_comp<NV>(c, dir) * nf + fc] = 0.5 * (Fl[c] + Fr[c]) + to_f64(Cv[c]);
        } else {
          const double fp = 0.5 * (Fl[c] + alpha_d * ql[c]);
          const double fm = 0.5 * (Fr[c] - alpha_d * qr[c]);
          A.fhat[perm_comp<NV>(c, dir) * nf + fc] = fp + fm + to_f64(Cv[c]);
        }
      }
    });
  } else {
    const int cnt = nts;
    for_items(lgTA, cnt, sfast, [&](const int a, const int t) {
      if (g.a0 + a >= g.na) return;
      const int e = G + t;
      const cell_t<NV> cell = ext0 + (cell_t<NV>)a * sa + (cell_t<NV>)e * sd;
      R r[NV];
      {
        R p0[NV], m1[NV], c1[NV], c0[NV];
        // per field: dF/2 of both of the cell's pairs (the centre part is in C)
        CV::load(dfp, cells, sidx(a, e - 1), p0);
        CV::load(FIELD ? dfp : dfm, cells, sidx(a, e), m1);
        CV::load(Cf, cells, sidx(a, e), c1);
        CV::load(Cf, cells, sidx(a, e - 1), c0);
#pragma unroll
        for (int c = 0; c < NV; ++c) {
          const R s = p0[c] + m1[c] + (c1[c] - c0[c]);
          r[c] = mul_rn(-s, inv_dx_r);
        }
      }
      // Every load of the cell comes first, each array's under one uniform
      // condition, so that all are in flight together; the stores follow (they
      // could alias the inputs as far as the compiler knows, and a load after
      // one would wait for it).
      const bool add = mode & kModeRhsAdd, combine = mode & kModeCombine;
      R o[NV];         // L(u) of the earlier axes
      double ui[NV];   // the stage's input
      float I[NV];     // FP32 bulk: the increment of the stage before
      double u0[NV];   // FP64: U^n
      if (add) {
#pragma unroll
        for (int c = 0; c < NV; ++c) o[c] = static_cast<const R*>(A.comp.rhs[c])[cell];
      }
      if (combine) {
        // (the batched kernel reads stage states it wrote itself: through L2)
#pragma unroll
        for (int c = 0; c < NV; ++c) {
          const double* p = A.comp.u_in[c] + cell;
          ui[c] = COHERENT ? __ldcg(p) : __ldg(p);
        }
        if (A.stage > 0) {
#pragma unroll
          for (int c = 0; c < NV; ++c) {
            if constexpr (FP32) {
              const float* p = A.comp.inc_in[c] + cell;
              I[c] = COHERENT ? __ldcg(p) : __ldg(p);
            } else {
              const double* p = A.comp.u0[c] + cell;
              u0[c] = COHERENT ? __ldcg(p) : __ldg(p);
            }
          }
        }
      }
      // L(u) summed over the axes in the bulk precision
      if (add) {
#pragma unroll
        for (int c = 0; c < NV; ++c) r[c] = o[c] + r[c];
      }
      if (!combine) {
#pragma unroll
        for (int c = 0; c < NV; ++c) static_cast<R*>(A.comp.rhs[c])[cell] = r[c];
        return;
      }
      double up[NV], unew[NV];
      float inc[NV];  // FP32 bulk: the increment this stage carries on
      if constexpr (FP32) {
        // Each stage as its own input u_i plus an FP32 increment, the step's
        // increments so far carried in FP32 (each is dt times an FP32-bulk
        // L(u)): with I0 = dt L(u0) and I1 = I0 + dt L(u1),
        //   u1 = u0 + I0
        //   u2 = u1 + (1/4 dt L(u1) - 3/4 I0)
        //   u3 = u2 + (2/3 dt L(u2) - 1/12 I1),
        // which are 3/4 u0 + 1/4 (u1 + dt L(u1)) and 1/3 u0 + 2/3 (u2 +
        // dt L(u2)) because u1 - u0 = I0 and u2 - u0 = I1 / 4 (up to FP64
        // rounding of u1 and u2).  One FP64 add per component (the FP64 unit
        // runs at 1/64 of the FP32 rate) and no read of U^n: the increments
        // take the bytes U^n took, and u_i was just read by phase 1.
        if (A.stage > 0) {
#pragma unroll
          for (int c = 0; c < NV; ++c) {
            inc[c] = fmaf(dt32, r[c], I[c]);  // I1 (stored by stage 1 only)
            up[c] = ui[c] + f64_of(fmaf(inc_w, I[c], wdt32 * r[c]));
          }
        } else {
#pragma unroll
          for (int c = 0; c < NV; ++c) {
            inc[c] = wdt32 * r[c];  // I0
            up[c] = ui[c] + f64_of(inc[c]);
          }
        }
      } else {
#pragma unroll
        for (int c = 0; c < NV; ++c) {
          const double Lk = to_f64(r[c]);
          if (A.stage == 0)
            up[c] = ui[c] + dt * Lk;
          else if (A.stage == 1)
            up[c] = 0.75 * u0[c] + 0.25 * (ui[c] + dt * Lk);
          else
            up[c] = (1.0 / 3.0) * u0[c] + (2.0 / 3.0) * (ui[c] + dt * Lk);
        }
      }
#pragma unroll
      for (int c = 0; c < NV; ++c) A.comp.u_out[c][cell] = up[c];
      if constexpr (FP32) {
        if (A.stage < 2) {
#pragma unroll
          for (int c = 0; c < NV; ++c) A.comp.inc_out[c][cell] = inc[c];
        }
      }
#pragma unroll
      for (int k = 0; k < NV; ++k) unew[k] = comp_of<NV>(up, k, dir);  // conserved order
      if constexpr (FP32) {
        bulk_state_check<NV>(A, cell, unew, mode, amax);
      } else if constexpr (NV > 1) {
        // non-physical check and next-step alpha on the new state; its FP64
        // operations (a division and a square root among them) only where
        // FP32 bounds leave either open
        double s[kAmax<FIELD>];
        if (!FIELD && state_is_plain<NV>(unew, A.gm1_f, mode & kModeAlpha, amax)) {
        } else if (!speeds64<NV, FIELD>(unew, A.gamma, s)) {
          atomicOr(&st->err, kErrNonPhys);
          atomicMin(&st->err_cell, cell);
        } else if (mode & kModeAlpha) {
#pragma unroll
          for (int k = 0; k < (FIELD ? 3 : 1) * (NV - 2); ++k) amax[k] = fmax(amax[k], s[k]);
        }
      } else {
        if (!isfinite(unew[0])) {
          atomicOr(&st->err, kErrNonPhys);
          atomicMin(&st->err_cell, cell);
        }
      }
    });
  }
  if constexpr (!FP32 && !FIELD && NV > 1) {
    // the maxima of a warp's lanes are each lane's from here on: the next
    // tile's cells below them need no FP64 speeds
    if (mode & kModeAlpha) {
#pragma unroll
      for (int d = 0; d < NV - 2; ++d)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
          amax[d] = fmax(amax[d], __shfl_xor_sync(0xffffffffu, amax[d], o));
    }
  }
  if constexpr (!TMA) hook();
  __syncthreads();
}

// Minimum resident blocks per SM asked of the compiler for the FP32-bulk
// sweep, which caps its registers at 65536 / (128 * min blocks): eight (64, a few
// spilled around the out-of-line calls) for ENO-AO5 and scalars, six (80) for
// ENO-AO7 of the Euler equations, whose selection spills at 64 (512^3 stage 29.1 ->
// 28.0 ms, 1024^2 jumps 237 -> 229 us, 512^2 noise, every face selected, 208 -> 201 us;
// where it was slower: 96^3 noise 0.99 -> 1.01 ms; scalars at 80: 1024^2 sine 44 ->
// 48 us).
#ifndef ENOAO_FP32_MIN_BLOCKS
#define ENOAO_FP32_MIN_BLOCKS 8
#endif
#ifndef ENOAO_FP32_MIN_BLOCKS_EULER7
#define ENOAO_FP32_MIN_BLOCKS_EULER7 6
#endif
// Per-field splitting keeps two projections per window cell live and takes
// four blocks (128 registers).  With a TMA-staged raw tile a block needs more
// shared memory, and four of them fill an SM: they get the registers (128, no
// spills; at 96 the thread-0 copy issue spills).
template <int NV, int ORDER, typename R, bool FIELD = false, bool TMA = false>
constexpr int sweep_min_blocks() {
  if (sizeof(R) == 8) return 1;
  if (FIELD || TMA) return 4;
  return NV > 1 && ORDER == 7 ? ENOAO_FP32_MIN_BLOCKS_EULER7 : ENOAO_FP32_MIN_BLOCKS;
}

// Bound on the polls of a TMA completion barrier (a copy of a few tens of KB
// lands in microseconds; this is about a second): beyond it the kernel sets
// the error word and returns instead of spinning on.
constexpr long long kTmaPollLimit = 1ll << 24;

// The end of a sweep launch, for every block: the last block to leave resets
// the tile queue (and the re-decision epoch), the FP64 re-decision count is
// added up, and the block's maxima of the new state's speeds go to alpha.
template <int NV, typename R, bool DEFER, bool FIELD>
__device__ __forceinline__ void sweep_epilogue(const SweepArgs& A, double (&amax)[kAmax<FIELD>],
                                               unsigned long long nfall) {
  constexpr int KA = kAmax<FIELD>;
  StepState* st = A.st;
  const int mode = A.mode;
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&st->blocks_done, 1u) == gridDim.x - 1) {
      st->tile_next = 0ull;
      st->blocks_done = 0u;
      if (DEFER) {
        // a new tag for the faces this sweep's re-decision pass marks (never 0,
        // the value of an unmarked face)
        const unsigned e = st->redo_epoch + 1u;
        st->redo_epoch = e ? e : 1u;
      }
      __threadfence();
    }
  }

  if constexpr (sizeof(R) == 4) {
    if (nfall) atomicAdd(&st->fallbacks, nfall);
  }
  if (NV > 1 && (mode & kModeAlpha)) {
    // block max of |u_d| + c (per field: |u_d - c|, |u_d|, |u_d + c|), then
    // one atomic per block and value
    __shared__ double red[KA][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int d = 0; d < KA; ++d) {
      double v = amax[d];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
      if (lane == 0) red[d][wid] = v;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
      for (int d = 0; d < KA; ++d) {
        double v = threadIdx.x < nw ? red[d][threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
        unsigned long long* acc;
        int axis;
        if constexpr (FIELD) {  // last stage only (per-field runs with per-step alpha)
          acc = &st->alpha_acc_f[st->par][0][0] + d;
          axis = d / 3;
        } else {
          acc = (A.stage == 2 ? st->alpha_acc[st->par] : st->alpha_stage) + d;
          axis = d;
        }
        if (threadIdx.x == 0 && axis < A.ndim && v > 0.0)
          atomicMax(acc, (unsigned long long)__double_as_longlong(v));
      }
    }
  }
}

// TMA: the tile's raw state (every component, the tile's lines, its cells and
// halo along the swept axis) is one box of the tensor map tmap, copied into
// the first A.tma_raw_bytes of dynamic shared memory by thread 0; the copy of
// the next tile is issued as soon as phase 1 of the current one is done, so
// it lands while phases 2 and 3 run.  Ghost cells outside the grid (the box
// reads zeros there) are then filled from the boundary map with plain loads.
template <int NV, int ORDER, typename R, bool DEFER = false, bool FIELD = false, bool TMA = false,
          int SHAPE = kShapeAny>
__global__ void __launch_bounds__(128, sweep_min_blocks<NV, ORDER, R, FIELD, TMA>())
    sweep_kernel(const __grid_constant__ SweepArgs A, const __grid_constant__ CUtensorMap tmap) {
  constexpr int G = Geo<ORDER>::G;
  StepState* st = A.st;
  if (st->skip) return;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ typename SweepConst<FIELD, R>::type s_k;
  if (threadIdx.x == 0) {
    tile_const<ORDER, R>(A, st->alpha[A.dir], st->dt, s_k);
    if constexpr (FIELD)
      for (int i = 0; i < 3; ++i) s_k.af[i] = (R)st->alpha_f[A.dir][i];
  }
  constexpr int KA = kAmax<FIELD>;
  double amax[KA];
#pragma unroll
  for (int i = 0; i < KA; ++i) amax[i] = 0.0;
  unsigned long long nfall = 0;
  // Dynamic tile queue: tiles differ in cost (slow faces and FP64
  // re-decisions cluster at discontinuities), so blocks pull their next tile
  // instead of striding.  Thread 0 asks for it as the current tile starts and
  // works out its geometry as that one ends, so that neither the atomic's
  // round trip nor the index arithmetic stands between two tiles.  The last
  // block to leave resets the queue for the next launch on the stream.
  if constexpr (!TMA) {
    __shared__ TileGeo s_geo[2];
    __shared__ bool s_more[2];
    if (threadIdx.x == 0) {
      s_geo[0] = tile_geo(A, blockIdx.x);  // the grid has at most a block per tile
      s_more[0] = true;
    }
    __syncthreads();
    for (int b = 0; s_more[b]; b ^= 1) {
      unsigned long long next = 0;
      if (threadIdx.x == 0) next = atomicAdd(&st->tile_next, 1ull) + gridDim.x;
      auto publish = [&]() {
        if (threadIdx.x == 0) {
          const bool more = next < (unsigned long long)A.ntiles;
          s_more[b ^ 1] = more;
          if (more) s_geo[b ^ 1] = tile_geo(A, (long long)next);
        }
      };
      sweep_tile<NV, ORDER, R, false, DEFER, FIELD, false, SHAPE, decltype(publish)>(
          A, s_geo[b], smem_raw, s_k, amax, nfall, RawTile{}, publish);
    }
  } else {
    __shared__ long long s_tile;
    __shared__ __align__(8) unsigned long long s_bar;
    double* raw = reinterpret_cast<double*>(smem_raw);
    unsigned char* smem = smem_raw + A.tma_raw_bytes;
    const int bx = A.tma_box;  // box extent along the swept axis
    RawTile rt;
    rt.p = raw;
    if (A.dir == 0) {  // box (x, lines, components)
      rt.re = 1, rt.ra = bx, rt.rc = bx * A.ta;
    } else {           // box (x = lines, [y,] swept axis, [z,] components)
      rt.re = A.ta, rt.ra = 1, rt.rc = A.ta * bx;
    }
    // thread 0: tile t's box on its way (x boxes start on the even x at or
    // below the tile's first extended cell, 16-byte aligned)
    auto issue = [&](long long t) {
      const TileGeo gg = tile_geo(A, t);
      const long long s_lo = gg.s0 - G;  // first extended cell along the swept axis
      fence_proxy_async();
      mbar_arrive_expect_tx(&s_bar, A.tma_bytes);
      if (A.dir == 0)
        tma_load_3d(raw, &tmap, (int)(s_lo - (s_lo & 1)), (int)gg.a0, 0, &s_bar);
      else if (A.dir == 1)
        tma_load_4d(raw, &tmap, (int)gg.a0, (int)s_lo, (int)gg.b, 0, &s_bar);
      else
        tma_load_4d(raw, &tmap, (int)gg.a0, (int)gg.b, (int)s_lo, 0, &s_bar);
    };
    if (threadIdx.x == 0) {
      mbar_init(&s_bar, 1);
      const long long t = (long long)atomicAdd(&st->tile_next, 1ull);
      s_tile = t;
      if (t < A.ntiles) issue(t);
    }
    __syncthreads();
    unsigned phase = 0;
    for (;;) {
      const long long tile = s_tile;
      if (tile >= A.ntiles) break;
      // the tile's box: a bounded wait, the same decision for the whole block
      bool late = true;
      for (long long it = 0; it < kTmaPollLimit; ++it)
        if (mbar_try_wait(&s_bar, phase)) {
          late = false;
          break;
        }
      if (__syncthreads_or(late)) {
        if (threadIdx.x == 0) atomicOr(&st->err, kErrTimeout);
        // the copy may still be in flight into this block's shared memory:
        // wait for it once more, again bounded, before leaving
        for (long long it = 0; it < kTmaPollLimit && !mbar_try_wait(&s_bar, phase); ++it) {
        }
        break;
      }
      phase ^= 1;
      const TileGeo g = tile_geo(A, tile);
      rt.xoff = A.dir == 0 ? (int)((g.s0 - G) & 1) : 0;
      // ghost cells beyond the grid along the swept axis (edge tiles only)
      if (g.s0 - G < 0 || g.s0 + g.nts + G > g.nd) {
        const int lgTA = __ffs(A.ta) - 1;
        for_items(lgTA, 2 * G, A.dir == 0, [&](const int a, const int k) {
          if (g.a0 + a >= g.na) return;
          const int e = k < G ? k : g.nts + k;
          const long long sg = g.s0 - G + e;
          if (sg >= 0 && sg < g.nd) return;
          double q[NV];
          load_state<NV, false>(
              A, g.base + (g.a0 + a) * g.stride_a + bc_map(sg, g.nd, A.bc) * g.stride_d, q);
          double* p = raw + a * rt.ra + (e + rt.xoff) * rt.re;
#pragma unroll
          for (int c = 0; c < NV; ++c) p[perm_comp<NV>(c, A.dir) * rt.rc] = q[c];
        });
        __syncthreads();
      }
      auto hook = [&]() {
        if (threadIdx.x == 0) {
          const long long t = (long long)atomicAdd(&st->tile_next, 1ull);
          s_tile = t;
          if (t < A.ntiles) issue(t);
        }
      };
      sweep_tile<NV, ORDER, R, false, DEFER, FIELD, true>(A, g, smem, s_k, amax, nfall, rt, hook);
    }
  }
  sweep_epilogue<NV, R, DEFER, FIELD>(A, amax, nfall);
}

// One Runge-Kutta stage of a 2D problem in one launch (FP32 bulk, one alpha,
// in-sweep re-decisions; Sec. 2's unsplit sum of the two axes' flux
// differences).  A block takes a 2D tile of Ax.ts x Ay.ts cells: first the x
// part of L(u) on it, as sub-tiles of Ax.ta rows that store it in the
// right-hand-side array like the x sweep, then, after the barrier that ends
// every sub-tile, the y part as sub-tiles of Ay.ta columns that add the
// stored x part and combine, like the y sweep.  A cell's x part is read back
// only by the block that wrote it, straight after writing it (from L2), so
// blocks never wait on one another.  Ax and Ay are the two axes' arguments
// as separate launches would take them; the host makes the 2D tile a whole
// number of both axes' sub-tiles (Ay.ts % Ax.ta == 0, Ax.ts % Ay.ta == 0).
// (ENO-AO7: five blocks, 96 registers for both parts in one kernel; 1024^2 jumps
// 1.04 -> 0.94 ms a stage)
template <int NV, int ORDER>
__global__ void __launch_bounds__(128, ORDER == 7 ? 5 : ENOAO_FP32_MIN_BLOCKS)
    fused2d_kernel(const __grid_constant__ SweepArgs Ax, const __grid_constant__ SweepArgs Ay) {
  using R = float;
  StepState* st = Ay.st;
  if (st->skip) return;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ TileConst<R> s_kx, s_ky;
  if (threadIdx.x == 0) {
    tile_const<ORDER, R>(Ax, st->alpha[0], st->dt, s_kx);
    tile_const<ORDER, R>(Ay, st->alpha[1], st->dt, s_ky);
  }
  double amax[3] = {0.0, 0.0, 0.0};
  unsigned long long nfall = 0;
  const long long tx = Ax.tiles_s, ty = Ay.tiles_s;  // 2D tiles along x and y
  const int kx = Ay.ts / Ax.ta, ky = Ax.ts / Ay.ta;   // sub-tiles per 2D tile
  __shared__ long long s_tile;
  for (;;) {
    if (threadIdx.x == 0) s_tile = (long long)atomicAdd(&st->tile_next, 1ull);
    __syncthreads();
    const long long T = s_tile;
    if (T >= tx * ty) break;
    const long long X = T % tx, Y = T / tx;
    for (int k = 0; k < kx; ++k) {
      const long long rows = Y * kx + k;  // row group of Ax.ta rows
      if (rows >= Ax.tiles_a) break;
      sweep_tile<NV, ORDER, R, false, false, false, false, kShapeXStore>(
          Ax, tile_geo(Ax, X + Ax.tiles_s * rows), smem_raw, s_kx, amax, nfall);
    }
    for (int m = 0; m < ky; ++m) {
      const long long cols = X * ky + m;  // column group of Ay.ta columns
      if (cols >= Ay.tiles_a) break;
      sweep_tile<NV, ORDER, R, false, false, false, false, kShapeYCombine>(
          Ay, tile_geo(Ay, Y + Ay.tiles_s * cols), smem_raw, s_ky, amax, nfall);
    }
  }
  sweep_epilogue<NV, R, false, false>(Ay, amax, nfall);
}

// ------------------------------------------------ grid-wide FP64 re-decisions
// Near-tie choices cluster at discontinuities and slip lines, in a few tiles
// whose SMs' FP64 units would then set a sweep's length.  With a list, the
// sweep instead lists every face that has flagged choices (its owner tile
// does), uses the FP32 choices throughout, and two passes over the whole grid
// follow it: redo_kernel re-decides the listed choices in FP64, one face per
// thread, and applies a change to the face's right cell; redo_apply_kernel
// then applies it to the face's left cell.  L(u) is linear in the face
// correction C, so a change dC of face F adds -dC/dx to cell F - 1 and +dC/dx
// to cell F.  Each cell takes its left face's change first, then its right
// face's, whatever tiles its faces fell in: the result does not depend on
// tiles.

// The line and the position along it of face fc (the face layout of the
// swept axis: nd + 1 faces per line, as tile_geo numbers them).
__device__ __forceinline__ void face_line(const SweepArgs& A, long long fc, long long& line,
                                          long long& F, long long& nd, long long& stride_d,
                                          long long& fstride_d) {
  const long long n0 = A.n[0], n1 = A.n[1];
  if (A.dir == 0) {
    nd = n0; stride_d = 1; fstride_d = 1;
    const long long li = fc / (n0 + 1);
    F = fc - li * (n0 + 1);
    line = li * n0;
  } else if (A.dir == 1) {
    nd = n1; stride_d = n0; fstride_d = n0;
    const long long b = fc / ((n1 + 1) * n0);
    const long long r = fc - b * (n1 + 1) * n0;
    F = r / n0;
    line = b * n1 * n0 + (r - F * n0);
  } else {
    nd = A.n[2]; stride_d = n0 * n1; fstride_d = n0 * n1;
    F = fc / (n0 * n1);
    line = fc - F * (n0 * n1);
  }
}

// Change of face F's correction C (sweep component order) when the choice of
// field v, sign sgn moves from the FP32 pick to pick64, added into dC: the
// FP32 window is rebuilt from the state with the arithmetic of phases 1 and
// 2, and the FP32 pick and value re-derived from it as phase 2b does.
template <int NV, int ORDER>
__device__ __forceinline__ void face_change32(const SweepArgs& A, const TileGeo& g, long long F,
                                              int v, int sgn, int pick64, double alpha_d,
                                              float (&dC)[NV], bool& changed) {
  using GE = Geo<ORDER>;
  const float gm1 = A.gm1_f, adv = A.adv_f;
  const float halpha = 0.5f * (float)alpha_d;
  auto cell = [&](long long gi, double (&q)[NV]) {
    load_state<NV, false>(A, g.base + bc_map(gi, g.nd, A.bc) * g.stride_d, q);
  };
  const bool shear = NV >= 4 && v >= 2 && v <= NV - 2;
  float L[NV], Rc[NV], w = 0.0f;
  if constexpr (NV > 1) {
    double ql64[NV], qr64[NV];
    cell(F - 1, ql64);
    cell(F, qr64);
    float ql[NV], qr[NV], pl[NV], prr[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) {
      ql[c] = to_bulk<float>(ql64[c]);  // the sweep's phase-1 narrowing
      qr[c] = to_bulk<float>(qr64[c]);
    }
    roe_prims<NV, float>(ql, gm1, inv_density<NV>(ql), pl);
    roe_prims<NV, float>(qr, gm1, inv_density<NV>(qr), prr);
    Eigen<NV, float> E;
    roe_eigen<NV, float>(pl, prr, gm1, E);
    left_row<NV, float>(E, v, L);
    right_col<NV, float>(E, v, Rc);
    if constexpr (NV >= 4) w = -L[0];
  } else {
    L[0] = 1.0f;
    Rc[0] = 1.0f;
  }
  // sign 0: d[i] is f^+ of cells (F-5+i, F-4+i); sign 1: -(f^- of (F+3-i, F+4-i))
  float d[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) d[i] = 0.0f;
#pragma unroll
  for (int i = GE::LO; i <= GE::HI; ++i) {
    const long long c0 = sgn == 0 ? F - 5 + i : F + 3 - i;
    double qa64[NV], qb64[NV];
    cell(c0, qa64);
    cell(c0 + 1, qb64);
    float qa[NV], qb[NV], fp[NV], fm[NV], x[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) {
      qa[c] = to_bulk<float>(qa64[c]);
      qb[c] = to_bulk<float>(qb64[c]);
    }
    split_diff<NV, float>(qa64, qb64, qa, qb, gm1, adv, halpha, inv_density<NV>(qa),
                          inv_density<NV>(qb), fp, fm);
#pragma unroll
    for (int c = 0; c < NV; ++c) x[c] = sgn == 0 ? fp[c] : fm[c];
    float acc = 0.0f;
    if constexpr (NV >= 4) {
      if (shear) {
        acc = fma(-w, x[0], shear_comp<NV>(x, v));
      } else {
#pragma unroll
        for (int c = 0; c < NV; ++c) acc = fma(L[c], x[c], acc);
      }
    } else {
#pragma unroll
      for (int c = 0; c < NV; ++c) acc = fma(L[c], x[c], acc);
    }
    d[i] = sgn == 0 ? acc : -acc;
  }
  int pick32;
  bool m;
  const float nomx[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  const float corr_old = eno_select<ORDER, float, false>(d, A.delta_f, A.tie_rel_f, nomx,
                                                         0.0f, pick32, m);
  if (pick64 == pick32) return;
  changed = true;
  float corr = 0.0f;
#pragma unroll
  for (int i = GE::LO; i <= GE::HI; ++i) corr = fma(bcoef<float>(pick64, i), d[i], corr);
  const float dv = corr - corr_old;
  if constexpr (NV >= 4) {
    if (shear) {  // column v of R is e_v + w e_{NV-1}
#pragma unroll
      for (int c = 2; c < NV - 1; ++c) dC[c] += c == v ? dv : 0.0f;
      dC[NV - 1] = fma(w, dv, dC[NV - 1]);
      return;
    }
  }
#pragma unroll
  for (int c = 0; c < NV; ++c) dC[c] = fma(Rc[c], dv, dC[c]);
}

// Adds s * dC (s = +-1/dx) to L(u) of one cell: to the stored L(u) of a
// non-final axis, or, on the final axis, to the combined state through the
// stage's weight of dt L (redo_coef) and to the FP32 increment the stage
// carries on (I0, I1: weight dt).
template <int NV>
__device__ __forceinline__ void apply_change(const SweepArgs& A, long long cell, float s,
                                             const float (&dC)[NV]) {
  const bool combine = (A.mode & kModeCombine) != 0;
  const double w = A.redo_coef * A.st->dt;
  const float dt32 = f32_rn(A.st->dt);
#pragma unroll
  for (int c = 0; c < NV; ++c) {
    const long long k = perm_comp<NV>(c, A.dir) * A.cstride + cell;
    const float dL = s * dC[c];
    if (combine) {
      A.u_out[k] += w * (double)dL;
      if (A.inc_out) A.inc_out[k] = fmaf(dt32, dL, A.inc_out[k]);  // I0, I1 carry dt L
    } else {
      reinterpret_cast<float*>(A.rhs)[k] += dL;
    }
  }
}

// The re-decision pass.  A warp takes CF listed faces at a time and spreads
// their flagged choices over its lanes, one choice per lane (32 per round):
// each lane re-decides its choice in FP64 alone (redo_lane), so that one warp
// instruction of the FP64 unit, whose cost does not shrink with fewer active
// lanes, serves up to 32 choices; it then re-derives the choice's FP32 pick
// and value, and each face's lane adds the changes of its choices in field /
// sign order.  A changed face stores its dC, marks itself with the sweep's
// epoch and applies the change to its right cell F.
template <int NV, int ORDER>
__global__ void __launch_bounds__(128) redo_kernel(const SweepArgs A) {
  constexpr int CF = 8;  // listed faces per warp round
  const unsigned FULL = 0xffffffffu;
  StepState* st = A.st;
  if (st->skip) return;
  const unsigned n = st->redo_n < A.redo_cap ? st->redo_n : (unsigned)A.redo_cap;
  const unsigned epoch = st->redo_epoch;
  const double alpha_d = st->alpha[A.dir];
  const float inv_dx = A.inv_dx_f;
  const int lane = threadIdx.x & 31;
  const unsigned nwarps = gridDim.x * (blockDim.x >> 5);
  unsigned long long nf = 0;
  for (unsigned base = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * CF; base < n;
       base += nwarps * CF) {
    // lane j < CF holds listed face base + j
    const unsigned i = base + lane;
    const bool hasf = lane < CF && i < n;
    const unsigned long long rec = hasf ? A.redo[i] : 0ull;
    const unsigned mask = (unsigned)(rec & 0xffffull);
    long long line, F, nd, stride_d, fstride_d;
    face_line(A, (long long)(rec >> 16), line, F, nd, stride_d, fstride_d);
    // choices of face j are numbers pre_j .. pre_j + m_j - 1 of the round
    const int m = __popc(mask);
    int incl = m;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += t;
    }
    const int pre = incl - m;
    const int T = __shfl_sync(FULL, incl, 31);
    float dC[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) dC[c] = 0.0f;
    bool changed = false;
    for (int c0 = 0; c0 < T; c0 += 32) {
      // lane l takes choice c0 + l: face j, field * 2 + sign k
      const int ci = c0 + lane;
      int j = 0;
#pragma unroll
      for (int q = 1; q < CF; ++q) {
        const int pq = __shfl_sync(FULL, pre, q);
        if (ci >= pq) j = q;
      }
      // every lane takes part in each shuffle (none inside a condition)
      const unsigned mj = __shfl_sync(FULL, mask, j);
      const int prej = __shfl_sync(FULL, pre, j);
      const long long lj = __shfl_sync(FULL, line, j), Fj = __shfl_sync(FULL, F, j);
      const int kb = ci < T ? nth_set_bit(mj, ci - prej) : -1;
      const bool valid = kb >= 0;
      const int k = valid ? kb : 0;
      const int cnt = T - c0 < 32 ? T - c0 : 32;
      float dk[NV];
#pragma unroll
      for (int c = 0; c < NV; ++c) dk[c] = 0.0f;
      bool ch = false;
      if (valid) {
        TileGeo g;  // the face's line, as redo_lane reads it
        g.base = lj;
        g.a0 = 0;
        g.stride_a = 0;
        g.stride_d = stride_d;
        g.nd = nd;
        const int pick64 = redo_lane<NV, ORDER, false>(A, g, 0, Fj - 1, k >> 1, k & 1, alpha_d);
        face_change32<NV, ORDER>(A, g, Fj, k >> 1, k & 1, pick64, alpha_d, dk, ch);
        ++nf;
      }
      // each face's lane adds its choices' changes in field / sign order
      for (int l = 0; l < cnt; ++l) {
        const int jl = __shfl_sync(FULL, j, l);
        const int chl = __shfl_sync(FULL, (int)ch, l);
        float v[NV];
#pragma unroll
        for (int c = 0; c < NV; ++c) v[c] = __shfl_sync(FULL, dk[c], l);
        if (lane == jl && chl) {
#pragma unroll
          for (int c = 0; c < NV; ++c) dC[c] += v[c];
          changed = true;
        }
      }
    }
    if (hasf) {
      const long long fc = (long long)(rec >> 16);
      A.redo_mark[fc] = changed ? epoch : 0u;
      if (changed) {
#pragma unroll
        for (int c = 0; c < NV; ++c) A.redo_dc[(long long)i * NV + c] = dC[c];
        if (F < nd) apply_change<NV>(A, line + F * stride_d, inv_dx, dC);
      }
    }
  }
  if (nf) atomicAdd(&st->fallbacks, nf);
}

// Second pass: each changed face applies its change to its left cell F - 1.
// On the final axis the cells a change touched are then checked and enter
// the next alpha (a cell whose right face also changed is checked by that
// face's thread, after both of its changes).  The last block to leave empties
// the list for the next sweep.
template <int NV>
__global__ void __launch_bounds__(128) redo_apply_kernel(const SweepArgs A) {
  StepState* st = A.st;
  const unsigned n = st->skip ? 0u : (st->redo_n < A.redo_cap ? st->redo_n : (unsigned)A.redo_cap);
  const unsigned epoch = st->redo_epoch;
  const float inv_dx = A.inv_dx_f;
  const bool check = (A.mode & kModeCombine) != 0;
  double amax[3] = {0.0, 0.0, 0.0};
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const long long fc = (long long)(A.redo[i] >> 16);
    if (A.redo_mark[fc] != epoch) continue;
    long long line, F, nd, stride_d, fstride_d;
    face_line(A, fc, line, F, nd, stride_d, fstride_d);
    float dC[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) dC[c] = A.redo_dc[(long long)i * NV + c];
    auto check_cell = [&](long long cell) {
      double u[NV];
#pragma unroll
      for (int c = 0; c < NV; ++c) u[c] = A.u_out[c * A.cstride + cell];
      bulk_state_check<NV>(A, cell, u, A.mode, amax);
    };
    if (F >= 1) {
      apply_change<NV>(A, line + (F - 1) * stride_d, -inv_dx, dC);
      if (check) check_cell(line + (F - 1) * stride_d);
    }
    if (check && F < nd && !(F + 1 <= nd && A.redo_mark[fc + fstride_d] == epoch))
      check_cell(line + F * stride_d);
  }
  if constexpr (NV > 1) {
    if (check && (A.mode & kModeAlpha)) {
      unsigned long long* acc = A.stage == 2 ? st->alpha_acc[st->par] : st->alpha_stage;
#pragma unroll
      for (int d = 0; d < 3; ++d)
        if (d < A.ndim && amax[d] > 0.0)
          atomicMax(&acc[d], (unsigned long long)__double_as_longlong(amax[d]));
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&st->redo_done, 1u) == gridDim.x - 1) {
      st->redo_n = 0u;
      st->redo_done = 0u;
      __threadfence();
    }
  }
}

}  // namespace enoao
