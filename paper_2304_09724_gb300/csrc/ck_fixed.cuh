// Cauchy-Kovalevskaya procedure of one point in block fixed point: scales and conversions around the
// generated recursions (ck_fixed_generated.cuh).
//
// Units.  Length: L = min(dx, dy) divided by 2^g; velocity: 2^eu; density: 2^e0; so a coefficient
// of total degree s of rho, (m, n), E is held times 2^-(e0 + g s), 2^-(e0 + eu + g s) and
// 2^-(e0 + 2 eu + g s), and the equations keep their form.  e0 and eu come from the leading
// state (rho0, |u0|, |v0|, sqrt(H0) <= 1 in these units); g >= 0 is the smallest growth for which
// every coefficient of degree s >= 1 is below 1 (the recursion then checks that everything stays
// below 1/4 and is repeated with a larger g where it does not), so that a steep point, whose
// coefficients grow with the degree, fits as a smooth one does.  What is rounded is 2^-62 of the
// field's scale times (2^g)^s, the size its coefficients of that degree have themselves; FP64
// rounds the leading coefficients at 2^-54.  A field whose values lie far below its scale keeps fewer bits
// than a double's.  Where that shows in a step, the recursion runs in FP64 (ck_euler1d, ck_euler2d):
//   - gamma above 3: p = (gamma - 1)(E - rho u^2 / 2) magnifies its rounding, and the growth that holds the
//     derivatives of p coarsens all others (steep random points: gamma 3 as FP64, 5 five times, 30 1e4 times
//     FP64's error);
//   - gamma near 1: sqrt(H0) is far above |u| + c then, and order k in time rounds at (sqrt(H0) / (|u| + c))^k
//     times what it should (gamma 1.02, half a cell per step: 1.6e-15 of the density, FP64 1e-20);
//   - a slow momentum along a 2D face where the energy does not vary (step2d_items.cuh);
//   - a density or velocity below 2^-300, where the exponents end.
// It does not show in a slow momentum across the face: the star state's energy is rounded there, in FP64
// too.  1D contacts, 100 cells, 8 steps, velocity 1e-2 / 1e-4 / 1e-8, error of the momentum against 64-bit
// mantissas: 1.18e-14 / 1.05e-12 / 6.3e-9, with the FP64 recursion 1.17e-14 / 1.05e-12 / 6.4e-9.  156 random shock
// tubes, shock-density waves, quadrants and double Mach reflections: 0.80 to 1.02 of its error in every field.
#pragma once
#include <cmath>

#include "ck_fixed_generated.cuh"

namespace shweno {

// Constants for one mesh.
struct CkFixed {
  CkFixedConst K;
  double iL;      // 1 / L: the time coefficients come in units of L
  double rx, ry;  // L / dx, L / dy: coordinates in units of L
  double gm1;     // gamma - 1, for the recursion in FP64
  // whether block fixed point is for this gas (Burgers: yes); below 1.0625 every point at rest has too fast a unit
  int32_t fixed;
};

// Most bits of a momentum along the face below its scale; a slower one is FP64's.  Shear flow with the recursion alone in
// fixed point, error of the drift's slope relative to FP64: 1.0 at 8 bits below, 1.1 at 9, 2 at 10, 3 at 11.
constexpr int CK_BELOW = 8;
constexpr int FX_STILL = 48;  // a momentum more bits than this below its scale counts as none
constexpr int CK_TINY = -300;  // least exponent of the units of density and velocity

FX_FN Fx fx_const(double x) {
  FxRange r{0};
  return fx_split(fx_from_double<FX_C>(x, 0) + FX_HALF, r);
}

inline void finalize_ck_fixed(CkFixed& C, int dim, double dx, double dy, double gamma) {
  const double L = dim == 2 && dy < dx ? dy : dx;
  C.rx = L / dx;
  C.ry = dim == 2 ? L / dy : 1.0;
  C.iL = 1.0 / L;
  C.K.third = fx_const(1.0 / 3.0);
  C.fixed = gamma >= 1.0625 && gamma <= 3.0;
  C.K.gm1 = fx_const(C.fixed ? gamma - 1.0 : 0.0);
  C.gm1 = gamma - 1.0;
}

FX_FN int fx_max(int a, int b) { return a > b ? a : b; }

// Leading state of a point as the scales need it (Euler): 1/rho0 and the high words (magnitude
// bits) of max(|u0|, |v0|), of H0 = (E0 + p0)/rho0 and of the sound speed.
struct CkLead {
  double ir;
  int32_t hu, hH, hc;
};
// Whether the unit of velocity 2^eu is more than 4 times the larger of velocity and sound speed (never for gamma
// of 1.4 and more); order 4 in time of half a cell per step then rounds at more than 16 quanta.  Or it is the
// least one: a state may lie anywhere below it.
FX_FN bool ck_off_unit(int eu, const CkLead& lead) {
  return eu > fx_max(fx_exp(lead.hu), fx_exp(lead.hc)) + 1 || eu <= CK_TINY;
}

// Scales of one point: the exponents of its fields and the growth.
template <int NC>
struct CkScale {
  static constexpr int NG = NC == 1 ? 1 : 3;  // groups: {u} or {rho}, {m, n}, {E}
  int base[NG], eu, g;
  bool finite;
  static FX_FN int group(int q) { return NC == 1 || q == 0 ? 0 : (q == NC - 1 ? 2 : 1); }
  FX_FN int of(int q, int s) const { return base[group(q)] + g * s; }
};

// Euler: whether the point's units of density and velocity do not fit it.
template <int NC>
FX_FN bool ck_off_units(const CkScale<NC>& S, const CkLead& lead) {
  return ck_off_unit(S.eu, lead) || S.base[0] <= CK_TINY;
}

// Scale of an Euler point from its leading state Ws and the exponents top[group][degree >= 1] of its
// other coefficients.
template <int NC>
FX_FN CkScale<NC> ck_scale_from(const double* Ws, const int (&top)[3][5], const CkLead& lead) {
  CkScale<NC> S;
  const int e0 = fx_max(fx_exp(fx_hi(Ws[0]) & 0x7fffffff), CK_TINY);  // an exact 0 then converts to 0 in every field
  const int eE = fx_exp(fx_hi(Ws[NC - 1]) & 0x7fffffff);
  int eh = fx_exp(lead.hH);
  // a negative density or pressure (E0 + p0 then no longer bounds E0 and the kinetic energy)
  const int ee = eE - e0 + 3;
  if (ee > eh + 3) eh = ee;
  S.eu = fx_max(fx_max(fx_exp(lead.hu), (eh + 1) >> 1), CK_TINY);
  S.base[0] = e0;
  S.base[1] = e0 + S.eu;
  S.base[2] = e0 + 2 * S.eu;
  S.finite = lead.hH < 0x7ff00000 && lead.hu < 0x7ff00000 && (fx_hi(lead.ir) & 0x7fffffff) < 0x7ff00000 &&
             e0 <= 1024 && eE <= 1024;
  S.g = 0;
#pragma unroll
  for (int s = 1; s < 5; ++s) {
    int d = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) d = fx_max(d, top[i][s] - S.base[i]);
    S.finite = S.finite && d < 3000;
    S.g = fx_max(S.g, (d + s - 1) / s);
  }
  return S;
}

// a(q, m*5+n) (m + n <= 4; n = 0 only when DIM == 1): spatial Taylor coefficients in cell units.
template <int NC, int DIM, typename Coef>
FX_FN CkScale<NC> ck_scale(const Coef& a, const CkLead& lead) {
  using Scale = CkScale<NC>;
  constexpr int NG = Scale::NG;
  int top[NG][5];  // largest high word (magnitude bits) by group and degree
#pragma unroll
  for (int i = 0; i < NG; ++i)
#pragma unroll
    for (int s = 0; s < 5; ++s) top[i][s] = 0;
#pragma unroll
  for (int q = 0; q < NC; ++q)
#pragma unroll
    for (int m = 0; m < 5; ++m)
#pragma unroll
      for (int n = 0; n + m < 5; ++n)
        if (DIM == 2 || n == 0) {
          int& t = top[Scale::group(q)][m + n];
          t = fx_max(t, fx_hi(a(q, m * 5 + n)) & 0x7fffffff);
        }
  int all = 0;
#pragma unroll
  for (int i = 0; i < NG; ++i)
#pragma unroll
    for (int s = 0; s < 5; ++s) {
      all = fx_max(all, top[i][s]);
      top[i][s] = fx_exp(top[i][s]);
    }
  Scale S;
  if constexpr (NC == 1) {
    // u0 may vanish; 2^-40 of the steepest coefficient is as good a scale then
    int e = top[0][0];
#pragma unroll
    for (int s = 1; s < 5; ++s) e = fx_max(e, top[0][s] - 40);
    S.base[0] = S.eu = fx_max(e, -900);  // an exact 0 then converts to 0
    S.g = 0;
#pragma unroll
    for (int s = 1; s < 5; ++s) S.g = fx_max(S.g, (fx_max(top[0][s] - S.base[0], 0) + s - 1) / s);
    S.finite = true;
  } else {
    double Ws[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) Ws[q] = a(q, 0);
    S = ck_scale_from<NC>(Ws, top, lead);
  }
  S.finite = S.finite && all < 0x7ff00000;
  return S;
}

// The same coefficient in a growth larger by one: X of total degree s divided by 2^s.
FX_FN Fx fx_regrow(Fx v, int s, FxRange& r) { return fx_split(((fx_join(v) + (int64_t(1) << (s - 1))) >> s) + FX_HALF, r); }

// Coefficient a of component q and degree s in the point's scale.
template <int NC>
FX_FN Fx ck_convert(const CkScale<NC>& S, double a, int q, int s, FxRange& r) {
  return fx_split(fx_from_double(a, S.of(q, s)) + FX_HALF, r);
}
template <int NC>
FX_FN Fx ck_ninv(const CkScale<NC>& S, const CkLead& lead) {
  FxRange r{0};
  return fx_split(fx_from_double<FX_C>(-lead.ir, -S.base[0]) + FX_HALF, r);
}

// Growths tried.  With inputs of degree s below 2^-11s, that is at the last one, no coefficient of any slice can
// leave the range: a majorant of the recursion (all signs equal, 1/rho0 = 2, gamma = 3) stays below 0.12.
constexpr int kCkTries = 12;

// Burgers and 1D Euler: the whole recursion in one thread's registers (2D Euler: step2d_items.cuh).  Writes tc[q][k],
// k = 1..4, per L^k (tc[q][0] is left to the caller); NaN where the input is not finite.
template <int NC, int DIM>
FX_FN void ck_fixed(const double (&a)[NC][25], const CkLead& lead, const CkFixed& C, double (&tc)[NC][5]) {
  const CkFixedConst& K = C.K;
  auto coef = [&a](int q, int mn) { return a[q][mn]; };
  CkScale<NC> S = ck_scale<NC, DIM>(coef, lead);
  if constexpr (NC == 3)
    if (!C.fixed || ck_off_units(S, lead)) return ck_euler1d(a, tc, C.gm1);
  Fx w[NC][25], ninv{0, 0};
  int64_t t[NC][5];
  if constexpr (NC > 1) ninv = ck_ninv<NC>(S, lead);
#pragma unroll 1
  for (int tries = 0; tries < kCkTries; ++tries, ++S.g) {
    FxRange r{0}, r0{0};
#pragma unroll
    for (int q = 0; q < NC; ++q)
#pragma unroll
      for (int m = 0; m < 5; ++m)
#pragma unroll
        for (int n = 0; n + m < 5; ++n)
          if (DIM == 2 || n == 0) w[q][m * 5 + n] = ck_convert<NC>(S, a[q][m * 5 + n], q, m + n, m + n ? r : r0);
    if constexpr (NC == 1 && DIM == 1) ck_burgers1d_fx(w, ninv, K, t, r);
    else if constexpr (NC == 1) ck_burgers2d_fx(w, ninv, K, t, r);
    else ck_euler1d_fx(w, ninv, K, t, r);
    if (!r.bad()) break;
    if (tries == kCkTries - 1) S.finite = false;
  }
#pragma unroll
  for (int q = 0; q < NC; ++q)
#pragma unroll
    for (int k = 1; k < 5; ++k)
      tc[q][k] = S.finite ? fx_to_double(t[q][k], S.of(q, 0) + k * (S.eu + S.g)) : fx_from_bits(0x7ff8000000000000ull);
}

}  // namespace shweno
