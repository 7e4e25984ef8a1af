// Generated by gen_ck.py -- do not edit.  The Cauchy-Kovalevskaya recursions
// in block fixed point (see fixed.cuh, ck_fixed.cuh and gen_ck.py for the method).
#pragma once
#include "fixed.cuh"

namespace shweno {

// Constants of the recursion: 1/3 and (gamma - 1) 2^-gshift.
struct CkFixedConst {
  Fx third, gm1;
  int32_t gshift;
};

// Minus z / k: from the flux derivatives of slice k - 1 to slice k.
template <int K>
FX_FN int64_t fx_time(int64_t z, Fx third) {
  if (K == 1) return -z;
  if (K == 2) return -((z + 1) >> 1);
  if (K == 4) return -((z + 2) >> 2);
  FxRange r0{0};
  FxAcc s = fx_zero<FX_C>();
  fx_mac(s, fx_split(FX_HALF - z, r0), third);
  return fx_sum<FX_C>(s);
}

// ck_burgers1d_fx: 1D burgers in block fixed point; inputs w[q][m*5+n], outputs t[q][k], k = 1..4, in
// the fields' units (fixed.cuh, ck_fixed.cuh); ninv = -1/rho0 in fixed point (Euler).
FX_FN void ck_burgers1d_fx(const Fx (&w)[1][25], Fx ninv, const CkFixedConst& K, int64_t (&t)[1][5], FxRange& r) {
  (void)ninv;
  int64_t f_100; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][5]); f_100 = fx_sum(s); }
  const Fx w0_001 = fx_split(fx_time<1>(1 * f_100, K.third) + FX_HALF, r);
  int64_t f_200; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][10]); f_200 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w[0][5], w[0][5]); f_200 += fx_sum(s) >> 1; }
  const Fx w0_101 = fx_split(fx_time<1>(2 * f_200, K.third) + FX_HALF, r);
  int64_t f_101; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_101); fx_mac(s, w0_001, w[0][5]); f_101 = fx_sum(s); }
  const Fx w0_002 = fx_split(fx_time<2>(1 * f_101, K.third) + FX_HALF, r);
  int64_t f_300; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][15]); fx_mac(s, w[0][5], w[0][10]); f_300 = fx_sum(s); }
  const Fx w0_201 = fx_split(fx_time<1>(3 * f_300, K.third) + FX_HALF, r);
  int64_t f_201; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_201); fx_mac(s, w0_001, w[0][10]); fx_mac(s, w[0][5], w0_101); f_201 = fx_sum(s); }
  const Fx w0_102 = fx_split(fx_time<2>(2 * f_201, K.third) + FX_HALF, r);
  int64_t f_102; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_102); fx_mac(s, w0_001, w0_101); fx_mac(s, w0_002, w[0][5]); f_102 = fx_sum(s); }
  const Fx w0_003 = fx_split(fx_time<3>(1 * f_102, K.third) + FX_HALF, r);
  int64_t f_400; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][20]); fx_mac(s, w[0][5], w[0][15]); f_400 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w[0][10], w[0][10]); f_400 += fx_sum(s) >> 1; }
  const Fx w0_301 = fx_split(fx_time<1>(4 * f_400, K.third) + FX_HALF, r);
  int64_t f_301; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_301); fx_mac(s, w0_001, w[0][15]); fx_mac(s, w[0][5], w0_201); fx_mac(s, w0_101, w[0][10]); f_301 = fx_sum(s); }
  const Fx w0_202 = fx_split(fx_time<2>(3 * f_301, K.third) + FX_HALF, r);
  int64_t f_202; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_202); fx_mac(s, w0_001, w0_201); fx_mac(s, w0_002, w[0][10]); fx_mac(s, w[0][5], w0_102); f_202 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w0_101, w0_101); f_202 += fx_sum(s) >> 1; }
  const Fx w0_103 = fx_split(fx_time<3>(2 * f_202, K.third) + FX_HALF, r);
  int64_t f_103; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_103); fx_mac(s, w0_001, w0_102); fx_mac(s, w0_002, w0_101); fx_mac(s, w0_003, w[0][5]); f_103 = fx_sum(s); }
  const Fx w0_004 = fx_split(fx_time<4>(1 * f_103, K.third) + FX_HALF, r);
  t[0][1] = fx_join(w0_001);
  t[0][2] = fx_join(w0_002);
  t[0][3] = fx_join(w0_003);
  t[0][4] = fx_join(w0_004);
}

// ck_burgers2d_fx: 2D burgers in block fixed point; inputs w[q][m*5+n], outputs t[q][k], k = 1..4, in
// the fields' units (fixed.cuh, ck_fixed.cuh); ninv = -1/rho0 in fixed point (Euler).
FX_FN void ck_burgers2d_fx(const Fx (&w)[1][25], Fx ninv, const CkFixedConst& K, int64_t (&t)[1][5], FxRange& r) {
  (void)ninv;
  int64_t f_100; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][5]); f_100 = fx_sum(s); }
  int64_t f_010; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][1]); f_010 = fx_sum(s); }
  const Fx w0_001 = fx_split(fx_time<1>(1 * f_100 + 1 * f_010, K.third) + FX_HALF, r);
  int64_t f_200; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][10]); f_200 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w[0][5], w[0][5]); f_200 += fx_sum(s) >> 1; }
  int64_t f_110; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][6]); fx_mac(s, w[0][1], w[0][5]); f_110 = fx_sum(s); }
  const Fx w0_101 = fx_split(fx_time<1>(2 * f_200 + 1 * f_110, K.third) + FX_HALF, r);
  int64_t f_101; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_101); fx_mac(s, w0_001, w[0][5]); f_101 = fx_sum(s); }
  int64_t f_020; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][2]); f_020 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w[0][1], w[0][1]); f_020 += fx_sum(s) >> 1; }
  const Fx w0_011 = fx_split(fx_time<1>(1 * f_110 + 2 * f_020, K.third) + FX_HALF, r);
  int64_t f_011; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_011); fx_mac(s, w0_001, w[0][1]); f_011 = fx_sum(s); }
  const Fx w0_002 = fx_split(fx_time<2>(1 * f_101 + 1 * f_011, K.third) + FX_HALF, r);
  int64_t f_300; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][15]); fx_mac(s, w[0][5], w[0][10]); f_300 = fx_sum(s); }
  int64_t f_210; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][11]); fx_mac(s, w[0][1], w[0][10]); fx_mac(s, w[0][5], w[0][6]); f_210 = fx_sum(s); }
  const Fx w0_201 = fx_split(fx_time<1>(3 * f_300 + 1 * f_210, K.third) + FX_HALF, r);
  int64_t f_201; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_201); fx_mac(s, w0_001, w[0][10]); fx_mac(s, w[0][5], w0_101); f_201 = fx_sum(s); }
  int64_t f_120; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][7]); fx_mac(s, w[0][1], w[0][6]); fx_mac(s, w[0][2], w[0][5]); f_120 = fx_sum(s); }
  const Fx w0_111 = fx_split(fx_time<1>(2 * f_210 + 2 * f_120, K.third) + FX_HALF, r);
  int64_t f_111; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_111); fx_mac(s, w0_001, w[0][6]); fx_mac(s, w[0][1], w0_101); fx_mac(s, w0_011, w[0][5]); f_111 = fx_sum(s); }
  const Fx w0_102 = fx_split(fx_time<2>(2 * f_201 + 1 * f_111, K.third) + FX_HALF, r);
  int64_t f_102; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_102); fx_mac(s, w0_001, w0_101); fx_mac(s, w0_002, w[0][5]); f_102 = fx_sum(s); }
  int64_t f_030; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][3]); fx_mac(s, w[0][1], w[0][2]); f_030 = fx_sum(s); }
  const Fx w0_021 = fx_split(fx_time<1>(1 * f_120 + 3 * f_030, K.third) + FX_HALF, r);
  int64_t f_021; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_021); fx_mac(s, w0_001, w[0][2]); fx_mac(s, w[0][1], w0_011); f_021 = fx_sum(s); }
  const Fx w0_012 = fx_split(fx_time<2>(1 * f_111 + 2 * f_021, K.third) + FX_HALF, r);
  int64_t f_012; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_012); fx_mac(s, w0_001, w0_011); fx_mac(s, w0_002, w[0][1]); f_012 = fx_sum(s); }
  const Fx w0_003 = fx_split(fx_time<3>(1 * f_102 + 1 * f_012, K.third) + FX_HALF, r);
  int64_t f_400; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][20]); fx_mac(s, w[0][5], w[0][15]); f_400 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w[0][10], w[0][10]); f_400 += fx_sum(s) >> 1; }
  int64_t f_310; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][16]); fx_mac(s, w[0][1], w[0][15]); fx_mac(s, w[0][5], w[0][11]); fx_mac(s, w[0][6], w[0][10]); f_310 = fx_sum(s); }
  const Fx w0_301 = fx_split(fx_time<1>(4 * f_400 + 1 * f_310, K.third) + FX_HALF, r);
  int64_t f_301; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_301); fx_mac(s, w0_001, w[0][15]); fx_mac(s, w[0][5], w0_201); fx_mac(s, w0_101, w[0][10]); f_301 = fx_sum(s); }
  int64_t f_220; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][12]); fx_mac(s, w[0][1], w[0][11]); fx_mac(s, w[0][2], w[0][10]); fx_mac(s, w[0][5], w[0][7]); f_220 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w[0][6], w[0][6]); f_220 += fx_sum(s) >> 1; }
  const Fx w0_211 = fx_split(fx_time<1>(3 * f_310 + 2 * f_220, K.third) + FX_HALF, r);
  int64_t f_211; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_211); fx_mac(s, w0_001, w[0][11]); fx_mac(s, w[0][1], w0_201); fx_mac(s, w0_011, w[0][10]); fx_mac(s, w[0][5], w0_111); fx_mac(s, w0_101, w[0][6]); f_211 = fx_sum(s); }
  const Fx w0_202 = fx_split(fx_time<2>(3 * f_301 + 1 * f_211, K.third) + FX_HALF, r);
  int64_t f_202; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_202); fx_mac(s, w0_001, w0_201); fx_mac(s, w0_002, w[0][10]); fx_mac(s, w[0][5], w0_102); f_202 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w0_101, w0_101); f_202 += fx_sum(s) >> 1; }
  int64_t f_130; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][8]); fx_mac(s, w[0][1], w[0][7]); fx_mac(s, w[0][2], w[0][6]); fx_mac(s, w[0][3], w[0][5]); f_130 = fx_sum(s); }
  const Fx w0_121 = fx_split(fx_time<1>(2 * f_220 + 3 * f_130, K.third) + FX_HALF, r);
  int64_t f_121; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_121); fx_mac(s, w0_001, w[0][7]); fx_mac(s, w[0][1], w0_111); fx_mac(s, w0_011, w[0][6]); fx_mac(s, w[0][2], w0_101); fx_mac(s, w0_021, w[0][5]); f_121 = fx_sum(s); }
  const Fx w0_112 = fx_split(fx_time<2>(2 * f_211 + 2 * f_121, K.third) + FX_HALF, r);
  int64_t f_112; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_112); fx_mac(s, w0_001, w0_111); fx_mac(s, w0_002, w[0][6]); fx_mac(s, w[0][1], w0_102); fx_mac(s, w0_011, w0_101); fx_mac(s, w0_012, w[0][5]); f_112 = fx_sum(s); }
  const Fx w0_103 = fx_split(fx_time<3>(2 * f_202 + 1 * f_112, K.third) + FX_HALF, r);
  int64_t f_103; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_103); fx_mac(s, w0_001, w0_102); fx_mac(s, w0_002, w0_101); fx_mac(s, w0_003, w[0][5]); f_103 = fx_sum(s); }
  int64_t f_040; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][4]); fx_mac(s, w[0][1], w[0][3]); f_040 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w[0][2], w[0][2]); f_040 += fx_sum(s) >> 1; }
  const Fx w0_031 = fx_split(fx_time<1>(1 * f_130 + 4 * f_040, K.third) + FX_HALF, r);
  int64_t f_031; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_031); fx_mac(s, w0_001, w[0][3]); fx_mac(s, w[0][1], w0_021); fx_mac(s, w0_011, w[0][2]); f_031 = fx_sum(s); }
  const Fx w0_022 = fx_split(fx_time<2>(1 * f_121 + 3 * f_031, K.third) + FX_HALF, r);
  int64_t f_022; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_022); fx_mac(s, w0_001, w0_021); fx_mac(s, w0_002, w[0][2]); fx_mac(s, w[0][1], w0_012); f_022 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w0_011, w0_011); f_022 += fx_sum(s) >> 1; }
  const Fx w0_013 = fx_split(fx_time<3>(1 * f_112 + 2 * f_022, K.third) + FX_HALF, r);
  int64_t f_013; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_013); fx_mac(s, w0_001, w0_012); fx_mac(s, w0_002, w0_011); fx_mac(s, w0_003, w[0][1]); f_013 = fx_sum(s); }
  const Fx w0_004 = fx_split(fx_time<4>(1 * f_103 + 1 * f_013, K.third) + FX_HALF, r);
  t[0][1] = fx_join(w0_001);
  t[0][2] = fx_join(w0_002);
  t[0][3] = fx_join(w0_003);
  t[0][4] = fx_join(w0_004);
}

// ck_euler1d_fx: 1D euler in block fixed point; inputs w[q][m*5+n], outputs t[q][k], k = 1..4, in
// the fields' units (fixed.cuh, ck_fixed.cuh); ninv = -1/rho0 in fixed point (Euler).
FX_FN void ck_euler1d_fx(const Fx (&w)[3][25], Fx ninv, const CkFixedConst& K, int64_t (&t)[3][5], FxRange& r) {
  (void)ninv;
  FxRange r0{0};  // leading coefficients are in range by their scales
  const int64_t z_w1_100 = fx_join(w[1][5]);
  const Fx w0_001 = fx_split(fx_time<1>(1 * (z_w1_100), K.third) + FX_HALF, r);
  Fx u_000n; { FxAcc s = fx_zero(true); fx_mac_int(s, w[1][0], -(1 << 30)); u_000n = fx_split(fx_sum(s), r0); }
  Fx u_000; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_000n, ninv); u_000 = fx_split(fx_sum<FX_C>(s), r0); }
  Fx u_100n; { FxAcc s = fx_zero(true); fx_mac_int(s, w[1][5], -(1 << 30)); fx_mac(s, w[0][5], u_000); u_100n = fx_split(fx_sum(s), r); }
  Fx u_100; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_100n, ninv); u_100 = fx_split(fx_sum<FX_C>(s), r); }
  Fx u_200n; { FxAcc s = fx_zero(true); fx_mac_int(s, w[1][10], -(1 << 30)); fx_mac(s, w[0][5], u_100); fx_mac(s, w[0][10], u_000); u_200n = fx_split(fx_sum(s), r); }
  Fx u_200; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_200n, ninv); u_200 = fx_split(fx_sum<FX_C>(s), r); }
  int64_t z_mu_200; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_200); fx_mac(s, w[1][5], u_100); fx_mac(s, w[1][10], u_000); z_mu_200 = fx_sum(s); }
  const int64_t z_w2_200 = fx_join(w[2][10]);
  const Fx e_200 = fx_split(((z_w2_200 - ((z_mu_200) >> 1)) << K.gshift) + FX_HALF, r);
  int64_t z_p_200; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_200, K.gm1); z_p_200 = fx_sum<FX_C>(s); }
  const Fx w1_101 = fx_split(fx_time<1>(2 * (z_mu_200 + z_p_200), K.third) + FX_HALF, r);
  const int64_t z_w1_101 = fx_join(w1_101);
  const Fx w0_002 = fx_split(fx_time<2>(1 * (z_w1_101), K.third) + FX_HALF, r);
  Fx u_300n; { FxAcc s = fx_zero(true); fx_mac_int(s, w[1][15], -(1 << 30)); fx_mac(s, w[0][5], u_200); fx_mac(s, w[0][10], u_100); fx_mac(s, w[0][15], u_000); u_300n = fx_split(fx_sum(s), r); }
  Fx u_300; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_300n, ninv); u_300 = fx_split(fx_sum<FX_C>(s), r); }
  int64_t z_mu_300; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_300); fx_mac(s, w[1][5], u_200); fx_mac(s, w[1][10], u_100); fx_mac(s, w[1][15], u_000); z_mu_300 = fx_sum(s); }
  const int64_t z_w2_300 = fx_join(w[2][15]);
  const Fx e_300 = fx_split(((z_w2_300 - ((z_mu_300) >> 1)) << K.gshift) + FX_HALF, r);
  int64_t z_p_300; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_300, K.gm1); z_p_300 = fx_sum<FX_C>(s); }
  const Fx w1_201 = fx_split(fx_time<1>(3 * (z_mu_300 + z_p_300), K.third) + FX_HALF, r);
  int64_t z_mu_100; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_100); fx_mac(s, w[1][5], u_000); z_mu_100 = fx_sum(s); }
  const int64_t z_w2_100 = fx_join(w[2][5]);
  const Fx e_100 = fx_split(((z_w2_100 - ((z_mu_100) >> 1)) << K.gshift) + FX_HALF, r);
  int64_t z_p_100; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_100, K.gm1); z_p_100 = fx_sum<FX_C>(s); }
  const Fx w1_001 = fx_split(fx_time<1>(1 * (z_mu_100 + z_p_100), K.third) + FX_HALF, r);
  Fx u_001n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_001, -(1 << 30)); fx_mac(s, w0_001, u_000); u_001n = fx_split(fx_sum(s), r); }
  Fx u_001; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_001n, ninv); u_001 = fx_split(fx_sum<FX_C>(s), r); }
  const int64_t z_w1_200 = fx_join(w[1][10]);
  const Fx w0_101 = fx_split(fx_time<1>(2 * (z_w1_200), K.third) + FX_HALF, r);
  Fx u_101n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_101, -(1 << 30)); fx_mac(s, w0_001, u_100); fx_mac(s, w[0][5], u_001); fx_mac(s, w0_101, u_000); u_101n = fx_split(fx_sum(s), r); }
  Fx u_101; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_101n, ninv); u_101 = fx_split(fx_sum<FX_C>(s), r); }
  const int64_t z_w1_300 = fx_join(w[1][15]);
  const Fx w0_201 = fx_split(fx_time<1>(3 * (z_w1_300), K.third) + FX_HALF, r);
  Fx u_201n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_201, -(1 << 30)); fx_mac(s, w0_001, u_200); fx_mac(s, w[0][5], u_101); fx_mac(s, w0_101, u_100); fx_mac(s, w[0][10], u_001); fx_mac(s, w0_201, u_000); u_201n = fx_split(fx_sum(s), r); }
  Fx u_201; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_201n, ninv); u_201 = fx_split(fx_sum<FX_C>(s), r); }
  int64_t z_mu_201; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_201); fx_mac(s, w1_001, u_200); fx_mac(s, w[1][5], u_101); fx_mac(s, w1_101, u_100); fx_mac(s, w[1][10], u_001); fx_mac(s, w1_201, u_000); z_mu_201 = fx_sum(s); }
  const Fx H_300 = fx_split(z_w2_300 + z_p_300 + FX_HALF, r);
  const Fx H_200 = fx_split(z_w2_200 + z_p_200 + FX_HALF, r);
  const Fx H_100 = fx_split(z_w2_100 + z_p_100 + FX_HALF, r);
  const int64_t z_w2_000 = fx_join(w[2][0]);
  int64_t z_mu_000; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_000); z_mu_000 = fx_sum(s); }
  const Fx e_000 = fx_split(((z_w2_000 - ((z_mu_000) >> 1)) << K.gshift) + FX_HALF, r0);
  int64_t z_p_000; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_000, K.gm1); z_p_000 = fx_sum<FX_C>(s); }
  const Fx H_000 = fx_split(z_w2_000 + z_p_000 + FX_HALF, r0);
  int64_t z_uH_300; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_300); fx_mac(s, u_100, H_200); fx_mac(s, u_200, H_100); fx_mac(s, u_300, H_000); z_uH_300 = fx_sum(s); }
  const Fx w2_201 = fx_split(fx_time<1>(3 * (z_uH_300), K.third) + FX_HALF, r);
  const int64_t z_w2_201 = fx_join(w2_201);
  const Fx e_201 = fx_split(((z_w2_201 - ((z_mu_201) >> 1)) << K.gshift) + FX_HALF, r);
  int64_t z_p_201; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_201, K.gm1); z_p_201 = fx_sum<FX_C>(s); }
  const Fx w1_102 = fx_split(fx_time<2>(2 * (z_mu_201 + z_p_201), K.third) + FX_HALF, r);
  const int64_t z_w1_102 = fx_join(w1_102);
  const Fx w0_003 = fx_split(fx_time<3>(1 * (z_w1_102), K.third) + FX_HALF, r);
  Fx u_400n; { FxAcc s = fx_zero(true); fx_mac_int(s, w[1][20], -(1 << 30)); fx_mac(s, w[0][5], u_300); fx_mac(s, w[0][10], u_200); fx_mac(s, w[0][15], u_100); fx_mac(s, w[0][20], u_000); u_400n = fx_split(fx_sum(s), r); }
  Fx u_400; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_400n, ninv); u_400 = fx_split(fx_sum<FX_C>(s), r); }
  int64_t z_mu_400; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_400); fx_mac(s, w[1][5], u_300); fx_mac(s, w[1][10], u_200); fx_mac(s, w[1][15], u_100); fx_mac(s, w[1][20], u_000); z_mu_400 = fx_sum(s); }
  const int64_t z_w2_400 = fx_join(w[2][20]);
  const Fx e_400 = fx_split(((z_w2_400 - ((z_mu_400) >> 1)) << K.gshift) + FX_HALF, r);
  int64_t z_p_400; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_400, K.gm1); z_p_400 = fx_sum<FX_C>(s); }
  const Fx w1_301 = fx_split(fx_time<1>(4 * (z_mu_400 + z_p_400), K.third) + FX_HALF, r);
  const int64_t z_w1_400 = fx_join(w[1][20]);
  const Fx w0_301 = fx_split(fx_time<1>(4 * (z_w1_400), K.third) + FX_HALF, r);
  Fx u_301n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_301, -(1 << 30)); fx_mac(s, w0_001, u_300); fx_mac(s, w[0][5], u_201); fx_mac(s, w0_101, u_200); fx_mac(s, w[0][10], u_101); fx_mac(s, w0_201, u_100); fx_mac(s, w[0][15], u_001); fx_mac(s, w0_301, u_000); u_301n = fx_split(fx_sum(s), r); }
  Fx u_301; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_301n, ninv); u_301 = fx_split(fx_sum<FX_C>(s), r); }
  int64_t z_mu_301; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_301); fx_mac(s, w1_001, u_300); fx_mac(s, w[1][5], u_201); fx_mac(s, w1_101, u_200); fx_mac(s, w[1][10], u_101); fx_mac(s, w1_201, u_100); fx_mac(s, w[1][15], u_001); fx_mac(s, w1_301, u_000); z_mu_301 = fx_sum(s); }
  const Fx H_400 = fx_split(z_w2_400 + z_p_400 + FX_HALF, r);
  int64_t z_uH_400; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_400); fx_mac(s, u_100, H_300); fx_mac(s, u_200, H_200); fx_mac(s, u_300, H_100); fx_mac(s, u_400, H_000); z_uH_400 = fx_sum(s); }
  const Fx w2_301 = fx_split(fx_time<1>(4 * (z_uH_400), K.third) + FX_HALF, r);
  const int64_t z_w2_301 = fx_join(w2_301);
  const Fx e_301 = fx_split(((z_w2_301 - ((z_mu_301) >> 1)) << K.gshift) + FX_HALF, r);
  int64_t z_p_301; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_301, K.gm1); z_p_301 = fx_sum<FX_C>(s); }
  const Fx w1_202 = fx_split(fx_time<2>(3 * (z_mu_301 + z_p_301), K.third) + FX_HALF, r);
  int64_t z_mu_101; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_101); fx_mac(s, w1_001, u_100); fx_mac(s, w[1][5], u_001); fx_mac(s, w1_101, u_000); z_mu_101 = fx_sum(s); }
  int64_t z_uH_200; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_200); fx_mac(s, u_100, H_100); fx_mac(s, u_200, H_000); z_uH_200 = fx_sum(s); }
  const Fx w2_101 = fx_split(fx_time<1>(2 * (z_uH_200), K.third) + FX_HALF, r);
  const int64_t z_w2_101 = fx_join(w2_101);
  const Fx e_101 = fx_split(((z_w2_101 - ((z_mu_101) >> 1)) << K.gshift) + FX_HALF, r);
  int64_t z_p_101; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_101, K.gm1); z_p_101 = fx_sum<FX_C>(s); }
  const Fx w1_002 = fx_split(fx_time<2>(1 * (z_mu_101 + z_p_101), K.third) + FX_HALF, r);
  Fx u_002n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_002, -(1 << 30)); fx_mac(s, w0_001, u_001); fx_mac(s, w0_002, u_000); u_002n = fx_split(fx_sum(s), r); }
  Fx u_002; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_002n, ninv); u_002 = fx_split(fx_sum<FX_C>(s), r); }
  const int64_t z_w1_201 = fx_join(w1_201);
  const Fx w0_102 = fx_split(fx_time<2>(2 * (z_w1_201), K.third) + FX_HALF, r);
  Fx u_102n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_102, -(1 << 30)); fx_mac(s, w0_001, u_101); fx_mac(s, w0_002, u_100); fx_mac(s, w[0][5], u_002); fx_mac(s, w0_101, u_001); fx_mac(s, w0_102, u_000); u_102n = fx_split(fx_sum(s), r); }
  Fx u_102; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_102n, ninv); u_102 = fx_split(fx_sum<FX_C>(s), r); }
  const int64_t z_w1_301 = fx_join(w1_301);
  const Fx w0_202 = fx_split(fx_time<2>(3 * (z_w1_301), K.third) + FX_HALF, r);
  Fx u_202n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_202, -(1 << 30)); fx_mac(s, w0_001, u_201); fx_mac(s, w0_002, u_200); fx_mac(s, w[0][5], u_102); fx_mac(s, w0_101, u_101); fx_mac(s, w0_102, u_100); fx_mac(s, w[0][10], u_002); fx_mac(s, w0_201, u_001); fx_mac(s, w0_202, u_000); u_202n = fx_split(fx_sum(s), r); }
  Fx u_202; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_202n, ninv); u_202 = fx_split(fx_sum<FX_C>(s), r); }
  int64_t z_mu_202; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_202); fx_mac(s, w1_001, u_201); fx_mac(s, w1_002, u_200); fx_mac(s, w[1][5], u_102); fx_mac(s, w1_101, u_101); fx_mac(s, w1_102, u_100); fx_mac(s, w[1][10], u_002); fx_mac(s, w1_201, u_001); fx_mac(s, w1_202, u_000); z_mu_202 = fx_sum(s); }
  const Fx H_301 = fx_split(z_w2_301 + z_p_301 + FX_HALF, r);
  const Fx H_201 = fx_split(z_w2_201 + z_p_201 + FX_HALF, r);
  const Fx H_101 = fx_split(z_w2_101 + z_p_101 + FX_HALF, r);
  int64_t z_uH_100; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_100); fx_mac(s, u_100, H_000); z_uH_100 = fx_sum(s); }
  const Fx w2_001 = fx_split(fx_time<1>(1 * (z_uH_100), K.third) + FX_HALF, r);
  const int64_t z_w2_001 = fx_join(w2_001);
  int64_t z_mu_001; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_001); fx_mac(s, w1_001, u_000); z_mu_001 = fx_sum(s); }
  const Fx e_001 = fx_split(((z_w2_001 - ((z_mu_001) >> 1)) << K.gshift) + FX_HALF, r);
  int64_t z_p_001; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_001, K.gm1); z_p_001 = fx_sum<FX_C>(s); }
  const Fx H_001 = fx_split(z_w2_001 + z_p_001 + FX_HALF, r);
  int64_t z_uH_301; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_301); fx_mac(s, u_001, H_300); fx_mac(s, u_100, H_201); fx_mac(s, u_101, H_200); fx_mac(s, u_200, H_101); fx_mac(s, u_201, H_100); fx_mac(s, u_300, H_001); fx_mac(s, u_301, H_000); z_uH_301 = fx_sum(s); }
  const Fx w2_202 = fx_split(fx_time<2>(3 * (z_uH_301), K.third) + FX_HALF, r);
  const int64_t z_w2_202 = fx_join(w2_202);
  const Fx e_202 = fx_split(((z_w2_202 - ((z_mu_202) >> 1)) << K.gshift) + FX_HALF, r);
  int64_t z_p_202; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_202, K.gm1); z_p_202 = fx_sum<FX_C>(s); }
  const Fx w1_103 = fx_split(fx_time<3>(2 * (z_mu_202 + z_p_202), K.third) + FX_HALF, r);
  const int64_t z_w1_103 = fx_join(w1_103);
  const Fx w0_004 = fx_split(fx_time<4>(1 * (z_w1_103), K.third) + FX_HALF, r);
  int64_t z_mu_102; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_102); fx_mac(s, w1_001, u_101); fx_mac(s, w1_002, u_100); fx_mac(s, w[1][5], u_002); fx_mac(s, w1_101, u_001); fx_mac(s, w1_102, u_000); z_mu_102 = fx_sum(s); }
  int64_t z_uH_201; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_201); fx_mac(s, u_001, H_200); fx_mac(s, u_100, H_101); fx_mac(s, u_101, H_100); fx_mac(s, u_200, H_001); fx_mac(s, u_201, H_000); z_uH_201 = fx_sum(s); }
  const Fx w2_102 = fx_split(fx_time<2>(2 * (z_uH_201), K.third) + FX_HALF, r);
  const int64_t z_w2_102 = fx_join(w2_102);
  const Fx e_102 = fx_split(((z_w2_102 - ((z_mu_102) >> 1)) << K.gshift) + FX_HALF, r);
  int64_t z_p_102; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_102, K.gm1); z_p_102 = fx_sum<FX_C>(s); }
  const Fx w1_003 = fx_split(fx_time<3>(1 * (z_mu_102 + z_p_102), K.third) + FX_HALF, r);
  Fx u_003n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_003, -(1 << 30)); fx_mac(s, w0_001, u_002); fx_mac(s, w0_002, u_001); fx_mac(s, w0_003, u_000); u_003n = fx_split(fx_sum(s), r); }
  Fx u_003; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_003n, ninv); u_003 = fx_split(fx_sum<FX_C>(s), r); }
  const int64_t z_w1_202 = fx_join(w1_202);
  const Fx w0_103 = fx_split(fx_time<3>(2 * (z_w1_202), K.third) + FX_HALF, r);
  Fx u_103n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_103, -(1 << 30)); fx_mac(s, w0_001, u_102); fx_mac(s, w0_002, u_101); fx_mac(s, w0_003, u_100); fx_mac(s, w[0][5], u_003); fx_mac(s, w0_101, u_002); fx_mac(s, w0_102, u_001); fx_mac(s, w0_103, u_000); u_103n = fx_split(fx_sum(s), r); }
  Fx u_103; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_103n, ninv); u_103 = fx_split(fx_sum<FX_C>(s), r); }
  int64_t z_mu_103; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_103); fx_mac(s, w1_001, u_102); fx_mac(s, w1_002, u_101); fx_mac(s, w1_003, u_100); fx_mac(s, w[1][5], u_003); fx_mac(s, w1_101, u_002); fx_mac(s, w1_102, u_001); fx_mac(s, w1_103, u_000); z_mu_103 = fx_sum(s); }
  const Fx H_202 = fx_split(z_w2_202 + z_p_202 + FX_HALF, r);
  const Fx H_102 = fx_split(z_w2_102 + z_p_102 + FX_HALF, r);
  int64_t z_uH_101; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_101); fx_mac(s, u_001, H_100); fx_mac(s, u_100, H_001); fx_mac(s, u_101, H_000); z_uH_101 = fx_sum(s); }
  const Fx w2_002 = fx_split(fx_time<2>(1 * (z_uH_101), K.third) + FX_HALF, r);
  const int64_t z_w2_002 = fx_join(w2_002);
  int64_t z_mu_002; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_002); fx_mac(s, w1_001, u_001); fx_mac(s, w1_002, u_000); z_mu_002 = fx_sum(s); }
  const Fx e_002 = fx_split(((z_w2_002 - ((z_mu_002) >> 1)) << K.gshift) + FX_HALF, r);
  int64_t z_p_002; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_002, K.gm1); z_p_002 = fx_sum<FX_C>(s); }
  const Fx H_002 = fx_split(z_w2_002 + z_p_002 + FX_HALF, r);
  int64_t z_uH_202; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_202); fx_mac(s, u_001, H_201); fx_mac(s, u_002, H_200); fx_mac(s, u_100, H_102); fx_mac(s, u_101, H_101); fx_mac(s, u_102, H_100); fx_mac(s, u_200, H_002); fx_mac(s, u_201, H_001); fx_mac(s, u_202, H_000); z_uH_202 = fx_sum(s); }
  const Fx w2_103 = fx_split(fx_time<3>(2 * (z_uH_202), K.third) + FX_HALF, r);
  const int64_t z_w2_103 = fx_join(w2_103);
  const Fx e_103 = fx_split(((z_w2_103 - ((z_mu_103) >> 1)) << K.gshift) + FX_HALF, r);
  int64_t z_p_103; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_103, K.gm1); z_p_103 = fx_sum<FX_C>(s); }
  const Fx w1_004 = fx_split(fx_time<4>(1 * (z_mu_103 + z_p_103), K.third) + FX_HALF, r);
  int64_t z_uH_102; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_102); fx_mac(s, u_001, H_101); fx_mac(s, u_002, H_100); fx_mac(s, u_100, H_002); fx_mac(s, u_101, H_001); fx_mac(s, u_102, H_000); z_uH_102 = fx_sum(s); }
  const Fx w2_003 = fx_split(fx_time<3>(1 * (z_uH_102), K.third) + FX_HALF, r);
  const Fx H_103 = fx_split(z_w2_103 + z_p_103 + FX_HALF, r);
  const int64_t z_w2_003 = fx_join(w2_003);
  int64_t z_mu_003; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_003); fx_mac(s, w1_001, u_002); fx_mac(s, w1_002, u_001); fx_mac(s, w1_003, u_000); z_mu_003 = fx_sum(s); }
  const Fx e_003 = fx_split(((z_w2_003 - ((z_mu_003) >> 1)) << K.gshift) + FX_HALF, r);
  int64_t z_p_003; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_003, K.gm1); z_p_003 = fx_sum<FX_C>(s); }
  const Fx H_003 = fx_split(z_w2_003 + z_p_003 + FX_HALF, r);
  int64_t z_uH_103; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_103); fx_mac(s, u_001, H_102); fx_mac(s, u_002, H_101); fx_mac(s, u_003, H_100); fx_mac(s, u_100, H_003); fx_mac(s, u_101, H_002); fx_mac(s, u_102, H_001); fx_mac(s, u_103, H_000); z_uH_103 = fx_sum(s); }
  const Fx w2_004 = fx_split(fx_time<4>(1 * (z_uH_103), K.third) + FX_HALF, r);
  t[0][1] = fx_join(w0_001);
  t[0][2] = fx_join(w0_002);
  t[0][3] = fx_join(w0_003);
  t[0][4] = fx_join(w0_004);
  t[1][1] = fx_join(w1_001);
  t[1][2] = fx_join(w1_002);
  t[1][3] = fx_join(w1_003);
  t[1][4] = fx_join(w1_004);
  t[2][1] = fx_join(w2_001);
  t[2][2] = fx_join(w2_002);
  t[2][3] = fx_join(w2_003);
  t[2][4] = fx_join(w2_004);
}

// 2D Euler, two lanes per point: S gives the shared series and constants, ninv = -1/rho0;
// S.next() takes the coefficients of the next slice.
template <typename Store>
FX_DEV void ck_euler2d_lane(Store& S, Fx ninv, Fx gm1, Fx third, int gshift, FxRange& r) {
  FxRange r0{0};  // leading coefficients are in range by their scales
  // ---- slice 0
  Fx vel000;
  Fx vel100;
  Fx vel010;
  Fx vel200;
  Fx vel110;
  Fx vel020;
  Fx vel300;
  Fx vel210;
  Fx vel120;
  Fx vel030;
  Fx vel400;
  Fx vel310;
  Fx vel220;
  Fx vel130;
  Fx vel040;
  {
  const Fx rho100 = S.ldrho(0, 1, 0);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 0, 0), -(1 << 30));
    const Fx n = fx_split(fx_sum(s), r0);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel000 = fx_split(fx_sum<FX_C>(z), r0); }
  const Fx rho010 = S.ldrho(0, 0, 1);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 1, 0), -(1 << 30));
    fx_mac(s, rho100, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel100 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho200 = S.ldrho(0, 2, 0);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 0, 1), -(1 << 30));
    fx_mac(s, rho010, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel010 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho110 = S.ldrho(0, 1, 1);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 2, 0), -(1 << 30));
    fx_mac(s, rho100, vel100);
    fx_mac(s, rho200, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel200 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho020 = S.ldrho(0, 0, 2);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 1, 1), -(1 << 30));
    fx_mac(s, rho010, vel100);
    fx_mac(s, rho100, vel010);
    fx_mac(s, rho110, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel110 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho300 = S.ldrho(0, 3, 0);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 0, 2), -(1 << 30));
    fx_mac(s, rho010, vel010);
    fx_mac(s, rho020, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel020 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho210 = S.ldrho(0, 2, 1);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 3, 0), -(1 << 30));
    fx_mac(s, rho100, vel200);
    fx_mac(s, rho200, vel100);
    fx_mac(s, rho300, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel300 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho120 = S.ldrho(0, 1, 2);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 2, 1), -(1 << 30));
    fx_mac(s, rho010, vel200);
    fx_mac(s, rho100, vel110);
    fx_mac(s, rho110, vel100);
    fx_mac(s, rho200, vel010);
    fx_mac(s, rho210, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel210 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho030 = S.ldrho(0, 0, 3);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 1, 2), -(1 << 30));
    fx_mac(s, rho010, vel110);
    fx_mac(s, rho020, vel100);
    fx_mac(s, rho100, vel020);
    fx_mac(s, rho110, vel010);
    fx_mac(s, rho120, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel120 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho400 = S.ldrho(0, 4, 0);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 0, 3), -(1 << 30));
    fx_mac(s, rho010, vel020);
    fx_mac(s, rho020, vel010);
    fx_mac(s, rho030, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel030 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho310 = S.ldrho(0, 3, 1);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 4, 0), -(1 << 30));
    fx_mac(s, rho100, vel300);
    fx_mac(s, rho200, vel200);
    fx_mac(s, rho300, vel100);
    fx_mac(s, rho400, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel400 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho220 = S.ldrho(0, 2, 2);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 3, 1), -(1 << 30));
    fx_mac(s, rho010, vel300);
    fx_mac(s, rho100, vel210);
    fx_mac(s, rho110, vel200);
    fx_mac(s, rho200, vel110);
    fx_mac(s, rho210, vel100);
    fx_mac(s, rho300, vel010);
    fx_mac(s, rho310, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel310 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho130 = S.ldrho(0, 1, 3);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 2, 2), -(1 << 30));
    fx_mac(s, rho010, vel210);
    fx_mac(s, rho020, vel200);
    fx_mac(s, rho100, vel120);
    fx_mac(s, rho110, vel110);
    fx_mac(s, rho120, vel100);
    fx_mac(s, rho200, vel020);
    fx_mac(s, rho210, vel010);
    fx_mac(s, rho220, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel220 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho040 = S.ldrho(0, 0, 4);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 1, 3), -(1 << 30));
    fx_mac(s, rho010, vel120);
    fx_mac(s, rho020, vel110);
    fx_mac(s, rho030, vel100);
    fx_mac(s, rho100, vel030);
    fx_mac(s, rho110, vel020);
    fx_mac(s, rho120, vel010);
    fx_mac(s, rho130, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel130 = fx_split(fx_sum<FX_C>(z), r); }
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 0, 4), -(1 << 30));
    fx_mac(s, rho010, vel030);
    fx_mac(s, rho020, vel020);
    fx_mac(s, rho030, vel010);
    fx_mac(s, rho040, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel040 = fx_split(fx_sum<FX_C>(z), r); }
  }
  int64_t k000;
  int64_t k100;
  int64_t k010;
  int64_t k200;
  int64_t k110;
  int64_t k020;
  int64_t k300;
  int64_t k210;
  int64_t k120;
  int64_t k030;
  int64_t k400;
  int64_t k310;
  int64_t k220;
  int64_t k130;
  int64_t k040;
  {
  const Fx mom000 = S.ldmom(0, 0, 0);
  const Fx mom100 = S.ldmom(0, 1, 0);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel000);
    k000 = fx_sum(s); }
  const Fx mom010 = S.ldmom(0, 0, 1);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel100);
    fx_mac(s, mom100, vel000);
    k100 = fx_sum(s); }
  const Fx mom200 = S.ldmom(0, 2, 0);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel010);
    fx_mac(s, mom010, vel000);
    k010 = fx_sum(s); }
  const Fx mom110 = S.ldmom(0, 1, 1);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel200);
    fx_mac(s, mom100, vel100);
    fx_mac(s, mom200, vel000);
    k200 = fx_sum(s); }
  const Fx mom020 = S.ldmom(0, 0, 2);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel110);
    fx_mac(s, mom010, vel100);
    fx_mac(s, mom100, vel010);
    fx_mac(s, mom110, vel000);
    k110 = fx_sum(s); }
  const Fx mom300 = S.ldmom(0, 3, 0);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel020);
    fx_mac(s, mom010, vel010);
    fx_mac(s, mom020, vel000);
    k020 = fx_sum(s); }
  const Fx mom210 = S.ldmom(0, 2, 1);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel300);
    fx_mac(s, mom100, vel200);
    fx_mac(s, mom200, vel100);
    fx_mac(s, mom300, vel000);
    k300 = fx_sum(s); }
  const Fx mom120 = S.ldmom(0, 1, 2);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel210);
    fx_mac(s, mom010, vel200);
    fx_mac(s, mom100, vel110);
    fx_mac(s, mom110, vel100);
    fx_mac(s, mom200, vel010);
    fx_mac(s, mom210, vel000);
    k210 = fx_sum(s); }
  const Fx mom030 = S.ldmom(0, 0, 3);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel120);
    fx_mac(s, mom010, vel110);
    fx_mac(s, mom020, vel100);
    fx_mac(s, mom100, vel020);
    fx_mac(s, mom110, vel010);
    fx_mac(s, mom120, vel000);
    k120 = fx_sum(s); }
  const Fx mom400 = S.ldmom(0, 4, 0);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel030);
    fx_mac(s, mom010, vel020);
    fx_mac(s, mom020, vel010);
    fx_mac(s, mom030, vel000);
    k030 = fx_sum(s); }
  const Fx mom310 = S.ldmom(0, 3, 1);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel400);
    fx_mac(s, mom100, vel300);
    fx_mac(s, mom200, vel200);
    fx_mac(s, mom300, vel100);
    fx_mac(s, mom400, vel000);
    k400 = fx_sum(s); }
  const Fx mom220 = S.ldmom(0, 2, 2);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel310);
    fx_mac(s, mom010, vel300);
    fx_mac(s, mom100, vel210);
    fx_mac(s, mom110, vel200);
    fx_mac(s, mom200, vel110);
    fx_mac(s, mom210, vel100);
    fx_mac(s, mom300, vel010);
    fx_mac(s, mom310, vel000);
    k310 = fx_sum(s); }
  const Fx mom130 = S.ldmom(0, 1, 3);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel220);
    fx_mac(s, mom010, vel210);
    fx_mac(s, mom020, vel200);
    fx_mac(s, mom100, vel120);
    fx_mac(s, mom110, vel110);
    fx_mac(s, mom120, vel100);
    fx_mac(s, mom200, vel020);
    fx_mac(s, mom210, vel010);
    fx_mac(s, mom220, vel000);
    k220 = fx_sum(s); }
  const Fx mom040 = S.ldmom(0, 0, 4);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel130);
    fx_mac(s, mom010, vel120);
    fx_mac(s, mom020, vel110);
    fx_mac(s, mom030, vel100);
    fx_mac(s, mom100, vel030);
    fx_mac(s, mom110, vel020);
    fx_mac(s, mom120, vel010);
    fx_mac(s, mom130, vel000);
    k130 = fx_sum(s); }
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel040);
    fx_mac(s, mom010, vel030);
    fx_mac(s, mom020, vel020);
    fx_mac(s, mom030, vel010);
    fx_mac(s, mom040, vel000);
    k040 = fx_sum(s); }
  }
  int64_t f100;
  int64_t f200;
  int64_t f110;
  int64_t f300;
  int64_t f210;
  int64_t f120;
  int64_t f400;
  int64_t f310;
  int64_t f220;
  int64_t f130;
  { const int64_t E = S.ldE(0, 0, 0);
    const Fx e = fx_split(((E - ((k000 + S.swap(k000)) >> 1)) << gshift) + FX_HALF, r0);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 0, 0, fx_split(E + p + FX_HALF, r0));
  }
  { const int64_t E = S.ldE(0, 1, 0);
    const Fx e = fx_split(((E - ((k100 + S.swap(k010)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 1, 0, fx_split(E + p + FX_HALF, r));
    f100 = k100 + p;
  }
  { const int64_t E = S.ldE(0, 0, 1);
    const Fx e = fx_split(((E - ((k010 + S.swap(k100)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 0, 1, fx_split(E + p + FX_HALF, r));
  }
  { const int64_t E = S.ldE(0, 2, 0);
    const Fx e = fx_split(((E - ((k200 + S.swap(k020)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 2, 0, fx_split(E + p + FX_HALF, r));
    f200 = k200 + p;
  }
  { const int64_t E = S.ldE(0, 1, 1);
    const Fx e = fx_split(((E - ((k110 + S.swap(k110)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 1, 1, fx_split(E + p + FX_HALF, r));
    f110 = k110 + p;
  }
  { const int64_t E = S.ldE(0, 0, 2);
    const Fx e = fx_split(((E - ((k020 + S.swap(k200)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 0, 2, fx_split(E + p + FX_HALF, r));
  }
  { const int64_t E = S.ldE(0, 3, 0);
    const Fx e = fx_split(((E - ((k300 + S.swap(k030)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 3, 0, fx_split(E + p + FX_HALF, r));
    f300 = k300 + p;
  }
  { const int64_t E = S.ldE(0, 2, 1);
    const Fx e = fx_split(((E - ((k210 + S.swap(k120)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 2, 1, fx_split(E + p + FX_HALF, r));
    f210 = k210 + p;
  }
  { const int64_t E = S.ldE(0, 1, 2);
    const Fx e = fx_split(((E - ((k120 + S.swap(k210)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 1, 2, fx_split(E + p + FX_HALF, r));
    f120 = k120 + p;
  }
  { const int64_t E = S.ldE(0, 0, 3);
    const Fx e = fx_split(((E - ((k030 + S.swap(k300)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 0, 3, fx_split(E + p + FX_HALF, r));
  }
  { const int64_t E = S.ldE(0, 4, 0);
    const Fx e = fx_split(((E - ((k400 + S.swap(k040)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 4, 0, fx_split(E + p + FX_HALF, r));
    f400 = k400 + p;
  }
  { const int64_t E = S.ldE(0, 3, 1);
    const Fx e = fx_split(((E - ((k310 + S.swap(k130)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 3, 1, fx_split(E + p + FX_HALF, r));
    f310 = k310 + p;
  }
  { const int64_t E = S.ldE(0, 2, 2);
    const Fx e = fx_split(((E - ((k220 + S.swap(k220)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 2, 2, fx_split(E + p + FX_HALF, r));
    f220 = k220 + p;
  }
  { const int64_t E = S.ldE(0, 1, 3);
    const Fx e = fx_split(((E - ((k130 + S.swap(k310)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 1, 3, fx_split(E + p + FX_HALF, r));
    f130 = k130 + p;
  }
  { const int64_t E = S.ldE(0, 0, 4);
    const Fx e = fx_split(((E - ((k040 + S.swap(k400)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 0, 4, fx_split(E + p + FX_HALF, r));
  }
  int64_t drho000;
  int64_t drho100;
  int64_t drho010;
  int64_t drho200;
  int64_t drho110;
  int64_t drho020;
  int64_t drho300;
  int64_t drho210;
  int64_t drho120;
  int64_t drho030;
  int64_t dmom000;
  int64_t dmom100;
  int64_t dmom010;
  int64_t dmom200;
  int64_t dmom110;
  int64_t dmom020;
  int64_t dmom300;
  int64_t dmom210;
  int64_t dmom120;
  int64_t dmom030;
  int64_t dE000;
  int64_t dE100;
  int64_t dE010;
  int64_t dE200;
  int64_t dE110;
  int64_t dE020;
  int64_t dE300;
  int64_t dE210;
  int64_t dE120;
  int64_t dE030;
  drho000 = 1 * fx_join(S.ldmom(0, 1, 0));
  dmom000 = 1 * f100;
  drho100 = 2 * fx_join(S.ldmom(0, 2, 0));
  dmom100 = 2 * f200;
  drho010 = 1 * fx_join(S.ldmom(0, 1, 1));
  dmom010 = 1 * f110;
  drho200 = 3 * fx_join(S.ldmom(0, 3, 0));
  dmom200 = 3 * f300;
  drho110 = 2 * fx_join(S.ldmom(0, 2, 1));
  dmom110 = 2 * f210;
  drho020 = 1 * fx_join(S.ldmom(0, 1, 2));
  dmom020 = 1 * f120;
  drho300 = 4 * fx_join(S.ldmom(0, 4, 0));
  dmom300 = 4 * f400;
  drho210 = 3 * fx_join(S.ldmom(0, 3, 1));
  dmom210 = 3 * f310;
  drho120 = 2 * fx_join(S.ldmom(0, 2, 2));
  dmom120 = 2 * f220;
  drho030 = 1 * fx_join(S.ldmom(0, 1, 3));
  dmom030 = 1 * f130;
  #pragma unroll 1
  for (int s = 0; s < 2; ++s) {
  const Fx ser000 = S.ldser(s, 0, 0, 0);
  const Fx ser100 = S.ldser(s, 0, 1, 0);
  const Fx ser200 = S.ldser(s, 0, 2, 0);
  int64_t z00;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel100);
    fx_mac(s, ser100, vel000);
    z00 = fx_sum(s); }
  dE000 = 1 * z00;
  const Fx ser010 = S.ldser(s, 0, 0, 1);
  const Fx ser110 = S.ldser(s, 0, 1, 1);
  int64_t z10;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel200);
    fx_mac(s, ser100, vel100);
    fx_mac(s, ser200, vel000);
    z10 = fx_sum(s); }
  dE100 = 2 * z10;
  const Fx ser300 = S.ldser(s, 0, 3, 0);
  int64_t z01;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel110);
    fx_mac(s, ser010, vel100);
    fx_mac(s, ser100, vel010);
    fx_mac(s, ser110, vel000);
    z01 = fx_sum(s); }
  dE010 = 1 * z01;
  const Fx ser210 = S.ldser(s, 0, 2, 1);
  int64_t z20;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel300);
    fx_mac(s, ser100, vel200);
    fx_mac(s, ser200, vel100);
    fx_mac(s, ser300, vel000);
    z20 = fx_sum(s); }
  dE200 = 3 * z20;
  const Fx ser020 = S.ldser(s, 0, 0, 2);
  const Fx ser120 = S.ldser(s, 0, 1, 2);
  int64_t z11;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel210);
    fx_mac(s, ser010, vel200);
    fx_mac(s, ser100, vel110);
    fx_mac(s, ser110, vel100);
    fx_mac(s, ser200, vel010);
    fx_mac(s, ser210, vel000);
    z11 = fx_sum(s); }
  dE110 = 2 * z11;
  const Fx ser400 = S.ldser(s, 0, 4, 0);
  int64_t z02;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel120);
    fx_mac(s, ser010, vel110);
    fx_mac(s, ser020, vel100);
    fx_mac(s, ser100, vel020);
    fx_mac(s, ser110, vel010);
    fx_mac(s, ser120, vel000);
    z02 = fx_sum(s); }
  dE020 = 1 * z02;
  const Fx ser310 = S.ldser(s, 0, 3, 1);
  int64_t z30;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel400);
    fx_mac(s, ser100, vel300);
    fx_mac(s, ser200, vel200);
    fx_mac(s, ser300, vel100);
    fx_mac(s, ser400, vel000);
    z30 = fx_sum(s); }
  dE300 = 4 * z30;
  const Fx ser220 = S.ldser(s, 0, 2, 2);
  int64_t z21;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel310);
    fx_mac(s, ser010, vel300);
    fx_mac(s, ser100, vel210);
    fx_mac(s, ser110, vel200);
    fx_mac(s, ser200, vel110);
    fx_mac(s, ser210, vel100);
    fx_mac(s, ser300, vel010);
    fx_mac(s, ser310, vel000);
    z21 = fx_sum(s); }
  dE210 = 3 * z21;
  const Fx ser030 = S.ldser(s, 0, 0, 3);
  const Fx ser130 = S.ldser(s, 0, 1, 3);
  int64_t z12;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel220);
    fx_mac(s, ser010, vel210);
    fx_mac(s, ser020, vel200);
    fx_mac(s, ser100, vel120);
    fx_mac(s, ser110, vel110);
    fx_mac(s, ser120, vel100);
    fx_mac(s, ser200, vel020);
    fx_mac(s, ser210, vel010);
    fx_mac(s, ser220, vel000);
    z12 = fx_sum(s); }
  dE120 = 2 * z12;
  int64_t z03;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel130);
    fx_mac(s, ser010, vel120);
    fx_mac(s, ser020, vel110);
    fx_mac(s, ser030, vel100);
    fx_mac(s, ser100, vel030);
    fx_mac(s, ser110, vel020);
    fx_mac(s, ser120, vel010);
    fx_mac(s, ser130, vel000);
    z03 = fx_sum(s); }
  dE030 = 1 * z03;
  if (s == 0) {
    S.stoth(1, 0, 0, dE000);
    S.stoth(1, 1, 0, dE100);
    S.stoth(1, 0, 1, dE010);
    S.stoth(1, 2, 0, dE200);
    S.stoth(1, 1, 1, dE110);
    S.stoth(1, 0, 2, dE020);
    S.stoth(1, 3, 0, dE300);
    S.stoth(1, 2, 1, dE210);
    S.stoth(1, 1, 2, dE120);
    S.stoth(1, 0, 3, dE030);
  } }
  S.sync();
  { const int64_t own = dmom000 + S.ldown(1, 0, 0);
    const int64_t both = S.pick(drho000, dE000) + S.swap(S.pick(dE000, drho000));
    S.next(1, 0, 0, fx_time<1>(own, third), fx_time<1>(both, third), r); }
  { const int64_t own = dmom100 + S.ldown(1, 1, 0);
    const int64_t both = S.pick(drho100, dE100) + S.swap(S.pick(dE010, drho010));
    S.next(1, 1, 0, fx_time<1>(own, third), fx_time<1>(both, third), r); }
  { const int64_t own = dmom010 + S.ldown(1, 0, 1);
    const int64_t both = S.pick(drho010, dE010) + S.swap(S.pick(dE100, drho100));
    S.next(1, 0, 1, fx_time<1>(own, third), fx_time<1>(both, third), r); }
  { const int64_t own = dmom200 + S.ldown(1, 2, 0);
    const int64_t both = S.pick(drho200, dE200) + S.swap(S.pick(dE020, drho020));
    S.next(1, 2, 0, fx_time<1>(own, third), fx_time<1>(both, third), r); }
  { const int64_t own = dmom110 + S.ldown(1, 1, 1);
    const int64_t both = S.pick(drho110, dE110) + S.swap(S.pick(dE110, drho110));
    S.next(1, 1, 1, fx_time<1>(own, third), fx_time<1>(both, third), r); }
  { const int64_t own = dmom020 + S.ldown(1, 0, 2);
    const int64_t both = S.pick(drho020, dE020) + S.swap(S.pick(dE200, drho200));
    S.next(1, 0, 2, fx_time<1>(own, third), fx_time<1>(both, third), r); }
  { const int64_t own = dmom300 + S.ldown(1, 3, 0);
    const int64_t both = S.pick(drho300, dE300) + S.swap(S.pick(dE030, drho030));
    S.next(1, 3, 0, fx_time<1>(own, third), fx_time<1>(both, third), r); }
  { const int64_t own = dmom210 + S.ldown(1, 2, 1);
    const int64_t both = S.pick(drho210, dE210) + S.swap(S.pick(dE120, drho120));
    S.next(1, 2, 1, fx_time<1>(own, third), fx_time<1>(both, third), r); }
  { const int64_t own = dmom120 + S.ldown(1, 1, 2);
    const int64_t both = S.pick(drho120, dE120) + S.swap(S.pick(dE210, drho210));
    S.next(1, 1, 2, fx_time<1>(own, third), fx_time<1>(both, third), r); }
  { const int64_t own = dmom030 + S.ldown(1, 0, 3);
    const int64_t both = S.pick(drho030, dE030) + S.swap(S.pick(dE300, drho300));
    S.next(1, 0, 3, fx_time<1>(own, third), fx_time<1>(both, third), r); }
  S.sync();
  const int64_t E001 = S.ldE(1, 0, 0);
  const int64_t E101 = S.ldE(1, 1, 0);
  const int64_t E011 = S.ldE(1, 0, 1);
  const int64_t E201 = S.ldE(1, 2, 0);
  const int64_t E111 = S.ldE(1, 1, 1);
  const int64_t E021 = S.ldE(1, 0, 2);
  const int64_t E301 = S.ldE(1, 3, 0);
  const int64_t E211 = S.ldE(1, 2, 1);
  const int64_t E121 = S.ldE(1, 1, 2);
  const int64_t E031 = S.ldE(1, 0, 3);
  // ---- slice 1
  Fx vel001;
  Fx vel101;
  Fx vel011;
  Fx vel201;
  Fx vel111;
  Fx vel021;
  Fx vel301;
  Fx vel211;
  Fx vel121;
  Fx vel031;
  {
  const Fx rho001 = S.ldrho(1, 0, 0);
  const Fx rho100 = S.ldrho(0, 1, 0);
  const Fx rho101 = S.ldrho(1, 1, 0);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(1, 0, 0), -(1 << 30));
    fx_mac(s, rho001, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel001 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho010 = S.ldrho(0, 0, 1);
  const Fx rho011 = S.ldrho(1, 0, 1);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(1, 1, 0), -(1 << 30));
    fx_mac(s, rho001, vel100);
    fx_mac(s, rho100, vel001);
    fx_mac(s, rho101, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel101 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho200 = S.ldrho(0, 2, 0);
  const Fx rho201 = S.ldrho(1, 2, 0);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(1, 0, 1), -(1 << 30));
    fx_mac(s, rho001, vel010);
    fx_mac(s, rho010, vel001);
    fx_mac(s, rho011, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel011 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho110 = S.ldrho(0, 1, 1);
  const Fx rho111 = S.ldrho(1, 1, 1);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(1, 2, 0), -(1 << 30));
    fx_mac(s, rho001, vel200);
    fx_mac(s, rho100, vel101);
    fx_mac(s, rho101, vel100);
    fx_mac(s, rho200, vel001);
    fx_mac(s, rho201, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel201 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho020 = S.ldrho(0, 0, 2);
  const Fx rho021 = S.ldrho(1, 0, 2);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(1, 1, 1), -(1 << 30));
    fx_mac(s, rho001, vel110);
    fx_mac(s, rho010, vel101);
    fx_mac(s, rho011, vel100);
    fx_mac(s, rho100, vel011);
    fx_mac(s, rho101, vel010);
    fx_mac(s, rho110, vel001);
    fx_mac(s, rho111, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel111 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho300 = S.ldrho(0, 3, 0);
  const Fx rho301 = S.ldrho(1, 3, 0);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(1, 0, 2), -(1 << 30));
    fx_mac(s, rho001, vel020);
    fx_mac(s, rho010, vel011);
    fx_mac(s, rho011, vel010);
    fx_mac(s, rho020, vel001);
    fx_mac(s, rho021, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel021 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho210 = S.ldrho(0, 2, 1);
  const Fx rho211 = S.ldrho(1, 2, 1);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(1, 3, 0), -(1 << 30));
    fx_mac(s, rho001, vel300);
    fx_mac(s, rho100, vel201);
    fx_mac(s, rho101, vel200);
    fx_mac(s, rho200, vel101);
    fx_mac(s, rho201, vel100);
    fx_mac(s, rho300, vel001);
    fx_mac(s, rho301, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel301 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho120 = S.ldrho(0, 1, 2);
  const Fx rho121 = S.ldrho(1, 1, 2);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(1, 2, 1), -(1 << 30));
    fx_mac(s, rho001, vel210);
    fx_mac(s, rho010, vel201);
    fx_mac(s, rho011, vel200);
    fx_mac(s, rho100, vel111);
    fx_mac(s, rho101, vel110);
    fx_mac(s, rho110, vel101);
    fx_mac(s, rho111, vel100);
    fx_mac(s, rho200, vel011);
    fx_mac(s, rho201, vel010);
    fx_mac(s, rho210, vel001);
    fx_mac(s, rho211, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel211 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho030 = S.ldrho(0, 0, 3);
  const Fx rho031 = S.ldrho(1, 0, 3);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(1, 1, 2), -(1 << 30));
    fx_mac(s, rho001, vel120);
    fx_mac(s, rho010, vel111);
    fx_mac(s, rho011, vel110);
    fx_mac(s, rho020, vel101);
    fx_mac(s, rho021, vel100);
    fx_mac(s, rho100, vel021);
    fx_mac(s, rho101, vel020);
    fx_mac(s, rho110, vel011);
    fx_mac(s, rho111, vel010);
    fx_mac(s, rho120, vel001);
    fx_mac(s, rho121, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel121 = fx_split(fx_sum<FX_C>(z), r); }
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(1, 0, 3), -(1 << 30));
    fx_mac(s, rho001, vel030);
    fx_mac(s, rho010, vel021);
    fx_mac(s, rho011, vel020);
    fx_mac(s, rho020, vel011);
    fx_mac(s, rho021, vel010);
    fx_mac(s, rho030, vel001);
    fx_mac(s, rho031, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel031 = fx_split(fx_sum<FX_C>(z), r); }
  }
  int64_t k001;
  int64_t k101;
  int64_t k011;
  int64_t k201;
  int64_t k111;
  int64_t k021;
  int64_t k301;
  int64_t k211;
  int64_t k121;
  int64_t k031;
  {
  const Fx mom000 = S.ldmom(0, 0, 0);
  const Fx mom001 = S.ldmom(1, 0, 0);
  const Fx mom100 = S.ldmom(0, 1, 0);
  const Fx mom101 = S.ldmom(1, 1, 0);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel001);
    fx_mac(s, mom001, vel000);
    k001 = fx_sum(s); }
  const Fx mom010 = S.ldmom(0, 0, 1);
  const Fx mom011 = S.ldmom(1, 0, 1);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel101);
    fx_mac(s, mom001, vel100);
    fx_mac(s, mom100, vel001);
    fx_mac(s, mom101, vel000);
    k101 = fx_sum(s); }
  const Fx mom200 = S.ldmom(0, 2, 0);
  const Fx mom201 = S.ldmom(1, 2, 0);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel011);
    fx_mac(s, mom001, vel010);
    fx_mac(s, mom010, vel001);
    fx_mac(s, mom011, vel000);
    k011 = fx_sum(s); }
  const Fx mom110 = S.ldmom(0, 1, 1);
  const Fx mom111 = S.ldmom(1, 1, 1);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel201);
    fx_mac(s, mom001, vel200);
    fx_mac(s, mom100, vel101);
    fx_mac(s, mom101, vel100);
    fx_mac(s, mom200, vel001);
    fx_mac(s, mom201, vel000);
    k201 = fx_sum(s); }
  const Fx mom020 = S.ldmom(0, 0, 2);
  const Fx mom021 = S.ldmom(1, 0, 2);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel111);
    fx_mac(s, mom001, vel110);
    fx_mac(s, mom010, vel101);
    fx_mac(s, mom011, vel100);
    fx_mac(s, mom100, vel011);
    fx_mac(s, mom101, vel010);
    fx_mac(s, mom110, vel001);
    fx_mac(s, mom111, vel000);
    k111 = fx_sum(s); }
  const Fx mom300 = S.ldmom(0, 3, 0);
  const Fx mom301 = S.ldmom(1, 3, 0);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel021);
    fx_mac(s, mom001, vel020);
    fx_mac(s, mom010, vel011);
    fx_mac(s, mom011, vel010);
    fx_mac(s, mom020, vel001);
    fx_mac(s, mom021, vel000);
    k021 = fx_sum(s); }
  const Fx mom210 = S.ldmom(0, 2, 1);
  const Fx mom211 = S.ldmom(1, 2, 1);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel301);
    fx_mac(s, mom001, vel300);
    fx_mac(s, mom100, vel201);
    fx_mac(s, mom101, vel200);
    fx_mac(s, mom200, vel101);
    fx_mac(s, mom201, vel100);
    fx_mac(s, mom300, vel001);
    fx_mac(s, mom301, vel000);
    k301 = fx_sum(s); }
  const Fx mom120 = S.ldmom(0, 1, 2);
  const Fx mom121 = S.ldmom(1, 1, 2);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel211);
    fx_mac(s, mom001, vel210);
    fx_mac(s, mom010, vel201);
    fx_mac(s, mom011, vel200);
    fx_mac(s, mom100, vel111);
    fx_mac(s, mom101, vel110);
    fx_mac(s, mom110, vel101);
    fx_mac(s, mom111, vel100);
    fx_mac(s, mom200, vel011);
    fx_mac(s, mom201, vel010);
    fx_mac(s, mom210, vel001);
    fx_mac(s, mom211, vel000);
    k211 = fx_sum(s); }
  const Fx mom030 = S.ldmom(0, 0, 3);
  const Fx mom031 = S.ldmom(1, 0, 3);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel121);
    fx_mac(s, mom001, vel120);
    fx_mac(s, mom010, vel111);
    fx_mac(s, mom011, vel110);
    fx_mac(s, mom020, vel101);
    fx_mac(s, mom021, vel100);
    fx_mac(s, mom100, vel021);
    fx_mac(s, mom101, vel020);
    fx_mac(s, mom110, vel011);
    fx_mac(s, mom111, vel010);
    fx_mac(s, mom120, vel001);
    fx_mac(s, mom121, vel000);
    k121 = fx_sum(s); }
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel031);
    fx_mac(s, mom001, vel030);
    fx_mac(s, mom010, vel021);
    fx_mac(s, mom011, vel020);
    fx_mac(s, mom020, vel011);
    fx_mac(s, mom021, vel010);
    fx_mac(s, mom030, vel001);
    fx_mac(s, mom031, vel000);
    k031 = fx_sum(s); }
  }
  int64_t f101;
  int64_t f201;
  int64_t f111;
  int64_t f301;
  int64_t f211;
  int64_t f121;
  { const int64_t E = E001;
    const Fx e = fx_split(((E - ((k001 + S.swap(k001)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 0, 0, fx_split(E + p + FX_HALF, r));
  }
  { const int64_t E = E101;
    const Fx e = fx_split(((E - ((k101 + S.swap(k011)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 1, 0, fx_split(E + p + FX_HALF, r));
    f101 = k101 + p;
  }
  { const int64_t E = E011;
    const Fx e = fx_split(((E - ((k011 + S.swap(k101)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 0, 1, fx_split(E + p + FX_HALF, r));
  }
  { const int64_t E = E201;
    const Fx e = fx_split(((E - ((k201 + S.swap(k021)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 2, 0, fx_split(E + p + FX_HALF, r));
    f201 = k201 + p;
  }
  { const int64_t E = E111;
    const Fx e = fx_split(((E - ((k111 + S.swap(k111)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 1, 1, fx_split(E + p + FX_HALF, r));
    f111 = k111 + p;
  }
  { const int64_t E = E021;
    const Fx e = fx_split(((E - ((k021 + S.swap(k201)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 0, 2, fx_split(E + p + FX_HALF, r));
  }
  { const int64_t E = E301;
    const Fx e = fx_split(((E - ((k301 + S.swap(k031)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 3, 0, fx_split(E + p + FX_HALF, r));
    f301 = k301 + p;
  }
  { const int64_t E = E211;
    const Fx e = fx_split(((E - ((k211 + S.swap(k121)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 2, 1, fx_split(E + p + FX_HALF, r));
    f211 = k211 + p;
  }
  { const int64_t E = E121;
    const Fx e = fx_split(((E - ((k121 + S.swap(k211)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 1, 2, fx_split(E + p + FX_HALF, r));
    f121 = k121 + p;
  }
  { const int64_t E = E031;
    const Fx e = fx_split(((E - ((k031 + S.swap(k301)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 0, 3, fx_split(E + p + FX_HALF, r));
  }
  int64_t drho001;
  int64_t drho101;
  int64_t drho011;
  int64_t drho201;
  int64_t drho111;
  int64_t drho021;
  int64_t dmom001;
  int64_t dmom101;
  int64_t dmom011;
  int64_t dmom201;
  int64_t dmom111;
  int64_t dmom021;
  int64_t dE001;
  int64_t dE101;
  int64_t dE011;
  int64_t dE201;
  int64_t dE111;
  int64_t dE021;
  drho001 = 1 * fx_join(S.ldmom(1, 1, 0));
  dmom001 = 1 * f101;
  drho101 = 2 * fx_join(S.ldmom(1, 2, 0));
  dmom101 = 2 * f201;
  drho011 = 1 * fx_join(S.ldmom(1, 1, 1));
  dmom011 = 1 * f111;
  drho201 = 3 * fx_join(S.ldmom(1, 3, 0));
  dmom201 = 3 * f301;
  drho111 = 2 * fx_join(S.ldmom(1, 2, 1));
  dmom111 = 2 * f211;
  drho021 = 1 * fx_join(S.ldmom(1, 1, 2));
  dmom021 = 1 * f121;
  #pragma unroll 1
  for (int s = 0; s < 2; ++s) {
  const Fx ser000 = S.ldser(s, 0, 0, 0);
  const Fx ser001 = S.ldser(s, 1, 0, 0);
  const Fx ser100 = S.ldser(s, 0, 1, 0);
  const Fx ser101 = S.ldser(s, 1, 1, 0);
  const Fx ser200 = S.ldser(s, 0, 2, 0);
  const Fx ser201 = S.ldser(s, 1, 2, 0);
  int64_t z00;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel101);
    fx_mac(s, ser001, vel100);
    fx_mac(s, ser100, vel001);
    fx_mac(s, ser101, vel000);
    z00 = fx_sum(s); }
  dE001 = 1 * z00;
  const Fx ser010 = S.ldser(s, 0, 0, 1);
  const Fx ser011 = S.ldser(s, 1, 0, 1);
  const Fx ser110 = S.ldser(s, 0, 1, 1);
  const Fx ser111 = S.ldser(s, 1, 1, 1);
  int64_t z10;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel201);
    fx_mac(s, ser001, vel200);
    fx_mac(s, ser100, vel101);
    fx_mac(s, ser101, vel100);
    fx_mac(s, ser200, vel001);
    fx_mac(s, ser201, vel000);
    z10 = fx_sum(s); }
  dE101 = 2 * z10;
  const Fx ser300 = S.ldser(s, 0, 3, 0);
  const Fx ser301 = S.ldser(s, 1, 3, 0);
  int64_t z01;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel111);
    fx_mac(s, ser001, vel110);
    fx_mac(s, ser010, vel101);
    fx_mac(s, ser011, vel100);
    fx_mac(s, ser100, vel011);
    fx_mac(s, ser101, vel010);
    fx_mac(s, ser110, vel001);
    fx_mac(s, ser111, vel000);
    z01 = fx_sum(s); }
  dE011 = 1 * z01;
  const Fx ser210 = S.ldser(s, 0, 2, 1);
  const Fx ser211 = S.ldser(s, 1, 2, 1);
  int64_t z20;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel301);
    fx_mac(s, ser001, vel300);
    fx_mac(s, ser100, vel201);
    fx_mac(s, ser101, vel200);
    fx_mac(s, ser200, vel101);
    fx_mac(s, ser201, vel100);
    fx_mac(s, ser300, vel001);
    fx_mac(s, ser301, vel000);
    z20 = fx_sum(s); }
  dE201 = 3 * z20;
  const Fx ser020 = S.ldser(s, 0, 0, 2);
  const Fx ser021 = S.ldser(s, 1, 0, 2);
  const Fx ser120 = S.ldser(s, 0, 1, 2);
  const Fx ser121 = S.ldser(s, 1, 1, 2);
  int64_t z11;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel211);
    fx_mac(s, ser001, vel210);
    fx_mac(s, ser010, vel201);
    fx_mac(s, ser011, vel200);
    fx_mac(s, ser100, vel111);
    fx_mac(s, ser101, vel110);
    fx_mac(s, ser110, vel101);
    fx_mac(s, ser111, vel100);
    fx_mac(s, ser200, vel011);
    fx_mac(s, ser201, vel010);
    fx_mac(s, ser210, vel001);
    fx_mac(s, ser211, vel000);
    z11 = fx_sum(s); }
  dE111 = 2 * z11;
  int64_t z02;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel121);
    fx_mac(s, ser001, vel120);
    fx_mac(s, ser010, vel111);
    fx_mac(s, ser011, vel110);
    fx_mac(s, ser020, vel101);
    fx_mac(s, ser021, vel100);
    fx_mac(s, ser100, vel021);
    fx_mac(s, ser101, vel020);
    fx_mac(s, ser110, vel011);
    fx_mac(s, ser111, vel010);
    fx_mac(s, ser120, vel001);
    fx_mac(s, ser121, vel000);
    z02 = fx_sum(s); }
  dE021 = 1 * z02;
  if (s == 0) {
    S.stoth(2, 0, 0, dE001);
    S.stoth(2, 1, 0, dE101);
    S.stoth(2, 0, 1, dE011);
    S.stoth(2, 2, 0, dE201);
    S.stoth(2, 1, 1, dE111);
    S.stoth(2, 0, 2, dE021);
  } }
  S.sync();
  { const int64_t own = dmom001 + S.ldown(2, 0, 0);
    const int64_t both = S.pick(drho001, dE001) + S.swap(S.pick(dE001, drho001));
    S.next(2, 0, 0, fx_time<2>(own, third), fx_time<2>(both, third), r); }
  { const int64_t own = dmom101 + S.ldown(2, 1, 0);
    const int64_t both = S.pick(drho101, dE101) + S.swap(S.pick(dE011, drho011));
    S.next(2, 1, 0, fx_time<2>(own, third), fx_time<2>(both, third), r); }
  { const int64_t own = dmom011 + S.ldown(2, 0, 1);
    const int64_t both = S.pick(drho011, dE011) + S.swap(S.pick(dE101, drho101));
    S.next(2, 0, 1, fx_time<2>(own, third), fx_time<2>(both, third), r); }
  { const int64_t own = dmom201 + S.ldown(2, 2, 0);
    const int64_t both = S.pick(drho201, dE201) + S.swap(S.pick(dE021, drho021));
    S.next(2, 2, 0, fx_time<2>(own, third), fx_time<2>(both, third), r); }
  { const int64_t own = dmom111 + S.ldown(2, 1, 1);
    const int64_t both = S.pick(drho111, dE111) + S.swap(S.pick(dE111, drho111));
    S.next(2, 1, 1, fx_time<2>(own, third), fx_time<2>(both, third), r); }
  { const int64_t own = dmom021 + S.ldown(2, 0, 2);
    const int64_t both = S.pick(drho021, dE021) + S.swap(S.pick(dE201, drho201));
    S.next(2, 0, 2, fx_time<2>(own, third), fx_time<2>(both, third), r); }
  S.sync();
  const int64_t E002 = S.ldE(2, 0, 0);
  const int64_t E102 = S.ldE(2, 1, 0);
  const int64_t E012 = S.ldE(2, 0, 1);
  const int64_t E202 = S.ldE(2, 2, 0);
  const int64_t E112 = S.ldE(2, 1, 1);
  const int64_t E022 = S.ldE(2, 0, 2);
  // ---- slice 2
  Fx vel002;
  Fx vel102;
  Fx vel012;
  Fx vel202;
  Fx vel112;
  Fx vel022;
  {
  const Fx rho001 = S.ldrho(1, 0, 0);
  const Fx rho002 = S.ldrho(2, 0, 0);
  const Fx rho100 = S.ldrho(0, 1, 0);
  const Fx rho101 = S.ldrho(1, 1, 0);
  const Fx rho102 = S.ldrho(2, 1, 0);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(2, 0, 0), -(1 << 30));
    fx_mac(s, rho001, vel001);
    fx_mac(s, rho002, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel002 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho010 = S.ldrho(0, 0, 1);
  const Fx rho011 = S.ldrho(1, 0, 1);
  const Fx rho012 = S.ldrho(2, 0, 1);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(2, 1, 0), -(1 << 30));
    fx_mac(s, rho001, vel101);
    fx_mac(s, rho002, vel100);
    fx_mac(s, rho100, vel002);
    fx_mac(s, rho101, vel001);
    fx_mac(s, rho102, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel102 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho200 = S.ldrho(0, 2, 0);
  const Fx rho201 = S.ldrho(1, 2, 0);
  const Fx rho202 = S.ldrho(2, 2, 0);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(2, 0, 1), -(1 << 30));
    fx_mac(s, rho001, vel011);
    fx_mac(s, rho002, vel010);
    fx_mac(s, rho010, vel002);
    fx_mac(s, rho011, vel001);
    fx_mac(s, rho012, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel012 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho110 = S.ldrho(0, 1, 1);
  const Fx rho111 = S.ldrho(1, 1, 1);
  const Fx rho112 = S.ldrho(2, 1, 1);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(2, 2, 0), -(1 << 30));
    fx_mac(s, rho001, vel201);
    fx_mac(s, rho002, vel200);
    fx_mac(s, rho100, vel102);
    fx_mac(s, rho101, vel101);
    fx_mac(s, rho102, vel100);
    fx_mac(s, rho200, vel002);
    fx_mac(s, rho201, vel001);
    fx_mac(s, rho202, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel202 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho020 = S.ldrho(0, 0, 2);
  const Fx rho021 = S.ldrho(1, 0, 2);
  const Fx rho022 = S.ldrho(2, 0, 2);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(2, 1, 1), -(1 << 30));
    fx_mac(s, rho001, vel111);
    fx_mac(s, rho002, vel110);
    fx_mac(s, rho010, vel102);
    fx_mac(s, rho011, vel101);
    fx_mac(s, rho012, vel100);
    fx_mac(s, rho100, vel012);
    fx_mac(s, rho101, vel011);
    fx_mac(s, rho102, vel010);
    fx_mac(s, rho110, vel002);
    fx_mac(s, rho111, vel001);
    fx_mac(s, rho112, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel112 = fx_split(fx_sum<FX_C>(z), r); }
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(2, 0, 2), -(1 << 30));
    fx_mac(s, rho001, vel021);
    fx_mac(s, rho002, vel020);
    fx_mac(s, rho010, vel012);
    fx_mac(s, rho011, vel011);
    fx_mac(s, rho012, vel010);
    fx_mac(s, rho020, vel002);
    fx_mac(s, rho021, vel001);
    fx_mac(s, rho022, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel022 = fx_split(fx_sum<FX_C>(z), r); }
  }
  int64_t k002;
  int64_t k102;
  int64_t k012;
  int64_t k202;
  int64_t k112;
  int64_t k022;
  {
  const Fx mom000 = S.ldmom(0, 0, 0);
  const Fx mom001 = S.ldmom(1, 0, 0);
  const Fx mom002 = S.ldmom(2, 0, 0);
  const Fx mom100 = S.ldmom(0, 1, 0);
  const Fx mom101 = S.ldmom(1, 1, 0);
  const Fx mom102 = S.ldmom(2, 1, 0);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel002);
    fx_mac(s, mom001, vel001);
    fx_mac(s, mom002, vel000);
    k002 = fx_sum(s); }
  const Fx mom010 = S.ldmom(0, 0, 1);
  const Fx mom011 = S.ldmom(1, 0, 1);
  const Fx mom012 = S.ldmom(2, 0, 1);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel102);
    fx_mac(s, mom001, vel101);
    fx_mac(s, mom002, vel100);
    fx_mac(s, mom100, vel002);
    fx_mac(s, mom101, vel001);
    fx_mac(s, mom102, vel000);
    k102 = fx_sum(s); }
  const Fx mom200 = S.ldmom(0, 2, 0);
  const Fx mom201 = S.ldmom(1, 2, 0);
  const Fx mom202 = S.ldmom(2, 2, 0);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel012);
    fx_mac(s, mom001, vel011);
    fx_mac(s, mom002, vel010);
    fx_mac(s, mom010, vel002);
    fx_mac(s, mom011, vel001);
    fx_mac(s, mom012, vel000);
    k012 = fx_sum(s); }
  const Fx mom110 = S.ldmom(0, 1, 1);
  const Fx mom111 = S.ldmom(1, 1, 1);
  const Fx mom112 = S.ldmom(2, 1, 1);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel202);
    fx_mac(s, mom001, vel201);
    fx_mac(s, mom002, vel200);
    fx_mac(s, mom100, vel102);
    fx_mac(s, mom101, vel101);
    fx_mac(s, mom102, vel100);
    fx_mac(s, mom200, vel002);
    fx_mac(s, mom201, vel001);
    fx_mac(s, mom202, vel000);
    k202 = fx_sum(s); }
  const Fx mom020 = S.ldmom(0, 0, 2);
  const Fx mom021 = S.ldmom(1, 0, 2);
  const Fx mom022 = S.ldmom(2, 0, 2);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel112);
    fx_mac(s, mom001, vel111);
    fx_mac(s, mom002, vel110);
    fx_mac(s, mom010, vel102);
    fx_mac(s, mom011, vel101);
    fx_mac(s, mom012, vel100);
    fx_mac(s, mom100, vel012);
    fx_mac(s, mom101, vel011);
    fx_mac(s, mom102, vel010);
    fx_mac(s, mom110, vel002);
    fx_mac(s, mom111, vel001);
    fx_mac(s, mom112, vel000);
    k112 = fx_sum(s); }
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel022);
    fx_mac(s, mom001, vel021);
    fx_mac(s, mom002, vel020);
    fx_mac(s, mom010, vel012);
    fx_mac(s, mom011, vel011);
    fx_mac(s, mom012, vel010);
    fx_mac(s, mom020, vel002);
    fx_mac(s, mom021, vel001);
    fx_mac(s, mom022, vel000);
    k022 = fx_sum(s); }
  }
  int64_t f102;
  int64_t f202;
  int64_t f112;
  { const int64_t E = E002;
    const Fx e = fx_split(((E - ((k002 + S.swap(k002)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(2, 0, 0, fx_split(E + p + FX_HALF, r));
  }
  { const int64_t E = E102;
    const Fx e = fx_split(((E - ((k102 + S.swap(k012)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(2, 1, 0, fx_split(E + p + FX_HALF, r));
    f102 = k102 + p;
  }
  { const int64_t E = E012;
    const Fx e = fx_split(((E - ((k012 + S.swap(k102)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(2, 0, 1, fx_split(E + p + FX_HALF, r));
  }
  { const int64_t E = E202;
    const Fx e = fx_split(((E - ((k202 + S.swap(k022)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(2, 2, 0, fx_split(E + p + FX_HALF, r));
    f202 = k202 + p;
  }
  { const int64_t E = E112;
    const Fx e = fx_split(((E - ((k112 + S.swap(k112)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(2, 1, 1, fx_split(E + p + FX_HALF, r));
    f112 = k112 + p;
  }
  { const int64_t E = E022;
    const Fx e = fx_split(((E - ((k022 + S.swap(k202)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(2, 0, 2, fx_split(E + p + FX_HALF, r));
  }
  int64_t drho002;
  int64_t drho102;
  int64_t drho012;
  int64_t dmom002;
  int64_t dmom102;
  int64_t dmom012;
  int64_t dE002;
  int64_t dE102;
  int64_t dE012;
  drho002 = 1 * fx_join(S.ldmom(2, 1, 0));
  dmom002 = 1 * f102;
  drho102 = 2 * fx_join(S.ldmom(2, 2, 0));
  dmom102 = 2 * f202;
  drho012 = 1 * fx_join(S.ldmom(2, 1, 1));
  dmom012 = 1 * f112;
  #pragma unroll 1
  for (int s = 0; s < 2; ++s) {
  const Fx ser000 = S.ldser(s, 0, 0, 0);
  const Fx ser001 = S.ldser(s, 1, 0, 0);
  const Fx ser002 = S.ldser(s, 2, 0, 0);
  const Fx ser100 = S.ldser(s, 0, 1, 0);
  const Fx ser101 = S.ldser(s, 1, 1, 0);
  const Fx ser102 = S.ldser(s, 2, 1, 0);
  const Fx ser200 = S.ldser(s, 0, 2, 0);
  const Fx ser201 = S.ldser(s, 1, 2, 0);
  const Fx ser202 = S.ldser(s, 2, 2, 0);
  int64_t z00;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel102);
    fx_mac(s, ser001, vel101);
    fx_mac(s, ser002, vel100);
    fx_mac(s, ser100, vel002);
    fx_mac(s, ser101, vel001);
    fx_mac(s, ser102, vel000);
    z00 = fx_sum(s); }
  dE002 = 1 * z00;
  const Fx ser010 = S.ldser(s, 0, 0, 1);
  const Fx ser011 = S.ldser(s, 1, 0, 1);
  const Fx ser012 = S.ldser(s, 2, 0, 1);
  const Fx ser110 = S.ldser(s, 0, 1, 1);
  const Fx ser111 = S.ldser(s, 1, 1, 1);
  const Fx ser112 = S.ldser(s, 2, 1, 1);
  int64_t z10;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel202);
    fx_mac(s, ser001, vel201);
    fx_mac(s, ser002, vel200);
    fx_mac(s, ser100, vel102);
    fx_mac(s, ser101, vel101);
    fx_mac(s, ser102, vel100);
    fx_mac(s, ser200, vel002);
    fx_mac(s, ser201, vel001);
    fx_mac(s, ser202, vel000);
    z10 = fx_sum(s); }
  dE102 = 2 * z10;
  int64_t z01;
  { FxAcc s = fx_zero();
    fx_mac(s, ser000, vel112);
    fx_mac(s, ser001, vel111);
    fx_mac(s, ser002, vel110);
    fx_mac(s, ser010, vel102);
    fx_mac(s, ser011, vel101);
    fx_mac(s, ser012, vel100);
    fx_mac(s, ser100, vel012);
    fx_mac(s, ser101, vel011);
    fx_mac(s, ser102, vel010);
    fx_mac(s, ser110, vel002);
    fx_mac(s, ser111, vel001);
    fx_mac(s, ser112, vel000);
    z01 = fx_sum(s); }
  dE012 = 1 * z01;
  if (s == 0) {
    S.stoth(3, 0, 0, dE002);
    S.stoth(3, 1, 0, dE102);
    S.stoth(3, 0, 1, dE012);
  } }
  S.sync();
  { const int64_t own = dmom002 + S.ldown(3, 0, 0);
    const int64_t both = S.pick(drho002, dE002) + S.swap(S.pick(dE002, drho002));
    S.next(3, 0, 0, fx_time<3>(own, third), fx_time<3>(both, third), r); }
  { const int64_t own = dmom102 + S.ldown(3, 1, 0);
    const int64_t both = S.pick(drho102, dE102) + S.swap(S.pick(dE012, drho012));
    S.next(3, 1, 0, fx_time<3>(own, third), fx_time<3>(both, third), r); }
  { const int64_t own = dmom012 + S.ldown(3, 0, 1);
    const int64_t both = S.pick(drho012, dE012) + S.swap(S.pick(dE102, drho102));
    S.next(3, 0, 1, fx_time<3>(own, third), fx_time<3>(both, third), r); }
  S.sync();
  const int64_t E003 = S.ldE(3, 0, 0);
  const int64_t E103 = S.ldE(3, 1, 0);
  const int64_t E013 = S.ldE(3, 0, 1);
  // ---- slice 3
  Fx vel003;
  Fx vel103;
  Fx vel013;
  {
  const Fx rho001 = S.ldrho(1, 0, 0);
  const Fx rho002 = S.ldrho(2, 0, 0);
  const Fx rho003 = S.ldrho(3, 0, 0);
  const Fx rho100 = S.ldrho(0, 1, 0);
  const Fx rho101 = S.ldrho(1, 1, 0);
  const Fx rho102 = S.ldrho(2, 1, 0);
  const Fx rho103 = S.ldrho(3, 1, 0);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(3, 0, 0), -(1 << 30));
    fx_mac(s, rho001, vel002);
    fx_mac(s, rho002, vel001);
    fx_mac(s, rho003, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel003 = fx_split(fx_sum<FX_C>(z), r); }
  const Fx rho010 = S.ldrho(0, 0, 1);
  const Fx rho011 = S.ldrho(1, 0, 1);
  const Fx rho012 = S.ldrho(2, 0, 1);
  const Fx rho013 = S.ldrho(3, 0, 1);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(3, 1, 0), -(1 << 30));
    fx_mac(s, rho001, vel102);
    fx_mac(s, rho002, vel101);
    fx_mac(s, rho003, vel100);
    fx_mac(s, rho100, vel003);
    fx_mac(s, rho101, vel002);
    fx_mac(s, rho102, vel001);
    fx_mac(s, rho103, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel103 = fx_split(fx_sum<FX_C>(z), r); }
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(3, 0, 1), -(1 << 30));
    fx_mac(s, rho001, vel012);
    fx_mac(s, rho002, vel011);
    fx_mac(s, rho003, vel010);
    fx_mac(s, rho010, vel003);
    fx_mac(s, rho011, vel002);
    fx_mac(s, rho012, vel001);
    fx_mac(s, rho013, vel000);
    const Fx n = fx_split(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel013 = fx_split(fx_sum<FX_C>(z), r); }
  }
  int64_t k003;
  int64_t k103;
  int64_t k013;
  {
  const Fx mom000 = S.ldmom(0, 0, 0);
  const Fx mom001 = S.ldmom(1, 0, 0);
  const Fx mom002 = S.ldmom(2, 0, 0);
  const Fx mom003 = S.ldmom(3, 0, 0);
  const Fx mom100 = S.ldmom(0, 1, 0);
  const Fx mom101 = S.ldmom(1, 1, 0);
  const Fx mom102 = S.ldmom(2, 1, 0);
  const Fx mom103 = S.ldmom(3, 1, 0);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel003);
    fx_mac(s, mom001, vel002);
    fx_mac(s, mom002, vel001);
    fx_mac(s, mom003, vel000);
    k003 = fx_sum(s); }
  const Fx mom010 = S.ldmom(0, 0, 1);
  const Fx mom011 = S.ldmom(1, 0, 1);
  const Fx mom012 = S.ldmom(2, 0, 1);
  const Fx mom013 = S.ldmom(3, 0, 1);
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel103);
    fx_mac(s, mom001, vel102);
    fx_mac(s, mom002, vel101);
    fx_mac(s, mom003, vel100);
    fx_mac(s, mom100, vel003);
    fx_mac(s, mom101, vel002);
    fx_mac(s, mom102, vel001);
    fx_mac(s, mom103, vel000);
    k103 = fx_sum(s); }
  { FxAcc s = fx_zero();
    fx_mac(s, mom000, vel013);
    fx_mac(s, mom001, vel012);
    fx_mac(s, mom002, vel011);
    fx_mac(s, mom003, vel010);
    fx_mac(s, mom010, vel003);
    fx_mac(s, mom011, vel002);
    fx_mac(s, mom012, vel001);
    fx_mac(s, mom013, vel000);
    k013 = fx_sum(s); }
  }
  int64_t f103;
  { const int64_t E = E003;
    const Fx e = fx_split(((E - ((k003 + S.swap(k003)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(3, 0, 0, fx_split(E + p + FX_HALF, r));
  }
  { const int64_t E = E103;
    const Fx e = fx_split(((E - ((k103 + S.swap(k013)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(3, 1, 0, fx_split(E + p + FX_HALF, r));
    f103 = k103 + p;
  }
  { const int64_t E = E013;
    const Fx e = fx_split(((E - ((k013 + S.swap(k103)) >> 1)) << gshift) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(3, 0, 1, fx_split(E + p + FX_HALF, r));
  }
  int64_t drho003;
  int64_t dmom003;
  int64_t dE003;
  int64_t doth003;
  drho003 = 1 * fx_join(S.ldmom(3, 1, 0));
  dmom003 = 1 * f103;
  {
  const Fx oth000 = S.ldoth(0, 0, 0);
  const Fx oth001 = S.ldoth(1, 0, 0);
  const Fx oth002 = S.ldoth(2, 0, 0);
  const Fx oth003 = S.ldoth(3, 0, 0);
  const Fx oth100 = S.ldoth(0, 1, 0);
  const Fx oth101 = S.ldoth(1, 1, 0);
  const Fx oth102 = S.ldoth(2, 1, 0);
  const Fx oth103 = S.ldoth(3, 1, 0);
  int64_t z;
  { FxAcc s = fx_zero();
    fx_mac(s, oth000, vel103);
    fx_mac(s, oth001, vel102);
    fx_mac(s, oth002, vel101);
    fx_mac(s, oth003, vel100);
    fx_mac(s, oth100, vel003);
    fx_mac(s, oth101, vel002);
    fx_mac(s, oth102, vel001);
    fx_mac(s, oth103, vel000);
    z = fx_sum(s); }
  doth003 = 1 * z;
  }
  {
  const Fx H000 = S.ldH(0, 0, 0);
  const Fx H001 = S.ldH(1, 0, 0);
  const Fx H002 = S.ldH(2, 0, 0);
  const Fx H003 = S.ldH(3, 0, 0);
  const Fx H100 = S.ldH(0, 1, 0);
  const Fx H101 = S.ldH(1, 1, 0);
  const Fx H102 = S.ldH(2, 1, 0);
  const Fx H103 = S.ldH(3, 1, 0);
  int64_t z;
  { FxAcc s = fx_zero();
    fx_mac(s, H000, vel103);
    fx_mac(s, H001, vel102);
    fx_mac(s, H002, vel101);
    fx_mac(s, H003, vel100);
    fx_mac(s, H100, vel003);
    fx_mac(s, H101, vel002);
    fx_mac(s, H102, vel001);
    fx_mac(s, H103, vel000);
    z = fx_sum(s); }
  dE003 = 1 * z;
  }
  { const int64_t own = dmom003 + S.swap(doth003);
    const int64_t both = S.pick(drho003, dE003) + S.swap(S.pick(dE003, drho003));
    S.next(4, 0, 0, fx_time<4>(own, third), fx_time<4>(both, third), r0); }
}

}  // namespace shweno
