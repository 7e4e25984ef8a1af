// Generated by gen_ck.py -- do not edit.  The Cauchy-Kovalevskaya recursions
// in block fixed point (see fixed.cuh, ck_fixed.cuh and gen_ck.py for the method).
#pragma once
#include "fixed.cuh"

namespace shweno {

// Constants of the recursion: 1/3 and gamma - 1.
struct CkFixedConst {
  Fx third, gm1;
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
  const Fx w0_001 = fx_split_any(fx_time<1>(1 * f_100, K.third) + FX_HALF, r);
  int64_t f_200; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][10]); f_200 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w[0][5], w[0][5]); f_200 += fx_sum(s) >> 1; }
  const Fx w0_101 = fx_split_any(fx_time<1>(2 * f_200, K.third) + FX_HALF, r);
  int64_t f_101; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_101); fx_mac(s, w0_001, w[0][5]); f_101 = fx_sum(s); }
  const Fx w0_002 = fx_split_any(fx_time<2>(1 * f_101, K.third) + FX_HALF, r);
  int64_t f_300; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][15]); fx_mac(s, w[0][5], w[0][10]); f_300 = fx_sum(s); }
  const Fx w0_201 = fx_split_any(fx_time<1>(3 * f_300, K.third) + FX_HALF, r);
  int64_t f_201; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_201); fx_mac(s, w0_001, w[0][10]); fx_mac(s, w[0][5], w0_101); f_201 = fx_sum(s); }
  const Fx w0_102 = fx_split_any(fx_time<2>(2 * f_201, K.third) + FX_HALF, r);
  int64_t f_102; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_102); fx_mac(s, w0_001, w0_101); fx_mac(s, w0_002, w[0][5]); f_102 = fx_sum(s); }
  const Fx w0_003 = fx_split_any(fx_time<3>(1 * f_102, K.third) + FX_HALF, r);
  int64_t f_400; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][20]); fx_mac(s, w[0][5], w[0][15]); f_400 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w[0][10], w[0][10]); f_400 += fx_sum(s) >> 1; }
  const Fx w0_301 = fx_split_any(fx_time<1>(4 * f_400, K.third) + FX_HALF, r);
  int64_t f_301; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_301); fx_mac(s, w0_001, w[0][15]); fx_mac(s, w[0][5], w0_201); fx_mac(s, w0_101, w[0][10]); f_301 = fx_sum(s); }
  const Fx w0_202 = fx_split_any(fx_time<2>(3 * f_301, K.third) + FX_HALF, r);
  int64_t f_202; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_202); fx_mac(s, w0_001, w0_201); fx_mac(s, w0_002, w[0][10]); fx_mac(s, w[0][5], w0_102); f_202 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w0_101, w0_101); f_202 += fx_sum(s) >> 1; }
  const Fx w0_103 = fx_split_any(fx_time<3>(2 * f_202, K.third) + FX_HALF, r);
  int64_t f_103; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_103); fx_mac(s, w0_001, w0_102); fx_mac(s, w0_002, w0_101); fx_mac(s, w0_003, w[0][5]); f_103 = fx_sum(s); }
  const Fx w0_004 = fx_split_any(fx_time<4>(1 * f_103, K.third) + FX_HALF, r);
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
  const Fx w0_001 = fx_split_any(fx_time<1>(1 * f_100 + 1 * f_010, K.third) + FX_HALF, r);
  int64_t f_200; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][10]); f_200 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w[0][5], w[0][5]); f_200 += fx_sum(s) >> 1; }
  int64_t f_110; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][6]); fx_mac(s, w[0][1], w[0][5]); f_110 = fx_sum(s); }
  const Fx w0_101 = fx_split_any(fx_time<1>(2 * f_200 + 1 * f_110, K.third) + FX_HALF, r);
  int64_t f_101; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_101); fx_mac(s, w0_001, w[0][5]); f_101 = fx_sum(s); }
  int64_t f_020; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][2]); f_020 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w[0][1], w[0][1]); f_020 += fx_sum(s) >> 1; }
  const Fx w0_011 = fx_split_any(fx_time<1>(1 * f_110 + 2 * f_020, K.third) + FX_HALF, r);
  int64_t f_011; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_011); fx_mac(s, w0_001, w[0][1]); f_011 = fx_sum(s); }
  const Fx w0_002 = fx_split_any(fx_time<2>(1 * f_101 + 1 * f_011, K.third) + FX_HALF, r);
  int64_t f_300; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][15]); fx_mac(s, w[0][5], w[0][10]); f_300 = fx_sum(s); }
  int64_t f_210; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][11]); fx_mac(s, w[0][1], w[0][10]); fx_mac(s, w[0][5], w[0][6]); f_210 = fx_sum(s); }
  const Fx w0_201 = fx_split_any(fx_time<1>(3 * f_300 + 1 * f_210, K.third) + FX_HALF, r);
  int64_t f_201; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_201); fx_mac(s, w0_001, w[0][10]); fx_mac(s, w[0][5], w0_101); f_201 = fx_sum(s); }
  int64_t f_120; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][7]); fx_mac(s, w[0][1], w[0][6]); fx_mac(s, w[0][2], w[0][5]); f_120 = fx_sum(s); }
  const Fx w0_111 = fx_split_any(fx_time<1>(2 * f_210 + 2 * f_120, K.third) + FX_HALF, r);
  int64_t f_111; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_111); fx_mac(s, w0_001, w[0][6]); fx_mac(s, w[0][1], w0_101); fx_mac(s, w0_011, w[0][5]); f_111 = fx_sum(s); }
  const Fx w0_102 = fx_split_any(fx_time<2>(2 * f_201 + 1 * f_111, K.third) + FX_HALF, r);
  int64_t f_102; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_102); fx_mac(s, w0_001, w0_101); fx_mac(s, w0_002, w[0][5]); f_102 = fx_sum(s); }
  int64_t f_030; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][3]); fx_mac(s, w[0][1], w[0][2]); f_030 = fx_sum(s); }
  const Fx w0_021 = fx_split_any(fx_time<1>(1 * f_120 + 3 * f_030, K.third) + FX_HALF, r);
  int64_t f_021; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_021); fx_mac(s, w0_001, w[0][2]); fx_mac(s, w[0][1], w0_011); f_021 = fx_sum(s); }
  const Fx w0_012 = fx_split_any(fx_time<2>(1 * f_111 + 2 * f_021, K.third) + FX_HALF, r);
  int64_t f_012; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_012); fx_mac(s, w0_001, w0_011); fx_mac(s, w0_002, w[0][1]); f_012 = fx_sum(s); }
  const Fx w0_003 = fx_split_any(fx_time<3>(1 * f_102 + 1 * f_012, K.third) + FX_HALF, r);
  int64_t f_400; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][20]); fx_mac(s, w[0][5], w[0][15]); f_400 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w[0][10], w[0][10]); f_400 += fx_sum(s) >> 1; }
  int64_t f_310; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][16]); fx_mac(s, w[0][1], w[0][15]); fx_mac(s, w[0][5], w[0][11]); fx_mac(s, w[0][6], w[0][10]); f_310 = fx_sum(s); }
  const Fx w0_301 = fx_split_any(fx_time<1>(4 * f_400 + 1 * f_310, K.third) + FX_HALF, r);
  int64_t f_301; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_301); fx_mac(s, w0_001, w[0][15]); fx_mac(s, w[0][5], w0_201); fx_mac(s, w0_101, w[0][10]); f_301 = fx_sum(s); }
  int64_t f_220; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][12]); fx_mac(s, w[0][1], w[0][11]); fx_mac(s, w[0][2], w[0][10]); fx_mac(s, w[0][5], w[0][7]); f_220 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w[0][6], w[0][6]); f_220 += fx_sum(s) >> 1; }
  const Fx w0_211 = fx_split_any(fx_time<1>(3 * f_310 + 2 * f_220, K.third) + FX_HALF, r);
  int64_t f_211; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_211); fx_mac(s, w0_001, w[0][11]); fx_mac(s, w[0][1], w0_201); fx_mac(s, w0_011, w[0][10]); fx_mac(s, w[0][5], w0_111); fx_mac(s, w0_101, w[0][6]); f_211 = fx_sum(s); }
  const Fx w0_202 = fx_split_any(fx_time<2>(3 * f_301 + 1 * f_211, K.third) + FX_HALF, r);
  int64_t f_202; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_202); fx_mac(s, w0_001, w0_201); fx_mac(s, w0_002, w[0][10]); fx_mac(s, w[0][5], w0_102); f_202 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w0_101, w0_101); f_202 += fx_sum(s) >> 1; }
  int64_t f_130; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][8]); fx_mac(s, w[0][1], w[0][7]); fx_mac(s, w[0][2], w[0][6]); fx_mac(s, w[0][3], w[0][5]); f_130 = fx_sum(s); }
  const Fx w0_121 = fx_split_any(fx_time<1>(2 * f_220 + 3 * f_130, K.third) + FX_HALF, r);
  int64_t f_121; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_121); fx_mac(s, w0_001, w[0][7]); fx_mac(s, w[0][1], w0_111); fx_mac(s, w0_011, w[0][6]); fx_mac(s, w[0][2], w0_101); fx_mac(s, w0_021, w[0][5]); f_121 = fx_sum(s); }
  const Fx w0_112 = fx_split_any(fx_time<2>(2 * f_211 + 2 * f_121, K.third) + FX_HALF, r);
  int64_t f_112; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_112); fx_mac(s, w0_001, w0_111); fx_mac(s, w0_002, w[0][6]); fx_mac(s, w[0][1], w0_102); fx_mac(s, w0_011, w0_101); fx_mac(s, w0_012, w[0][5]); f_112 = fx_sum(s); }
  const Fx w0_103 = fx_split_any(fx_time<3>(2 * f_202 + 1 * f_112, K.third) + FX_HALF, r);
  int64_t f_103; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_103); fx_mac(s, w0_001, w0_102); fx_mac(s, w0_002, w0_101); fx_mac(s, w0_003, w[0][5]); f_103 = fx_sum(s); }
  int64_t f_040; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w[0][4]); fx_mac(s, w[0][1], w[0][3]); f_040 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w[0][2], w[0][2]); f_040 += fx_sum(s) >> 1; }
  const Fx w0_031 = fx_split_any(fx_time<1>(1 * f_130 + 4 * f_040, K.third) + FX_HALF, r);
  int64_t f_031; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_031); fx_mac(s, w0_001, w[0][3]); fx_mac(s, w[0][1], w0_021); fx_mac(s, w0_011, w[0][2]); f_031 = fx_sum(s); }
  const Fx w0_022 = fx_split_any(fx_time<2>(1 * f_121 + 3 * f_031, K.third) + FX_HALF, r);
  int64_t f_022; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_022); fx_mac(s, w0_001, w0_021); fx_mac(s, w0_002, w[0][2]); fx_mac(s, w[0][1], w0_012); f_022 = fx_sum(s); }{ FxAcc s = fx_zero(); fx_mac(s, w0_011, w0_011); f_022 += fx_sum(s) >> 1; }
  const Fx w0_013 = fx_split_any(fx_time<3>(1 * f_112 + 2 * f_022, K.third) + FX_HALF, r);
  int64_t f_013; { FxAcc s = fx_zero(); fx_mac(s, w[0][0], w0_013); fx_mac(s, w0_001, w0_012); fx_mac(s, w0_002, w0_011); fx_mac(s, w0_003, w[0][1]); f_013 = fx_sum(s); }
  const Fx w0_004 = fx_split_any(fx_time<4>(1 * f_103 + 1 * f_013, K.third) + FX_HALF, r);
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
  const Fx w0_001 = fx_split_any(fx_time<1>(1 * (z_w1_100), K.third) + FX_HALF, r);
  Fx u_000n; { FxAcc s = fx_zero(true); fx_mac_int(s, w[1][0], -(1 << 30)); u_000n = fx_split(fx_sum(s), r0); }
  Fx u_000; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_000n, ninv); u_000 = fx_split(fx_sum<FX_C>(s), r0); }
  Fx u_100n; { FxAcc s = fx_zero(true); fx_mac_int(s, w[1][5], -(1 << 30)); fx_mac(s, w[0][5], u_000); u_100n = fx_split(fx_sum(s), r); }
  Fx u_100; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_100n, ninv); u_100 = fx_split(fx_sum<FX_C>(s), r); }
  Fx u_200n; { FxAcc s = fx_zero(true); fx_mac_int(s, w[1][10], -(1 << 30)); fx_mac(s, w[0][5], u_100); fx_mac(s, w[0][10], u_000); u_200n = fx_split(fx_sum(s), r); }
  Fx u_200; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_200n, ninv); u_200 = fx_split(fx_sum<FX_C>(s), r); }
  int64_t z_mu_200; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_200); fx_mac(s, w[1][5], u_100); fx_mac(s, w[1][10], u_000); z_mu_200 = fx_sum(s); }
  const int64_t z_w2_200 = fx_join(w[2][10]);
  const Fx e_200 = fx_split(z_w2_200 - ((z_mu_200) >> 1) + FX_HALF, r);
  int64_t z_p_200; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_200, K.gm1); z_p_200 = fx_sum<FX_C>(s); }
  const Fx w1_101 = fx_split_any(fx_time<1>(2 * (z_mu_200 + z_p_200), K.third) + FX_HALF, r);
  const int64_t z_w1_101 = fx_join(w1_101);
  const Fx w0_002 = fx_split_any(fx_time<2>(1 * (z_w1_101), K.third) + FX_HALF, r);
  Fx u_300n; { FxAcc s = fx_zero(true); fx_mac_int(s, w[1][15], -(1 << 30)); fx_mac(s, w[0][5], u_200); fx_mac(s, w[0][10], u_100); fx_mac(s, w[0][15], u_000); u_300n = fx_split(fx_sum(s), r); }
  Fx u_300; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_300n, ninv); u_300 = fx_split(fx_sum<FX_C>(s), r); }
  int64_t z_mu_300; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_300); fx_mac(s, w[1][5], u_200); fx_mac(s, w[1][10], u_100); fx_mac(s, w[1][15], u_000); z_mu_300 = fx_sum(s); }
  const int64_t z_w2_300 = fx_join(w[2][15]);
  const Fx e_300 = fx_split(z_w2_300 - ((z_mu_300) >> 1) + FX_HALF, r);
  int64_t z_p_300; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_300, K.gm1); z_p_300 = fx_sum<FX_C>(s); }
  const Fx w1_201 = fx_split_any(fx_time<1>(3 * (z_mu_300 + z_p_300), K.third) + FX_HALF, r);
  int64_t z_mu_100; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_100); fx_mac(s, w[1][5], u_000); z_mu_100 = fx_sum(s); }
  const int64_t z_w2_100 = fx_join(w[2][5]);
  const Fx e_100 = fx_split(z_w2_100 - ((z_mu_100) >> 1) + FX_HALF, r);
  int64_t z_p_100; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_100, K.gm1); z_p_100 = fx_sum<FX_C>(s); }
  const Fx w1_001 = fx_split_any(fx_time<1>(1 * (z_mu_100 + z_p_100), K.third) + FX_HALF, r);
  Fx u_001n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_001, -(1 << 30)); fx_mac(s, w0_001, u_000); u_001n = fx_split(fx_sum(s), r); }
  Fx u_001; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_001n, ninv); u_001 = fx_split(fx_sum<FX_C>(s), r); }
  const int64_t z_w1_200 = fx_join(w[1][10]);
  const Fx w0_101 = fx_split_any(fx_time<1>(2 * (z_w1_200), K.third) + FX_HALF, r);
  Fx u_101n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_101, -(1 << 30)); fx_mac(s, w0_001, u_100); fx_mac(s, w[0][5], u_001); fx_mac(s, w0_101, u_000); u_101n = fx_split(fx_sum(s), r); }
  Fx u_101; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_101n, ninv); u_101 = fx_split(fx_sum<FX_C>(s), r); }
  const int64_t z_w1_300 = fx_join(w[1][15]);
  const Fx w0_201 = fx_split_any(fx_time<1>(3 * (z_w1_300), K.third) + FX_HALF, r);
  Fx u_201n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_201, -(1 << 30)); fx_mac(s, w0_001, u_200); fx_mac(s, w[0][5], u_101); fx_mac(s, w0_101, u_100); fx_mac(s, w[0][10], u_001); fx_mac(s, w0_201, u_000); u_201n = fx_split(fx_sum(s), r); }
  Fx u_201; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_201n, ninv); u_201 = fx_split(fx_sum<FX_C>(s), r); }
  int64_t z_mu_201; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_201); fx_mac(s, w1_001, u_200); fx_mac(s, w[1][5], u_101); fx_mac(s, w1_101, u_100); fx_mac(s, w[1][10], u_001); fx_mac(s, w1_201, u_000); z_mu_201 = fx_sum(s); }
  const Fx H_300 = fx_split(z_w2_300 + z_p_300 + FX_HALF, r);
  const Fx H_200 = fx_split(z_w2_200 + z_p_200 + FX_HALF, r);
  const Fx H_100 = fx_split(z_w2_100 + z_p_100 + FX_HALF, r);
  const int64_t z_w2_000 = fx_join(w[2][0]);
  int64_t z_mu_000; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_000); z_mu_000 = fx_sum(s); }
  const Fx e_000 = fx_split(z_w2_000 - ((z_mu_000) >> 1) + FX_HALF, r0);
  int64_t z_p_000; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_000, K.gm1); z_p_000 = fx_sum<FX_C>(s); }
  const Fx H_000 = fx_split(z_w2_000 + z_p_000 + FX_HALF, r0);
  int64_t z_uH_300; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_300); fx_mac(s, u_100, H_200); fx_mac(s, u_200, H_100); fx_mac(s, u_300, H_000); z_uH_300 = fx_sum(s); }
  const Fx w2_201 = fx_split_any(fx_time<1>(3 * (z_uH_300), K.third) + FX_HALF, r);
  const int64_t z_w2_201 = fx_join(w2_201);
  const Fx e_201 = fx_split(z_w2_201 - ((z_mu_201) >> 1) + FX_HALF, r);
  int64_t z_p_201; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_201, K.gm1); z_p_201 = fx_sum<FX_C>(s); }
  const Fx w1_102 = fx_split_any(fx_time<2>(2 * (z_mu_201 + z_p_201), K.third) + FX_HALF, r);
  const int64_t z_w1_102 = fx_join(w1_102);
  const Fx w0_003 = fx_split_any(fx_time<3>(1 * (z_w1_102), K.third) + FX_HALF, r);
  Fx u_400n; { FxAcc s = fx_zero(true); fx_mac_int(s, w[1][20], -(1 << 30)); fx_mac(s, w[0][5], u_300); fx_mac(s, w[0][10], u_200); fx_mac(s, w[0][15], u_100); fx_mac(s, w[0][20], u_000); u_400n = fx_split(fx_sum(s), r); }
  Fx u_400; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_400n, ninv); u_400 = fx_split(fx_sum<FX_C>(s), r); }
  int64_t z_mu_400; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_400); fx_mac(s, w[1][5], u_300); fx_mac(s, w[1][10], u_200); fx_mac(s, w[1][15], u_100); fx_mac(s, w[1][20], u_000); z_mu_400 = fx_sum(s); }
  const int64_t z_w2_400 = fx_join(w[2][20]);
  const Fx e_400 = fx_split(z_w2_400 - ((z_mu_400) >> 1) + FX_HALF, r);
  int64_t z_p_400; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_400, K.gm1); z_p_400 = fx_sum<FX_C>(s); }
  const Fx w1_301 = fx_split_any(fx_time<1>(4 * (z_mu_400 + z_p_400), K.third) + FX_HALF, r);
  const int64_t z_w1_400 = fx_join(w[1][20]);
  const Fx w0_301 = fx_split_any(fx_time<1>(4 * (z_w1_400), K.third) + FX_HALF, r);
  Fx u_301n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_301, -(1 << 30)); fx_mac(s, w0_001, u_300); fx_mac(s, w[0][5], u_201); fx_mac(s, w0_101, u_200); fx_mac(s, w[0][10], u_101); fx_mac(s, w0_201, u_100); fx_mac(s, w[0][15], u_001); fx_mac(s, w0_301, u_000); u_301n = fx_split(fx_sum(s), r); }
  Fx u_301; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_301n, ninv); u_301 = fx_split(fx_sum<FX_C>(s), r); }
  int64_t z_mu_301; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_301); fx_mac(s, w1_001, u_300); fx_mac(s, w[1][5], u_201); fx_mac(s, w1_101, u_200); fx_mac(s, w[1][10], u_101); fx_mac(s, w1_201, u_100); fx_mac(s, w[1][15], u_001); fx_mac(s, w1_301, u_000); z_mu_301 = fx_sum(s); }
  const Fx H_400 = fx_split(z_w2_400 + z_p_400 + FX_HALF, r);
  int64_t z_uH_400; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_400); fx_mac(s, u_100, H_300); fx_mac(s, u_200, H_200); fx_mac(s, u_300, H_100); fx_mac(s, u_400, H_000); z_uH_400 = fx_sum(s); }
  const Fx w2_301 = fx_split_any(fx_time<1>(4 * (z_uH_400), K.third) + FX_HALF, r);
  const int64_t z_w2_301 = fx_join(w2_301);
  const Fx e_301 = fx_split(z_w2_301 - ((z_mu_301) >> 1) + FX_HALF, r);
  int64_t z_p_301; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_301, K.gm1); z_p_301 = fx_sum<FX_C>(s); }
  const Fx w1_202 = fx_split_any(fx_time<2>(3 * (z_mu_301 + z_p_301), K.third) + FX_HALF, r);
  int64_t z_mu_101; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_101); fx_mac(s, w1_001, u_100); fx_mac(s, w[1][5], u_001); fx_mac(s, w1_101, u_000); z_mu_101 = fx_sum(s); }
  int64_t z_uH_200; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_200); fx_mac(s, u_100, H_100); fx_mac(s, u_200, H_000); z_uH_200 = fx_sum(s); }
  const Fx w2_101 = fx_split_any(fx_time<1>(2 * (z_uH_200), K.third) + FX_HALF, r);
  const int64_t z_w2_101 = fx_join(w2_101);
  const Fx e_101 = fx_split(z_w2_101 - ((z_mu_101) >> 1) + FX_HALF, r);
  int64_t z_p_101; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_101, K.gm1); z_p_101 = fx_sum<FX_C>(s); }
  const Fx w1_002 = fx_split_any(fx_time<2>(1 * (z_mu_101 + z_p_101), K.third) + FX_HALF, r);
  Fx u_002n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_002, -(1 << 30)); fx_mac(s, w0_001, u_001); fx_mac(s, w0_002, u_000); u_002n = fx_split(fx_sum(s), r); }
  Fx u_002; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_002n, ninv); u_002 = fx_split(fx_sum<FX_C>(s), r); }
  const int64_t z_w1_201 = fx_join(w1_201);
  const Fx w0_102 = fx_split_any(fx_time<2>(2 * (z_w1_201), K.third) + FX_HALF, r);
  Fx u_102n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_102, -(1 << 30)); fx_mac(s, w0_001, u_101); fx_mac(s, w0_002, u_100); fx_mac(s, w[0][5], u_002); fx_mac(s, w0_101, u_001); fx_mac(s, w0_102, u_000); u_102n = fx_split(fx_sum(s), r); }
  Fx u_102; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_102n, ninv); u_102 = fx_split(fx_sum<FX_C>(s), r); }
  const int64_t z_w1_301 = fx_join(w1_301);
  const Fx w0_202 = fx_split_any(fx_time<2>(3 * (z_w1_301), K.third) + FX_HALF, r);
  Fx u_202n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_202, -(1 << 30)); fx_mac(s, w0_001, u_201); fx_mac(s, w0_002, u_200); fx_mac(s, w[0][5], u_102); fx_mac(s, w0_101, u_101); fx_mac(s, w0_102, u_100); fx_mac(s, w[0][10], u_002); fx_mac(s, w0_201, u_001); fx_mac(s, w0_202, u_000); u_202n = fx_split(fx_sum(s), r); }
  Fx u_202; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_202n, ninv); u_202 = fx_split(fx_sum<FX_C>(s), r); }
  int64_t z_mu_202; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_202); fx_mac(s, w1_001, u_201); fx_mac(s, w1_002, u_200); fx_mac(s, w[1][5], u_102); fx_mac(s, w1_101, u_101); fx_mac(s, w1_102, u_100); fx_mac(s, w[1][10], u_002); fx_mac(s, w1_201, u_001); fx_mac(s, w1_202, u_000); z_mu_202 = fx_sum(s); }
  const Fx H_301 = fx_split(z_w2_301 + z_p_301 + FX_HALF, r);
  const Fx H_201 = fx_split(z_w2_201 + z_p_201 + FX_HALF, r);
  const Fx H_101 = fx_split(z_w2_101 + z_p_101 + FX_HALF, r);
  int64_t z_uH_100; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_100); fx_mac(s, u_100, H_000); z_uH_100 = fx_sum(s); }
  const Fx w2_001 = fx_split_any(fx_time<1>(1 * (z_uH_100), K.third) + FX_HALF, r);
  const int64_t z_w2_001 = fx_join(w2_001);
  int64_t z_mu_001; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_001); fx_mac(s, w1_001, u_000); z_mu_001 = fx_sum(s); }
  const Fx e_001 = fx_split(z_w2_001 - ((z_mu_001) >> 1) + FX_HALF, r);
  int64_t z_p_001; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_001, K.gm1); z_p_001 = fx_sum<FX_C>(s); }
  const Fx H_001 = fx_split(z_w2_001 + z_p_001 + FX_HALF, r);
  int64_t z_uH_301; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_301); fx_mac(s, u_001, H_300); fx_mac(s, u_100, H_201); fx_mac(s, u_101, H_200); fx_mac(s, u_200, H_101); fx_mac(s, u_201, H_100); fx_mac(s, u_300, H_001); fx_mac(s, u_301, H_000); z_uH_301 = fx_sum(s); }
  const Fx w2_202 = fx_split_any(fx_time<2>(3 * (z_uH_301), K.third) + FX_HALF, r);
  const int64_t z_w2_202 = fx_join(w2_202);
  const Fx e_202 = fx_split(z_w2_202 - ((z_mu_202) >> 1) + FX_HALF, r);
  int64_t z_p_202; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_202, K.gm1); z_p_202 = fx_sum<FX_C>(s); }
  const Fx w1_103 = fx_split_any(fx_time<3>(2 * (z_mu_202 + z_p_202), K.third) + FX_HALF, r);
  const int64_t z_w1_103 = fx_join(w1_103);
  const Fx w0_004 = fx_split_any(fx_time<4>(1 * (z_w1_103), K.third) + FX_HALF, r);
  int64_t z_mu_102; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_102); fx_mac(s, w1_001, u_101); fx_mac(s, w1_002, u_100); fx_mac(s, w[1][5], u_002); fx_mac(s, w1_101, u_001); fx_mac(s, w1_102, u_000); z_mu_102 = fx_sum(s); }
  int64_t z_uH_201; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_201); fx_mac(s, u_001, H_200); fx_mac(s, u_100, H_101); fx_mac(s, u_101, H_100); fx_mac(s, u_200, H_001); fx_mac(s, u_201, H_000); z_uH_201 = fx_sum(s); }
  const Fx w2_102 = fx_split_any(fx_time<2>(2 * (z_uH_201), K.third) + FX_HALF, r);
  const int64_t z_w2_102 = fx_join(w2_102);
  const Fx e_102 = fx_split(z_w2_102 - ((z_mu_102) >> 1) + FX_HALF, r);
  int64_t z_p_102; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_102, K.gm1); z_p_102 = fx_sum<FX_C>(s); }
  const Fx w1_003 = fx_split_any(fx_time<3>(1 * (z_mu_102 + z_p_102), K.third) + FX_HALF, r);
  Fx u_003n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_003, -(1 << 30)); fx_mac(s, w0_001, u_002); fx_mac(s, w0_002, u_001); fx_mac(s, w0_003, u_000); u_003n = fx_split(fx_sum(s), r); }
  Fx u_003; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_003n, ninv); u_003 = fx_split(fx_sum<FX_C>(s), r); }
  const int64_t z_w1_202 = fx_join(w1_202);
  const Fx w0_103 = fx_split_any(fx_time<3>(2 * (z_w1_202), K.third) + FX_HALF, r);
  Fx u_103n; { FxAcc s = fx_zero(true); fx_mac_int(s, w1_103, -(1 << 30)); fx_mac(s, w0_001, u_102); fx_mac(s, w0_002, u_101); fx_mac(s, w0_003, u_100); fx_mac(s, w[0][5], u_003); fx_mac(s, w0_101, u_002); fx_mac(s, w0_102, u_001); fx_mac(s, w0_103, u_000); u_103n = fx_split(fx_sum(s), r); }
  Fx u_103; { FxAcc s = fx_zero<FX_C>(true); fx_mac(s, u_103n, ninv); u_103 = fx_split(fx_sum<FX_C>(s), r); }
  int64_t z_mu_103; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_103); fx_mac(s, w1_001, u_102); fx_mac(s, w1_002, u_101); fx_mac(s, w1_003, u_100); fx_mac(s, w[1][5], u_003); fx_mac(s, w1_101, u_002); fx_mac(s, w1_102, u_001); fx_mac(s, w1_103, u_000); z_mu_103 = fx_sum(s); }
  const Fx H_202 = fx_split(z_w2_202 + z_p_202 + FX_HALF, r);
  const Fx H_102 = fx_split(z_w2_102 + z_p_102 + FX_HALF, r);
  int64_t z_uH_101; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_101); fx_mac(s, u_001, H_100); fx_mac(s, u_100, H_001); fx_mac(s, u_101, H_000); z_uH_101 = fx_sum(s); }
  const Fx w2_002 = fx_split_any(fx_time<2>(1 * (z_uH_101), K.third) + FX_HALF, r);
  const int64_t z_w2_002 = fx_join(w2_002);
  int64_t z_mu_002; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_002); fx_mac(s, w1_001, u_001); fx_mac(s, w1_002, u_000); z_mu_002 = fx_sum(s); }
  const Fx e_002 = fx_split(z_w2_002 - ((z_mu_002) >> 1) + FX_HALF, r);
  int64_t z_p_002; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_002, K.gm1); z_p_002 = fx_sum<FX_C>(s); }
  const Fx H_002 = fx_split(z_w2_002 + z_p_002 + FX_HALF, r);
  int64_t z_uH_202; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_202); fx_mac(s, u_001, H_201); fx_mac(s, u_002, H_200); fx_mac(s, u_100, H_102); fx_mac(s, u_101, H_101); fx_mac(s, u_102, H_100); fx_mac(s, u_200, H_002); fx_mac(s, u_201, H_001); fx_mac(s, u_202, H_000); z_uH_202 = fx_sum(s); }
  const Fx w2_103 = fx_split_any(fx_time<3>(2 * (z_uH_202), K.third) + FX_HALF, r);
  const int64_t z_w2_103 = fx_join(w2_103);
  const Fx e_103 = fx_split(z_w2_103 - ((z_mu_103) >> 1) + FX_HALF, r);
  int64_t z_p_103; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_103, K.gm1); z_p_103 = fx_sum<FX_C>(s); }
  const Fx w1_004 = fx_split_any(fx_time<4>(1 * (z_mu_103 + z_p_103), K.third) + FX_HALF, r);
  int64_t z_uH_102; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_102); fx_mac(s, u_001, H_101); fx_mac(s, u_002, H_100); fx_mac(s, u_100, H_002); fx_mac(s, u_101, H_001); fx_mac(s, u_102, H_000); z_uH_102 = fx_sum(s); }
  const Fx w2_003 = fx_split_any(fx_time<3>(1 * (z_uH_102), K.third) + FX_HALF, r);
  const Fx H_103 = fx_split(z_w2_103 + z_p_103 + FX_HALF, r);
  const int64_t z_w2_003 = fx_join(w2_003);
  int64_t z_mu_003; { FxAcc s = fx_zero(); fx_mac(s, w[1][0], u_003); fx_mac(s, w1_001, u_002); fx_mac(s, w1_002, u_001); fx_mac(s, w1_003, u_000); z_mu_003 = fx_sum(s); }
  const Fx e_003 = fx_split(z_w2_003 - ((z_mu_003) >> 1) + FX_HALF, r);
  int64_t z_p_003; { FxAcc s = fx_zero<FX_C>(); fx_mac(s, e_003, K.gm1); z_p_003 = fx_sum<FX_C>(s); }
  const Fx H_003 = fx_split(z_w2_003 + z_p_003 + FX_HALF, r);
  int64_t z_uH_103; { FxAcc s = fx_zero(); fx_mac(s, u_000, H_103); fx_mac(s, u_001, H_102); fx_mac(s, u_002, H_101); fx_mac(s, u_003, H_100); fx_mac(s, u_100, H_003); fx_mac(s, u_101, H_002); fx_mac(s, u_102, H_001); fx_mac(s, u_103, H_000); z_uH_103 = fx_sum(s); }
  const Fx w2_004 = fx_split_any(fx_time<4>(1 * (z_uH_103), K.third) + FX_HALF, r);
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
FX_DEV void ck_euler2d_lane(Store& S, Fx ninv, Fx gm1, Fx third, FxRange& r) {
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
    const Fx n = fx_split_any(fx_sum(s), r0);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel000 = fx_split_any(fx_sum<FX_C>(z), r0); }
  const Fx rho010 = S.ldrho(0, 0, 1);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 1, 0), -(1 << 30));
    fx_mac(s, rho100, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel100 = fx_split_any(fx_sum<FX_C>(z), r); }
  const Fx rho200 = S.ldrho(0, 2, 0);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 0, 1), -(1 << 30));
    fx_mac(s, rho010, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel010 = fx_split_any(fx_sum<FX_C>(z), r); }
  const Fx rho110 = S.ldrho(0, 1, 1);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 2, 0), -(1 << 30));
    fx_mac(s, rho100, vel100);
    fx_mac(s, rho200, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel200 = fx_split_any(fx_sum<FX_C>(z), r); }
  const Fx rho020 = S.ldrho(0, 0, 2);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 1, 1), -(1 << 30));
    fx_mac(s, rho010, vel100);
    fx_mac(s, rho100, vel010);
    fx_mac(s, rho110, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel110 = fx_split_any(fx_sum<FX_C>(z), r); }
  const Fx rho300 = S.ldrho(0, 3, 0);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 0, 2), -(1 << 30));
    fx_mac(s, rho010, vel010);
    fx_mac(s, rho020, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel020 = fx_split_any(fx_sum<FX_C>(z), r); }
  const Fx rho210 = S.ldrho(0, 2, 1);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 3, 0), -(1 << 30));
    fx_mac(s, rho100, vel200);
    fx_mac(s, rho200, vel100);
    fx_mac(s, rho300, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel300 = fx_split_any(fx_sum<FX_C>(z), r); }
  const Fx rho120 = S.ldrho(0, 1, 2);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 2, 1), -(1 << 30));
    fx_mac(s, rho010, vel200);
    fx_mac(s, rho100, vel110);
    fx_mac(s, rho110, vel100);
    fx_mac(s, rho200, vel010);
    fx_mac(s, rho210, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel210 = fx_split_any(fx_sum<FX_C>(z), r); }
  const Fx rho030 = S.ldrho(0, 0, 3);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 1, 2), -(1 << 30));
    fx_mac(s, rho010, vel110);
    fx_mac(s, rho020, vel100);
    fx_mac(s, rho100, vel020);
    fx_mac(s, rho110, vel010);
    fx_mac(s, rho120, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel120 = fx_split_any(fx_sum<FX_C>(z), r); }
  const Fx rho400 = S.ldrho(0, 4, 0);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 0, 3), -(1 << 30));
    fx_mac(s, rho010, vel020);
    fx_mac(s, rho020, vel010);
    fx_mac(s, rho030, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel030 = fx_split_any(fx_sum<FX_C>(z), r); }
  const Fx rho310 = S.ldrho(0, 3, 1);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 4, 0), -(1 << 30));
    fx_mac(s, rho100, vel300);
    fx_mac(s, rho200, vel200);
    fx_mac(s, rho300, vel100);
    fx_mac(s, rho400, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel400 = fx_split_any(fx_sum<FX_C>(z), r); }
  const Fx rho220 = S.ldrho(0, 2, 2);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 3, 1), -(1 << 30));
    fx_mac(s, rho010, vel300);
    fx_mac(s, rho100, vel210);
    fx_mac(s, rho110, vel200);
    fx_mac(s, rho200, vel110);
    fx_mac(s, rho210, vel100);
    fx_mac(s, rho300, vel010);
    fx_mac(s, rho310, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel310 = fx_split_any(fx_sum<FX_C>(z), r); }
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
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel220 = fx_split_any(fx_sum<FX_C>(z), r); }
  const Fx rho040 = S.ldrho(0, 0, 4);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 1, 3), -(1 << 30));
    fx_mac(s, rho010, vel120);
    fx_mac(s, rho020, vel110);
    fx_mac(s, rho030, vel100);
    fx_mac(s, rho100, vel030);
    fx_mac(s, rho110, vel020);
    fx_mac(s, rho120, vel010);
    fx_mac(s, rho130, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel130 = fx_split_any(fx_sum<FX_C>(z), r); }
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(0, 0, 4), -(1 << 30));
    fx_mac(s, rho010, vel030);
    fx_mac(s, rho020, vel020);
    fx_mac(s, rho030, vel010);
    fx_mac(s, rho040, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel040 = fx_split_any(fx_sum<FX_C>(z), r); }
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
    const Fx e = fx_split_any(E - ((k000 + S.swap(k000)) >> 1) + FX_HALF, r0);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 0, 0, fx_split_any(E + p + FX_HALF, r0));
  }
  { const int64_t E = S.ldE(0, 1, 0);
    const Fx e = fx_split_any(E - ((k100 + S.swap(k010)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 1, 0, fx_split_any(E + p + FX_HALF, r));
    f100 = k100 + p;
  }
  { const int64_t E = S.ldE(0, 0, 1);
    const Fx e = fx_split_any(E - ((k010 + S.swap(k100)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 0, 1, fx_split_any(E + p + FX_HALF, r));
  }
  { const int64_t E = S.ldE(0, 2, 0);
    const Fx e = fx_split_any(E - ((k200 + S.swap(k020)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 2, 0, fx_split_any(E + p + FX_HALF, r));
    f200 = k200 + p;
  }
  { const int64_t E = S.ldE(0, 1, 1);
    const Fx e = fx_split_any(E - ((k110 + S.swap(k110)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 1, 1, fx_split_any(E + p + FX_HALF, r));
    f110 = k110 + p;
  }
  { const int64_t E = S.ldE(0, 0, 2);
    const Fx e = fx_split_any(E - ((k020 + S.swap(k200)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 0, 2, fx_split_any(E + p + FX_HALF, r));
  }
  { const int64_t E = S.ldE(0, 3, 0);
    const Fx e = fx_split_any(E - ((k300 + S.swap(k030)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 3, 0, fx_split_any(E + p + FX_HALF, r));
    f300 = k300 + p;
  }
  { const int64_t E = S.ldE(0, 2, 1);
    const Fx e = fx_split_any(E - ((k210 + S.swap(k120)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 2, 1, fx_split_any(E + p + FX_HALF, r));
    f210 = k210 + p;
  }
  { const int64_t E = S.ldE(0, 1, 2);
    const Fx e = fx_split_any(E - ((k120 + S.swap(k210)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 1, 2, fx_split_any(E + p + FX_HALF, r));
    f120 = k120 + p;
  }
  { const int64_t E = S.ldE(0, 0, 3);
    const Fx e = fx_split_any(E - ((k030 + S.swap(k300)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 0, 3, fx_split_any(E + p + FX_HALF, r));
  }
  { const int64_t E = S.ldE(0, 4, 0);
    const Fx e = fx_split_any(E - ((k400 + S.swap(k040)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 4, 0, fx_split_any(E + p + FX_HALF, r));
    f400 = k400 + p;
  }
  { const int64_t E = S.ldE(0, 3, 1);
    const Fx e = fx_split_any(E - ((k310 + S.swap(k130)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 3, 1, fx_split_any(E + p + FX_HALF, r));
    f310 = k310 + p;
  }
  { const int64_t E = S.ldE(0, 2, 2);
    const Fx e = fx_split_any(E - ((k220 + S.swap(k220)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 2, 2, fx_split_any(E + p + FX_HALF, r));
    f220 = k220 + p;
  }
  { const int64_t E = S.ldE(0, 1, 3);
    const Fx e = fx_split_any(E - ((k130 + S.swap(k310)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 1, 3, fx_split_any(E + p + FX_HALF, r));
    f130 = k130 + p;
  }
  { const int64_t E = S.ldE(0, 0, 4);
    const Fx e = fx_split_any(E - ((k040 + S.swap(k400)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(0, 0, 4, fx_split_any(E + p + FX_HALF, r));
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
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel001 = fx_split_any(fx_sum<FX_C>(z), r); }
  const Fx rho010 = S.ldrho(0, 0, 1);
  const Fx rho011 = S.ldrho(1, 0, 1);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(1, 1, 0), -(1 << 30));
    fx_mac(s, rho001, vel100);
    fx_mac(s, rho100, vel001);
    fx_mac(s, rho101, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel101 = fx_split_any(fx_sum<FX_C>(z), r); }
  const Fx rho200 = S.ldrho(0, 2, 0);
  const Fx rho201 = S.ldrho(1, 2, 0);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(1, 0, 1), -(1 << 30));
    fx_mac(s, rho001, vel010);
    fx_mac(s, rho010, vel001);
    fx_mac(s, rho011, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel011 = fx_split_any(fx_sum<FX_C>(z), r); }
  const Fx rho110 = S.ldrho(0, 1, 1);
  const Fx rho111 = S.ldrho(1, 1, 1);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(1, 2, 0), -(1 << 30));
    fx_mac(s, rho001, vel200);
    fx_mac(s, rho100, vel101);
    fx_mac(s, rho101, vel100);
    fx_mac(s, rho200, vel001);
    fx_mac(s, rho201, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel201 = fx_split_any(fx_sum<FX_C>(z), r); }
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
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel111 = fx_split_any(fx_sum<FX_C>(z), r); }
  const Fx rho300 = S.ldrho(0, 3, 0);
  const Fx rho301 = S.ldrho(1, 3, 0);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(1, 0, 2), -(1 << 30));
    fx_mac(s, rho001, vel020);
    fx_mac(s, rho010, vel011);
    fx_mac(s, rho011, vel010);
    fx_mac(s, rho020, vel001);
    fx_mac(s, rho021, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel021 = fx_split_any(fx_sum<FX_C>(z), r); }
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
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel301 = fx_split_any(fx_sum<FX_C>(z), r); }
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
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel211 = fx_split_any(fx_sum<FX_C>(z), r); }
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
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel121 = fx_split_any(fx_sum<FX_C>(z), r); }
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(1, 0, 3), -(1 << 30));
    fx_mac(s, rho001, vel030);
    fx_mac(s, rho010, vel021);
    fx_mac(s, rho011, vel020);
    fx_mac(s, rho020, vel011);
    fx_mac(s, rho021, vel010);
    fx_mac(s, rho030, vel001);
    fx_mac(s, rho031, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel031 = fx_split_any(fx_sum<FX_C>(z), r); }
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
    const Fx e = fx_split_any(E - ((k001 + S.swap(k001)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 0, 0, fx_split_any(E + p + FX_HALF, r));
  }
  { const int64_t E = E101;
    const Fx e = fx_split_any(E - ((k101 + S.swap(k011)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 1, 0, fx_split_any(E + p + FX_HALF, r));
    f101 = k101 + p;
  }
  { const int64_t E = E011;
    const Fx e = fx_split_any(E - ((k011 + S.swap(k101)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 0, 1, fx_split_any(E + p + FX_HALF, r));
  }
  { const int64_t E = E201;
    const Fx e = fx_split_any(E - ((k201 + S.swap(k021)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 2, 0, fx_split_any(E + p + FX_HALF, r));
    f201 = k201 + p;
  }
  { const int64_t E = E111;
    const Fx e = fx_split_any(E - ((k111 + S.swap(k111)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 1, 1, fx_split_any(E + p + FX_HALF, r));
    f111 = k111 + p;
  }
  { const int64_t E = E021;
    const Fx e = fx_split_any(E - ((k021 + S.swap(k201)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 0, 2, fx_split_any(E + p + FX_HALF, r));
  }
  { const int64_t E = E301;
    const Fx e = fx_split_any(E - ((k301 + S.swap(k031)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 3, 0, fx_split_any(E + p + FX_HALF, r));
    f301 = k301 + p;
  }
  { const int64_t E = E211;
    const Fx e = fx_split_any(E - ((k211 + S.swap(k121)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 2, 1, fx_split_any(E + p + FX_HALF, r));
    f211 = k211 + p;
  }
  { const int64_t E = E121;
    const Fx e = fx_split_any(E - ((k121 + S.swap(k211)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 1, 2, fx_split_any(E + p + FX_HALF, r));
    f121 = k121 + p;
  }
  { const int64_t E = E031;
    const Fx e = fx_split_any(E - ((k031 + S.swap(k301)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(1, 0, 3, fx_split_any(E + p + FX_HALF, r));
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
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel002 = fx_split_any(fx_sum<FX_C>(z), r); }
  const Fx rho010 = S.ldrho(0, 0, 1);
  const Fx rho011 = S.ldrho(1, 0, 1);
  const Fx rho012 = S.ldrho(2, 0, 1);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(2, 1, 0), -(1 << 30));
    fx_mac(s, rho001, vel101);
    fx_mac(s, rho002, vel100);
    fx_mac(s, rho100, vel002);
    fx_mac(s, rho101, vel001);
    fx_mac(s, rho102, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel102 = fx_split_any(fx_sum<FX_C>(z), r); }
  const Fx rho200 = S.ldrho(0, 2, 0);
  const Fx rho201 = S.ldrho(1, 2, 0);
  const Fx rho202 = S.ldrho(2, 2, 0);
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(2, 0, 1), -(1 << 30));
    fx_mac(s, rho001, vel011);
    fx_mac(s, rho002, vel010);
    fx_mac(s, rho010, vel002);
    fx_mac(s, rho011, vel001);
    fx_mac(s, rho012, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel012 = fx_split_any(fx_sum<FX_C>(z), r); }
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
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel202 = fx_split_any(fx_sum<FX_C>(z), r); }
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
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel112 = fx_split_any(fx_sum<FX_C>(z), r); }
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(2, 0, 2), -(1 << 30));
    fx_mac(s, rho001, vel021);
    fx_mac(s, rho002, vel020);
    fx_mac(s, rho010, vel012);
    fx_mac(s, rho011, vel011);
    fx_mac(s, rho012, vel010);
    fx_mac(s, rho020, vel002);
    fx_mac(s, rho021, vel001);
    fx_mac(s, rho022, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel022 = fx_split_any(fx_sum<FX_C>(z), r); }
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
    const Fx e = fx_split_any(E - ((k002 + S.swap(k002)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(2, 0, 0, fx_split_any(E + p + FX_HALF, r));
  }
  { const int64_t E = E102;
    const Fx e = fx_split_any(E - ((k102 + S.swap(k012)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(2, 1, 0, fx_split_any(E + p + FX_HALF, r));
    f102 = k102 + p;
  }
  { const int64_t E = E012;
    const Fx e = fx_split_any(E - ((k012 + S.swap(k102)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(2, 0, 1, fx_split_any(E + p + FX_HALF, r));
  }
  { const int64_t E = E202;
    const Fx e = fx_split_any(E - ((k202 + S.swap(k022)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(2, 2, 0, fx_split_any(E + p + FX_HALF, r));
    f202 = k202 + p;
  }
  { const int64_t E = E112;
    const Fx e = fx_split_any(E - ((k112 + S.swap(k112)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(2, 1, 1, fx_split_any(E + p + FX_HALF, r));
    f112 = k112 + p;
  }
  { const int64_t E = E022;
    const Fx e = fx_split_any(E - ((k022 + S.swap(k202)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(2, 0, 2, fx_split_any(E + p + FX_HALF, r));
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
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel003 = fx_split_any(fx_sum<FX_C>(z), r); }
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
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel103 = fx_split_any(fx_sum<FX_C>(z), r); }
  { FxAcc s = fx_zero(true); fx_mac_int(s, S.ldmom(3, 0, 1), -(1 << 30));
    fx_mac(s, rho001, vel012);
    fx_mac(s, rho002, vel011);
    fx_mac(s, rho003, vel010);
    fx_mac(s, rho010, vel003);
    fx_mac(s, rho011, vel002);
    fx_mac(s, rho012, vel001);
    fx_mac(s, rho013, vel000);
    const Fx n = fx_split_any(fx_sum(s), r);
    FxAcc z = fx_zero<FX_C>(true); fx_mac(z, n, ninv); vel013 = fx_split_any(fx_sum<FX_C>(z), r); }
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
    const Fx e = fx_split_any(E - ((k003 + S.swap(k003)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(3, 0, 0, fx_split_any(E + p + FX_HALF, r));
  }
  { const int64_t E = E103;
    const Fx e = fx_split_any(E - ((k103 + S.swap(k013)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(3, 1, 0, fx_split_any(E + p + FX_HALF, r));
    f103 = k103 + p;
  }
  { const int64_t E = E013;
    const Fx e = fx_split_any(E - ((k013 + S.swap(k103)) >> 1) + FX_HALF, r);
    FxAcc s = fx_zero<FX_C>(); fx_mac(s, e, gm1); const int64_t p = fx_sum<FX_C>(s);
    S.stH(3, 0, 1, fx_split_any(E + p + FX_HALF, r));
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

// ck_euler1d: 1D Euler in FP64; inputs a[q][m*5+n] and outputs tc[q][k], k = 1..4, in units of L.
FX_FN void ck_euler1d(const double (&a)[3][25], double (&tc)[3][5], double gm1) {
  const double inv_r0 = 1.0 / a[0][0];
  const double w1_100 = a[1][5];
  const double F0_100 = w1_100;
  const double w0_001 = -(F0_100);
  const double w1_000 = a[1][0];
  const double w1_200 = a[1][10];
  const double w0_100 = a[0][5];
  const double u_000 = w1_000 * inv_r0;
  const double u_100 = (w1_100 - w0_100 * u_000) * inv_r0;
  const double w0_200 = a[0][10];
  const double u_200 = (w1_200 - w0_100 * u_100 - w0_200 * u_000) * inv_r0;
  const double mu_200 = w1_000 * u_200 + w1_100 * u_100 + w1_200 * u_000;
  const double w2_200 = a[2][10];
  const double p_200 = gm1 * (w2_200 - 0.5 * mu_200);
  const double F1_200 = mu_200 + p_200;
  const double w1_101 = -(2.0 * F1_200);
  const double F0_101 = w1_101;
  const double w0_002 = -((1.0 / 2.0) * F0_101);
  const double w1_300 = a[1][15];
  const double w0_300 = a[0][15];
  const double u_300 = (w1_300 - w0_100 * u_200 - w0_200 * u_100 - w0_300 * u_000) * inv_r0;
  const double mu_300 = w1_000 * u_300 + w1_100 * u_200 + w1_200 * u_100 + w1_300 * u_000;
  const double w2_300 = a[2][15];
  const double p_300 = gm1 * (w2_300 - 0.5 * mu_300);
  const double F1_300 = mu_300 + p_300;
  const double w1_201 = -(3.0 * F1_300);
  const double mu_100 = w1_000 * u_100 + w1_100 * u_000;
  const double w2_100 = a[2][5];
  const double p_100 = gm1 * (w2_100 - 0.5 * mu_100);
  const double F1_100 = mu_100 + p_100;
  const double w1_001 = -(F1_100);
  const double u_001 = (w1_001 - w0_001 * u_000) * inv_r0;
  const double F0_200 = w1_200;
  const double w0_101 = -(2.0 * F0_200);
  const double u_101 = (w1_101 - w0_001 * u_100 - w0_100 * u_001 - w0_101 * u_000) * inv_r0;
  const double F0_300 = w1_300;
  const double w0_201 = -(3.0 * F0_300);
  const double u_201 = (w1_201 - w0_001 * u_200 - w0_100 * u_101 - w0_101 * u_100 - w0_200 * u_001 - w0_201 * u_000) * inv_r0;
  const double mu_201 = w1_000 * u_201 + w1_001 * u_200 + w1_100 * u_101 + w1_101 * u_100 + w1_200 * u_001 + w1_201 * u_000;
  const double H_300 = w2_300 + p_300;
  const double H_200 = w2_200 + p_200;
  const double H_100 = w2_100 + p_100;
  const double w2_000 = a[2][0];
  const double mu_000 = w1_000 * u_000;
  const double p_000 = gm1 * (w2_000 - 0.5 * mu_000);
  const double H_000 = w2_000 + p_000;
  const double uH_300 = u_000 * H_300 + u_100 * H_200 + u_200 * H_100 + u_300 * H_000;
  const double F2_300 = uH_300;
  const double w2_201 = -(3.0 * F2_300);
  const double p_201 = gm1 * (w2_201 - 0.5 * mu_201);
  const double F1_201 = mu_201 + p_201;
  const double w1_102 = -(F1_201);
  const double F0_102 = w1_102;
  const double w0_003 = -((1.0 / 3.0) * F0_102);
  const double w1_400 = a[1][20];
  const double w0_400 = a[0][20];
  const double u_400 = (w1_400 - w0_100 * u_300 - w0_200 * u_200 - w0_300 * u_100 - w0_400 * u_000) * inv_r0;
  const double mu_400 = w1_000 * u_400 + w1_100 * u_300 + w1_200 * u_200 + w1_300 * u_100 + w1_400 * u_000;
  const double w2_400 = a[2][20];
  const double p_400 = gm1 * (w2_400 - 0.5 * mu_400);
  const double F1_400 = mu_400 + p_400;
  const double w1_301 = -(4.0 * F1_400);
  const double F0_400 = w1_400;
  const double w0_301 = -(4.0 * F0_400);
  const double u_301 = (w1_301 - w0_001 * u_300 - w0_100 * u_201 - w0_101 * u_200 - w0_200 * u_101 - w0_201 * u_100 - w0_300 * u_001 - w0_301 * u_000) * inv_r0;
  const double mu_301 = w1_000 * u_301 + w1_001 * u_300 + w1_100 * u_201 + w1_101 * u_200 + w1_200 * u_101 + w1_201 * u_100 + w1_300 * u_001 + w1_301 * u_000;
  const double H_400 = w2_400 + p_400;
  const double uH_400 = u_000 * H_400 + u_100 * H_300 + u_200 * H_200 + u_300 * H_100 + u_400 * H_000;
  const double F2_400 = uH_400;
  const double w2_301 = -(4.0 * F2_400);
  const double p_301 = gm1 * (w2_301 - 0.5 * mu_301);
  const double F1_301 = mu_301 + p_301;
  const double w1_202 = -((3.0 / 2.0) * F1_301);
  const double mu_101 = w1_000 * u_101 + w1_001 * u_100 + w1_100 * u_001 + w1_101 * u_000;
  const double uH_200 = u_000 * H_200 + u_100 * H_100 + u_200 * H_000;
  const double F2_200 = uH_200;
  const double w2_101 = -(2.0 * F2_200);
  const double p_101 = gm1 * (w2_101 - 0.5 * mu_101);
  const double F1_101 = mu_101 + p_101;
  const double w1_002 = -((1.0 / 2.0) * F1_101);
  const double u_002 = (w1_002 - w0_001 * u_001 - w0_002 * u_000) * inv_r0;
  const double F0_201 = w1_201;
  const double w0_102 = -(F0_201);
  const double u_102 = (w1_102 - w0_001 * u_101 - w0_002 * u_100 - w0_100 * u_002 - w0_101 * u_001 - w0_102 * u_000) * inv_r0;
  const double F0_301 = w1_301;
  const double w0_202 = -((3.0 / 2.0) * F0_301);
  const double u_202 = (w1_202 - w0_001 * u_201 - w0_002 * u_200 - w0_100 * u_102 - w0_101 * u_101 - w0_102 * u_100 - w0_200 * u_002 - w0_201 * u_001 - w0_202 * u_000) * inv_r0;
  const double mu_202 = w1_000 * u_202 + w1_001 * u_201 + w1_002 * u_200 + w1_100 * u_102 + w1_101 * u_101 + w1_102 * u_100 + w1_200 * u_002 + w1_201 * u_001 + w1_202 * u_000;
  const double H_301 = w2_301 + p_301;
  const double H_201 = w2_201 + p_201;
  const double H_101 = w2_101 + p_101;
  const double uH_100 = u_000 * H_100 + u_100 * H_000;
  const double F2_100 = uH_100;
  const double w2_001 = -(F2_100);
  const double mu_001 = w1_000 * u_001 + w1_001 * u_000;
  const double p_001 = gm1 * (w2_001 - 0.5 * mu_001);
  const double H_001 = w2_001 + p_001;
  const double uH_301 = u_000 * H_301 + u_001 * H_300 + u_100 * H_201 + u_101 * H_200 + u_200 * H_101 + u_201 * H_100 + u_300 * H_001 + u_301 * H_000;
  const double F2_301 = uH_301;
  const double w2_202 = -((3.0 / 2.0) * F2_301);
  const double p_202 = gm1 * (w2_202 - 0.5 * mu_202);
  const double F1_202 = mu_202 + p_202;
  const double w1_103 = -((2.0 / 3.0) * F1_202);
  const double F0_103 = w1_103;
  const double w0_004 = -((1.0 / 4.0) * F0_103);
  const double mu_102 = w1_000 * u_102 + w1_001 * u_101 + w1_002 * u_100 + w1_100 * u_002 + w1_101 * u_001 + w1_102 * u_000;
  const double uH_201 = u_000 * H_201 + u_001 * H_200 + u_100 * H_101 + u_101 * H_100 + u_200 * H_001 + u_201 * H_000;
  const double F2_201 = uH_201;
  const double w2_102 = -(F2_201);
  const double p_102 = gm1 * (w2_102 - 0.5 * mu_102);
  const double F1_102 = mu_102 + p_102;
  const double w1_003 = -((1.0 / 3.0) * F1_102);
  const double u_003 = (w1_003 - w0_001 * u_002 - w0_002 * u_001 - w0_003 * u_000) * inv_r0;
  const double F0_202 = w1_202;
  const double w0_103 = -((2.0 / 3.0) * F0_202);
  const double u_103 = (w1_103 - w0_001 * u_102 - w0_002 * u_101 - w0_003 * u_100 - w0_100 * u_003 - w0_101 * u_002 - w0_102 * u_001 - w0_103 * u_000) * inv_r0;
  const double mu_103 = w1_000 * u_103 + w1_001 * u_102 + w1_002 * u_101 + w1_003 * u_100 + w1_100 * u_003 + w1_101 * u_002 + w1_102 * u_001 + w1_103 * u_000;
  const double H_202 = w2_202 + p_202;
  const double H_102 = w2_102 + p_102;
  const double uH_101 = u_000 * H_101 + u_001 * H_100 + u_100 * H_001 + u_101 * H_000;
  const double F2_101 = uH_101;
  const double w2_002 = -((1.0 / 2.0) * F2_101);
  const double mu_002 = w1_000 * u_002 + w1_001 * u_001 + w1_002 * u_000;
  const double p_002 = gm1 * (w2_002 - 0.5 * mu_002);
  const double H_002 = w2_002 + p_002;
  const double uH_202 = u_000 * H_202 + u_001 * H_201 + u_002 * H_200 + u_100 * H_102 + u_101 * H_101 + u_102 * H_100 + u_200 * H_002 + u_201 * H_001 + u_202 * H_000;
  const double F2_202 = uH_202;
  const double w2_103 = -((2.0 / 3.0) * F2_202);
  const double p_103 = gm1 * (w2_103 - 0.5 * mu_103);
  const double F1_103 = mu_103 + p_103;
  const double w1_004 = -((1.0 / 4.0) * F1_103);
  const double uH_102 = u_000 * H_102 + u_001 * H_101 + u_002 * H_100 + u_100 * H_002 + u_101 * H_001 + u_102 * H_000;
  const double F2_102 = uH_102;
  const double w2_003 = -((1.0 / 3.0) * F2_102);
  const double H_103 = w2_103 + p_103;
  const double mu_003 = w1_000 * u_003 + w1_001 * u_002 + w1_002 * u_001 + w1_003 * u_000;
  const double p_003 = gm1 * (w2_003 - 0.5 * mu_003);
  const double H_003 = w2_003 + p_003;
  const double uH_103 = u_000 * H_103 + u_001 * H_102 + u_002 * H_101 + u_003 * H_100 + u_100 * H_003 + u_101 * H_002 + u_102 * H_001 + u_103 * H_000;
  const double F2_103 = uH_103;
  const double w2_004 = -((1.0 / 4.0) * F2_103);
  tc[0][1] = w0_001;
  tc[0][2] = w0_002;
  tc[0][3] = w0_003;
  tc[0][4] = w0_004;
  tc[1][1] = w1_001;
  tc[1][2] = w1_002;
  tc[1][3] = w1_003;
  tc[1][4] = w1_004;
  tc[2][1] = w2_001;
  tc[2][2] = w2_002;
  tc[2][3] = w2_003;
  tc[2][4] = w2_004;
}

// ck_euler2d: 2D Euler in FP64; inputs a[q][m*5+n] and outputs tc[q][k], k = 1..4, in units of L.
FX_FN void ck_euler2d(const double (&a)[4][25], double (&tc)[4][5], double gm1) {
  const double inv_r0 = 1.0 / a[0][0];
  const double w1_100 = a[1][5];
  const double F0_100 = w1_100;
  const double w2_010 = a[2][1];
  const double G0_010 = w2_010;
  const double w0_001 = -(F0_100 + G0_010);
  const double w1_000 = a[1][0];
  const double w1_200 = a[1][10];
  const double w0_100 = a[0][5];
  const double u_000 = w1_000 * inv_r0;
  const double u_100 = (w1_100 - w0_100 * u_000) * inv_r0;
  const double w0_200 = a[0][10];
  const double u_200 = (w1_200 - w0_100 * u_100 - w0_200 * u_000) * inv_r0;
  const double mu_200 = w1_000 * u_200 + w1_100 * u_100 + w1_200 * u_000;
  const double w3_200 = a[3][10];
  const double w2_000 = a[2][0];
  const double w2_200 = a[2][10];
  const double w2_100 = a[2][5];
  const double v_000 = w2_000 * inv_r0;
  const double v_100 = (w2_100 - w0_100 * v_000) * inv_r0;
  const double v_200 = (w2_200 - w0_100 * v_100 - w0_200 * v_000) * inv_r0;
  const double nv_200 = w2_000 * v_200 + w2_100 * v_100 + w2_200 * v_000;
  const double p_200 = gm1 * (w3_200 - 0.5 * (mu_200 + nv_200));
  const double F1_200 = mu_200 + p_200;
  const double w2_110 = a[2][6];
  const double w0_010 = a[0][1];
  const double v_010 = (w2_010 - w0_010 * v_000) * inv_r0;
  const double w0_110 = a[0][6];
  const double v_110 = (w2_110 - w0_010 * v_100 - w0_100 * v_010 - w0_110 * v_000) * inv_r0;
  const double w1_010 = a[1][1];
  const double w1_110 = a[1][6];
  const double mv_110 = w1_000 * v_110 + w1_010 * v_100 + w1_100 * v_010 + w1_110 * v_000;
  const double G1_110 = mv_110;
  const double w1_101 = -(2.0 * F1_200 + G1_110);
  const double F0_101 = w1_101;
  const double F2_110 = mv_110;
  const double w2_020 = a[2][2];
  const double w0_020 = a[0][2];
  const double v_020 = (w2_020 - w0_010 * v_010 - w0_020 * v_000) * inv_r0;
  const double nv_020 = w2_000 * v_020 + w2_010 * v_010 + w2_020 * v_000;
  const double w3_020 = a[3][2];
  const double w1_020 = a[1][2];
  const double u_010 = (w1_010 - w0_010 * u_000) * inv_r0;
  const double u_020 = (w1_020 - w0_010 * u_010 - w0_020 * u_000) * inv_r0;
  const double mu_020 = w1_000 * u_020 + w1_010 * u_010 + w1_020 * u_000;
  const double p_020 = gm1 * (w3_020 - 0.5 * (mu_020 + nv_020));
  const double G2_020 = nv_020 + p_020;
  const double w2_011 = -(F2_110 + 2.0 * G2_020);
  const double G0_011 = w2_011;
  const double w0_002 = -((1.0 / 2.0) * F0_101 + (1.0 / 2.0) * G0_011);
  const double w1_300 = a[1][15];
  const double w0_300 = a[0][15];
  const double u_300 = (w1_300 - w0_100 * u_200 - w0_200 * u_100 - w0_300 * u_000) * inv_r0;
  const double mu_300 = w1_000 * u_300 + w1_100 * u_200 + w1_200 * u_100 + w1_300 * u_000;
  const double w3_300 = a[3][15];
  const double w2_300 = a[2][15];
  const double v_300 = (w2_300 - w0_100 * v_200 - w0_200 * v_100 - w0_300 * v_000) * inv_r0;
  const double nv_300 = w2_000 * v_300 + w2_100 * v_200 + w2_200 * v_100 + w2_300 * v_000;
  const double p_300 = gm1 * (w3_300 - 0.5 * (mu_300 + nv_300));
  const double F1_300 = mu_300 + p_300;
  const double w2_210 = a[2][11];
  const double w0_210 = a[0][11];
  const double v_210 = (w2_210 - w0_010 * v_200 - w0_100 * v_110 - w0_110 * v_100 - w0_200 * v_010 - w0_210 * v_000) * inv_r0;
  const double w1_210 = a[1][11];
  const double mv_210 = w1_000 * v_210 + w1_010 * v_200 + w1_100 * v_110 + w1_110 * v_100 + w1_200 * v_010 + w1_210 * v_000;
  const double G1_210 = mv_210;
  const double w1_201 = -(3.0 * F1_300 + G1_210);
  const double mu_100 = w1_000 * u_100 + w1_100 * u_000;
  const double w3_100 = a[3][5];
  const double nv_100 = w2_000 * v_100 + w2_100 * v_000;
  const double p_100 = gm1 * (w3_100 - 0.5 * (mu_100 + nv_100));
  const double F1_100 = mu_100 + p_100;
  const double mv_010 = w1_000 * v_010 + w1_010 * v_000;
  const double G1_010 = mv_010;
  const double w1_001 = -(F1_100 + G1_010);
  const double u_001 = (w1_001 - w0_001 * u_000) * inv_r0;
  const double F0_200 = w1_200;
  const double G0_110 = w2_110;
  const double w0_101 = -(2.0 * F0_200 + G0_110);
  const double u_101 = (w1_101 - w0_001 * u_100 - w0_100 * u_001 - w0_101 * u_000) * inv_r0;
  const double F0_300 = w1_300;
  const double G0_210 = w2_210;
  const double w0_201 = -(3.0 * F0_300 + G0_210);
  const double u_201 = (w1_201 - w0_001 * u_200 - w0_100 * u_101 - w0_101 * u_100 - w0_200 * u_001 - w0_201 * u_000) * inv_r0;
  const double mu_201 = w1_000 * u_201 + w1_001 * u_200 + w1_100 * u_101 + w1_101 * u_100 + w1_200 * u_001 + w1_201 * u_000;
  const double H_300 = w3_300 + p_300;
  const double H_200 = w3_200 + p_200;
  const double H_100 = w3_100 + p_100;
  const double w3_000 = a[3][0];
  const double mu_000 = w1_000 * u_000;
  const double nv_000 = w2_000 * v_000;
  const double p_000 = gm1 * (w3_000 - 0.5 * (mu_000 + nv_000));
  const double H_000 = w3_000 + p_000;
  const double uH_300 = u_000 * H_300 + u_100 * H_200 + u_200 * H_100 + u_300 * H_000;
  const double F3_300 = uH_300;
  const double w3_210 = a[3][11];
  const double u_110 = (w1_110 - w0_010 * u_100 - w0_100 * u_010 - w0_110 * u_000) * inv_r0;
  const double u_210 = (w1_210 - w0_010 * u_200 - w0_100 * u_110 - w0_110 * u_100 - w0_200 * u_010 - w0_210 * u_000) * inv_r0;
  const double mu_210 = w1_000 * u_210 + w1_010 * u_200 + w1_100 * u_110 + w1_110 * u_100 + w1_200 * u_010 + w1_210 * u_000;
  const double nv_210 = w2_000 * v_210 + w2_010 * v_200 + w2_100 * v_110 + w2_110 * v_100 + w2_200 * v_010 + w2_210 * v_000;
  const double p_210 = gm1 * (w3_210 - 0.5 * (mu_210 + nv_210));
  const double H_210 = w3_210 + p_210;
  const double w3_110 = a[3][6];
  const double mu_110 = w1_000 * u_110 + w1_010 * u_100 + w1_100 * u_010 + w1_110 * u_000;
  const double nv_110 = w2_000 * v_110 + w2_010 * v_100 + w2_100 * v_010 + w2_110 * v_000;
  const double p_110 = gm1 * (w3_110 - 0.5 * (mu_110 + nv_110));
  const double H_110 = w3_110 + p_110;
  const double w3_010 = a[3][1];
  const double mu_010 = w1_000 * u_010 + w1_010 * u_000;
  const double nv_010 = w2_000 * v_010 + w2_010 * v_000;
  const double p_010 = gm1 * (w3_010 - 0.5 * (mu_010 + nv_010));
  const double H_010 = w3_010 + p_010;
  const double vH_210 = v_000 * H_210 + v_010 * H_200 + v_100 * H_110 + v_110 * H_100 + v_200 * H_010 + v_210 * H_000;
  const double G3_210 = vH_210;
  const double w3_201 = -(3.0 * F3_300 + G3_210);
  const double mv_300 = w1_000 * v_300 + w1_100 * v_200 + w1_200 * v_100 + w1_300 * v_000;
  const double F2_300 = mv_300;
  const double G2_210 = nv_210 + p_210;
  const double w2_201 = -(3.0 * F2_300 + G2_210);
  const double mv_200 = w1_000 * v_200 + w1_100 * v_100 + w1_200 * v_000;
  const double F2_200 = mv_200;
  const double G2_110 = nv_110 + p_110;
  const double w2_101 = -(2.0 * F2_200 + G2_110);
  const double mv_100 = w1_000 * v_100 + w1_100 * v_000;
  const double F2_100 = mv_100;
  const double G2_010 = nv_010 + p_010;
  const double w2_001 = -(F2_100 + G2_010);
  const double v_001 = (w2_001 - w0_001 * v_000) * inv_r0;
  const double v_101 = (w2_101 - w0_001 * v_100 - w0_100 * v_001 - w0_101 * v_000) * inv_r0;
  const double v_201 = (w2_201 - w0_001 * v_200 - w0_100 * v_101 - w0_101 * v_100 - w0_200 * v_001 - w0_201 * v_000) * inv_r0;
  const double nv_201 = w2_000 * v_201 + w2_001 * v_200 + w2_100 * v_101 + w2_101 * v_100 + w2_200 * v_001 + w2_201 * v_000;
  const double p_201 = gm1 * (w3_201 - 0.5 * (mu_201 + nv_201));
  const double F1_201 = mu_201 + p_201;
  const double F2_210 = mv_210;
  const double w2_120 = a[2][7];
  const double w0_120 = a[0][7];
  const double v_120 = (w2_120 - w0_010 * v_110 - w0_020 * v_100 - w0_100 * v_020 - w0_110 * v_010 - w0_120 * v_000) * inv_r0;
  const double nv_120 = w2_000 * v_120 + w2_010 * v_110 + w2_020 * v_100 + w2_100 * v_020 + w2_110 * v_010 + w2_120 * v_000;
  const double w3_120 = a[3][7];
  const double w1_120 = a[1][7];
  const double u_120 = (w1_120 - w0_010 * u_110 - w0_020 * u_100 - w0_100 * u_020 - w0_110 * u_010 - w0_120 * u_000) * inv_r0;
  const double mu_120 = w1_000 * u_120 + w1_010 * u_110 + w1_020 * u_100 + w1_100 * u_020 + w1_110 * u_010 + w1_120 * u_000;
  const double p_120 = gm1 * (w3_120 - 0.5 * (mu_120 + nv_120));
  const double G2_120 = nv_120 + p_120;
  const double w2_111 = -(2.0 * F2_210 + 2.0 * G2_120);
  const double F0_110 = w1_110;
  const double G0_020 = w2_020;
  const double w0_011 = -(F0_110 + 2.0 * G0_020);
  const double v_011 = (w2_011 - w0_001 * v_010 - w0_010 * v_001 - w0_011 * v_000) * inv_r0;
  const double F0_210 = w1_210;
  const double G0_120 = w2_120;
  const double w0_111 = -(2.0 * F0_210 + 2.0 * G0_120);
  const double v_111 = (w2_111 - w0_001 * v_110 - w0_010 * v_101 - w0_011 * v_100 - w0_100 * v_011 - w0_101 * v_010 - w0_110 * v_001 - w0_111 * v_000) * inv_r0;
  const double F1_110 = mu_110 + p_110;
  const double mv_020 = w1_000 * v_020 + w1_010 * v_010 + w1_020 * v_000;
  const double G1_020 = mv_020;
  const double w1_011 = -(F1_110 + 2.0 * G1_020);
  const double F1_210 = mu_210 + p_210;
  const double mv_120 = w1_000 * v_120 + w1_010 * v_110 + w1_020 * v_100 + w1_100 * v_020 + w1_110 * v_010 + w1_120 * v_000;
  const double G1_120 = mv_120;
  const double w1_111 = -(2.0 * F1_210 + 2.0 * G1_120);
  const double mv_111 = w1_000 * v_111 + w1_001 * v_110 + w1_010 * v_101 + w1_011 * v_100 + w1_100 * v_011 + w1_101 * v_010 + w1_110 * v_001 + w1_111 * v_000;
  const double G1_111 = mv_111;
  const double w1_102 = -(F1_201 + (1.0 / 2.0) * G1_111);
  const double F0_102 = w1_102;
  const double F2_111 = mv_111;
  const double F2_120 = mv_120;
  const double w2_030 = a[2][3];
  const double w0_030 = a[0][3];
  const double v_030 = (w2_030 - w0_010 * v_020 - w0_020 * v_010 - w0_030 * v_000) * inv_r0;
  const double nv_030 = w2_000 * v_030 + w2_010 * v_020 + w2_020 * v_010 + w2_030 * v_000;
  const double w3_030 = a[3][3];
  const double w1_030 = a[1][3];
  const double u_030 = (w1_030 - w0_010 * u_020 - w0_020 * u_010 - w0_030 * u_000) * inv_r0;
  const double mu_030 = w1_000 * u_030 + w1_010 * u_020 + w1_020 * u_010 + w1_030 * u_000;
  const double p_030 = gm1 * (w3_030 - 0.5 * (mu_030 + nv_030));
  const double G2_030 = nv_030 + p_030;
  const double w2_021 = -(F2_120 + 3.0 * G2_030);
  const double F0_120 = w1_120;
  const double G0_030 = w2_030;
  const double w0_021 = -(F0_120 + 3.0 * G0_030);
  const double v_021 = (w2_021 - w0_001 * v_020 - w0_010 * v_011 - w0_011 * v_010 - w0_020 * v_001 - w0_021 * v_000) * inv_r0;
  const double nv_021 = w2_000 * v_021 + w2_001 * v_020 + w2_010 * v_011 + w2_011 * v_010 + w2_020 * v_001 + w2_021 * v_000;
  const double H_120 = w3_120 + p_120;
  const double H_020 = w3_020 + p_020;
  const double uH_120 = u_000 * H_120 + u_010 * H_110 + u_020 * H_100 + u_100 * H_020 + u_110 * H_010 + u_120 * H_000;
  const double F3_120 = uH_120;
  const double H_030 = w3_030 + p_030;
  const double vH_030 = v_000 * H_030 + v_010 * H_020 + v_020 * H_010 + v_030 * H_000;
  const double G3_030 = vH_030;
  const double w3_021 = -(F3_120 + 3.0 * G3_030);
  const double F1_120 = mu_120 + p_120;
  const double mv_030 = w1_000 * v_030 + w1_010 * v_020 + w1_020 * v_010 + w1_030 * v_000;
  const double G1_030 = mv_030;
  const double w1_021 = -(F1_120 + 3.0 * G1_030);
  const double u_011 = (w1_011 - w0_001 * u_010 - w0_010 * u_001 - w0_011 * u_000) * inv_r0;
  const double u_021 = (w1_021 - w0_001 * u_020 - w0_010 * u_011 - w0_011 * u_010 - w0_020 * u_001 - w0_021 * u_000) * inv_r0;
  const double mu_021 = w1_000 * u_021 + w1_001 * u_020 + w1_010 * u_011 + w1_011 * u_010 + w1_020 * u_001 + w1_021 * u_000;
  const double p_021 = gm1 * (w3_021 - 0.5 * (mu_021 + nv_021));
  const double G2_021 = nv_021 + p_021;
  const double w2_012 = -((1.0 / 2.0) * F2_111 + G2_021);
  const double G0_012 = w2_012;
  const double w0_003 = -((1.0 / 3.0) * F0_102 + (1.0 / 3.0) * G0_012);
  const double w1_400 = a[1][20];
  const double w0_400 = a[0][20];
  const double u_400 = (w1_400 - w0_100 * u_300 - w0_200 * u_200 - w0_300 * u_100 - w0_400 * u_000) * inv_r0;
  const double mu_400 = w1_000 * u_400 + w1_100 * u_300 + w1_200 * u_200 + w1_300 * u_100 + w1_400 * u_000;
  const double w3_400 = a[3][20];
  const double w2_400 = a[2][20];
  const double v_400 = (w2_400 - w0_100 * v_300 - w0_200 * v_200 - w0_300 * v_100 - w0_400 * v_000) * inv_r0;
  const double nv_400 = w2_000 * v_400 + w2_100 * v_300 + w2_200 * v_200 + w2_300 * v_100 + w2_400 * v_000;
  const double p_400 = gm1 * (w3_400 - 0.5 * (mu_400 + nv_400));
  const double F1_400 = mu_400 + p_400;
  const double w2_310 = a[2][16];
  const double w0_310 = a[0][16];
  const double v_310 = (w2_310 - w0_010 * v_300 - w0_100 * v_210 - w0_110 * v_200 - w0_200 * v_110 - w0_210 * v_100 - w0_300 * v_010 - w0_310 * v_000) * inv_r0;
  const double w1_310 = a[1][16];
  const double mv_310 = w1_000 * v_310 + w1_010 * v_300 + w1_100 * v_210 + w1_110 * v_200 + w1_200 * v_110 + w1_210 * v_100 + w1_300 * v_010 + w1_310 * v_000;
  const double G1_310 = mv_310;
  const double w1_301 = -(4.0 * F1_400 + G1_310);
  const double F0_400 = w1_400;
  const double G0_310 = w2_310;
  const double w0_301 = -(4.0 * F0_400 + G0_310);
  const double u_301 = (w1_301 - w0_001 * u_300 - w0_100 * u_201 - w0_101 * u_200 - w0_200 * u_101 - w0_201 * u_100 - w0_300 * u_001 - w0_301 * u_000) * inv_r0;
  const double mu_301 = w1_000 * u_301 + w1_001 * u_300 + w1_100 * u_201 + w1_101 * u_200 + w1_200 * u_101 + w1_201 * u_100 + w1_300 * u_001 + w1_301 * u_000;
  const double H_400 = w3_400 + p_400;
  const double uH_400 = u_000 * H_400 + u_100 * H_300 + u_200 * H_200 + u_300 * H_100 + u_400 * H_000;
  const double F3_400 = uH_400;
  const double w3_310 = a[3][16];
  const double u_310 = (w1_310 - w0_010 * u_300 - w0_100 * u_210 - w0_110 * u_200 - w0_200 * u_110 - w0_210 * u_100 - w0_300 * u_010 - w0_310 * u_000) * inv_r0;
  const double mu_310 = w1_000 * u_310 + w1_010 * u_300 + w1_100 * u_210 + w1_110 * u_200 + w1_200 * u_110 + w1_210 * u_100 + w1_300 * u_010 + w1_310 * u_000;
  const double nv_310 = w2_000 * v_310 + w2_010 * v_300 + w2_100 * v_210 + w2_110 * v_200 + w2_200 * v_110 + w2_210 * v_100 + w2_300 * v_010 + w2_310 * v_000;
  const double p_310 = gm1 * (w3_310 - 0.5 * (mu_310 + nv_310));
  const double H_310 = w3_310 + p_310;
  const double vH_310 = v_000 * H_310 + v_010 * H_300 + v_100 * H_210 + v_110 * H_200 + v_200 * H_110 + v_210 * H_100 + v_300 * H_010 + v_310 * H_000;
  const double G3_310 = vH_310;
  const double w3_301 = -(4.0 * F3_400 + G3_310);
  const double mv_400 = w1_000 * v_400 + w1_100 * v_300 + w1_200 * v_200 + w1_300 * v_100 + w1_400 * v_000;
  const double F2_400 = mv_400;
  const double G2_310 = nv_310 + p_310;
  const double w2_301 = -(4.0 * F2_400 + G2_310);
  const double v_301 = (w2_301 - w0_001 * v_300 - w0_100 * v_201 - w0_101 * v_200 - w0_200 * v_101 - w0_201 * v_100 - w0_300 * v_001 - w0_301 * v_000) * inv_r0;
  const double nv_301 = w2_000 * v_301 + w2_001 * v_300 + w2_100 * v_201 + w2_101 * v_200 + w2_200 * v_101 + w2_201 * v_100 + w2_300 * v_001 + w2_301 * v_000;
  const double p_301 = gm1 * (w3_301 - 0.5 * (mu_301 + nv_301));
  const double F1_301 = mu_301 + p_301;
  const double F2_310 = mv_310;
  const double w2_220 = a[2][12];
  const double w0_220 = a[0][12];
  const double v_220 = (w2_220 - w0_010 * v_210 - w0_020 * v_200 - w0_100 * v_120 - w0_110 * v_110 - w0_120 * v_100 - w0_200 * v_020 - w0_210 * v_010 - w0_220 * v_000) * inv_r0;
  const double nv_220 = w2_000 * v_220 + w2_010 * v_210 + w2_020 * v_200 + w2_100 * v_120 + w2_110 * v_110 + w2_120 * v_100 + w2_200 * v_020 + w2_210 * v_010 + w2_220 * v_000;
  const double w3_220 = a[3][12];
  const double w1_220 = a[1][12];
  const double u_220 = (w1_220 - w0_010 * u_210 - w0_020 * u_200 - w0_100 * u_120 - w0_110 * u_110 - w0_120 * u_100 - w0_200 * u_020 - w0_210 * u_010 - w0_220 * u_000) * inv_r0;
  const double mu_220 = w1_000 * u_220 + w1_010 * u_210 + w1_020 * u_200 + w1_100 * u_120 + w1_110 * u_110 + w1_120 * u_100 + w1_200 * u_020 + w1_210 * u_010 + w1_220 * u_000;
  const double p_220 = gm1 * (w3_220 - 0.5 * (mu_220 + nv_220));
  const double G2_220 = nv_220 + p_220;
  const double w2_211 = -(3.0 * F2_310 + 2.0 * G2_220);
  const double F0_310 = w1_310;
  const double G0_220 = w2_220;
  const double w0_211 = -(3.0 * F0_310 + 2.0 * G0_220);
  const double v_211 = (w2_211 - w0_001 * v_210 - w0_010 * v_201 - w0_011 * v_200 - w0_100 * v_111 - w0_101 * v_110 - w0_110 * v_101 - w0_111 * v_100 - w0_200 * v_011 - w0_201 * v_010 - w0_210 * v_001 - w0_211 * v_000) * inv_r0;
  const double F1_310 = mu_310 + p_310;
  const double mv_220 = w1_000 * v_220 + w1_010 * v_210 + w1_020 * v_200 + w1_100 * v_120 + w1_110 * v_110 + w1_120 * v_100 + w1_200 * v_020 + w1_210 * v_010 + w1_220 * v_000;
  const double G1_220 = mv_220;
  const double w1_211 = -(3.0 * F1_310 + 2.0 * G1_220);
  const double mv_211 = w1_000 * v_211 + w1_001 * v_210 + w1_010 * v_201 + w1_011 * v_200 + w1_100 * v_111 + w1_101 * v_110 + w1_110 * v_101 + w1_111 * v_100 + w1_200 * v_011 + w1_201 * v_010 + w1_210 * v_001 + w1_211 * v_000;
  const double G1_211 = mv_211;
  const double w1_202 = -((3.0 / 2.0) * F1_301 + (1.0 / 2.0) * G1_211);
  const double mu_101 = w1_000 * u_101 + w1_001 * u_100 + w1_100 * u_001 + w1_101 * u_000;
  const double uH_200 = u_000 * H_200 + u_100 * H_100 + u_200 * H_000;
  const double F3_200 = uH_200;
  const double vH_110 = v_000 * H_110 + v_010 * H_100 + v_100 * H_010 + v_110 * H_000;
  const double G3_110 = vH_110;
  const double w3_101 = -(2.0 * F3_200 + G3_110);
  const double nv_101 = w2_000 * v_101 + w2_001 * v_100 + w2_100 * v_001 + w2_101 * v_000;
  const double p_101 = gm1 * (w3_101 - 0.5 * (mu_101 + nv_101));
  const double F1_101 = mu_101 + p_101;
  const double mv_011 = w1_000 * v_011 + w1_001 * v_010 + w1_010 * v_001 + w1_011 * v_000;
  const double G1_011 = mv_011;
  const double w1_002 = -((1.0 / 2.0) * F1_101 + (1.0 / 2.0) * G1_011);
  const double u_002 = (w1_002 - w0_001 * u_001 - w0_002 * u_000) * inv_r0;
  const double F0_201 = w1_201;
  const double G0_111 = w2_111;
  const double w0_102 = -(F0_201 + (1.0 / 2.0) * G0_111);
  const double u_102 = (w1_102 - w0_001 * u_101 - w0_002 * u_100 - w0_100 * u_002 - w0_101 * u_001 - w0_102 * u_000) * inv_r0;
  const double F0_301 = w1_301;
  const double G0_211 = w2_211;
  const double w0_202 = -((3.0 / 2.0) * F0_301 + (1.0 / 2.0) * G0_211);
  const double u_202 = (w1_202 - w0_001 * u_201 - w0_002 * u_200 - w0_100 * u_102 - w0_101 * u_101 - w0_102 * u_100 - w0_200 * u_002 - w0_201 * u_001 - w0_202 * u_000) * inv_r0;
  const double mu_202 = w1_000 * u_202 + w1_001 * u_201 + w1_002 * u_200 + w1_100 * u_102 + w1_101 * u_101 + w1_102 * u_100 + w1_200 * u_002 + w1_201 * u_001 + w1_202 * u_000;
  const double H_301 = w3_301 + p_301;
  const double H_201 = w3_201 + p_201;
  const double H_101 = w3_101 + p_101;
  const double uH_100 = u_000 * H_100 + u_100 * H_000;
  const double F3_100 = uH_100;
  const double vH_010 = v_000 * H_010 + v_010 * H_000;
  const double G3_010 = vH_010;
  const double w3_001 = -(F3_100 + G3_010);
  const double mu_001 = w1_000 * u_001 + w1_001 * u_000;
  const double nv_001 = w2_000 * v_001 + w2_001 * v_000;
  const double p_001 = gm1 * (w3_001 - 0.5 * (mu_001 + nv_001));
  const double H_001 = w3_001 + p_001;
  const double uH_301 = u_000 * H_301 + u_001 * H_300 + u_100 * H_201 + u_101 * H_200 + u_200 * H_101 + u_201 * H_100 + u_300 * H_001 + u_301 * H_000;
  const double F3_301 = uH_301;
  const double uH_310 = u_000 * H_310 + u_010 * H_300 + u_100 * H_210 + u_110 * H_200 + u_200 * H_110 + u_210 * H_100 + u_300 * H_010 + u_310 * H_000;
  const double F3_310 = uH_310;
  const double H_220 = w3_220 + p_220;
  const double vH_220 = v_000 * H_220 + v_010 * H_210 + v_020 * H_200 + v_100 * H_120 + v_110 * H_110 + v_120 * H_100 + v_200 * H_020 + v_210 * H_010 + v_220 * H_000;
  const double G3_220 = vH_220;
  const double w3_211 = -(3.0 * F3_310 + 2.0 * G3_220);
  const double u_111 = (w1_111 - w0_001 * u_110 - w0_010 * u_101 - w0_011 * u_100 - w0_100 * u_011 - w0_101 * u_010 - w0_110 * u_001 - w0_111 * u_000) * inv_r0;
  const double u_211 = (w1_211 - w0_001 * u_210 - w0_010 * u_201 - w0_011 * u_200 - w0_100 * u_111 - w0_101 * u_110 - w0_110 * u_101 - w0_111 * u_100 - w0_200 * u_011 - w0_201 * u_010 - w0_210 * u_001 - w0_211 * u_000) * inv_r0;
  const double mu_211 = w1_000 * u_211 + w1_001 * u_210 + w1_010 * u_201 + w1_011 * u_200 + w1_100 * u_111 + w1_101 * u_110 + w1_110 * u_101 + w1_111 * u_100 + w1_200 * u_011 + w1_201 * u_010 + w1_210 * u_001 + w1_211 * u_000;
  const double nv_211 = w2_000 * v_211 + w2_001 * v_210 + w2_010 * v_201 + w2_011 * v_200 + w2_100 * v_111 + w2_101 * v_110 + w2_110 * v_101 + w2_111 * v_100 + w2_200 * v_011 + w2_201 * v_010 + w2_210 * v_001 + w2_211 * v_000;
  const double p_211 = gm1 * (w3_211 - 0.5 * (mu_211 + nv_211));
  const double H_211 = w3_211 + p_211;
  const double uH_210 = u_000 * H_210 + u_010 * H_200 + u_100 * H_110 + u_110 * H_100 + u_200 * H_010 + u_210 * H_000;
  const double F3_210 = uH_210;
  const double vH_120 = v_000 * H_120 + v_010 * H_110 + v_020 * H_100 + v_100 * H_020 + v_110 * H_010 + v_120 * H_000;
  const double G3_120 = vH_120;
  const double w3_111 = -(2.0 * F3_210 + 2.0 * G3_120);
  const double mu_111 = w1_000 * u_111 + w1_001 * u_110 + w1_010 * u_101 + w1_011 * u_100 + w1_100 * u_011 + w1_101 * u_010 + w1_110 * u_001 + w1_111 * u_000;
  const double nv_111 = w2_000 * v_111 + w2_001 * v_110 + w2_010 * v_101 + w2_011 * v_100 + w2_100 * v_011 + w2_101 * v_010 + w2_110 * v_001 + w2_111 * v_000;
  const double p_111 = gm1 * (w3_111 - 0.5 * (mu_111 + nv_111));
  const double H_111 = w3_111 + p_111;
  const double uH_110 = u_000 * H_110 + u_010 * H_100 + u_100 * H_010 + u_110 * H_000;
  const double F3_110 = uH_110;
  const double vH_020 = v_000 * H_020 + v_010 * H_010 + v_020 * H_000;
  const double G3_020 = vH_020;
  const double w3_011 = -(F3_110 + 2.0 * G3_020);
  const double mu_011 = w1_000 * u_011 + w1_001 * u_010 + w1_010 * u_001 + w1_011 * u_000;
  const double nv_011 = w2_000 * v_011 + w2_001 * v_010 + w2_010 * v_001 + w2_011 * v_000;
  const double p_011 = gm1 * (w3_011 - 0.5 * (mu_011 + nv_011));
  const double H_011 = w3_011 + p_011;
  const double vH_211 = v_000 * H_211 + v_001 * H_210 + v_010 * H_201 + v_011 * H_200 + v_100 * H_111 + v_101 * H_110 + v_110 * H_101 + v_111 * H_100 + v_200 * H_011 + v_201 * H_010 + v_210 * H_001 + v_211 * H_000;
  const double G3_211 = vH_211;
  const double w3_202 = -((3.0 / 2.0) * F3_301 + (1.0 / 2.0) * G3_211);
  const double mv_301 = w1_000 * v_301 + w1_001 * v_300 + w1_100 * v_201 + w1_101 * v_200 + w1_200 * v_101 + w1_201 * v_100 + w1_300 * v_001 + w1_301 * v_000;
  const double F2_301 = mv_301;
  const double G2_211 = nv_211 + p_211;
  const double w2_202 = -((3.0 / 2.0) * F2_301 + (1.0 / 2.0) * G2_211);
  const double mv_201 = w1_000 * v_201 + w1_001 * v_200 + w1_100 * v_101 + w1_101 * v_100 + w1_200 * v_001 + w1_201 * v_000;
  const double F2_201 = mv_201;
  const double G2_111 = nv_111 + p_111;
  const double w2_102 = -(F2_201 + (1.0 / 2.0) * G2_111);
  const double mv_101 = w1_000 * v_101 + w1_001 * v_100 + w1_100 * v_001 + w1_101 * v_000;
  const double F2_101 = mv_101;
  const double G2_011 = nv_011 + p_011;
  const double w2_002 = -((1.0 / 2.0) * F2_101 + (1.0 / 2.0) * G2_011);
  const double v_002 = (w2_002 - w0_001 * v_001 - w0_002 * v_000) * inv_r0;
  const double v_102 = (w2_102 - w0_001 * v_101 - w0_002 * v_100 - w0_100 * v_002 - w0_101 * v_001 - w0_102 * v_000) * inv_r0;
  const double v_202 = (w2_202 - w0_001 * v_201 - w0_002 * v_200 - w0_100 * v_102 - w0_101 * v_101 - w0_102 * v_100 - w0_200 * v_002 - w0_201 * v_001 - w0_202 * v_000) * inv_r0;
  const double nv_202 = w2_000 * v_202 + w2_001 * v_201 + w2_002 * v_200 + w2_100 * v_102 + w2_101 * v_101 + w2_102 * v_100 + w2_200 * v_002 + w2_201 * v_001 + w2_202 * v_000;
  const double p_202 = gm1 * (w3_202 - 0.5 * (mu_202 + nv_202));
  const double F1_202 = mu_202 + p_202;
  const double F2_211 = mv_211;
  const double F2_220 = mv_220;
  const double w2_130 = a[2][8];
  const double w0_130 = a[0][8];
  const double v_130 = (w2_130 - w0_010 * v_120 - w0_020 * v_110 - w0_030 * v_100 - w0_100 * v_030 - w0_110 * v_020 - w0_120 * v_010 - w0_130 * v_000) * inv_r0;
  const double nv_130 = w2_000 * v_130 + w2_010 * v_120 + w2_020 * v_110 + w2_030 * v_100 + w2_100 * v_030 + w2_110 * v_020 + w2_120 * v_010 + w2_130 * v_000;
  const double w3_130 = a[3][8];
  const double w1_130 = a[1][8];
  const double u_130 = (w1_130 - w0_010 * u_120 - w0_020 * u_110 - w0_030 * u_100 - w0_100 * u_030 - w0_110 * u_020 - w0_120 * u_010 - w0_130 * u_000) * inv_r0;
  const double mu_130 = w1_000 * u_130 + w1_010 * u_120 + w1_020 * u_110 + w1_030 * u_100 + w1_100 * u_030 + w1_110 * u_020 + w1_120 * u_010 + w1_130 * u_000;
  const double p_130 = gm1 * (w3_130 - 0.5 * (mu_130 + nv_130));
  const double G2_130 = nv_130 + p_130;
  const double w2_121 = -(2.0 * F2_220 + 3.0 * G2_130);
  const double F0_220 = w1_220;
  const double G0_130 = w2_130;
  const double w0_121 = -(2.0 * F0_220 + 3.0 * G0_130);
  const double v_121 = (w2_121 - w0_001 * v_120 - w0_010 * v_111 - w0_011 * v_110 - w0_020 * v_101 - w0_021 * v_100 - w0_100 * v_021 - w0_101 * v_020 - w0_110 * v_011 - w0_111 * v_010 - w0_120 * v_001 - w0_121 * v_000) * inv_r0;
  const double nv_121 = w2_000 * v_121 + w2_001 * v_120 + w2_010 * v_111 + w2_011 * v_110 + w2_020 * v_101 + w2_021 * v_100 + w2_100 * v_021 + w2_101 * v_020 + w2_110 * v_011 + w2_111 * v_010 + w2_120 * v_001 + w2_121 * v_000;
  const double uH_220 = u_000 * H_220 + u_010 * H_210 + u_020 * H_200 + u_100 * H_120 + u_110 * H_110 + u_120 * H_100 + u_200 * H_020 + u_210 * H_010 + u_220 * H_000;
  const double F3_220 = uH_220;
  const double H_130 = w3_130 + p_130;
  const double vH_130 = v_000 * H_130 + v_010 * H_120 + v_020 * H_110 + v_030 * H_100 + v_100 * H_030 + v_110 * H_020 + v_120 * H_010 + v_130 * H_000;
  const double G3_130 = vH_130;
  const double w3_121 = -(2.0 * F3_220 + 3.0 * G3_130);
  const double F1_220 = mu_220 + p_220;
  const double mv_130 = w1_000 * v_130 + w1_010 * v_120 + w1_020 * v_110 + w1_030 * v_100 + w1_100 * v_030 + w1_110 * v_020 + w1_120 * v_010 + w1_130 * v_000;
  const double G1_130 = mv_130;
  const double w1_121 = -(2.0 * F1_220 + 3.0 * G1_130);
  const double u_121 = (w1_121 - w0_001 * u_120 - w0_010 * u_111 - w0_011 * u_110 - w0_020 * u_101 - w0_021 * u_100 - w0_100 * u_021 - w0_101 * u_020 - w0_110 * u_011 - w0_111 * u_010 - w0_120 * u_001 - w0_121 * u_000) * inv_r0;
  const double mu_121 = w1_000 * u_121 + w1_001 * u_120 + w1_010 * u_111 + w1_011 * u_110 + w1_020 * u_101 + w1_021 * u_100 + w1_100 * u_021 + w1_101 * u_020 + w1_110 * u_011 + w1_111 * u_010 + w1_120 * u_001 + w1_121 * u_000;
  const double p_121 = gm1 * (w3_121 - 0.5 * (mu_121 + nv_121));
  const double G2_121 = nv_121 + p_121;
  const double w2_112 = -(F2_211 + G2_121);
  const double F0_111 = w1_111;
  const double G0_021 = w2_021;
  const double w0_012 = -((1.0 / 2.0) * F0_111 + G0_021);
  const double v_012 = (w2_012 - w0_001 * v_011 - w0_002 * v_010 - w0_010 * v_002 - w0_011 * v_001 - w0_012 * v_000) * inv_r0;
  const double F0_211 = w1_211;
  const double G0_121 = w2_121;
  const double w0_112 = -(F0_211 + G0_121);
  const double v_112 = (w2_112 - w0_001 * v_111 - w0_002 * v_110 - w0_010 * v_102 - w0_011 * v_101 - w0_012 * v_100 - w0_100 * v_012 - w0_101 * v_011 - w0_102 * v_010 - w0_110 * v_002 - w0_111 * v_001 - w0_112 * v_000) * inv_r0;
  const double F1_111 = mu_111 + p_111;
  const double mv_021 = w1_000 * v_021 + w1_001 * v_020 + w1_010 * v_011 + w1_011 * v_010 + w1_020 * v_001 + w1_021 * v_000;
  const double G1_021 = mv_021;
  const double w1_012 = -((1.0 / 2.0) * F1_111 + G1_021);
  const double F1_211 = mu_211 + p_211;
  const double mv_121 = w1_000 * v_121 + w1_001 * v_120 + w1_010 * v_111 + w1_011 * v_110 + w1_020 * v_101 + w1_021 * v_100 + w1_100 * v_021 + w1_101 * v_020 + w1_110 * v_011 + w1_111 * v_010 + w1_120 * v_001 + w1_121 * v_000;
  const double G1_121 = mv_121;
  const double w1_112 = -(F1_211 + G1_121);
  const double mv_112 = w1_000 * v_112 + w1_001 * v_111 + w1_002 * v_110 + w1_010 * v_102 + w1_011 * v_101 + w1_012 * v_100 + w1_100 * v_012 + w1_101 * v_011 + w1_102 * v_010 + w1_110 * v_002 + w1_111 * v_001 + w1_112 * v_000;
  const double G1_112 = mv_112;
  const double w1_103 = -((2.0 / 3.0) * F1_202 + (1.0 / 3.0) * G1_112);
  const double F0_103 = w1_103;
  const double F2_112 = mv_112;
  const double F2_121 = mv_121;
  const double F2_130 = mv_130;
  const double w2_040 = a[2][4];
  const double w0_040 = a[0][4];
  const double v_040 = (w2_040 - w0_010 * v_030 - w0_020 * v_020 - w0_030 * v_010 - w0_040 * v_000) * inv_r0;
  const double nv_040 = w2_000 * v_040 + w2_010 * v_030 + w2_020 * v_020 + w2_030 * v_010 + w2_040 * v_000;
  const double w3_040 = a[3][4];
  const double w1_040 = a[1][4];
  const double u_040 = (w1_040 - w0_010 * u_030 - w0_020 * u_020 - w0_030 * u_010 - w0_040 * u_000) * inv_r0;
  const double mu_040 = w1_000 * u_040 + w1_010 * u_030 + w1_020 * u_020 + w1_030 * u_010 + w1_040 * u_000;
  const double p_040 = gm1 * (w3_040 - 0.5 * (mu_040 + nv_040));
  const double G2_040 = nv_040 + p_040;
  const double w2_031 = -(F2_130 + 4.0 * G2_040);
  const double F0_130 = w1_130;
  const double G0_040 = w2_040;
  const double w0_031 = -(F0_130 + 4.0 * G0_040);
  const double v_031 = (w2_031 - w0_001 * v_030 - w0_010 * v_021 - w0_011 * v_020 - w0_020 * v_011 - w0_021 * v_010 - w0_030 * v_001 - w0_031 * v_000) * inv_r0;
  const double nv_031 = w2_000 * v_031 + w2_001 * v_030 + w2_010 * v_021 + w2_011 * v_020 + w2_020 * v_011 + w2_021 * v_010 + w2_030 * v_001 + w2_031 * v_000;
  const double uH_130 = u_000 * H_130 + u_010 * H_120 + u_020 * H_110 + u_030 * H_100 + u_100 * H_030 + u_110 * H_020 + u_120 * H_010 + u_130 * H_000;
  const double F3_130 = uH_130;
  const double H_040 = w3_040 + p_040;
  const double vH_040 = v_000 * H_040 + v_010 * H_030 + v_020 * H_020 + v_030 * H_010 + v_040 * H_000;
  const double G3_040 = vH_040;
  const double w3_031 = -(F3_130 + 4.0 * G3_040);
  const double F1_130 = mu_130 + p_130;
  const double mv_040 = w1_000 * v_040 + w1_010 * v_030 + w1_020 * v_020 + w1_030 * v_010 + w1_040 * v_000;
  const double G1_040 = mv_040;
  const double w1_031 = -(F1_130 + 4.0 * G1_040);
  const double u_031 = (w1_031 - w0_001 * u_030 - w0_010 * u_021 - w0_011 * u_020 - w0_020 * u_011 - w0_021 * u_010 - w0_030 * u_001 - w0_031 * u_000) * inv_r0;
  const double mu_031 = w1_000 * u_031 + w1_001 * u_030 + w1_010 * u_021 + w1_011 * u_020 + w1_020 * u_011 + w1_021 * u_010 + w1_030 * u_001 + w1_031 * u_000;
  const double p_031 = gm1 * (w3_031 - 0.5 * (mu_031 + nv_031));
  const double G2_031 = nv_031 + p_031;
  const double w2_022 = -((1.0 / 2.0) * F2_121 + (3.0 / 2.0) * G2_031);
  const double F0_121 = w1_121;
  const double G0_031 = w2_031;
  const double w0_022 = -((1.0 / 2.0) * F0_121 + (3.0 / 2.0) * G0_031);
  const double v_022 = (w2_022 - w0_001 * v_021 - w0_002 * v_020 - w0_010 * v_012 - w0_011 * v_011 - w0_012 * v_010 - w0_020 * v_002 - w0_021 * v_001 - w0_022 * v_000) * inv_r0;
  const double nv_022 = w2_000 * v_022 + w2_001 * v_021 + w2_002 * v_020 + w2_010 * v_012 + w2_011 * v_011 + w2_012 * v_010 + w2_020 * v_002 + w2_021 * v_001 + w2_022 * v_000;
  const double H_121 = w3_121 + p_121;
  const double H_021 = w3_021 + p_021;
  const double uH_121 = u_000 * H_121 + u_001 * H_120 + u_010 * H_111 + u_011 * H_110 + u_020 * H_101 + u_021 * H_100 + u_100 * H_021 + u_101 * H_020 + u_110 * H_011 + u_111 * H_010 + u_120 * H_001 + u_121 * H_000;
  const double F3_121 = uH_121;
  const double H_031 = w3_031 + p_031;
  const double vH_031 = v_000 * H_031 + v_001 * H_030 + v_010 * H_021 + v_011 * H_020 + v_020 * H_011 + v_021 * H_010 + v_030 * H_001 + v_031 * H_000;
  const double G3_031 = vH_031;
  const double w3_022 = -((1.0 / 2.0) * F3_121 + (3.0 / 2.0) * G3_031);
  const double F1_121 = mu_121 + p_121;
  const double mv_031 = w1_000 * v_031 + w1_001 * v_030 + w1_010 * v_021 + w1_011 * v_020 + w1_020 * v_011 + w1_021 * v_010 + w1_030 * v_001 + w1_031 * v_000;
  const double G1_031 = mv_031;
  const double w1_022 = -((1.0 / 2.0) * F1_121 + (3.0 / 2.0) * G1_031);
  const double u_012 = (w1_012 - w0_001 * u_011 - w0_002 * u_010 - w0_010 * u_002 - w0_011 * u_001 - w0_012 * u_000) * inv_r0;
  const double u_022 = (w1_022 - w0_001 * u_021 - w0_002 * u_020 - w0_010 * u_012 - w0_011 * u_011 - w0_012 * u_010 - w0_020 * u_002 - w0_021 * u_001 - w0_022 * u_000) * inv_r0;
  const double mu_022 = w1_000 * u_022 + w1_001 * u_021 + w1_002 * u_020 + w1_010 * u_012 + w1_011 * u_011 + w1_012 * u_010 + w1_020 * u_002 + w1_021 * u_001 + w1_022 * u_000;
  const double p_022 = gm1 * (w3_022 - 0.5 * (mu_022 + nv_022));
  const double G2_022 = nv_022 + p_022;
  const double w2_013 = -((1.0 / 3.0) * F2_112 + (2.0 / 3.0) * G2_022);
  const double G0_013 = w2_013;
  const double w0_004 = -((1.0 / 4.0) * F0_103 + (1.0 / 4.0) * G0_013);
  const double mu_102 = w1_000 * u_102 + w1_001 * u_101 + w1_002 * u_100 + w1_100 * u_002 + w1_101 * u_001 + w1_102 * u_000;
  const double uH_201 = u_000 * H_201 + u_001 * H_200 + u_100 * H_101 + u_101 * H_100 + u_200 * H_001 + u_201 * H_000;
  const double F3_201 = uH_201;
  const double vH_111 = v_000 * H_111 + v_001 * H_110 + v_010 * H_101 + v_011 * H_100 + v_100 * H_011 + v_101 * H_010 + v_110 * H_001 + v_111 * H_000;
  const double G3_111 = vH_111;
  const double w3_102 = -(F3_201 + (1.0 / 2.0) * G3_111);
  const double nv_102 = w2_000 * v_102 + w2_001 * v_101 + w2_002 * v_100 + w2_100 * v_002 + w2_101 * v_001 + w2_102 * v_000;
  const double p_102 = gm1 * (w3_102 - 0.5 * (mu_102 + nv_102));
  const double F1_102 = mu_102 + p_102;
  const double mv_012 = w1_000 * v_012 + w1_001 * v_011 + w1_002 * v_010 + w1_010 * v_002 + w1_011 * v_001 + w1_012 * v_000;
  const double G1_012 = mv_012;
  const double w1_003 = -((1.0 / 3.0) * F1_102 + (1.0 / 3.0) * G1_012);
  const double u_003 = (w1_003 - w0_001 * u_002 - w0_002 * u_001 - w0_003 * u_000) * inv_r0;
  const double F0_202 = w1_202;
  const double G0_112 = w2_112;
  const double w0_103 = -((2.0 / 3.0) * F0_202 + (1.0 / 3.0) * G0_112);
  const double u_103 = (w1_103 - w0_001 * u_102 - w0_002 * u_101 - w0_003 * u_100 - w0_100 * u_003 - w0_101 * u_002 - w0_102 * u_001 - w0_103 * u_000) * inv_r0;
  const double mu_103 = w1_000 * u_103 + w1_001 * u_102 + w1_002 * u_101 + w1_003 * u_100 + w1_100 * u_003 + w1_101 * u_002 + w1_102 * u_001 + w1_103 * u_000;
  const double H_202 = w3_202 + p_202;
  const double H_102 = w3_102 + p_102;
  const double uH_101 = u_000 * H_101 + u_001 * H_100 + u_100 * H_001 + u_101 * H_000;
  const double F3_101 = uH_101;
  const double vH_011 = v_000 * H_011 + v_001 * H_010 + v_010 * H_001 + v_011 * H_000;
  const double G3_011 = vH_011;
  const double w3_002 = -((1.0 / 2.0) * F3_101 + (1.0 / 2.0) * G3_011);
  const double mu_002 = w1_000 * u_002 + w1_001 * u_001 + w1_002 * u_000;
  const double nv_002 = w2_000 * v_002 + w2_001 * v_001 + w2_002 * v_000;
  const double p_002 = gm1 * (w3_002 - 0.5 * (mu_002 + nv_002));
  const double H_002 = w3_002 + p_002;
  const double uH_202 = u_000 * H_202 + u_001 * H_201 + u_002 * H_200 + u_100 * H_102 + u_101 * H_101 + u_102 * H_100 + u_200 * H_002 + u_201 * H_001 + u_202 * H_000;
  const double F3_202 = uH_202;
  const double uH_211 = u_000 * H_211 + u_001 * H_210 + u_010 * H_201 + u_011 * H_200 + u_100 * H_111 + u_101 * H_110 + u_110 * H_101 + u_111 * H_100 + u_200 * H_011 + u_201 * H_010 + u_210 * H_001 + u_211 * H_000;
  const double F3_211 = uH_211;
  const double vH_121 = v_000 * H_121 + v_001 * H_120 + v_010 * H_111 + v_011 * H_110 + v_020 * H_101 + v_021 * H_100 + v_100 * H_021 + v_101 * H_020 + v_110 * H_011 + v_111 * H_010 + v_120 * H_001 + v_121 * H_000;
  const double G3_121 = vH_121;
  const double w3_112 = -(F3_211 + G3_121);
  const double u_112 = (w1_112 - w0_001 * u_111 - w0_002 * u_110 - w0_010 * u_102 - w0_011 * u_101 - w0_012 * u_100 - w0_100 * u_012 - w0_101 * u_011 - w0_102 * u_010 - w0_110 * u_002 - w0_111 * u_001 - w0_112 * u_000) * inv_r0;
  const double mu_112 = w1_000 * u_112 + w1_001 * u_111 + w1_002 * u_110 + w1_010 * u_102 + w1_011 * u_101 + w1_012 * u_100 + w1_100 * u_012 + w1_101 * u_011 + w1_102 * u_010 + w1_110 * u_002 + w1_111 * u_001 + w1_112 * u_000;
  const double nv_112 = w2_000 * v_112 + w2_001 * v_111 + w2_002 * v_110 + w2_010 * v_102 + w2_011 * v_101 + w2_012 * v_100 + w2_100 * v_012 + w2_101 * v_011 + w2_102 * v_010 + w2_110 * v_002 + w2_111 * v_001 + w2_112 * v_000;
  const double p_112 = gm1 * (w3_112 - 0.5 * (mu_112 + nv_112));
  const double H_112 = w3_112 + p_112;
  const double uH_111 = u_000 * H_111 + u_001 * H_110 + u_010 * H_101 + u_011 * H_100 + u_100 * H_011 + u_101 * H_010 + u_110 * H_001 + u_111 * H_000;
  const double F3_111 = uH_111;
  const double vH_021 = v_000 * H_021 + v_001 * H_020 + v_010 * H_011 + v_011 * H_010 + v_020 * H_001 + v_021 * H_000;
  const double G3_021 = vH_021;
  const double w3_012 = -((1.0 / 2.0) * F3_111 + G3_021);
  const double mu_012 = w1_000 * u_012 + w1_001 * u_011 + w1_002 * u_010 + w1_010 * u_002 + w1_011 * u_001 + w1_012 * u_000;
  const double nv_012 = w2_000 * v_012 + w2_001 * v_011 + w2_002 * v_010 + w2_010 * v_002 + w2_011 * v_001 + w2_012 * v_000;
  const double p_012 = gm1 * (w3_012 - 0.5 * (mu_012 + nv_012));
  const double H_012 = w3_012 + p_012;
  const double vH_112 = v_000 * H_112 + v_001 * H_111 + v_002 * H_110 + v_010 * H_102 + v_011 * H_101 + v_012 * H_100 + v_100 * H_012 + v_101 * H_011 + v_102 * H_010 + v_110 * H_002 + v_111 * H_001 + v_112 * H_000;
  const double G3_112 = vH_112;
  const double w3_103 = -((2.0 / 3.0) * F3_202 + (1.0 / 3.0) * G3_112);
  const double mv_202 = w1_000 * v_202 + w1_001 * v_201 + w1_002 * v_200 + w1_100 * v_102 + w1_101 * v_101 + w1_102 * v_100 + w1_200 * v_002 + w1_201 * v_001 + w1_202 * v_000;
  const double F2_202 = mv_202;
  const double G2_112 = nv_112 + p_112;
  const double w2_103 = -((2.0 / 3.0) * F2_202 + (1.0 / 3.0) * G2_112);
  const double mv_102 = w1_000 * v_102 + w1_001 * v_101 + w1_002 * v_100 + w1_100 * v_002 + w1_101 * v_001 + w1_102 * v_000;
  const double F2_102 = mv_102;
  const double G2_012 = nv_012 + p_012;
  const double w2_003 = -((1.0 / 3.0) * F2_102 + (1.0 / 3.0) * G2_012);
  const double v_003 = (w2_003 - w0_001 * v_002 - w0_002 * v_001 - w0_003 * v_000) * inv_r0;
  const double v_103 = (w2_103 - w0_001 * v_102 - w0_002 * v_101 - w0_003 * v_100 - w0_100 * v_003 - w0_101 * v_002 - w0_102 * v_001 - w0_103 * v_000) * inv_r0;
  const double nv_103 = w2_000 * v_103 + w2_001 * v_102 + w2_002 * v_101 + w2_003 * v_100 + w2_100 * v_003 + w2_101 * v_002 + w2_102 * v_001 + w2_103 * v_000;
  const double p_103 = gm1 * (w3_103 - 0.5 * (mu_103 + nv_103));
  const double F1_103 = mu_103 + p_103;
  const double F0_112 = w1_112;
  const double G0_022 = w2_022;
  const double w0_013 = -((1.0 / 3.0) * F0_112 + (2.0 / 3.0) * G0_022);
  const double v_013 = (w2_013 - w0_001 * v_012 - w0_002 * v_011 - w0_003 * v_010 - w0_010 * v_003 - w0_011 * v_002 - w0_012 * v_001 - w0_013 * v_000) * inv_r0;
  const double F1_112 = mu_112 + p_112;
  const double mv_022 = w1_000 * v_022 + w1_001 * v_021 + w1_002 * v_020 + w1_010 * v_012 + w1_011 * v_011 + w1_012 * v_010 + w1_020 * v_002 + w1_021 * v_001 + w1_022 * v_000;
  const double G1_022 = mv_022;
  const double w1_013 = -((1.0 / 3.0) * F1_112 + (2.0 / 3.0) * G1_022);
  const double mv_013 = w1_000 * v_013 + w1_001 * v_012 + w1_002 * v_011 + w1_003 * v_010 + w1_010 * v_003 + w1_011 * v_002 + w1_012 * v_001 + w1_013 * v_000;
  const double G1_013 = mv_013;
  const double w1_004 = -((1.0 / 4.0) * F1_103 + (1.0 / 4.0) * G1_013);
  const double mv_103 = w1_000 * v_103 + w1_001 * v_102 + w1_002 * v_101 + w1_003 * v_100 + w1_100 * v_003 + w1_101 * v_002 + w1_102 * v_001 + w1_103 * v_000;
  const double F2_103 = mv_103;
  const double nv_013 = w2_000 * v_013 + w2_001 * v_012 + w2_002 * v_011 + w2_003 * v_010 + w2_010 * v_003 + w2_011 * v_002 + w2_012 * v_001 + w2_013 * v_000;
  const double uH_112 = u_000 * H_112 + u_001 * H_111 + u_002 * H_110 + u_010 * H_102 + u_011 * H_101 + u_012 * H_100 + u_100 * H_012 + u_101 * H_011 + u_102 * H_010 + u_110 * H_002 + u_111 * H_001 + u_112 * H_000;
  const double F3_112 = uH_112;
  const double H_022 = w3_022 + p_022;
  const double vH_022 = v_000 * H_022 + v_001 * H_021 + v_002 * H_020 + v_010 * H_012 + v_011 * H_011 + v_012 * H_010 + v_020 * H_002 + v_021 * H_001 + v_022 * H_000;
  const double G3_022 = vH_022;
  const double w3_013 = -((1.0 / 3.0) * F3_112 + (2.0 / 3.0) * G3_022);
  const double u_013 = (w1_013 - w0_001 * u_012 - w0_002 * u_011 - w0_003 * u_010 - w0_010 * u_003 - w0_011 * u_002 - w0_012 * u_001 - w0_013 * u_000) * inv_r0;
  const double mu_013 = w1_000 * u_013 + w1_001 * u_012 + w1_002 * u_011 + w1_003 * u_010 + w1_010 * u_003 + w1_011 * u_002 + w1_012 * u_001 + w1_013 * u_000;
  const double p_013 = gm1 * (w3_013 - 0.5 * (mu_013 + nv_013));
  const double G2_013 = nv_013 + p_013;
  const double w2_004 = -((1.0 / 4.0) * F2_103 + (1.0 / 4.0) * G2_013);
  const double uH_102 = u_000 * H_102 + u_001 * H_101 + u_002 * H_100 + u_100 * H_002 + u_101 * H_001 + u_102 * H_000;
  const double F3_102 = uH_102;
  const double vH_012 = v_000 * H_012 + v_001 * H_011 + v_002 * H_010 + v_010 * H_002 + v_011 * H_001 + v_012 * H_000;
  const double G3_012 = vH_012;
  const double w3_003 = -((1.0 / 3.0) * F3_102 + (1.0 / 3.0) * G3_012);
  const double H_103 = w3_103 + p_103;
  const double mu_003 = w1_000 * u_003 + w1_001 * u_002 + w1_002 * u_001 + w1_003 * u_000;
  const double nv_003 = w2_000 * v_003 + w2_001 * v_002 + w2_002 * v_001 + w2_003 * v_000;
  const double p_003 = gm1 * (w3_003 - 0.5 * (mu_003 + nv_003));
  const double H_003 = w3_003 + p_003;
  const double uH_103 = u_000 * H_103 + u_001 * H_102 + u_002 * H_101 + u_003 * H_100 + u_100 * H_003 + u_101 * H_002 + u_102 * H_001 + u_103 * H_000;
  const double F3_103 = uH_103;
  const double H_013 = w3_013 + p_013;
  const double vH_013 = v_000 * H_013 + v_001 * H_012 + v_002 * H_011 + v_003 * H_010 + v_010 * H_003 + v_011 * H_002 + v_012 * H_001 + v_013 * H_000;
  const double G3_013 = vH_013;
  const double w3_004 = -((1.0 / 4.0) * F3_103 + (1.0 / 4.0) * G3_013);
  tc[0][1] = w0_001;
  tc[0][2] = w0_002;
  tc[0][3] = w0_003;
  tc[0][4] = w0_004;
  tc[1][1] = w1_001;
  tc[1][2] = w1_002;
  tc[1][3] = w1_003;
  tc[1][4] = w1_004;
  tc[2][1] = w2_001;
  tc[2][2] = w2_002;
  tc[2][3] = w2_003;
  tc[2][4] = w2_004;
  tc[3][1] = w3_001;
  tc[3][2] = w3_002;
  tc[3][3] = w3_003;
  tc[3][4] = w3_004;
}

}  // namespace shweno
