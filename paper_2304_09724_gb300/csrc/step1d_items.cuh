// Device functions of the 1D step, shared by the one-mesh kernel (step1d.cu) and the batched
// kernels (batch.cu): a warp advances up to W1D neighbouring cells by one step.
//
// Lane l owns cell c0 - 1 + l and the face between it and the next lane's cell.  Each cell's
// polynomial is formed once and evaluated at both of its ends (a face that formed both of its
// neighbours' polynomials did that part twice); the left ends travel to the face's lane, and the
// fluxes to the cells' lanes, by shuffles, so nothing but the state is read or written and a step
// is one kernel.  The price is the two halo lanes (32 lanes for 30 cells).
//
// Bound: the FP64 pipe (64 clocks per warp instruction and scheduler), and for meshes that do not
// fill the GPU the latency of one warp's chain of those instructions.
#pragma once
#include "shweno_device.cuh"

namespace shweno {

constexpr int W1D = 30;  // cells a warp advances

// Taylor coefficients 0..4 of the cell's polynomial at its right and left end, one component.  The
// values come from the combined monomial coefficients by Horner's rule: the derivative averages
// are differences of these values over dx, so that on a fine mesh their rounding shows.
template <bool Q>
__device__ __forceinline__ void ends1d(const Params& P, double Wm, double W0, double Wp, double vm, double v0,
                                       double vp, int nonlinear, double eR[5], double eL[5]) {
  double c[6], l[6], r[6];
  p1_coeffs_t<Q>(Wm, W0, Wp, vm, v0, vp, c);
  mix_coeffs_t<Q>(shweno_mix_t<Q>(P, Wm, W0, Wp, c, nonlinear), Wm, W0, Wp, c, r);
#pragma unroll
  for (int m = 0; m < (Q ? 6 : 5); ++m) l[m] = r[m];
  taylor_shift_d<Q ? 5 : 4>(r, 0.5);
  taylor_shift_d<Q ? 5 : 4>(l, -0.5);
#pragma unroll
  for (int m = 0; m < 5; ++m) {
    eR[m] = r[m];
    eL[m] = l[m];
  }
}

// Stencil of cell i, component q: W-, W0, W+ and h times the derivative averages.  (Mapping the
// ghost cells costs a branch per load, so cells inside the mesh load straight.)
struct Stencil1D {
  double Wm, W0, Wp, vm, v0, vp;
};
template <int NC, bool Q>
__device__ __forceinline__ Stencil1D load_stencil1d(const Params& P, const double* st, int q, int i, double t) {
  Stencil1D d;
  if (i >= 1 && i + 1 < P.nx) {
    const double *w = st + (size_t)q * P.nx + i, *v = w + (size_t)NC * P.nx;
    d.Wm = __ldcg(w - 1); d.W0 = __ldcg(w); d.Wp = __ldcg(w + 1);
    d.vm = __ldcg(v - 1); d.v0 = Q ? __ldcg(v) : 0.0; d.vp = __ldcg(v + 1);
  } else {
    d.Wm = fetch(P, st, 0, q, i - 1, 0, t); d.W0 = fetch(P, st, 0, q, i, 0, t); d.Wp = fetch(P, st, 0, q, i + 1, 0, t);
    d.vm = fetch(P, st, 1, q, i - 1, 0, t); d.v0 = Q ? fetch(P, st, 1, q, i, 0, t) : 0.0; d.vp = fetch(P, st, 1, q, i + 1, 0, t);
  }
  d.vm *= P.dx; d.v0 *= P.dx; d.vp *= P.dx;
  return d;
}

// Characteristic-wise option: the Taylor coefficients on the side of a face towards `cell`,
// reconstructed in the fields of basis B.
template <int NC, bool Q>
__device__ __forceinline__ void char_side1d(const Params& P, const double* st, const uint8_t* __restrict__ flag,
                                            int cell, bool right_end, double t, const CharBasis<NC>& B,
                                            double e[NC][5]) {
  const int nonlinear = cell_flag(P, flag, cell, 0);
  constexpr int ND = Q ? 6 : 5;
  double d[ND][NC], x[ND][NC];  // W-, W0, W+, h V-, h V+ (, h V0): physical, then fields
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    d[0][q] = fetch(P, st, 0, q, cell - 1, 0, t);
    d[1][q] = fetch(P, st, 0, q, cell, 0, t);
    d[2][q] = fetch(P, st, 0, q, cell + 1, 0, t);
    d[3][q] = P.dx * fetch(P, st, 1, q, cell - 1, 0, t);
    d[4][q] = P.dx * fetch(P, st, 1, q, cell + 1, 0, t);
    if constexpr (Q) d[5][q] = P.dx * fetch(P, st, 1, q, cell, 0, t);
  }
#pragma unroll
  for (int r = 0; r < ND; ++r) B.to_fields(d[r], x[r]);
  double f[NC][5];
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    double eR[5], eL[5];
    ends1d<Q>(P, x[0][k], x[1][k], x[2][k], x[3][k], Q ? x[ND - 1][k] : 0.0, x[4][k], nonlinear, eR, eL);
#pragma unroll
    for (int m = 0; m < 5; ++m) f[k][m] = right_end ? eR[m] : eL[m];
  }
#pragma unroll
  for (int m = 0; m < 5; ++m) {
    double xm[NC], ym[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) xm[k] = f[k][m];
    B.to_physical(xm, ym);
#pragma unroll
    for (int q = 0; q < NC; ++q) e[q][m] = ym[q];
  }
}

// State and flux at node al of the Lobatto rule in time.  Every node divides on its own: the
// division that the 2D kernels' nodes share moves the flux by a few units in its last place, which
// a fine mesh turns into noise of the derivative averages two steps on (2e-9 of their size at
// 4 M cells), and costs 3 % of the kernel to keep out.
template <int NC>
__device__ __forceinline__ void lobatto_node(const double tc[NC][5], double dt, double g, int al, double W[NC], double F[NC]) {
  using namespace shweno_tables;
  const double tau = al == 1 ? LOB_L1 * dt : al == 2 ? LOB_L2 * dt : dt;
#pragma unroll
  for (int q = 0; q < NC; ++q)
    W[q] = al == 0 ? tc[q][0] : (((tc[q][4] * tau + tc[q][3]) * tau + tc[q][2]) * tau + tc[q][1]) * tau + tc[q][0];
  phys_flux<NC>(W, g, 0, F);
}
__device__ __forceinline__ double lobatto_weight(int al) {
  return al == 0 || al == 3 ? shweno_tables::LOB_W0 : shweno_tables::LOB_W1;
}

// Leading term, derivative problems, Cauchy-Kovalevskaya and Lobatto flux of one face from the
// Taylor coefficients on its two sides: time-averaged flux Fh and the state We at t + dt.
template <int NC>
__device__ __forceinline__ void face1d(const Params& P, const double l[NC][5], const double r[NC][5], double dt,
                                       double Fh[NC], double We[NC]) {
  double a[NC][25], Ws[NC], WL[NC], WR[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    WL[q] = l[q][0];
    WR[q] = r[q][0];
  }
  if constexpr (NC == 1) Ws[0] = burgers_godunov(WL[0], WR[0]);
  else hllc_state<NC>(WL, WR, P.gamma, 0, Ws);
  Upwinder<NC> U;
  U.setup(Ws, P.gamma, 0, NC == 1 ? fmax(fabs(WL[0]), fabs(WR[0])) : 0.0);
#pragma unroll
  for (int m = 1; m < 5; ++m) {
    double x[NC], y[NC], o[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) { x[q] = l[q][m]; y[q] = r[q][m]; }
    U.apply(x, y, o);
#pragma unroll
    for (int q = 0; q < NC; ++q) a[q][m * 5] = o[q];
  }
  double tc[NC][5];
#pragma unroll
  for (int q = 0; q < NC; ++q) a[q][0] = tc[q][0] = Ws[q];
  ck_fixed<NC, 1>(a, U.lead, P.ck, tc);
#pragma unroll
  for (int q = 0; q < NC; ++q) Fh[q] = 0.0;
#pragma unroll
  for (int al = 0; al < 4; ++al) {
    double F[NC];
    lobatto_node<NC>(tc, dt * P.ck.iL, P.gamma, al, We, F);  // the coefficients' unit of time is L = dx
#pragma unroll
    for (int q = 0; q < NC; ++q) Fh[q] += lobatto_weight(al) * F[q];
  }
}

// Update of a warp's cells from the fluxes Fh and states We of the faces right of its lanes' cells
// (Eq. 2.2, 2.11); returns the lane's signal speed as step1d_warp.
template <int NC>
__device__ __forceinline__ double update1d_warp(const Params& P, Ctl* ctl, const double* st, double* out, int i,
                                                bool mine, double dt, const double Fh[NC], const double We[NC]) {
  double Wn[NC], speed = 0.0;
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    const double Fm = __shfl_up_sync(0xffffffffu, Fh[q], 1), Wm = __shfl_up_sync(0xffffffffu, We[q], 1);
    if (mine) {
      Wn[q] = __ldcg(st + (size_t)q * P.nx + i) - dt / P.dx * (Fh[q] - Fm);
      out[(size_t)q * P.nx + i] = Wn[q];
      out[(size_t)(NC + q) * P.nx + i] = (We[q] - Wm) * P.idx;  // 1 / dx from the host
    }
  }
  if (mine) {
    speed = signal_speed1d<NC>(P, Wn);
    if (speed < 0.0) {
      atomicCAS(&ctl->err, ERR_NONE, ERR_NONPHYSICAL);
      __threadfence();  // before this CTA counts as done
      speed = 0.0;
    }
  }
  return speed;
}

// One step of the cells c0 .. c0 + n - 1 (n <= W1D) of state st into out, by one warp; every lane
// calls.  Returns the largest signal speed of the lane's new cell (0: no cell) and raises the
// control block's error word for a non-physical one.
template <int NC, bool Q>
__device__ __forceinline__ double step1d_warp(const Params& P, Ctl* ctl, const double* st, double* out,
                                              const uint8_t* __restrict__ flag, int c0, int n, double t, double dt) {
  const int lane = threadIdx.x & 31, i = c0 - 1 + lane;
  const bool has_cell = lane <= n + 1, has_face = lane <= n;
  double l[NC][5], r[NC][5], Fh[NC], We[NC];
  if (NC > 1 && P.charwise) {
    if constexpr (NC > 1)
      if (has_face) {  // basis at the mean of the two cells next to the face
        double Wref[NC];
#pragma unroll
        for (int q = 0; q < NC; ++q) Wref[q] = 0.5 * (fetch(P, st, 0, q, i, 0, t) + fetch(P, st, 0, q, i + 1, 0, t));
        CharBasis<NC> B;
        B.setup(Wref, P.gamma, 0);
        char_side1d<NC, Q>(P, st, flag, i, true, t, B, l);
        char_side1d<NC, Q>(P, st, flag, i + 1, false, t, B, r);
      }
  } else {
    if (has_cell) {
      const int nonlinear = cell_flag(P, flag, i, 0);
#pragma unroll
      for (int q = 0; q < NC; ++q) {
        const auto d = load_stencil1d<NC, Q>(P, st, q, i, t);
        ends1d<Q>(P, d.Wm, d.W0, d.Wp, d.vm, d.v0, d.vp, nonlinear, l[q], r[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < NC; ++q)
#pragma unroll
      for (int m = 0; m < 5; ++m) r[q][m] = __shfl_down_sync(0xffffffffu, r[q][m], 1);
  }
  if (has_face) face1d<NC>(P, l, r, dt, Fh, We);
  return update1d_warp<NC>(P, ctl, st, out, i, lane >= 1 && lane <= n, dt, Fh, We);
}

// Raises the step's next rate (max of |u| + c over dx) to the warp's largest signal speed.
__device__ __forceinline__ void report_speed1d(const Params& P, Ctl* ctl, double speed) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) speed = fmax(speed, __shfl_xor_sync(0xffffffffu, speed, o));
  if ((threadIdx.x & 31) == 0 && speed > 0.0) {
    const double rate = speed / P.dx;  // non-negative doubles order as their bit patterns
    const unsigned long long bits = (unsigned long long)__double_as_longlong(rate);
    if (bits > *(volatile unsigned long long*)&ctl->rate_next) atomicMax(&ctl->rate_next, bits);
  }
}

// The same step of W1D Euler cells by the four warps of a CTA, for meshes too small to give every
// scheduler a warp of its own cells: what is independent within a cell or face is spread over the
// warps, each of which has a scheduler's FP64 unit to itself (components in the reconstruction,
// derivative orders in the upwinding, Lobatto nodes in the flux; the leading term and the
// Cauchy-Kovalevskaya recursion run in all four).  Same operations on the same numbers as
// step1d_warp, half as many FP64 instructions one after the other (656 -> about 320).
struct Small1D {
  double end[3][2][5][32];  // Taylor coefficients at the cells' right and left ends
  double a[3][4][32];       // upwinded derivatives of the faces
  double F[4][3][32], We[3][32];
};
template <bool Q>
__device__ __forceinline__ double step1d_cta(const Params& P, Ctl* ctl, const double* st, double* out,
                                             const uint8_t* __restrict__ flag, int c0, int n, double t, double dt,
                                             Small1D& S) {
  constexpr int NC = 3;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, i = c0 - 1 + lane;
  const bool has_face = lane <= n;
  if (w < NC && lane <= n + 1) {
    double r[5], l[5];
    const auto d = load_stencil1d<NC, Q>(P, st, w, i, t);
    ends1d<Q>(P, d.Wm, d.W0, d.Wp, d.vm, d.v0, d.vp, cell_flag(P, flag, i, 0), r, l);
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      S.end[w][0][m][lane] = r[m];
      S.end[w][1][m][lane] = l[m];
    }
  }
  __syncthreads();
  double Ws[NC];
  Upwinder<NC> U;
  if (has_face) {
    double L[NC], R[NC], o[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) { L[q] = S.end[q][0][0][lane]; R[q] = S.end[q][1][0][lane + 1]; }
    hllc_state<NC>(L, R, P.gamma, 0, Ws);
    U.setup(Ws, P.gamma, 0);
#pragma unroll
    for (int q = 0; q < NC; ++q) { L[q] = S.end[q][0][w + 1][lane]; R[q] = S.end[q][1][w + 1][lane + 1]; }
    U.apply(L, R, o);
#pragma unroll
    for (int q = 0; q < NC; ++q) S.a[q][w][lane] = o[q];
  }
  __syncthreads();
  if (has_face) {
    double a[NC][25], tc[NC][5], W[NC], F[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      a[q][0] = tc[q][0] = Ws[q];
#pragma unroll
      for (int m = 1; m < 5; ++m) a[q][m * 5] = S.a[q][m - 1][lane];
    }
    ck_fixed<NC, 1>(a, U.lead, P.ck, tc);
    lobatto_node<NC>(tc, dt * P.ck.iL, P.gamma, w, W, F);
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      S.F[w][q][lane] = F[q];
      if (w == 3) S.We[q][lane] = W[q];
    }
  }
  __syncthreads();
  if (w > 0) return 0.0;
  double Fh[NC], We[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    Fh[q] = 0.0;
    We[q] = S.We[q][lane];
#pragma unroll
    for (int al = 0; al < 4; ++al) Fh[q] += lobatto_weight(al) * S.F[al][q][lane];
  }
  return update1d_warp<NC>(P, ctl, st, out, i, lane >= 1 && lane <= n, dt, Fh, We);
}

}  // namespace shweno
