// One ADER-SHWENO time step in two space dimensions (Section 3; Section 4 Steps 1-5).
//
// The SHWENO reconstruction runs dimension by dimension (Section 3.2): a first 1D pass along
// the face gives line averages of W and of its normal derivative as polynomials in the
// tangential coordinate, a second pass across the face gives all mixed derivatives
// d^{m+n}W/dx^m dy^n (m + n <= 4) on both sides of each face quadrature point.
//
//   coef2d   one thread per cell (ghost ring included) and reconstruction: the first-pass
//            polynomials, y-pass on {W, Y} and {V, Z}, x-pass on {W, V} and {Y, Z}, one of the
//            four to a CTA (blockIdx.z); the stencil tile (2 fields x NC components with a
//            one-cell halo) is staged in shared memory.
//   xface2d  one CTA per SEG x-faces of a row, or of several rows where they are short or leave a
//            remainder (FaceSplit), and one Gauss point (or the corner row): the CTA evaluates the
//            y-pass polynomials of the columns it needs at eta_g into shared memory, then each
//            thread owns one face point (the Euler recursion: two threads): x-pass, leading term
//            (Eq. 3.6: HLLC, or the exact Burgers state), eigen-upwinded derivatives (Eq. 3.7),
//            Cauchy-Kovalevskaya (Section 3.1), Lobatto flux (Eq. 3.8) and W(t_{n+1})
//            (Eq. 3.11).  The corner row averages the y-pass traces of the rows below and above
//            and keeps only W(t_{n+1}).
//   yface2d  the same for y-faces along the columns.
//   update2d one thread per cell: Eq. (3.2) and Eq. (3.10), physical check, CFL rate; the last CTA
//            ends the step and begins the next.
// Every kernel is instantiated for NC = 1 (scalar Burgers) and NC = 4 (Euler), and for reading
// R1 (quartic p1) in step2d.cu and the R1' option (quintic p1) in step2d_quintic.cu, so the two
// translation units compile in parallel.
#pragma once
#include <cuda_runtime.h>

#include "shweno_kernels.h"
#include "step2d_items.cuh"

namespace shweno {

constexpr int TY = 8;        // tile height of coef2d and update2d
constexpr int TY_SMALL = 4;  // the same where the mesh has fewer tiles than the GPU has CTA slots: a
                             // tile's warps then share fewer schedulers' FP64 units, or none at all

template <int NC, bool Q, int TYK>
__global__ void __launch_bounds__(TX * TYK) coef2d_kernel(Params P, const Ctl* __restrict__ ctl,
                                                         const double* s0, const double* s1,
                                                         const uint8_t* __restrict__ flag,
                                                         double* __restrict__ ycoef,
                                                         double* __restrict__ xcoef) {
  __shared__ double tile[2 * NC][TYK + 2][TX + 2];
  if (!ctl->active) return;
  coef2d_item<NC, TYK, Q>(P, step_view(ctl), s0, s1, flag, ycoef, xcoef, blockIdx.z, blockIdx.x * TX - 2, blockIdx.y * TYK - 2, tile,
                  threadIdx.x, threadIdx.y);
}

template <int NC, bool FLAGS, bool CHAR, bool Q>
__global__ void __launch_bounds__(SEG, NC == 1 ? 3 : 2) xface2d_kernel(Params P, const Ctl* __restrict__ ctl,
                                                      const double* s0, const double* s1,
                                                      const double* __restrict__ ycoef,
                                                      const uint8_t* __restrict__ flag,
                                                      double* __restrict__ FX,
                                                      double* __restrict__ WX,
                                                      double* __restrict__ WC) {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  if (!ctl->active) return;
  const int slice = blockIdx.y;  // 0..2: Gauss point of the rows; 3: corner rows
  if (slice < 3 && (int)blockIdx.x >= FaceSplit(P.nx + 1).ctas(P.ny)) return;
  const StepView sv = step_view(ctl);
  xface_item<NC, FLAGS, CHAR, Q>(P, sv, sv.odd ? s1 : s0, ycoef, flag, FX, WX, WC, blockIdx.x, slice, dyn_smem);
}

template <int NC, bool FLAGS, bool CHAR, bool Q>
__global__ void __launch_bounds__(SEG, NC == 1 ? 3 : 2) yface2d_kernel(Params P, const Ctl* __restrict__ ctl,
                                                      const double* s0, const double* s1,
                                                      const double* __restrict__ xcoef,
                                                      const uint8_t* __restrict__ flag,
                                                      double* __restrict__ FY,
                                                      double* __restrict__ WY) {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  if (!ctl->active) return;
  const StepView sv = step_view(ctl);
  yface_item<NC, FLAGS, CHAR, Q>(P, sv, sv.odd ? s1 : s0, xcoef, flag, FY, WY, blockIdx.x, blockIdx.y, dyn_smem);
}

template <int NC>
__global__ void __launch_bounds__(256) update2d_kernel(Params P, Ctl* __restrict__ ctl,
                                                       const double* s0, const double* s1,
                                                       double* o0, double* o1,
                                                       const double* __restrict__ FX,
                                                       const double* __restrict__ WX,
                                                       const double* __restrict__ FY,
                                                       const double* __restrict__ WY,
                                                       const double* __restrict__ WC) {
  __shared__ double red[32];
  if (!ctl->active) return;
  const int i = blockIdx.x * TX + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
  const StepView sv = step_view(ctl);
  double rate = 0.0;
  if (i < P.nx && j < P.ny) rate = update2d_cell<NC>(P, ctl, sv, sv.odd ? s1 : s0, sv.odd ? o0 : o1, FX, WX, FY, WY, WC, i, j);
  block_max_rate(rate, &ctl->rate_next, red);  // holds a barrier: every cell's error has been raised
  if (threadIdx.x == 0 && threadIdx.y == 0) ctl_commit_last(ctl, gridDim.x * gridDim.y);
}

// ------------------------------------------------------------------ host side (templates)
// Dynamic shared memory limits of the face kernels; returns the first failing call's status.
template <int NC, bool CHAR, bool Q>
static cudaError_t init_kernels2d_nc() {
  cudaError_t e = cudaSuccess;
  auto set = [&e](const void* f, size_t bytes) {
    const cudaError_t r = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) e = r;
  };
  set((const void*)xface2d_kernel<NC, false, CHAR, Q>, face_smem<NC>());
  set((const void*)yface2d_kernel<NC, false, CHAR, Q>, face_smem<NC>());
  set((const void*)xface2d_kernel<NC, true, CHAR, Q>, face_smem<NC>());
  set((const void*)yface2d_kernel<NC, true, CHAR, Q>, face_smem<NC>());
  return e;
}

// Attributes of every face kernel of one reading (Q = false: R1, true: R1').
template <bool Q>
static cudaError_t init_kernels2d_reading() {
  cudaError_t e = init_kernels2d_nc<1, false, Q>();
  if (e == cudaSuccess) e = init_kernels2d_nc<4, false, Q>();
  if (e == cudaSuccess) e = init_kernels2d_nc<4, true, Q>();
  return e;
}


// The two face kernels of a step (x-faces with the corner rows, then y-faces).
template <int NC, bool CHAR, bool Q>
static void launch_faces2d(const Params& P, Ctl* ctl, const double* s0, const double* s1,
                           const uint8_t* flag, const Scratch2D& S, cudaStream_t st, cudaEvent_t* ev) {
  dim3 xg(FaceSplit(P.nx + 1).ctas(P.ny + 1), 4), yg(FaceSplit(P.ny + 1).ctas(P.nx), 3);
  // Both kernels read the first-pass tables and write arrays of their own.  Where one does not fill
  // the GPU (the handle then has a second stream) the y-faces go beside the x-faces: 40^2 cells, 112
  // and 101 us one after the other, about 115 together.
  const bool beside = !ev && S.aux;
  cudaStream_t sy = st;
  if (beside) {
    sy = S.aux;
    cudaEventRecord(S.fork, st);
    cudaStreamWaitEvent(sy, S.fork, 0);
  }
  if (P.flag_mode == FLAG_ALL_NONLINEAR)
    xface2d_kernel<NC, false, CHAR, Q><<<xg, SEG, face_smem<NC>(), st>>>(P, ctl, s0, s1, S.ycoef, flag, S.FX, S.WX, S.WC);
  else
    xface2d_kernel<NC, true, CHAR, Q><<<xg, SEG, face_smem<NC>(), st>>>(P, ctl, s0, s1, S.ycoef, flag, S.FX, S.WX, S.WC);
  if (ev) cudaEventRecord(ev[2], st);
  if (P.flag_mode == FLAG_ALL_NONLINEAR)
    yface2d_kernel<NC, false, CHAR, Q><<<yg, SEG, face_smem<NC>(), sy>>>(P, ctl, s0, s1, S.xcoef, flag, S.FY, S.WY);
  else
    yface2d_kernel<NC, true, CHAR, Q><<<yg, SEG, face_smem<NC>(), sy>>>(P, ctl, s0, s1, S.xcoef, flag, S.FY, S.WY);
  if (beside) {
    cudaEventRecord(S.join, sy);
    cudaStreamWaitEvent(st, S.join, 0);
  }
}

template <int NC, bool Q>
static void launch_step2d_nc(const Params& P, Ctl* ctl, const double* s0, const double* s1,
                             double* o0, double* o1, const uint8_t* flag, const Scratch2D& S,
                             cudaStream_t st, cudaEvent_t* ev) {
  // 40^2 cells: coef2d 38 -> 29 us, update2d 27 -> 21 us with the low tiles
  const bool small = ((P.nx + TX - 1) / TX) * ((P.ny + TY - 1) / TY) < 2 * kSMs;
  const int th = small ? TY_SMALL : TY;
  const dim3 cb(TX, th), cg((P.nx + 4 + TX - 1) / TX, (P.ny + 4 + th - 1) / th, 4);
  if (ev) cudaEventRecord(ev[0], st);
  if (small) coef2d_kernel<NC, Q, TY_SMALL><<<cg, cb, 0, st>>>(P, ctl, s0, s1, flag, S.ycoef, S.xcoef);
  else coef2d_kernel<NC, Q, TY><<<cg, cb, 0, st>>>(P, ctl, s0, s1, flag, S.ycoef, S.xcoef);
  if (ev) cudaEventRecord(ev[1], st);
  if constexpr (NC == 4) {
    if (P.charwise) launch_faces2d<NC, true, Q>(P, ctl, s0, s1, flag, S, st, ev);
    else launch_faces2d<NC, false, Q>(P, ctl, s0, s1, flag, S, st, ev);
  } else {
    launch_faces2d<NC, false, Q>(P, ctl, s0, s1, flag, S, st, ev);
  }
  if (ev) cudaEventRecord(ev[3], st);
  const int uh = small ? 2 : TY;
  const dim3 ub(TX, uh), ug((P.nx + TX - 1) / TX, (P.ny + uh - 1) / uh);
  update2d_kernel<NC><<<ug, ub, 0, st>>>(P, ctl, s0, s1, o0, o1, S.FX, S.WX, S.FY, S.WY, S.WC);
  if (ev) cudaEventRecord(ev[4], st);
}

// Both component counts of one reading.
template <bool Q>
static void launch_step2d_reading(const Params& P, Ctl* ctl, const double* s0, const double* s1,
                                  double* o0, double* o1, const uint8_t* flag, const Scratch2D& S,
                                  cudaStream_t st, cudaEvent_t* ev) {
  if (P.ncomp == 1) launch_step2d_nc<1, Q>(P, ctl, s0, s1, o0, o1, flag, S, st, ev);
  else launch_step2d_nc<4, Q>(P, ctl, s0, s1, o0, o1, flag, S, st, ev);
}

}  // namespace shweno
