// One ADER-SHWENO time step in one space dimension (Section 2; Section 4 Steps 1-5), one kernel:
// each warp advances W1D cells (step1d_items.cuh: SHWENO reconstruction of Section 2.4, leading
// term of Eq. 2.5, derivative problems of Eq. 2.8, Cauchy-Kovalevskaya of Eq. 2.6, Lobatto flux of
// Eq. 2.9 and Remark 2, the state at t_{n+1} of Eq. 2.12, updates of Eq. 2.2 and 2.11, physical
// check and CFL rate); the last CTA ends the step and begins the next.
#include <cuda_runtime.h>

#include "shweno_kernels.h"
#include "step1d_items.cuh"

namespace shweno {

template <int NC, bool Q>
__global__ void __launch_bounds__(128, 3) step1d_kernel(Params P, Ctl* __restrict__ ctl, const double* s0,
                                                     const double* s1, double* o0, double* o1,
                                                     const uint8_t* __restrict__ flag) {
  if (!ctl->active) return;
  const StepView sv = step_view(ctl);
  const int c0 = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * W1D;
  if (c0 < P.nx) {
    const double speed = step1d_warp<NC, Q>(P, ctl, sv.odd ? s1 : s0, sv.odd ? o0 : o1, flag, c0,
                                            min(W1D, P.nx - c0), sv.t, sv.dt);
    report_speed1d(P, ctl, speed);
  }
  __threadfence();  // each warp's report before the CTA counts as done
  __syncthreads();
  if (threadIdx.x == 0) ctl_commit_last(ctl, gridDim.x);
}

template <bool Q>
__global__ void __launch_bounds__(128) step1d_small_kernel(Params P, Ctl* __restrict__ ctl, const double* s0,
                                                           const double* s1, double* o0, double* o1,
                                                           const uint8_t* __restrict__ flag) {
  __shared__ Small1D S;
  if (!ctl->active) return;
  const StepView sv = step_view(ctl);
  const int c0 = blockIdx.x * W1D;
  const double speed = step1d_cta<Q>(P, ctl, sv.odd ? s1 : s0, sv.odd ? o0 : o1, flag, c0, min(W1D, P.nx - c0),
                                     sv.t, sv.dt, S);
  if (threadIdx.x >= 32) return;  // the first warp updated the cells
  report_speed1d(P, ctl, speed);
  __syncwarp();
  if (threadIdx.x == 0) ctl_commit_last(ctl, gridDim.x);
}

void launch_step1d(const Params& P, Ctl* ctl, const double* s0, const double* s1, double* o0,
                   double* o1, const uint8_t* flag, cudaStream_t st, cudaEvent_t* ev) {
  const int warps = (P.nx + W1D - 1) / W1D;
  if (ev) cudaEventRecord(ev[0], st);
  if (P.ncomp == 3 && !P.charwise && warps <= 2 * kSMs) {
    // Four warps for W1D cells: the latency of one chain of FP64 instructions is all there is, so it
    // is shortened.  Lax, 200 cells, whole run: 9.1 -> 5.6 ms against one warp per CTA.  The line is
    // two CTAs per SM, as many as its registers hold, in one wave (9120 cells).  Per step, one warp per
    // CTA / four: 4561 cells 40.3 / 33.9 us, 9120 cells 41.1 / 34.7, 18240 cells (a second wave)
    // 43.3 / 64.7.
    if (P.quintic) step1d_small_kernel<true><<<warps, 128, 0, st>>>(P, ctl, s0, s1, o0, o1, flag);
    else step1d_small_kernel<false><<<warps, 128, 0, st>>>(P, ctl, s0, s1, o0, o1, flag);
  } else {
    // One warp per CTA while the mesh does not fill the GPU: the CTAs then go to different SMs, each
    // warp has a scheduler's FP64 unit to itself.  From two warps per scheduler on, four:
    // three such CTAs per SM (4M cells: 13.9 ms with two, 12.0 with three).
    const int per = warps < 8 * kSMs ? 1 : 4;
    const dim3 g((warps + per - 1) / per), b(32 * per);
    if (P.ncomp == 1) {
      if (P.quintic) step1d_kernel<1, true><<<g, b, 0, st>>>(P, ctl, s0, s1, o0, o1, flag);
      else step1d_kernel<1, false><<<g, b, 0, st>>>(P, ctl, s0, s1, o0, o1, flag);
    } else {
      if (P.quintic) step1d_kernel<3, true><<<g, b, 0, st>>>(P, ctl, s0, s1, o0, o1, flag);
      else step1d_kernel<3, false><<<g, b, 0, st>>>(P, ctl, s0, s1, o0, o1, flag);
    }
  }
  if (ev) cudaEventRecord(ev[1], st);
}

}  // namespace shweno
