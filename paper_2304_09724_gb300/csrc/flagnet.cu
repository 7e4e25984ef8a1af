// Learned troubled-cell flag: a small MLP decides per cell whether the SHWENO reconstructions
// anchored on it need the nonlinear weights (flag 1) or may use the linear weights (flag 0),
// which makes them exactly the big-stencil polynomial p1 and skips the smoothness indicators.
// The paper has no such component; it is the learned layer put on top of the method.
//
//   features2d   22 inputs per cell from the committed state (FP64 arithmetic, stored FP32):
//                for rho and E, the eight 3x3 neighbours minus the centre and dx V, dy Y of the
//                centre, divided by (stencil range + 1e-12 |centre| + 1e-300), and
//                log10(range / (|centre| + 1e-30) + 1e-16) / 8.
//   wdev2d       label source: per cell, the largest relative deviation
//                max_l |w_l - gamma_l| / gamma_l of the 16 first-pass reconstructions anchored
//                on it (the plain scheme's own weights).
//   fdev2d       training label source: per cell, the largest change those weights make to the
//                reconstructions' end values, |p(+-1/2) - p1(+-1/2)|, relative to the range of the
//                reconstruction's three averages plus the caller's floor times |W0|.
//   mlp_forward / mlp_grad / mlp_adam   FP32 network 22 -> 32 -> 32 -> 1 (ReLU, ReLU, sigmoid),
//                binary cross-entropy with a positive-class weight, Adam.
//   infer2d + dilate2d   each step, before the reconstruction: flag = net(features) > threshold,
//                then dilated by one cell (3x3 OR), imposed-state ghost cells count as troubled.
#include <cuda_runtime.h>

#include "device_once.h"
#include "flagnet_items.cuh"
#include "shweno_kernels.h"

namespace shweno {

__global__ void features2d_kernel(Params P, const Ctl* __restrict__ ctl, const double* s0,
                                  const double* s1, float* __restrict__ out) {
  const size_t cells = (size_t)P.nx * P.ny;
  const size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cells) return;
  const double* st = (ctl->nsteps & 1) ? s1 : s0;
  float f[NIN];
  cell_features(P, st, (int)(c % P.nx), (int)(c / P.nx), ctl->t, f);
#pragma unroll
  for (int k = 0; k < NIN; ++k) out[c * NIN + k] = f[k];
}

__global__ void wdev2d_kernel(Params P, const Ctl* __restrict__ ctl, const double* s0,
                              const double* s1, double* __restrict__ out) {
  const size_t cells = (size_t)P.nx * P.ny;
  const size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cells) return;
  const double* st = (ctl->nsteps & 1) ? s1 : s0;
  const int i = (int)(c % P.nx), j = (int)(c / P.nx);
  const double t = ctl->t;
  double dev = 0.0;
  for (int pass = 0; pass < 2; ++pass)
    for (int set = 0; set < 2; ++set)
      for (int q = 0; q < P.ncomp; ++q) {
        const int fa = pass == 0 ? (set == 0 ? 0 : 1) : (set == 0 ? 0 : 2);
        const int fd = pass == 0 ? (set == 0 ? 2 : 3) : (set == 0 ? 1 : 3);
        const int di = pass == 1, dj = pass == 0;
        const double h = pass == 0 ? P.dy : P.dx;
        const double Wm = fetch(P, st, fa, q, i - di, j - dj, t), W0 = fetch(P, st, fa, q, i, j, t);
        const double Wp = fetch(P, st, fa, q, i + di, j + dj, t);
        double cf[5];
        p1_coeffs(Wm, W0, Wp, h * fetch(P, st, fd, q, i - di, j - dj, t), h * fetch(P, st, fd, q, i + di, j + dj, t), cf);
        const Mix m = shweno_mix(P, Wm, W0, Wp, cf, 1);
        // back from (A, B, C) to the weights: w1 = A g1, w2 = B + A g2, w3 = C + A g3
        const double w[3] = {m.A * P.gam[0], m.B + m.A * P.gam[1], m.C + m.A * P.gam[2]};
        for (int l = 0; l < 3; ++l) dev = fmax(dev, fabs(w[l] - P.gam[l]) / P.gam[l]);
      }
  out[c] = dev;
}

__global__ void fdev2d_kernel(Params P, const Ctl* __restrict__ ctl, const double* s0,
                              const double* s1, double floor_rel, double* __restrict__ out) {
  const size_t cells = (size_t)P.nx * P.ny;
  const size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cells) return;
  const double* st = (ctl->nsteps & 1) ? s1 : s0;
  const int i = (int)(c % P.nx), j = (int)(c / P.nx);
  const double t = ctl->t;
  double dev = 0.0;
  for (int pass = 0; pass < 2; ++pass)
    for (int set = 0; set < 2; ++set)
      for (int q = 0; q < P.ncomp; ++q) {
        const int fa = pass == 0 ? (set == 0 ? 0 : 1) : (set == 0 ? 0 : 2);
        const int fd = pass == 0 ? (set == 0 ? 2 : 3) : (set == 0 ? 1 : 3);
        const int di = pass == 1, dj = pass == 0;
        const double h = pass == 0 ? P.dy : P.dx;
        const double Wm = fetch(P, st, fa, q, i - di, j - dj, t), W0 = fetch(P, st, fa, q, i, j, t);
        const double Wp = fetch(P, st, fa, q, i + di, j + dj, t);
        double cf[5];
        p1_coeffs(Wm, W0, Wp, h * fetch(P, st, fd, q, i - di, j - dj, t), h * fetch(P, st, fd, q, i + di, j + dj, t), cf);
        const Mix m = shweno_mix(P, Wm, W0, Wp, cf, 1);
        // p - p1 = (A - 1) p1 + B p2 + C p3 at xi = +-1/2 (p2 = W0 + (W0 - W-) xi, p3 = W0 + (W+ - W0) xi)
        const double even = cf[0] + 0.25 * cf[2] + 0.0625 * cf[4], odd = 0.5 * cf[1] + 0.125 * cf[3];
        const double s2 = 0.5 * (W0 - Wm), s3 = 0.5 * (Wp - W0);
        const double scale = fmax(Wm, fmax(W0, Wp)) - fmin(Wm, fmin(W0, Wp)) + floor_rel * fabs(W0) + 1e-300;
        const double dR = (m.A - 1.0) * (even + odd) + m.B * (W0 + s2) + m.C * (W0 + s3);
        const double dL = (m.A - 1.0) * (even - odd) + m.B * (W0 - s2) + m.C * (W0 - s3);
        dev = fmax(dev, fmax(fabs(dR), fabs(dL)) / scale);
      }
  out[c] = dev;
}

__global__ void mlp_forward_kernel(const float* __restrict__ params, const float* __restrict__ X,
                                   int64_t n, float* __restrict__ prob) {
  __shared__ float p[NPARAM];
  load_params(params, p);
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= n) return;
  float x[NIN];
#pragma unroll
  for (int j = 0; j < NIN; ++j) x[j] = X[b * NIN + j];
  prob[b] = 1.f / (1.f + expf(-net_logit(p, x)));
}

// Gradient of mean BCE over n samples.  A CTA handles GB samples: each thread runs forward and
// backward for one sample, keeping its activations and their gradients transposed in shared memory
// ([unit][sample], rows padded by four words so that neither the threads' stores nor the 16-byte
// reads of the sums collide), then the CTA sums every parameter's gradient over its samples, eight
// parameters of a column to a thread, and adds it to grad with one atomicAdd per parameter.  The
// weights are read 16 bytes at a time (the first layer's rows padded from 22 to 24).  Bound by the
// chain of one warp per scheduler: about 2800 multiply-adds forward and backward, 2300 in the sums;
// one training step of 16384 samples: 40.5 -> 27.7 us (rows of 32 floats put all 32 lanes' stores on one bank before, and
// every multiply-add of the sums read both factors).
constexpr int GB = 128;
constexpr int GROW = GB + 4;
constexpr int NINP = 24;
struct __align__(16) GradSmem {
  float w1[NH][NINP], w2[NH][NH], b1[NH], b2[NH], w3[NH], b3;
  float pad[3];
  float x[NIN][GROW], h1[NH][GROW], h2[NH][GROW], d1[NH][GROW], d2[NH][GROW], d3[GROW];
  float red[GB / 32];
};

__global__ void mlp_zero_kernel(float* __restrict__ grad, float* __restrict__ loss) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < NPARAM) grad[k] = 0.f;
  if (k == NPARAM) *loss = 0.f;
}

// s[0..7] = sum over the samples of d[i0 + u] * y
__device__ __forceinline__ void grad_sums(const float (*d)[GROW], const float* y, int i0, float s[8]) {
#pragma unroll
  for (int u = 0; u < 8; ++u) s[u] = 0.f;
#pragma unroll 4
  for (int b = 0; b < GB; b += 4) {
    const float4 v = *reinterpret_cast<const float4*>(y + b);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const float4 w = *reinterpret_cast<const float4*>(&d[i0 + u][b]);
      s[u] = fmaf(w.x, v.x, s[u]);
      s[u] = fmaf(w.y, v.y, s[u]);
      s[u] = fmaf(w.z, v.z, s[u]);
      s[u] = fmaf(w.w, v.w, s[u]);
    }
  }
}

__global__ void __launch_bounds__(GB) mlp_grad_kernel(const float* __restrict__ params,
                                                      const float* __restrict__ X,
                                                      const float* __restrict__ y, int64_t n,
                                                      float pw, float* __restrict__ grad,
                                                      float* __restrict__ loss) {
  extern __shared__ __align__(16) unsigned char raw[];
  GradSmem& S = *reinterpret_cast<GradSmem*>(raw);
  const int tid = threadIdx.x;
  for (int k = tid; k < NPARAM; k += GB) {
    const float v = params[k];
    if (k < OFF_B1) S.w1[k / NIN][k % NIN] = v;
    else if (k < OFF_W2) S.b1[k - OFF_B1] = v;
    else if (k < OFF_B2) (&S.w2[0][0])[k - OFF_W2] = v;
    else if (k < OFF_W3) S.b2[k - OFF_B2] = v;
    else if (k < OFF_B3) S.w3[k - OFF_W3] = v;
    else S.b3 = v;
  }
  if (tid < NH) S.w1[tid][NIN] = S.w1[tid][NIN + 1] = 0.f;
  const int64_t b0 = (int64_t)blockIdx.x * GB;
  const int64_t b = b0 + tid;
  // the CTA's samples lie one after the other
  const int cnt = (int)(n - b0 < GB ? n - b0 : GB);
  for (int k = tid; k < GB * NIN; k += GB) S.x[k % NIN][k / NIN] = k < cnt * NIN ? X[b0 * NIN + k] : 0.f;
  __syncthreads();
  float l = 0.f;
  if (b < n) {
    float x[NINP], h1[NH];
#pragma unroll
    for (int j = 0; j < NINP; ++j) x[j] = j < NIN ? S.x[j][tid] : 0.f;
#pragma unroll 4
    for (int i = 0; i < NH; ++i) {
      float z = S.b1[i];
#pragma unroll
      for (int j = 0; j < NINP; j += 4) {
        const float4 w = *reinterpret_cast<const float4*>(&S.w1[i][j]);
        z = fmaf(w.x, x[j], z);
        z = fmaf(w.y, x[j + 1], z);
        if (j + 2 < NIN) {
          z = fmaf(w.z, x[j + 2], z);
          z = fmaf(w.w, x[j + 3], z);
        }
      }
      S.h1[i][tid] = fmaxf(z, 0.f);
    }
#pragma unroll
    for (int j = 0; j < NH; ++j) h1[j] = S.h1[j][tid];
    float z3 = S.b3;
    unsigned on2 = 0;  // units of the second layer that pass
#pragma unroll 4
    for (int i = 0; i < NH; ++i) {
      float z = S.b2[i];
#pragma unroll
      for (int j = 0; j < NH; j += 4) {
        const float4 w = *reinterpret_cast<const float4*>(&S.w2[i][j]);
        z = fmaf(w.x, h1[j], z);
        z = fmaf(w.y, h1[j + 1], z);
        z = fmaf(w.z, h1[j + 2], z);
        z = fmaf(w.w, h1[j + 3], z);
      }
      on2 |= z > 0.f ? 1u << i : 0u;
      S.h2[i][tid] = fmaxf(z, 0.f);
      z3 = fmaf(S.w3[i], fmaxf(z, 0.f), z3);
    }
    const float yy = y[b];
    const float sg = 1.f / (1.f + expf(-z3));
    // per-sample loss, stable: -pw y log(sig) - (1 - y) log(1 - sig)
    const float sp_neg = log1pf(expf(-fabsf(z3))) + fmaxf(-z3, 0.f);  // -log(sig(z))
    const float sp_pos = sp_neg + z3;                                    // -log(1 - sig(z))
    l = pw * yy * sp_neg + (1.f - yy) * sp_pos;
    const float d3 = (-pw * yy * (1.f - sg) + (1.f - yy) * sg) / (float)n;
    S.d3[tid] = d3;
    float s[NH];
#pragma unroll
    for (int j = 0; j < NH; ++j) s[j] = 0.f;
#pragma unroll 4
    for (int i = 0; i < NH; ++i) {
      const float d2 = S.d2[i][tid] = on2 >> i & 1u ? d3 * S.w3[i] : 0.f;
#pragma unroll
      for (int j = 0; j < NH; j += 4) {
        const float4 w = *reinterpret_cast<const float4*>(&S.w2[i][j]);
        s[j] = fmaf(w.x, d2, s[j]);
        s[j + 1] = fmaf(w.y, d2, s[j + 1]);
        s[j + 2] = fmaf(w.z, d2, s[j + 2]);
        s[j + 3] = fmaf(w.w, d2, s[j + 3]);
      }
    }
#pragma unroll
    for (int j = 0; j < NH; ++j) S.d1[j][tid] = h1[j] > 0.f ? s[j] : 0.f;
  } else {
    for (int i = 0; i < NH; ++i) S.h1[i][tid] = S.h2[i][tid] = S.d1[i][tid] = S.d2[i][tid] = 0.f;
    S.d3[tid] = 0.f;
  }
  // loss: block sum, one atomic per CTA
  for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  if ((tid & 31) == 0) S.red[tid >> 5] = l;
  __syncthreads();
  if (tid == 0) {
    float s = 0.f;
    for (int w = 0; w < GB / 32; ++w) s += S.red[w];
    atomicAdd(loss, s / (float)n);
  }
  // parameter gradients: sums over the CTA's samples, warp w the rows 8 w .. 8 w + 7 of both layers
  const int lane = tid & 31, i0 = (tid >> 5) * 8;
  float s[8];
  grad_sums(S.d2, S.h1[lane], i0, s);
#pragma unroll
  for (int u = 0; u < 8; ++u) atomicAdd(&grad[OFF_W2 + (i0 + u) * NH + lane], s[u]);
  if (lane < NIN) {
    grad_sums(S.d1, S.x[lane], i0, s);
#pragma unroll
    for (int u = 0; u < 8; ++u) atomicAdd(&grad[OFF_W1 + (i0 + u) * NIN + lane], s[u]);
  } else if (lane < NIN + 8) {  // the biases of the warp's rows
    float t1 = 0.f, t2 = 0.f, t3 = 0.f;
    const int i = i0 + lane - NIN;
    for (int bb = 0; bb < GB; ++bb) {
      t1 += S.d1[i][bb];
      t2 += S.d2[i][bb];
      t3 = fmaf(S.d3[bb], S.h2[i][bb], t3);
    }
    atomicAdd(&grad[OFF_B1 + i], t1);
    atomicAdd(&grad[OFF_B2 + i], t2);
    atomicAdd(&grad[OFF_W3 + i], t3);
  } else if (tid == NIN + 8) {
    float t = 0.f;
    for (int bb = 0; bb < GB; ++bb) t += S.d3[bb];
    atomicAdd(&grad[OFF_B3], t);
  }
}

__global__ void mlp_adam_kernel(float* __restrict__ params, const float* __restrict__ grad,
                                float* __restrict__ m, float* __restrict__ v, float lr, float b1,
                                float b2, float eps, float bc1, float bc2) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= NPARAM) return;
  const float g = grad[k];
  const float mk = b1 * m[k] + (1.f - b1) * g;
  const float vk = b2 * v[k] + (1.f - b2) * g * g;
  m[k] = mk;
  v[k] = vk;
  params[k] -= lr * (mk / bc1) / (sqrtf(vk / bc2) + eps);
}

// ------------------------------------------------------------------ per-step inference
__global__ void infer2d_kernel(Params P, const Ctl* __restrict__ ctl, const double* s0,
                               const double* s1, const float* __restrict__ params, float logit_thr,
                               uint8_t* __restrict__ raw) {
  __shared__ float p[NPARAM];
  if (!ctl->active) return;
  load_params(params, p);
  const size_t cells = (size_t)P.nx * P.ny;
  const size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cells) return;
  const double* st = (ctl->nsteps & 1) ? s1 : s0;
  float f[NIN];
  cell_features(P, st, (int)(c % P.nx), (int)(c / P.nx), ctl->t, f);
  raw[c] = net_logit(p, f) > logit_thr ? 1 : 0;
}

__global__ void dilate2d_kernel(Params P, const Ctl* __restrict__ ctl, const uint8_t* __restrict__ raw,
                                uint8_t* __restrict__ flags) {
  if (!ctl->active) return;
  const size_t cells = (size_t)P.nx * P.ny;
  const size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cells) return;
  const int i = (int)(c % P.nx), j = (int)(c / P.nx);
  int f = 0;
  for (int dj = -1; dj <= 1; ++dj)
    for (int di = -1; di <= 1; ++di) f |= raw_flag(P, raw, i + di, j + dj);
  flags[c] = (uint8_t)f;
}

// ------------------------------------------------------------------ host launchers
void launch_features2d(const Params& P, const Ctl* ctl, const double* s0, const double* s1,
                       float* out, cudaStream_t st) {
  const size_t cells = (size_t)P.nx * P.ny;
  features2d_kernel<<<(unsigned)((cells + 127) / 128), 128, 0, st>>>(P, ctl, s0, s1, out);
}
void launch_fdev2d(const Params& P, const Ctl* ctl, const double* s0, const double* s1,
                   double floor_rel, double* out, cudaStream_t st) {
  const size_t cells = (size_t)P.nx * P.ny;
  fdev2d_kernel<<<(unsigned)((cells + 127) / 128), 128, 0, st>>>(P, ctl, s0, s1, floor_rel, out);
}

void launch_wdev2d(const Params& P, const Ctl* ctl, const double* s0, const double* s1,
                   double* out, cudaStream_t st) {
  const size_t cells = (size_t)P.nx * P.ny;
  wdev2d_kernel<<<(unsigned)((cells + 127) / 128), 128, 0, st>>>(P, ctl, s0, s1, out);
}
void launch_infer2d(const Params& P, const Ctl* ctl, const double* s0, const double* s1,
                    const float* params, float logit_thr, uint8_t* raw, uint8_t* flags,
                    cudaStream_t st) {
  const size_t cells = (size_t)P.nx * P.ny;
  const unsigned g = (unsigned)((cells + 255) / 256);
  infer2d_kernel<<<g, 256, 0, st>>>(P, ctl, s0, s1, params, logit_thr, raw);
  dilate2d_kernel<<<g, 256, 0, st>>>(P, ctl, raw, flags);
}
void mlp_forward(const float* params, const float* X, int64_t n, float* prob, cudaStream_t st) {
  if (n > 0) mlp_forward_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(params, X, n, prob);
}
cudaError_t mlp_grad(const float* params, const float* X, const float* y, int64_t n, float pw,
                     float* grad, float* loss, cudaStream_t st) {
  static DeviceOnce limit;  // the kernel's shared-memory limit belongs to the device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (limit.needed(dev)) {
    e = cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradSmem));
    if (e != cudaSuccess) return e;
    limit.done(dev);
  }
  mlp_zero_kernel<<<(NPARAM + 256) / 256, 256, 0, st>>>(grad, loss);
  if (n > 0)
    mlp_grad_kernel<<<(unsigned)((n + GB - 1) / GB), GB, sizeof(GradSmem), st>>>(params, X, y, n, pw, grad, loss);
  return cudaGetLastError();
}
void mlp_adam(float* params, const float* grad, float* m, float* v, float lr, float b1, float b2,
              float eps, float bc1, float bc2, cudaStream_t st) {
  mlp_adam_kernel<<<(NPARAM + 255) / 256, 256, 0, st>>>(params, grad, m, v, lr, b1, b2, eps, bc1, bc2);
}

}  // namespace shweno
