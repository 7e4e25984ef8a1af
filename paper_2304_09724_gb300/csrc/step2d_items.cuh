// Per-item device functions of the 2D step, shared by the one-mesh kernels (step2d.cu) and the
// batched persistent kernel (batch.cu).  See step2d.cu for the structure of the step.
#pragma once
#include "shweno_device.cuh"

namespace shweno {

constexpr int SEG = 128;          // threads of a face CTA
constexpr int NFACE = SEG - 1;    // most faces of a face CTA: its threads own the SEG cells next to them
constexpr int SPAN = 144;         // first-pass evaluations a CTA has room for
constexpr int TX = 32;            // first-pass tile width

// ------------------------------------------------------------------ the faces of a CTA
// A line of n faces is cut into segments of NFACE faces, one CTA each; what remains of the lines
// (rem faces each) goes together, per lines to a CTA, so that short lines and ragged ends fill
// their warps too (an FP64 instruction costs a warp the same for one lane as for 32; 401 faces:
// 3 segments and 20 faces that had a CTA and two CTA slots' worth of waiting to themselves).
// A CTA's faces are runs of nf faces on nrun neighbouring lines; thread t owns the cell
// t % (nf + 1) of run t / (nf + 1) and, but for the last cell of a run, the face right of it.
struct FaceSplit {
  int nfull, rem, per;
  __host__ __device__ explicit FaceSplit(int n) : nfull(n / NFACE), rem(n % NFACE), per(1) {
    if (rem > 0) per = SEG / (rem + 1) < SPAN / (rem + 3) ? SEG / (rem + 1) : SPAN / (rem + 3);
  }
  __host__ __device__ int ctas(int lines) const { return nfull * lines + (rem > 0 ? (lines + per - 1) / per : 0); }
};
struct FaceRuns {
  int f0, nf, line, nrun;  // first face, faces per run, first line, runs
  int run, ct, col;        // this thread's run, cell in it and stencil column (run * (nf + 3) + ct + 1)
  bool has_cell, has_face;
  __device__ __forceinline__ FaceRuns(int n, int lines, int b) {
    const FaceSplit S(n);
    if (b < S.nfull * lines) {
      line = b / S.nfull; f0 = (b % S.nfull) * NFACE; nf = NFACE; nrun = 1;
    } else {
      line = (b - S.nfull * lines) * S.per; f0 = S.nfull * NFACE; nf = S.rem; nrun = min(S.per, lines - line);
    }
    run = threadIdx.x / (nf + 1);
    ct = threadIdx.x % (nf + 1);
    col = run * (nf + 3) + ct + 1;
    has_cell = run < nrun;
    has_face = has_cell && ct < nf;
  }
};

// ------------------------------------------------------------------ second pass, cell by cell
// Second pass across the face.  ev[set*NC+q][k][col] holds the first-pass Taylor coefficients
// (order k along the face) of a row of stencil columns; column c holds the cell whose stencil is
// columns c-1..c+1.  Each cell's weights come from its order-0 data and serve every order
// (remark ending Section 2.1.2) and both of the cell's ends, so one thread per cell forms its
// weights once and then, order by order, the Taylor coefficients across the face at both ends
// (EndTable); one thread per face then reads the left cell's right end and the right cell's left
// end.  The two ends of a cell share their arithmetic: with s = W- + W+, a = W+ - W-,
// dv = v+ - v-, sv = v- + v+, p1's coefficient p at xi = +-1/2 is U_p + V_p and (-1)^p (U_p - V_p)
// (U_p from the even monomials, V_p from the odd ones; end_u / end_v of recon_tables.cuh).
template <int NC>
struct EndTable {
  // left ends (xi = -1/2) of the cells, two buffers (orders of even / odd K) so that one barrier
  // per order suffices: [buffer][comp][p][slot], the cell of thread t at slot t
  double L[2][NC][5][SEG];
};
// Flags of the cells next to the faces, for the characteristic-wise path (whose weights belong to
// each face point): lin[c] = 1 when the cell in column c uses the linear weights.
struct FlagTable {
  int lin[SPAN];
};

template <int NC>
constexpr size_t ev_bytes() { return sizeof(double) * 2 * NC * 5 * SPAN; }
template <int NC>
constexpr size_t table_bytes() {
  return ev_bytes<NC>() + (sizeof(EndTable<NC>) > sizeof(FlagTable) ? sizeof(EndTable<NC>) : sizeof(FlagTable));
}

// Weights of one cell's reconstruction across the face: p = A p1 + B p2 + C p3 per component.
template <int NC>
struct CellMix {
  double A[NC], B[NC], C[NC];
  bool lin;  // linear weights: p = p1 (A = 1, B = C = 0)
};

template <int NC, bool Q>
__device__ __forceinline__ void cell_mix(const Params& P, const double (*ev)[5][SPAN], int c, bool lin,
                                         CellMix<NC>& m) {
  m.lin = lin;
  if (lin) {  // one branch for the whole cell: a warp of linear cells skips the weights
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      m.A[q] = 1.0;
      m.B[q] = m.C[q] = 0.0;
    }
    return;
  }
  if constexpr (NC == 4 && !Q) {
    // the four components' weights normalised in pairs: 1/S0 = S1 / (S0 S1), 1/S1 = S0 / (S0 S1)
    // (two divisions instead of four; the sums are products of smoothness indicators, far from
    // the range where their product could overflow)
    RawWeights rw[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      const double Wm = ev[q][0][c - 1], W0 = ev[q][0][c], Wp = ev[q][0][c + 1];
      double cf[6];
      p1_coeffs_t<Q>(Wm, W0, Wp, ev[NC + q][0][c - 1], ev[NC + q][0][c], ev[NC + q][0][c + 1], cf);
      rw[q] = shweno_raw_weights(P, Wm, W0, Wp, cf);
    }
#pragma unroll
    for (int h = 0; h < NC; h += 2) {
      const double r = 1.0 / (rw[h].sum * rw[h + 1].sum);
      const Mix m0 = mix_from_raw(P, rw[h], r * rw[h + 1].sum), m1 = mix_from_raw(P, rw[h + 1], r * rw[h].sum);
      m.A[h] = m0.A; m.B[h] = m0.B; m.C[h] = m0.C;
      m.A[h + 1] = m1.A; m.B[h + 1] = m1.B; m.C[h + 1] = m1.C;
    }
  } else {
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      const double Wm = ev[q][0][c - 1], W0 = ev[q][0][c], Wp = ev[q][0][c + 1];
      double cf[6];
      p1_coeffs_t<Q>(Wm, W0, Wp, ev[NC + q][0][c - 1], ev[NC + q][0][c], ev[NC + q][0][c + 1], cf);
      const Mix mm = shweno_mix_t<Q>(P, Wm, W0, Wp, cf, 1);
      m.A[q] = mm.A;
      m.B[q] = mm.B;
      m.C[q] = mm.C;
    }
  }
}

// Taylor coefficients p = 0..4-K across the face of tangential order K at both ends of the cell in
// column c, into the thread's slot of the EndTable.  The small stencils p2 = W0 + (W0 - W-) xi and
// p3 = W0 + (W+ - W0) xi add h +- g/2 to the value and g to the slope at the ends, with
// h = (B + C) W0 and g = B (W0 - W-) + C (W+ - W0).  LIN: a cell with the linear weights (p = p1,
// A = 1, B = C = 0; the general form gives the same values bit for bit with more operations).
template <int NC, bool LIN, bool Q, int K>
__device__ __forceinline__ void cell_ends_t(const double (*ev)[5][SPAN], int c, const CellMix<NC>& m,
                                            EndTable<NC>& et, double eRo[NC][5]) {
  using namespace shweno_tables;
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    const double Wm = ev[q][K][c - 1], W0 = ev[q][K][c], Wp = ev[q][K][c + 1];
    const double vm = ev[NC + q][K][c - 1], vp = ev[NC + q][K][c + 1];
    const double v0 = Q ? ev[NC + q][K][c] : 0.0;
    const double s = Wm + Wp, a = Wp - Wm, dv = vp - vm, sv = vm + vp;
    const double A = m.A[q];
    double g = 0.0, hR = 0.0, hL = 0.0;
    if (!LIN) {
      g = m.B[q] * (W0 - Wm) + m.C[q] * (Wp - W0);
      const double h = (m.B[q] + m.C[q]) * W0;
      hR = fma(0.5, g, h);
      hL = fma(-0.5, g, h);
    }
#pragma unroll
    for (int p = 0; p + K <= 4; ++p) {
      const double U = end_u(p, W0, s, dv);
      double eR, eL;
      if (!Q && p == 4) {  // V_4 = 0 for the quartic: both ends are U_4
        eR = eL = LIN ? U : A * U;
      } else {
        const double V = Q ? qend_v(p, a, sv, v0) : end_v(p, a, sv);
        if (LIN) {
          eR = U + V;
          eL = (p & 1) ? V - U : U - V;
        } else if (p == 0) {
          eR = fma(A, V, fma(A, U, hR));
          eL = fma(-A, V, fma(A, U, hL));
        } else if (p == 1) {
          eR = fma(A, V, fma(A, U, g));
          eL = fma(A, V, fma(-A, U, g));
        } else {
          const double AU = A * U;
          eR = fma(A, V, AU);
          eL = (p & 1) ? fma(A, V, -AU) : fma(-A, V, AU);
        }
      }
      eRo[q][p] = eR;
      et.L[K & 1][q][p][threadIdx.x] = eL;
    }
  }
}
// FLAGS = false: every cell is nonlinear (no branch on the flag); otherwise one branch per cell.
template <int NC, bool FLAGS, bool Q, int K>
__device__ __forceinline__ void cell_ends(const double (*ev)[5][SPAN], int c, const CellMix<NC>& m,
                                          EndTable<NC>& et, double eR[NC][5]) {
  if (FLAGS && m.lin) cell_ends_t<NC, true, Q, K>(ev, c, m, et, eR);
  else cell_ends_t<NC, false, Q, K>(ev, c, m, et, eR);
}

// Order K of the face point of thread f (its cell and thread f + 1's): the two sides from the
// EndTable; at K = 0 the leading term (Burgers: exact Godunov state; Euler: HLLC) and the
// eigen-decomposition of the upwinding; every derivative vector upwinded into a[q][m*5+n]
// (m along x, n along y; dir = 0: x-face, p across = m; dir = 1: y-face, p across = n).
template <int NC, int K>
__device__ __forceinline__ void face_order(const Params& P, const EndTable<NC>& et, const double eR[NC][5], int f,
                                           int dir, double Ws[NC], Upwinder<NC>& U, double a[NC][25]) {
  double dr[NC][5];
#pragma unroll
  for (int q = 0; q < NC; ++q)
#pragma unroll
    for (int p = 0; p + K <= 4; ++p) dr[q][p] = et.L[K & 1][q][p][f + 1];
  if constexpr (K == 0) {
    double WL[NC], WR[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) { WL[q] = eR[q][0]; WR[q] = dr[q][0]; }
    if constexpr (NC == 1) Ws[0] = burgers_godunov(WL[0], WR[0]);  // the same flux u^2/2 along x and y
    else hllc_state<NC>(WL, WR, P.gamma, dir, Ws);
    U.setup(Ws, P.gamma, dir, NC == 1 ? fmax(fabs(WL[0]), fabs(WR[0])) : 0.0);
  }
#pragma unroll
  for (int p = 0; p + K <= 4; ++p) {
    if (p == 0 && K == 0) continue;
    double x[NC], y[NC], o[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) { x[q] = eR[q][p]; y[q] = dr[q][p]; }
    U.apply(x, y, o);
    const int idx = dir == 0 ? p * 5 + K : K * 5 + p;
#pragma unroll
    for (int q = 0; q < NC; ++q) a[q][idx] = o[q];
  }
}

// One order of the two-phase second pass: every cell thread keeps its right ends and publishes its
// left ends (buffer K & 1), one barrier, then every face thread upwinds its own cell's right end
// against the next cell's left end.  The next order writes the other buffer, so a thread still
// reading this one cannot be overtaken.  Called by all threads of the CTA (it holds the barrier).
template <int NC, bool FLAGS, bool Q, int K>
__device__ __forceinline__ void pass_order(const Params& P, const double (*ev)[5][SPAN], EndTable<NC>& et,
                                           const FaceRuns& fr, const CellMix<NC>& m,
                                           int dir, double Ws[NC], Upwinder<NC>& U, double a[NC][25]) {
  double eR[NC][5];
  if (fr.has_cell) cell_ends<NC, FLAGS, Q, K>(ev, fr.col, m, et, eR);
  __syncthreads();
  if (fr.has_face) face_order<NC, K>(P, et, eR, threadIdx.x, dir, Ws, U, a);
}

// ------------------------------------------------------------------ Cauchy-Kovalevskaya of the points
// The points of a CTA go through the recursion in fixed point (ck_fixed.cuh) on the integer pipe.
// Euler: the owner of a point converts its 60 coefficients into shared memory (in the place of the
// first- and second-pass tables, which no thread reads any more), then each warp takes 16 points
// at a time, two lanes a point (ck_euler2d_lane: one lane per direction, 16 lanes apart, so that a
// half-warp reads 128 consecutive bytes), and the owner converts the results back.  One thread
// cannot hold the recursion's series in registers beside its accumulators (10 KB of spills);
// split over two lanes and shared memory it needs about 5500 instructions a lane and no spills.
// In FP64 (ck_points64) one thread does hold it.
constexpr int CKP = 64;               // points in work at a time
constexpr int kCkRow = CKP * 8;       // bytes of one coefficient of them
constexpr int kCkIn = 0;              // [2 halves][4 comps][15] level 0 (in the end: the results)
constexpr int kCkLev = kCkIn + 2 * 60 * kCkRow;  // [rho, m, n, H][10 + 6 + 3] levels 1..3
constexpr int kCkH0 = kCkLev + 4 * 19 * kCkRow;  // [15] H, level 0
constexpr int kCkE = kCkH0 + 15 * kCkRow;        // [10] E of the level in work, 64-bit
constexpr int kCkNinv = kCkE + 10 * kCkRow;      // [SEG] -1/rho0
constexpr int kCkGrow = kCkNinv + SEG * 8;       // [SEG] growth added on the way
constexpr size_t kCkBytes = kCkGrow + SEG * 4;
constexpr int kCkLost = 1 << 20;                 // growth of a point whose values never fitted: its result is NaN

template <int NC>
constexpr size_t face_smem() {
  return NC == 4 && kCkBytes > table_bytes<NC>() ? kCkBytes : table_bytes<NC>();
}

__host__ __device__ constexpr int ck_pair(int i, int j) { return (i + j) * (i + j + 1) / 2 + j; }
__host__ __device__ constexpr int ck_level_row(int t) { return t == 1 ? 0 : t == 2 ? 10 : 16; }

__device__ __forceinline__ Fx ck_ld(int at) {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  const int2 v = *reinterpret_cast<const int2*>(dyn_smem + at);
  return Fx{v.x, v.y};
}
__device__ __forceinline__ int64_t ck_ld64(int at) {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  return *reinterpret_cast<const long long*>(dyn_smem + at);
}
__device__ __forceinline__ void ck_st64(int at, int64_t v) {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  *reinterpret_cast<long long*>(dyn_smem + at) = v;
}
__device__ __forceinline__ void ck_st(int at, Fx v) {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  *reinterpret_cast<int2*>(dyn_smem + at) = make_int2(v.h, v.l);
}

// A lane's view of its point's series in shared memory, in the lane's own coordinates.
struct CkLane {
  int off[15];                    // row offset of the coefficient (i, j) of the lane's directions
  int in, lev, h0, e0;            // the point's column in the four areas
  int mom0, oth0, momL, othL;     // the lane's momentum and the other one, level 0 and above
  int dir;
  int64_t mom_out[4], both_out[4];  // results: the lane's momentum; density (x) or energy (y)
  __device__ __forceinline__ CkLane(int half, int pt, int d) : dir(d) {
#pragma unroll
    for (int s = 0; s < 5; ++s)
#pragma unroll
      for (int j = 0; j <= s; ++j) off[ck_pair(s - j, j)] = (dir ? ck_pair(j, s - j) : ck_pair(s - j, j)) * kCkRow;
    in = kCkIn + half * 60 * kCkRow + pt * 8;
    lev = kCkLev + pt * 8;
    h0 = kCkH0 + pt * 8;
    e0 = kCkE + pt * 8;
    mom0 = in + (1 + dir) * 15 * kCkRow;
    oth0 = in + (2 - dir) * 15 * kCkRow;
    momL = lev + (1 + dir) * 19 * kCkRow;
    othL = lev + (2 - dir) * 19 * kCkRow;
  }
  __device__ __forceinline__ int at(int base0, int baseL, int t, int i, int j) const {
    return (t == 0 ? base0 : baseL + ck_level_row(t) * kCkRow) + off[ck_pair(i, j)];
  }
  __device__ __forceinline__ Fx ldrho(int t, int i, int j) const { return ck_ld(at(in, lev, t, i, j)); }
  __device__ __forceinline__ Fx ldmom(int t, int i, int j) const { return ck_ld(at(mom0, momL, t, i, j)); }
  __device__ __forceinline__ Fx ldoth(int t, int i, int j) const { return ck_ld(at(oth0, othL, t, i, j)); }
  __device__ __forceinline__ Fx ldH(int t, int i, int j) const { return ck_ld(at(h0, lev + 57 * kCkRow, t, i, j)); }
  // the other momentum (s = 0) or H (s = 1)
  __device__ __forceinline__ Fx ldser(int s, int t, int i, int j) const {
    return ck_ld(at(s ? h0 : oth0, s ? lev + 57 * kCkRow : othL, t, i, j));
  }
  // the lane's part of the other momentum's coefficient (i, j) of slice n, and the other lane's part
  // of its own
  __device__ __forceinline__ void stoth(int n, int i, int j, int64_t z) const {
    ck_st64(othL + ck_level_row(n) * kCkRow + off[ck_pair(i, j)], z);
  }
  __device__ __forceinline__ int64_t ldown(int n, int i, int j) const {
    return ck_ld64(momL + ck_level_row(n) * kCkRow + off[ck_pair(i, j)]);
  }
  // both lanes of a point compute and write the same H
  __device__ __forceinline__ void stH(int t, int i, int j, Fx v) const { ck_st(at(h0, lev + 57 * kCkRow, t, i, j), v); }
  __device__ __forceinline__ int64_t ldE(int t, int i, int j) const {
    if (t == 0) return fx_join(ck_ld(in + 45 * kCkRow + off[ck_pair(i, j)]));
    return ck_ld64(e0 + off[ck_pair(i, j)]);
  }
  __device__ __forceinline__ int64_t pick(int64_t x, int64_t y) const { return dir ? y : x; }
  // the other lane's value
  __device__ __forceinline__ int64_t swap(int64_t z) const { return __shfl_xor_sync(0xffffffffu, (long long)z, 16); }
  __device__ __forceinline__ void sync() const { __syncwarp(); }
  // coefficient (i, j) of slice n: the lane's momentum, and density (lane x) or energy (lane y)
  __device__ __forceinline__ void next(int n, int i, int j, int64_t own, int64_t both, FxRange& r) {
    if (i + j == 0) {
      mom_out[n - 1] = own;
      both_out[n - 1] = both;
    }
    if (n == 4) return;
    ck_st(momL + ck_level_row(n) * kCkRow + off[ck_pair(i, j)], fx_split_any(own + FX_HALF, r));
    FxRange rb{0};
    const Fx v = fx_split_any(both + FX_HALF, rb);
    r.t |= dir ? 0u : rb.t;
    const Fx e = Fx{(int32_t)((uint64_t)both & 0xffffffffu), (int32_t)(both >> 32)};  // low word first
    ck_st((dir ? e0 : lev + ck_level_row(n) * kCkRow) + off[ck_pair(i, j)], dir ? e : v);
  }
};

// The recursion of the 16 points p0.. of a half (valid: points that exist), by one whole warp.
// Results: t[q][k] (64-bit, k = 1..4) in row q * 4 + k - 1 of the point's column of the half's input.
// Out of line: one copy of the recursion for all kernels of a translation unit.
static __device__ __noinline__ void ck_warp_euler2d(int half, int p0, int valid, Fx third, Fx gm1) {
  const int lane = threadIdx.x & 31, dir = lane >> 4, pt = p0 + (lane & 15);
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  CkLane S(half, pt, dir);
  const Fx ninv = ck_ld(kCkNinv + (half * CKP + pt) * 8);
#pragma unroll 1
  for (int tries = 1;; ++tries) {
    FxRange r{0};
    ck_euler2d_lane(S, ninv, gm1, third, r);
    int bad = (lane & 15) < valid && r.bad() ? 1 : 0;
    bad |= __shfl_xor_sync(0xffffffffu, bad, 16);
    if (!__any_sync(0xffffffffu, bad)) break;
    if (tries == kCkTries) {
      if (bad && dir == 0) *reinterpret_cast<int*>(dyn_smem + kCkGrow + (half * CKP + pt) * 4) = kCkLost;
      break;
    }
    __syncwarp();
    if (bad) {  // divide the coefficients of degree s by 2^s: each lane half of the components
      FxRange none{0};
#pragma unroll 1
      for (int q = 2 * dir; q < 2 * dir + 2; ++q)
#pragma unroll
        for (int s = 1; s < 5; ++s)
#pragma unroll
          for (int j = 0; j <= s; ++j) {
            const int at = S.in + (q * 15 + ck_pair(s - j, j)) * kCkRow;
            ck_st(at, fx_regrow(ck_ld(at), s, none));
          }
      if (dir == 0) *reinterpret_cast<int*>(dyn_smem + kCkGrow + (half * CKP + pt) * 4) += 1;
    }
    __syncwarp();
  }
  __syncwarp();  // the inputs are read no more
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    ck_st64(S.in + ((1 + dir) * 4 + k) * kCkRow, S.mom_out[k]);
    ck_st64(S.in + (dir * 12 + k) * kCkRow, S.both_out[k]);
  }
}

// Both coordinates in units of L (dx != dy): factors of the spatial coefficients.
template <int NC>
__device__ __forceinline__ void ck_unit_lengths(const Params& P, double (&a)[NC][25]) {
  if (P.ck.rx == P.ck.ry) return;
  double fx = 1.0;
#pragma unroll
  for (int m = 0; m < 5; ++m, fx *= P.ck.rx) {
    double f = fx;
#pragma unroll
    for (int n = 0; n + m < 5; ++n, f *= P.ck.ry)
#pragma unroll
      for (int q = 0; q < NC; ++q) a[q][m * 5 + n] *= f;
  }
}

// Time-Taylor coefficients per unit L^k (P.ck.iL = 1 / L) of the CTA's points (threads 0 .. npt - 1, those
// with has_face) for 2D Euler; called by every thread after the barrier that ends the use of the
// tables.  S: the point's scale, conv(q, m*5+n) its coefficients in that scale, Ws the leading state.
template <typename Conv>
__device__ __forceinline__ void ck_points4(const Params& P, int npt, bool has_face, CkScale<4> S, const Conv& conv,
                                           const CkLead& lead, const double* Ws, double (&tc)[4][5]) {
  const int tid = threadIdx.x;
  const int col = kCkIn + (tid / CKP) * 60 * kCkRow + (tid % CKP) * 8;
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  if (has_face) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int s = 0; s < 5; ++s)
#pragma unroll
        for (int n = 0; n <= s; ++n) ck_st(col + (q * 15 + ck_pair(s - n, n)) * kCkRow, conv(q, (s - n) * 5 + n));
    ck_st(kCkNinv + tid * 8, ck_ninv<4>(S, lead));
    *reinterpret_cast<int*>(dyn_smem + kCkGrow + tid * 4) = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) tc[q][0] = Ws[q];
  } else if (tid < npt) {  // the last cell of a run: zeros stay zeros
#pragma unroll 1
    for (int k = 0; k < 60; ++k) ck_st(col + k * kCkRow, Fx{0, 0});
    ck_st(kCkNinv + tid * 8, Fx{0, 0});
  }
  __syncthreads();
  const int p0 = (tid >> 5) * 16;
#pragma unroll 1
  for (int half = 0; half * CKP < npt; ++half) {
    const int valid = npt - half * CKP - p0;
    if (valid > 0) ck_warp_euler2d(half, p0, valid, P.ck.K.third, P.ck.K.gm1);
    __syncwarp();
  }
  __syncthreads();
  if (!has_face) return;
  const int grown = *reinterpret_cast<const int*>(dyn_smem + kCkGrow + tid * 4);
  S.g += grown;
  S.finite = S.finite && grown != kCkLost;
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int k = 1; k < 5; ++k) {
      const int64_t t = ck_ld64(col + (q * 4 + k - 1) * kCkRow);
      tc[q][k] = S.finite ? fx_to_double(t, S.of(q, 0) + k * (S.eu + S.g)) : fx_from_bits(0x7ff8000000000000ull);
    }
}

// The same in FP64, one thread a point, from the coefficients a[q][m*5+n] in units of L.
__device__ __forceinline__ void ck_points64(const Params& P, bool has_face, const double (&a)[4][25], double (&tc)[4][5]) {
  if (!has_face) return;
  ck_euler2d(a, tc, P.ck.gm1);
#pragma unroll
  for (int q = 0; q < 4; ++q) tc[q][0] = a[q][0];
}

// Whether a point of a face across direction dir has a slow momentum along the face that FP64 holds better (see
// cell_exponents).
__device__ __forceinline__ bool ck_coarse2d(const double (&a)[4][25], int dir) {
  auto mag = [&a](int q, int mn) { return fx_hi(a[q][mn]) & 0x7fffffff; };
  const int n0 = fx_exp(mag(0, 0)), n3 = fx_exp(mag(3, 0)), nm = (n0 + n3 + 1) >> 1;
  int E = 0, mom = 0;  // the energy's coefficients along the face, the momentum
#pragma unroll
  for (int m = 0; m < 5; ++m)
#pragma unroll
    for (int n = 0; n + m < 5; ++n) {
      if ((dir ? m : n) > 0) E = max(E, mag(3, m * 5 + n));
      mom = max(mom, mag(2 - dir, m * 5 + n));
    }
  const int below = nm - fx_exp(mom);
  return mom > 0 && below > CK_BELOW && below <= FX_STILL && fx_exp(E) < n3 - FX_STILL;
}

// The same from FP64 coefficients a[q][m*5+n] in cell units, Burgers or Euler; called while the tables may still
// be in use.
template <int NC>
__device__ __forceinline__ void ck_points(const Params& P, int npt, bool has_face, int dir, double (&a)[NC][25],
                                          const CkLead& lead, double (&tc)[NC][5]) {
  ck_unit_lengths<NC>(P, a);
  if constexpr (NC == 1) {
    if (!has_face) return;
    ck_fixed<1, 2>(a, lead, P.ck, tc);
    tc[0][0] = a[0][0];
  } else {
    CkScale<4> S{};
    if (has_face) S = ck_scale<4, 2>([&a](int q, int mn) { return a[q][mn]; }, lead);
    if (__syncthreads_or(!P.ck.fixed || (has_face && (ck_off_units(S, lead) || ck_coarse2d(a, dir))) ? 1 : 0)) return ck_points64(P, has_face, a, tc);
    const double Ws[4] = {a[0][0], a[1][0], a[2][0], a[3][0]};
    FxRange none{0};  // the recursion checks its operands
    ck_points4(P, npt, has_face, S, [&](int q, int mn) { return ck_convert<4>(S, a[q][mn], q, mn / 5 + mn % 5, none); },
               lead, Ws, tc);
  }
}

// ------------------------------------------------------------------ second pass in fixed point
// 2D Euler, reading R1, componentwise: the end values, their differences and the upwinding in 64-bit
// integers instead of FP64 (about 790 of a face point's 1680 remaining FP64 instructions).  A cell's
// data (first-pass coefficients of its three columns) are converted in a scale of each component's
// own, the largest of them in [1/2, 1), 57 fraction bits (its double has 53).  The
// end values are sums of shifted data (their coefficients are eighths, but for the value's) times the
// cell's weights; a face brings both sides to a scale that fits its units of density and velocity
// and upwinds there with the FP64 eigenvectors, converted.  What the format would hold worse than FP64
// does is noticed and the CTA takes the FP64 pass instead: before any work, data that are not finite or
// not of one size (cell_exponents); on the way (FxRange), face units far above the density or energy,
// eigenvectors beyond 2^4 in them, end values above 8 times the data, weights of 4 and more.
constexpr int FX_ABOVE = 4;       // most bits of a cell's data above the size its own state gives the component
constexpr int FX_BELOW = 6;       // a momentum more bits than this below that size is a slow one,
                                  // and one more than FX_STILL counts as none
constexpr int FX_UNIT = 5;        // most bits of a face's density and energy below their units
constexpr int FX_EL = FX_D - 53;  // most bits that the projections' scale takes off
constexpr int FX_TINY = CK_TINY;  // least exponent of a scale
struct CellMixFx {
  Fx A[4], B[4], C[4];
  int h[4];  // exponents of the cell's data
  bool lin;
};

// x 2^-58 c + ..., c a constant with FX_C fraction bits
__device__ __forceinline__ int64_t fx_scaled(Fx x, Fx c) {
  FxAcc s = fx_zero<FX_C>();
  fx_mac(s, x, c);
  return fx_sum<FX_C>(s);
}

// Exponents of the cell's data over all orders and its three columns; false if FP64 holds them better.
// FP64 rounds every value by its own size, a block by its largest.  The lines below lie where the error of a whole
// step against 64-bit mantissas begins to exceed that of the FP64 pass.
//   A cold cell beside a hot one, which the weights cut off, rounds at 2^-57 of the hot one (energy 2.5
// beside 564: 1.4e-14 of the cold cell's end value, in FP64 3e-16; beside 1e12: 5e-6).  So no value may be
// more than FX_ABOVE bits above the cell's own density, energy, or the momentum sqrt(rho E) they allow.  Cells beside
// a block of 2^k times their density and energy, error of their slopes relative to the FP64 pass, mean of
// three flows: 1.0 at k = 3, 1.1 at 4, 1.6 at 5, 2.7 at 6, 3.8 at 7, 13 at 10.
//   A slow momentum rounds at 2^-57 of that one: less than what the rounding of the pressure, 2^-53 of
// rho c^2, does in every step to the momentum across the face, and to the one along the face where the energy
// varies along it.  Where it does not (a shear layer), the pressure moves nothing and FP64 carries
// the momentum with all its bits.  Shear flow, three steps, error of the drift's slope relative to the FP64
// pass: 0.9 at 6 bits below, 1.2 at 7, 1.4 at 8, 2.5 at 9, 6 at 10, 10 at 11.
//   Share of the CTAs that go to FP64: vortex, smooth flows 0; quadrants 0 to 0.6 % (400^2, 300 steps), random ones
// (rho, p in [0.1, 2]) 0 to 13 %; double Mach reflection 11 % (1024 x 256, 400 steps), whose step takes 8.5 ms (8.7
// with every CTA in fixed point).  If any slow momentum went there: quadrants 16 to 65 %.  Testing the cells:
// 0.2 % of the vortex step (2048^2).  Drift of a shear flow at 1e-6 of the sound speed, three steps, error
// against 64-bit mantissas: 2.0e-13 -> 7.5e-17.
__device__ __forceinline__ bool cell_exponents(const double (*ev)[5][SPAN], int c, int dir, int h[4]) {
  auto mag = [&](int f, int k, int col) { return fx_hi(ev[f][k][col]) & 0x7fffffff; };
  const int n0 = fx_exp(mag(0, 0, c)), n3 = fx_exp(mag(3, 0, c)), nm = (n0 + n3 + 1) >> 1;
  int along = 0;  // the energy's coefficients along the face
#pragma unroll
  for (int k = 1; k < 5; ++k) along = max(along, max(mag(3, k, c - 1), max(mag(3, k, c), mag(3, k, c + 1))));
  const bool even = fx_exp(along) < n3 - FX_STILL;
  int all = 0;
  bool ok = true;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    int top = 0;
#pragma unroll
    for (int k = 0; k < 5; ++k)
      top = max(top, max(max(mag(q, k, c - 1), max(mag(q, k, c), mag(q, k, c + 1))), max(mag(4 + q, k, c - 1), mag(4 + q, k, c + 1))));
    all = max(all, top);
    const int e = fx_exp(top);
    const bool momentum = q == 1 || q == 2;
    if (top > 0 && !(momentum && e < nm - FX_STILL)) {
      ok = ok && e >= FX_TINY && e <= (q == 0 ? n0 : q == 3 ? n3 : nm) + FX_ABOVE;
      if (q == 2 - dir) ok = ok && !(even && e < nm - FX_BELOW);
    }
    h[q] = max(e, FX_TINY);  // an exact 0 then converts to 0
  }
  return ok && all < 0x7ff00000;
}

// Order K of the thread's cell: its ends into the tables L and R (units of the cell's h).  The
// components and the orders share one copy of the code: unrolled, the pass alone would overflow the
// instruction cache (128 KB), which the kernel then waits for.
template <bool LIN>
__device__ __forceinline__ void cell_ends_fx(const double (*ev)[5][SPAN], int K, int c, const CellMixFx& m,
                                             int64_t (*L)[5][SEG], int64_t (*R)[5][SEG], FxRange& r) {
  const Fx u0w{85004561, 143165568}, u0s{24606583, 1002159032}, u0d{-6710886, -858993460};  // 19/30, 11/60, -1/20
#pragma unroll 1
  for (int q = 0; q < 4; ++q) {
    const int h = m.h[q];
    const int64_t Wm = fx_from_double<FX_D>(ev[q][K][c - 1], h), W0 = fx_from_double<FX_D>(ev[q][K][c], h);
    const int64_t Wp = fx_from_double<FX_D>(ev[q][K][c + 1], h);
    const int64_t vm = fx_from_double<FX_D>(ev[4 + q][K][c - 1], h), vp = fx_from_double<FX_D>(ev[4 + q][K][c + 1], h);
    const int64_t s = Wm + Wp, a = Wp - Wm, dv = vp - vm, sv = vm + vp;
    FxRange in{0};  // the data themselves are in range by their scale
    const Fx w0 = fx_split(W0 + FX_HALF, in);
    int64_t g = 0, hh = 0;
    if (!LIN) {
      const Fx d2 = fx_split(W0 - Wm + FX_HALF, in), d3 = fx_split(Wp - W0 + FX_HALF, in);
      FxAcc z = fx_zero<FX_C>();
      fx_mac(z, d2, m.B[q]);
      fx_mac(z, d3, m.C[q]);
      g = fx_sum<FX_C>(z);
      z = fx_zero<FX_C>();
      fx_mac(z, w0, m.B[q]);
      fx_mac(z, w0, m.C[q]);
      hh = fx_sum<FX_C>(z);
    }
#pragma unroll
    for (int p = 0; p < 5; ++p) {
      if (p + K > 4) break;
      int64_t U, V = 0;
      if (p == 0) {
        FxAcc z = fx_zero<FX_C>();
        fx_mac(z, w0, u0w);
        fx_mac(z, fx_split(s + FX_HALF, in), u0s);
        fx_mac(z, fx_split(dv + FX_HALF, in), u0d);
        U = fx_sum<FX_C>(z);
        V = (3 * a - sv + 4) >> 3;
      } else if (p == 1) {
        U = s - 2 * W0 - ((dv + 2) >> 2);
        V = (5 * a - sv + 4) >> 3;
      } else if (p == 2) {
        U = ((s + 1) >> 1) - W0;
        V = (3 * (sv - a) + 4) >> 3;
      } else if (p == 3) {
        U = 2 * W0 - s + ((dv + 1) >> 1);
        V = (sv - a + 2) >> 2;
      } else {
        U = W0 - ((s + 1) >> 1) + ((dv + 2) >> 2);
      }
      if (!LIN) {
        U = fx_scaled(fx_split_wide(U + FX_HALF, r), m.A[q]);
        if (p < 4) V = fx_scaled(fx_split_wide(V + FX_HALF, r), m.A[q]);
        if (p == 0) { U += hh; V += g >> 1; }
        if (p == 1) U += g;
      }
      // odd p: the slope terms have one sign at both ends, so g is added after the mirror image
      R[q][p][threadIdx.x] = U + V;
      int64_t eL = (p & 1) ? V - U : U - V;
      if (!LIN && p == 1) eL += 2 * g;
      L[q][p][threadIdx.x] = eL;
    }
  }
}

// The face's upwinding in fixed point.  The linearised problem's solution (Upwinder) is
// d* = base + sum_k s_k (l_k . d) r_k, d = dL - dR.  The entropy and shear waves share their speed, so
// their s (call it c), and the four projections add up to the identity: d* = base + c d +
// sum over the two acoustic waves of (s_k - c) (l_k . d) r_k.  A moving subsonic face needs one acoustic
// wave and c = 0, a standing one (c = +-1/2) both; which one it is differs from lane to lane and is
// chosen by the vectors, not by a branch.
struct UpwindFx {
  Fx l[2][4], r[2][4];  // (s_k - c) l_k times 2^-el, and r_k, in the face's units
  int waves, c2;        // waves that contribute; 2 c
  int el, base_left;
  int f[4], sl[4], sr[4];  // the face's exponents; right shifts of the two sides' end values
};

// Order K of the thread's face: upwinded derivatives a[q][m*5+n] in units of f (a in local memory: K is
// a loop's).
__device__ __forceinline__ void face_order_fx(const int64_t (*L)[5][SEG], const int64_t (*R)[5][SEG], int K, int dir,
                                              const UpwindFx& U, int64_t (&a)[4][25], FxRange& r) {
#pragma unroll
  for (int p = 0; p < 5; ++p) {
    if (p + K > 4) break;
    if (p == 0 && K == 0) continue;
    const int idx = dir == 0 ? p * 5 + K : K * 5 + p;
    int64_t base[4];
    Fx d[4];
    FxAcc out[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int64_t x = R[q][p][threadIdx.x] >> U.sl[q], y = L[q][p][threadIdx.x + 1] >> U.sr[q];
      d[q] = fx_split_wide(x - y + FX_HALF, r);
      out[q] = fx_zero<FX_C>();
      base[q] = (U.base_left ? x : y) + ((U.c2 * (x - y)) >> 1);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (U.waves <= k) continue;
      FxAcc z = fx_zero<FX_C>();
#pragma unroll
      for (int q = 0; q < 4; ++q) fx_mac(z, d[q], U.l[k][q]);
      const int64_t w = fx_sum<FX_C>(z);
      if (((w ^ (w >> 63)) >> (59 - U.el)) != 0) r.h |= 0x80000000u;
      const Fx al = fx_split((int64_t)((uint64_t)w << U.el) + FX_HALF, r);
#pragma unroll
      for (int q = 0; q < 4; ++q) fx_mac(out[q], al, U.r[k][q]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) a[q][idx] = base[q] + fx_sum<FX_C>(out[q]);
  }
}

// Leading term and acoustic eigenvectors of the thread's face (FP64), its units, the converted waves.
__device__ __forceinline__ void face_setup_fx(const Params& P, const int64_t (*L)[5][SEG], const int64_t (*R)[5][SEG],
                                              const int hL[4], const int* hs, int dir, double Ws[4], CkLead& lead,
                                              UpwindFx& X, FxRange& r) {
  int hR[4];
  double WL[4], WR[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    hR[q] = hs[q * SEG + threadIdx.x + 1];
    WL[q] = fx_to_double(R[q][0][threadIdx.x], hL[q] + FX_Q - FX_D);
    WR[q] = fx_to_double(L[q][0][threadIdx.x + 1], hR[q] + FX_Q - FX_D);
  }
  hllc_state<4>(WL, WR, P.gamma, dir, Ws);
  const Prim S = euler_prim(Ws, 4, P.gamma);
  lead = prim_lead<4>(S);
  double rv[4][4], lv[4][4], lam[4], s[4];
  euler_eigvecs<4>(S, P.gamma, dir, rv, lv, lam);
  X.base_left = wave_coefficients<4>(lam, 1e-12 * S.c, s);
  X.c2 = (int)(2.0 * s[1]);
  const double b0 = s[0] - s[1], b3 = s[3] - s[1];
  const bool low = b0 != 0.0;  // the first wave that contributes is u - c
  X.waves = (low ? 1 : 0) + (b3 != 0.0 ? 1 : 0);
  const int f0 = max(hL[0], hR[0]);
  int F = max(max(max(hL[1], hR[1]), max(hL[2], hR[2])) - f0, (max(hL[3], hR[3]) - f0 + 1) >> 1);
  F = max(F, max(fx_exp(lead.hu), (fx_exp(lead.hH) + 1) >> 1));
  int top = 0, el = -2000;
  bool coarse = ck_off_unit(F, lead);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int u = q == 0 ? 0 : q == 3 ? 2 * F : F;
    X.f[q] = f0 + u;
    X.sl[q] = min(X.f[q] - hL[q], 63);
    X.sr[q] = min(X.f[q] - hR[q], 63);
    if (q == 0 || q == 3) coarse = coarse || X.f[q] - max(hL[q], hR[q]) > FX_UNIT;
    const int hi = max(fx_hi(lv[0][q]) & 0x7fffffff, fx_hi(lv[3][q]) & 0x7fffffff);
    top = max(top, hi);
    el = max(el, fx_exp(hi) + u);
  }
  X.el = max(el, 0);
  if (coarse || top >= 0x7ff00000 || X.el > FX_EL || lead.hH >= 0x7ff00000 || lead.hu >= 0x7ff00000) {
    r.h |= 0x80000000u;
    X.el = 0;
  }
  FxRange in{0};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int u = q == 0 ? 0 : q == 3 ? 2 * F : F;
    X.l[0][q] = fx_split(fx_from_double<FX_C>(low ? b0 * lv[0][q] : b3 * lv[3][q], X.el - u) + FX_HALF, in);
    X.l[1][q] = fx_split(fx_from_double<FX_C>(b3 * lv[3][q], X.el - u) + FX_HALF, in);
    X.r[0][q] = fx_split(fx_from_double<FX_C>(low ? rv[0][q] : rv[3][q], u) + FX_HALF, in);
    X.r[1][q] = fx_split(fx_from_double<FX_C>(rv[3][q], u) + FX_HALF, in);
  }
}

static_assert(ev_bytes<4>() + sizeof(EndTable<4>) + 4 * SEG * sizeof(int) + 4 * 5 * SEG * 8 <= kCkBytes, "tables");
// The whole pass of the CTA; false (for all threads) if something left the format.
template <bool FLAGS>
__device__ __forceinline__ bool second_pass_fx(const Params& P, unsigned char* smem_raw, const FaceRuns& fr, int dir,
                                               bool nl, double (&tc)[4][5]) {
  const double(*ev)[5][SPAN] = reinterpret_cast<const double(*)[5][SPAN]>(smem_raw);
  unsigned char* tables = smem_raw + ev_bytes<4>();
  FxRange r{0};
  CellMixFx m;
  if (!P.ck.fixed) return false;
  const bool ok = !fr.has_cell || cell_exponents(ev, fr.col, dir, m.h);
  if (__syncthreads_or(ok ? 0 : 1)) return false;
  if (fr.has_cell) {
    CellMix<4> w;
    cell_mix<4, false>(P, ev, fr.col, FLAGS && !nl, w);
    m.lin = w.lin;
    int top = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      top = max(top, max(fx_hi(w.A[q]) & 0x7fffffff, max(fx_hi(w.B[q]) & 0x7fffffff, fx_hi(w.C[q]) & 0x7fffffff)));
    if (top >= 0x40100000) r.h = 0x80000000u;  // weights are at most 1 / gam[0] unless they overflowed
    FxRange in{0};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      m.A[q] = fx_split(fx_from_double<FX_C>(w.A[q], 0) + FX_HALF, in);
      m.B[q] = fx_split(fx_from_double<FX_C>(w.B[q], 0) + FX_HALF, in);
      m.C[q] = fx_split(fx_from_double<FX_C>(w.C[q], 0) + FX_HALF, in);
    }
  }
  int64_t a[4][25];
  double Ws[4];
  CkLead lead{};
  UpwindFx X;
  int* hs = reinterpret_cast<int*>(tables + sizeof(EndTable<4>));
  auto R = reinterpret_cast<int64_t(*)[5][SEG]>(tables + sizeof(EndTable<4>) + 4 * SEG * sizeof(int));  // each thread its own
#pragma unroll 1
  for (int K = 0; K < 5; ++K) {  // one barrier per order, as in pass_order
    auto L = reinterpret_cast<int64_t(*)[5][SEG]>(tables) + (K & 1) * 4;
    if (fr.has_cell) {
      if (FLAGS && m.lin) cell_ends_fx<true>(ev, K, fr.col, m, L, R, r);
      else cell_ends_fx<false>(ev, K, fr.col, m, L, R, r);
      if (K == 0)
#pragma unroll
        for (int q = 0; q < 4; ++q) hs[q * SEG + threadIdx.x] = m.h[q];
    }
    __syncthreads();
    if (fr.has_face) {
      if (K == 0) face_setup_fx(P, L, R, m.h, hs, dir, Ws, lead, X, r);
      face_order_fx(L, R, K, dir, X, a, r);
    }
  }
  if (__syncthreads_or(r.bad() ? 1 : 0)) return false;
  CkScale<4> S{};
  if (fr.has_face) {
    int top[3][5];  // exponents by group and degree
    uint64_t bits[3][5];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int s = 0; s < 5; ++s) bits[i][s] = 0;
    if (P.ck.rx != P.ck.ry) {  // dx != dy: both coordinates in units of L (one factor is 1)
      const bool along_x = P.ck.rx != 1.0;
      double f = 1.0;
#pragma unroll
      for (int i = 1; i < 5; ++i) {
        f *= along_x ? P.ck.rx : P.ck.ry;
        const Fx c = fx_const(f);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int j = 0; j + i < 5; ++j) {
            FxRange in{0};
            int64_t& z = a[q][along_x ? i * 5 + j : j * 5 + i];
            z = fx_scaled(fx_split(z + FX_HALF, in), c);
          }
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int s = 1; s < 5; ++s)
#pragma unroll
        for (int n = 0; n <= s; ++n) {
          const int64_t z = a[q][(s - n) * 5 + n];
          bits[CkScale<4>::group(q)][s] |= (uint64_t)(z ^ (z >> 63));
        }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int q = i == 0 ? 0 : i == 1 ? 1 : 3;
      top[i][0] = 0;
#pragma unroll
      for (int s = 1; s < 5; ++s) top[i][s] = X.f[q] - FX_D + 64 - fx_clz(bits[i][s]);
    }
    S = ck_scale_from<4>(Ws, top, lead);
  }
  ck_points4(P, fr.nrun * (fr.nf + 1), fr.has_face, S,
             [&](int q, int mn) {
               FxRange none{0};
               const int s = mn / 5 + mn % 5;
               if (s == 0) return ck_convert<4>(S, Ws[q], q, 0, none);
               const int n = FX_Q - FX_D + X.f[q] - S.of(q, s);  // left shift
               const int64_t z = a[q][mn];
               const int64_t x = n >= 0 ? (int64_t)((uint64_t)z << min(n, 63))
                                        : ((z >> min(-n - 1, 62)) + 1) >> 1;
               return fx_split(x + FX_HALF, none);
             },
             lead, Ws, tc);
  return true;
}

// Second pass, leading term, upwinding and CK of the CTA's faces.  A thread with a face gets in
// tc[q][0..4] the time-Taylor coefficients of its face point per L^k.  nl: whether the thread's cell
// uses the nonlinear weights.
template <int NC, bool FLAGS, bool Q>
__device__ __forceinline__ void second_pass_cells(const Params& P, unsigned char* smem_raw, const FaceRuns& fr, int dir,
                                                  bool nl, double (&tc)[NC][5]) {
  if constexpr (NC == 4 && !Q)
    if (second_pass_fx<FLAGS>(P, smem_raw, fr, dir, nl, tc)) return;
  const double(*ev)[5][SPAN] = reinterpret_cast<const double(*)[5][SPAN]>(smem_raw);
  EndTable<NC>& et = *reinterpret_cast<EndTable<NC>*>(smem_raw + ev_bytes<NC>());
  CellMix<NC> m;
  if (fr.has_cell) cell_mix<NC, Q>(P, ev, fr.col, FLAGS && !nl, m);
  double a[NC][25], Ws[NC];
  Upwinder<NC> U;
  pass_order<NC, FLAGS, Q, 0>(P, ev, et, fr, m, dir, Ws, U, a);
  pass_order<NC, FLAGS, Q, 1>(P, ev, et, fr, m, dir, Ws, U, a);
  pass_order<NC, FLAGS, Q, 2>(P, ev, et, fr, m, dir, Ws, U, a);
  pass_order<NC, FLAGS, Q, 3>(P, ev, et, fr, m, dir, Ws, U, a);
  pass_order<NC, FLAGS, Q, 4>(P, ev, et, fr, m, dir, Ws, U, a);
  if (fr.has_face)
#pragma unroll
    for (int q = 0; q < NC; ++q) a[q][0] = Ws[q];
  if constexpr (NC == 4 && !Q) {
    ck_unit_lengths<NC>(P, a);
    ck_points64(P, fr.has_face, a, tc);
  } else {
    ck_points<NC>(P, fr.nrun * (fr.nf + 1), fr.has_face, dir, a, U.lead, tc);
  }
}

// ------------------------------------------------------------------ characteristic-wise face point
// Cross-face Taylor coefficients e[p] (p <= 4 - k) of tangential order k at the right end
// (PLUS, xi = +1/2) or left end of a cell, from its field data d = (W-, W0, W+, v-, v+) of that
// order ((W-, W0, W+, v-, v0, v+) for reading R1', Q): e[p] = A * END[p] . d + (small-stencil
// terms for p <= 1).
template <bool PLUS, bool Q = false>
__device__ __forceinline__ void side_out_d(const double* d, int k, double A, double B, double C,
                                           bool lin, double e[5]) {
  using namespace shweno_tables;
  if (lin) {  // linear weights: p = p1
#pragma unroll
    for (int p = 0; p + k <= 4; ++p) e[p] = Q ? qend_dot<PLUS>(p, d) : end_dot<PLUS>(p, d);
    return;
  }
#pragma unroll
  for (int p = 0; p + k <= 4; ++p) e[p] = A * (Q ? qend_dot<PLUS>(p, d) : end_dot<PLUS>(p, d));
  // p2 = W0 + (W0 - W-) xi and p3 = W0 + (W+ - W0) xi: value and slope at the end
  if (PLUS) e[0] += (1.5 * B + 0.5 * C) * d[1] - 0.5 * B * d[0] + 0.5 * C * d[2];
  else e[0] += (0.5 * B + 1.5 * C) * d[1] + 0.5 * B * d[0] - 0.5 * C * d[2];
  if (k <= 3) e[1] += (B - C) * d[1] - B * d[0] + C * d[2];
}

// Characteristic-wise counterpart for one face point (Euler, NC = 4): the first-pass data of
// tangential order k of the four stencil columns c0..c0+3, projected onto the fields of basis
// Bs; xw[c][f] from {W, Y} (x-face) or {W, V} (y-face), xv[c][f] from the derivative set.
template <int NC>
__device__ __forceinline__ void fields_at(const double (*ev)[5][SPAN], const CharBasis<NC>& Bs, int c0,
                                          int k, double xw[4][NC], double xv[4][NC]) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    double w[NC], v[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) { w[q] = ev[q][k][c0 + c]; v[q] = ev[NC + q][k][c0 + c]; }
    Bs.to_fields(w, xw[c]);
    Bs.to_fields(v, xv[c]);
  }
}
// Cross-face Taylor coefficients of both sides in physical variables, tangential order k, from
// the field data: left cell = column 1 (stencil 0..2), right cell = column 2 (stencil 1..3).
template <int NC, bool Q>
__device__ __forceinline__ void char_sides(const CharBasis<NC>& Bs, const double xw[4][NC],
                                           const double xv[4][NC], int k, const double* AL,
                                           const double* BL, const double* CL, bool linL,
                                           const double* AR, const double* BR, const double* CR,
                                           bool linR, double dl[NC][5], double dr[NC][5]) {
  double el[NC][5], er[NC][5];
#pragma unroll
  for (int f = 0; f < NC; ++f) {
    if constexpr (Q) {
      const double dL[6] = {xw[0][f], xw[1][f], xw[2][f], xv[0][f], xv[1][f], xv[2][f]};
      const double dR[6] = {xw[1][f], xw[2][f], xw[3][f], xv[1][f], xv[2][f], xv[3][f]};
      side_out_d<true, true>(dL, k, AL[f], BL[f], CL[f], linL, el[f]);
      side_out_d<false, true>(dR, k, AR[f], BR[f], CR[f], linR, er[f]);
    } else {
      const double dL5[5] = {xw[0][f], xw[1][f], xw[2][f], xv[0][f], xv[2][f]};
      const double dR5[5] = {xw[1][f], xw[2][f], xw[3][f], xv[1][f], xv[3][f]};
      side_out_d<true>(dL5, k, AL[f], BL[f], CL[f], linL, el[f]);
      side_out_d<false>(dR5, k, AR[f], BR[f], CR[f], linR, er[f]);
    }
  }
#pragma unroll
  for (int p = 0; p + k <= 4; ++p) {
    double x[NC], y[NC];
#pragma unroll
    for (int f = 0; f < NC; ++f) x[f] = el[f][p];
    Bs.to_physical(x, y);
#pragma unroll
    for (int q = 0; q < NC; ++q) dl[q][p] = y[q];
#pragma unroll
    for (int f = 0; f < NC; ++f) x[f] = er[f][p];
    Bs.to_physical(x, y);
#pragma unroll
    for (int q = 0; q < NC; ++q) dr[q][p] = y[q];
  }
}

// Face point of the characteristic-wise option (Euler): the second pass across the face runs in
// the characteristic fields of the Jacobian along the face normal at Wref (the mean of the cell
// averages next to the point), with its own weights per field and side; then the leading term
// (HLLC) and the upwinding.  Left cell in column c0 + 1, right cell in c0 + 2; dir = 0:
// x-face (first pass along y), 1: y-face.  Returns the spatial Taylor coefficients a[q][m*5+n] and
// the scales of the leading state.
template <int NC, bool FLAGS, bool Q>
__device__ __forceinline__ void char_face_point(const Params& P, const double (*ev)[5][SPAN],
                                                const FlagTable& ft, int c0, int dir, double (&a)[NC][25],
                                                CkLead& lead, const double* Wref) {
  static_assert(NC == 4, "characteristic fields are for the Euler system");
  const double g = P.gamma;
  double dl[NC][5], dr[NC][5];
  double AL[NC], BL[NC], CL[NC], AR[NC], BR[NC], CR[NC];
  // FLAGS = false: every cell uses the nonlinear weights (compile-time, no branch)
  const bool linL = FLAGS && ft.lin[c0 + 1], linR = FLAGS && ft.lin[c0 + 2];
  CharBasis<NC> Bs;
  Bs.setup(Wref, g, dir);
  {
    double xw[4][NC], xv[4][NC];
    fields_at<NC>(ev, Bs, c0, 0, xw, xv);
#pragma unroll
    for (int f = 0; f < NC; ++f) {
      AL[f] = AR[f] = 1.0;
      BL[f] = CL[f] = BR[f] = CR[f] = 0.0;
      if (!linL) {
        double cf[6];
        p1_coeffs_t<Q>(xw[0][f], xw[1][f], xw[2][f], xv[0][f], xv[1][f], xv[2][f], cf);
        const Mix m = shweno_mix_t<Q>(P, xw[0][f], xw[1][f], xw[2][f], cf, 1);
        AL[f] = m.A; BL[f] = m.B; CL[f] = m.C;
      }
      if (!linR) {
        double cf[6];
        p1_coeffs_t<Q>(xw[1][f], xw[2][f], xw[3][f], xv[1][f], xv[2][f], xv[3][f], cf);
        const Mix m = shweno_mix_t<Q>(P, xw[1][f], xw[2][f], xw[3][f], cf, 1);
        AR[f] = m.A; BR[f] = m.B; CR[f] = m.C;
      }
    }
    char_sides<NC, Q>(Bs, xw, xv, 0, AL, BL, CL, linL, AR, BR, CR, linR, dl, dr);
  }
  double WL[NC], WR[NC], Ws[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) { WL[q] = dl[q][0]; WR[q] = dr[q][0]; }
  hllc_state<NC>(WL, WR, g, dir, Ws);
  Upwinder<NC> U;
  U.setup(Ws, g, dir);
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    if (k > 0) {
      double xw[4][NC], xv[4][NC];
      fields_at<NC>(ev, Bs, c0, k, xw, xv);
      char_sides<NC, Q>(Bs, xw, xv, k, AL, BL, CL, linL, AR, BR, CR, linR, dl, dr);
    }
#pragma unroll
    for (int p = 0; p + k <= 4; ++p) {
      if (p == 0 && k == 0) continue;
      double x[NC], y[NC], o[NC];
#pragma unroll
      for (int q = 0; q < NC; ++q) { x[q] = dl[q][p]; y[q] = dr[q][p]; }
      U.apply(x, y, o);
      // p is the order across the face, k the order along it
      const int idx = dir == 0 ? p * 5 + k : k * 5 + p;
#pragma unroll
      for (int q = 0; q < NC; ++q) a[q][idx] = o[q];
    }
  }
#pragma unroll
  for (int q = 0; q < NC; ++q) a[q][0] = Ws[q];
  lead = U.lead;
}

// Combined coefficients C[u] of NU = 1 or 2 components of one cell from their stencil averages
// w[u] = (W-, W0, W+) and p1 coefficients c[u] (C = c for a cell with the linear weights).  PAIR
// (Euler, reading R1): the two components' weights share one division, 1/S0 = S1 / (S0 S1) and
// 1/S1 = S0 / (S0 S1), as in the second pass.
template <bool Q, bool PAIR>
__device__ __forceinline__ void first_pass_mix(const Params& P, int nl, const double (*w)[3], const double (*c)[6],
                                               double (*C)[6]) {
  constexpr int NU = PAIR ? 2 : 1;
  if (!nl) {
#pragma unroll
    for (int u = 0; u < NU; ++u)
#pragma unroll
      for (int k = 0; k < 6; ++k) C[u][k] = c[u][k];
    return;
  }
  if constexpr (PAIR) {
    const RawWeights r0 = shweno_raw_weights(P, w[0][0], w[0][1], w[0][2], c[0]);
    const RawWeights r1 = shweno_raw_weights(P, w[1][0], w[1][1], w[1][2], c[1]);
    const double inv = 1.0 / (r0.sum * r1.sum);
    mix_coeffs_t<Q>(mix_from_raw(P, r0, inv * r1.sum), w[0][0], w[0][1], w[0][2], c[0], C[0]);
    mix_coeffs_t<Q>(mix_from_raw(P, r1, inv * r0.sum), w[1][0], w[1][1], w[1][2], c[1], C[1]);
  } else {
    mix_coeffs_t<Q>(shweno_mix_t<Q>(P, w[0][0], w[0][1], w[0][2], c[0], 1), w[0][0], w[0][1], w[0][2], c[0], C[0]);
  }
}

// First-pass polynomials of the cells of one tile, one of the four reconstructions (unit 0: y-pass
// on {W, Y}, 1: y-pass on {V, Z}, 2: x-pass on {W, V}, 3: x-pass on {Y, Z}): thread (tx, ty) of a
// TX x TYB block owns the extended cell (bx + tx, by + ty); the unit's 2 * NC fields of the tile plus a
// one-cell halo are staged in shared memory `tile` (room for 8) by all threads first.  The units are
// independent, so a small mesh spreads over four times as many CTAs (40^2 cells: 104 -> 38 us) and a
// large one runs more warps per SM.  Q: reading R1', whose quintic p1 also uses the cell's own
// derivative average; it stores six coefficients per polynomial instead of five (the scratch
// layout's KC).
template <int NC, int TYB, bool Q = false>
__device__ __forceinline__ void coef2d_item(const Params& P, const StepView& sv, const double* s0,
                                            const double* s1, const uint8_t* __restrict__ flag,
                                            double* __restrict__ ycoef, double* __restrict__ xcoef, int unit,
                                            int bx, int by, double (*tile)[TYB + 2][TX + 2], int tx,
                                            int ty) {
  const double* st = sv.odd ? s1 : s0;
  const double t = sv.t;
  const bool ypass = unit < 2;
  const int s = unit & 1;
  const int fa = s == 0 ? 0 : (ypass ? 1 : 2), fd = s == 1 ? 3 : (ypass ? 2 : 1);
  const int tid = ty * TX + tx;
  for (int idx = tid; idx < 2 * NC * (TYB + 2) * (TX + 2); idx += TX * TYB) {
    const int xx = idx % (TX + 2), rest = idx / (TX + 2);
    const int yy = rest % (TYB + 2), fq = rest / (TYB + 2);
    const int i = bx - 1 + xx, j = by - 1 + yy;
    double v = 0.0;
    if (i >= -3 && i <= P.nx + 2 && j >= -3 && j <= P.ny + 2) v = fetch(P, st, fq < NC ? fa : fd, fq % NC, i, j, t);
    tile[fq][yy][xx] = v;
  }
  __syncthreads();
  const int ic = bx + tx, jr = by + ty;
  if (ypass ? !(ic <= P.nx + 1 && jr >= -1 && jr <= P.ny) : !(ic >= 0 && ic < P.nx && jr <= P.ny + 1)) return;
  const int lx = tx + 1, ly = ty + 1;
  const int dx = ypass ? 0 : 1, dy = ypass ? 1 : 0;
  constexpr int KC = Q ? 6 : 5;
  constexpr bool PAIR = NC == 4 && !Q;
  constexpr int NU = PAIR ? 2 : 1;
  const int nl = cell_flag(P, flag, ic, jr);
  const double h = ypass ? P.dy : P.dx;
  const double sc = ypass ? P.dx : P.dy;  // set 1: derivative data of the pass across, h avg
  const size_t NX4 = P.nx + 4, NY2 = P.ny + 2, NY4 = P.ny + 4;
  double* out = ypass ? ycoef + (size_t)(jr + 1) * NX4 + (ic + 2) : xcoef + (size_t)ic * NY4 + (jr + 2);
  const size_t plane = ypass ? NY2 * NX4 : (size_t)P.nx * NY4;
#pragma unroll
  for (int q0 = 0; q0 < NC; q0 += NU) {
    double w[NU][3], c[NU][6], C[NU][6];
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      const int q = q0 + u;
      w[u][0] = tile[q][ly - dy][lx - dx]; w[u][1] = tile[q][ly][lx]; w[u][2] = tile[q][ly + dy][lx + dx];
      const double vm = h * tile[NC + q][ly - dy][lx - dx], vp = h * tile[NC + q][ly + dy][lx + dx];
      const double v0 = Q ? h * tile[NC + q][ly][lx] : 0.0;
      p1_coeffs_t<Q>(w[u][0], w[u][1], w[u][2], vm, v0, vp, c[u]);
    }
    first_pass_mix<Q, PAIR>(P, nl, w, c, C);
    if (s == 1)
#pragma unroll
      for (int u = 0; u < NU; ++u)
#pragma unroll
        for (int k = 0; k < KC; ++k) C[u][k] *= sc;
#pragma unroll
    for (int u = 0; u < NU; ++u)
#pragma unroll
      for (int k = 0; k < KC; ++k) out[((size_t)(s * NC + q0 + u) * KC + k) * plane] = C[u][k];
  }
}

// x-face Gauss points (slice 0..2; lines are cell rows) or corner points (slice 3; lines are corner
// rows, row r at y_{r-1/2}) of CTA b of the slice; SEG threads, smem_raw of face_smem<NC>() bytes.
template <int NC, bool FLAGS, bool CHAR = false, bool Q = false>
__device__ __forceinline__ void xface_item(const Params& P, const StepView& sv, const double* st,
                                           const double* __restrict__ ycoef,
                                           const uint8_t* __restrict__ flag, double* __restrict__ FX,
                                           double* __restrict__ WX, double* __restrict__ WC, int b,
                                           int slice, unsigned char* smem_raw) {
  double(*ev)[5][SPAN] = reinterpret_cast<double(*)[5][SPAN]>(smem_raw);
  const int NX4 = P.nx + 4, NY2 = P.ny + 2;
  using namespace shweno_tables;
  const FaceRuns fr(P.nx + 1, slice < 3 ? P.ny : P.ny + 1, b);
  // a run's faces x_{f0-1/2} .. x_{f0+nf-3/2} have stencils that span its columns 0 .. nf + 2
  const int w = fr.nf + 3, ncol = fr.nrun * w;
  for (int it = threadIdx.x; it < 2 * NC * ncol; it += SEG) {
    const int col = it % ncol, rq = it / ncol;
    const int tcol = fr.f0 + col % w, row = fr.line + col / w;
    double e[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    if constexpr (Q) {  // six coefficients per polynomial (reading R1')
      if (slice < 3) {
        const double* src = ycoef + ((size_t)(rq * 6) * NY2 + (row + 1)) * NX4 + tcol;
#pragma unroll
        for (int k = 0; k < 6; ++k) e[k] = __ldcg(src + (size_t)k * NY2 * NX4);
        if (slice != 1) taylor_shift_d<5>(e, slice == 0 ? -GAUSS_G : GAUSS_G);
      } else {
        double lo[6], hi[6];
        const double* slo = ycoef + ((size_t)(rq * 6) * NY2 + row) * NX4 + tcol;
        const double* shi = slo + NX4;
#pragma unroll
        for (int k = 0; k < 6; ++k) { lo[k] = __ldcg(slo + (size_t)k * NY2 * NX4); hi[k] = __ldcg(shi + (size_t)k * NY2 * NX4); }
        taylor_shift_d<5>(lo, 0.5);
        taylor_shift_d<5>(hi, -0.5);
#pragma unroll
        for (int k = 0; k < 5; ++k) e[k] = 0.5 * (lo[k] + hi[k]);
      }
    } else if (slice < 3) {
      const double* src = ycoef + ((size_t)(rq * 5) * NY2 + (row + 1)) * NX4 + tcol;
#pragma unroll
      for (int k = 0; k < 5; ++k) e[k] = __ldcg(src + (size_t)k * NY2 * NX4);
      if (slice != 1) taylor_shift(e, slice == 0 ? -GAUSS_G : GAUSS_G, 4);
    } else {
      double lo[5], hi[5];
      const double* slo = ycoef + ((size_t)(rq * 5) * NY2 + row) * NX4 + tcol;
      const double* shi = slo + NX4;
#pragma unroll
      for (int k = 0; k < 5; ++k) { lo[k] = __ldcg(slo + (size_t)k * NY2 * NX4); hi[k] = __ldcg(shi + (size_t)k * NY2 * NX4); }
      taylor_shift(lo, 0.5, 4);
      taylor_shift(hi, -0.5, 4);
#pragma unroll
      for (int k = 0; k < 5; ++k) e[k] = 0.5 * (lo[k] + hi[k]);
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) ev[rq][k][col] = e[k];
  }
  __syncthreads();
  // a run's column c holds cell i = f0 + c - 2; a corner row uses the rows below and above
  auto nl = [&](int i, int row) {
    return slice < 3 ? cell_flag(P, flag, i, row)
                     : (cell_flag(P, flag, i, row - 1) | cell_flag(P, flag, i, row));
  };
  const int fi = fr.f0 + fr.ct, row = fr.line + fr.run;  // face x_{fi-1/2}
  double tc[NC][5];
  if constexpr (CHAR) {
    FlagTable& ft = *reinterpret_cast<FlagTable*>(smem_raw + ev_bytes<NC>());
    for (int c = threadIdx.x; c < ncol; c += SEG) ft.lin[c] = !nl(fr.f0 + c % w - 2, fr.line + c / w);
    __syncthreads();
    double a[NC][25], Wref[NC];  // Wref: cells next to the face point (the four around a corner)
    CkLead lead;
    if (fr.has_face) {
#pragma unroll
      for (int q = 0; q < NC; ++q) {
        if (slice < 3)
          Wref[q] = 0.5 * (fetch(P, st, 0, q, fi - 1, row, sv.t) + fetch(P, st, 0, q, fi, row, sv.t));
        else
          Wref[q] = 0.25 * (fetch(P, st, 0, q, fi - 1, row - 1, sv.t) + fetch(P, st, 0, q, fi, row - 1, sv.t) +
                            fetch(P, st, 0, q, fi - 1, row, sv.t) + fetch(P, st, 0, q, fi, row, sv.t));
      }
      char_face_point<NC, FLAGS, Q>(P, ev, ft, fr.col - 1, 0, a, lead, Wref);
    }
    ck_points<NC>(P, fr.nrun * (fr.nf + 1), fr.has_face, 0, a, lead, tc);
  } else {
    second_pass_cells<NC, FLAGS, Q>(P, smem_raw, fr, 0, FLAGS && fr.has_cell && nl(fi - 1, row), tc);
  }
  if (!fr.has_face) return;
  const double dt = sv.dt * P.ck.iL;  // in the coefficients' unit of time
  if (slice < 3) {
    double Fh[NC], We[NC];
    lobatto<NC>(tc, dt, P.gamma, 0, Fh, We);
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      const size_t o = ((size_t)(slice * NC + q) * P.ny + row) * (P.nx + 1) + fi;
      FX[o] = Fh[q];
      WX[o] = We[q];
    }
  } else {
#pragma unroll
    for (int q = 0; q < NC; ++q) WC[((size_t)q * (P.ny + 1) + row) * (P.nx + 1) + fi] = state_at(tc[q], dt);
  }
}

// y-face Gauss points (slice 0..2; lines are cell columns) of CTA b of the slice.
template <int NC, bool FLAGS, bool CHAR = false, bool Q = false>
__device__ __forceinline__ void yface_item(const Params& P, const StepView& sv, const double* st,
                                           const double* __restrict__ xcoef,
                                           const uint8_t* __restrict__ flag, double* __restrict__ FY,
                                           double* __restrict__ WY, int b, int slice,
                                           unsigned char* smem_raw) {
  double(*ev)[5][SPAN] = reinterpret_cast<double(*)[5][SPAN]>(smem_raw);
  const int NY4 = P.ny + 4;
  using namespace shweno_tables;
  const FaceRuns fr(P.ny + 1, P.nx, b);
  // a run's faces y_{f0-1/2} .. y_{f0+nf-3/2} have stencils that span its rows 0 .. nf + 2
  const int w = fr.nf + 3, nrow = fr.nrun * w;
  for (int it = threadIdx.x; it < 2 * NC * nrow; it += SEG) {
    const int r = it % nrow, rq = it / nrow;
    const int trow = fr.f0 + r % w, col = fr.line + r / w;
    double e[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    {
      constexpr int KC = Q ? 6 : 5;
      const double* src = xcoef + ((size_t)(rq * KC) * P.nx + col) * NY4 + trow;
#pragma unroll
      for (int k = 0; k < KC; ++k) e[k] = __ldcg(src + (size_t)k * P.nx * NY4);
      if constexpr (Q) {
        if (slice != 1) taylor_shift_d<5>(e, slice == 0 ? -GAUSS_G : GAUSS_G);
      } else {
        if (slice != 1) taylor_shift(e, slice == 0 ? -GAUSS_G : GAUSS_G, 4);
      }
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) ev[rq][k][r] = e[k];
  }
  __syncthreads();
  const int fj = fr.f0 + fr.ct, col = fr.line + fr.run;  // face y_{fj-1/2}
  double tc[NC][5];
  if constexpr (CHAR) {
    FlagTable& ft = *reinterpret_cast<FlagTable*>(smem_raw + ev_bytes<NC>());
    for (int c = threadIdx.x; c < nrow; c += SEG) ft.lin[c] = !cell_flag(P, flag, fr.line + c / w, fr.f0 + c % w - 2);
    __syncthreads();
    double a[NC][25], Wref[NC];
    CkLead lead;
    if (fr.has_face) {
#pragma unroll
      for (int q = 0; q < NC; ++q)
        Wref[q] = 0.5 * (fetch(P, st, 0, q, col, fj - 1, sv.t) + fetch(P, st, 0, q, col, fj, sv.t));
      char_face_point<NC, FLAGS, Q>(P, ev, ft, fr.col - 1, 1, a, lead, Wref);
    }
    ck_points<NC>(P, fr.nrun * (fr.nf + 1), fr.has_face, 1, a, lead, tc);
  } else {
    second_pass_cells<NC, FLAGS, Q>(P, smem_raw, fr, 1, FLAGS && fr.has_cell && cell_flag(P, flag, col, fj - 1), tc);
  }
  if (!fr.has_face) return;
  double Gh[NC], We[NC];
  lobatto<NC>(tc, sv.dt * P.ck.iL, P.gamma, 1, Gh, We);
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    const size_t o = ((size_t)(slice * NC + q) * (P.ny + 1) + fj) * P.nx + col;
    FY[o] = Gh[q];
    WY[o] = We[q];
  }
}

// Update of cell (i, j) (Eq. 3.2, 3.10) into `out`; returns the cell's CFL rate (0 when the new
// state is non-physical, which raises the control block's error word).
template <int NC>
__device__ __forceinline__ double update2d_cell(const Params& P, Ctl* __restrict__ ctl, const StepView& sv,
                                                const double* st,
                                                double* out, const double* __restrict__ FX,
                                                const double* __restrict__ WX,
                                                const double* __restrict__ FY,
                                                const double* __restrict__ WY,
                                                const double* __restrict__ WC, int i, int j) {
  const double dt = sv.dt;
  const int nx = P.nx, ny = P.ny;
  using namespace shweno_tables;
  const double gw[3] = {GAUSS_W0, GAUSS_W1, GAUSS_W0};
  double Wn[NC];
  const size_t cells = (size_t)nx * ny, c = (size_t)j * nx + i;
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    double fl = 0.0, fr = 0.0, gb = 0.0, gt = 0.0, wl = 0.0, wr = 0.0, wb = 0.0, wt = 0.0;
#pragma unroll
    for (int g = 0; g < 3; ++g) {
      const size_t ox = ((size_t)(g * NC + q) * ny + j) * (nx + 1) + i;
      const size_t oy = ((size_t)(g * NC + q) * (ny + 1) + j) * nx + i;
      fl += gw[g] * __ldcg(FX + ox);
      fr += gw[g] * __ldcg(FX + ox + 1);
      wl += gw[g] * __ldcg(WX + ox);
      wr += gw[g] * __ldcg(WX + ox + 1);
      gb += gw[g] * __ldcg(FY + oy);
      gt += gw[g] * __ldcg(FY + oy + nx);
      wb += gw[g] * __ldcg(WY + oy);
      wt += gw[g] * __ldcg(WY + oy + nx);
    }
    const size_t oc = ((size_t)q * (ny + 1) + j) * (nx + 1) + i;
    // the derivative averages scale by reciprocals of the mesh widths (set by the host), which
    // spares the FP64 pipe twelve divisions per cell
    const double z = (__ldcg(WC + oc + (nx + 1) + 1) - __ldcg(WC + oc + (nx + 1)) - __ldcg(WC + oc + 1) + __ldcg(WC + oc)) * P.idxy;
    Wn[q] = __ldcg(st + q * cells + c) - dt / P.dx * (fr - fl) - dt / P.dy * (gt - gb);
    out[q * cells + c] = Wn[q];
    out[(NC + q) * cells + c] = (wr - wl) * P.idx;
    out[(2 * NC + q) * cells + c] = (wt - wb) * P.idy;
    out[(3 * NC + q) * cells + c] = z;
  }
  if (!cell_physical(P, Wn)) {
    atomicCAS(&ctl->err, ERR_NONE, ERR_NONPHYSICAL);
    __threadfence();  // before this CTA counts as done
    return 0.0;
  }
  return cell_rate(P, Wn);
}

}  // namespace shweno
