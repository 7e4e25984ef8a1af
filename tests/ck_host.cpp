// Host program of tests/test_ck_host.py: one step of the 1D Euler recursion at random points, the
// library's form (ck_fixed.cuh) and FP64 throughout against long double.  Prints, per gamma, the largest
// error of each component of the state after the step, relative to rho, rho c and E: library, FP64; and the
// same for steep points (every coefficient as large as the state) of any velocity up to Mach 0.7, root mean
// square, relative to the sum of the time series' terms.
#include <cmath>
#include <cstdio>
#include <random>

#include "ck_fixed.cuh"

using namespace shweno;
typedef long double T;

static void recursion(const double (&a)[3][25], T g, T (&tc)[3][5]) {
  T S[3][5][5], u[5][5], mu[5][5], p[5][5], H[5][5], F[3][5];
  for (int q = 0; q < 3; ++q)
    for (int m = 0; m < 5; ++m) S[q][m][0] = a[q][m * 5];
  for (int k = 0; k < 4; ++k) {
    for (int m = 0; m + k < 5; ++m) {
      T s = S[1][m][k];
      for (int i = 0; i <= m; ++i)
        for (int t = 0; t <= k; ++t)
          if (i + t) s -= S[0][i][t] * u[m - i][k - t];
      u[m][k] = s / S[0][0][0];
      mu[m][k] = 0;
      for (int i = 0; i <= m; ++i)
        for (int t = 0; t <= k; ++t) mu[m][k] += S[1][i][t] * u[m - i][k - t];
      p[m][k] = (g - 1) * (S[2][m][k] - mu[m][k] / 2);
      H[m][k] = S[2][m][k] + p[m][k];
      F[0][m] = S[1][m][k];
      F[1][m] = mu[m][k] + p[m][k];
      F[2][m] = 0;
      for (int i = 0; i <= m; ++i)
        for (int t = 0; t <= k; ++t) F[2][m] += u[i][t] * H[m - i][k - t];
    }
    for (int q = 0; q < 3; ++q)
      for (int m = 0; m + k < 4; ++m) S[q][m][k + 1] = -(m + 1) * F[q][m + 1] / (k + 1);
  }
  for (int q = 0; q < 3; ++q)
    for (int k = 0; k < 5; ++k) tc[q][k] = S[q][0][k];
}

// Largest difference between the library's step at a state and at the same state in other units (powers of two,
// which FP64 carries exactly), relative to the state: small or large density and velocity.
static void units() {
  std::mt19937_64 rng(3);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  CkFixed C;
  finalize_ck_fixed(C, 1, 1.0, 1.0, 1.4);
  for (int er : {0, -200, -299, -301, -330, -400, 300, 500})
    for (int ev : {0, 20, -20, -100, -290, -305}) {
      double worst = 0.0;
      for (int it = 0; it < 200; ++it) {
        double a[2][3][25] = {}, t[2][3][5];
        const double W[3] = {1.0 + 0.3 * U(rng), 0.4 * U(rng), 2.5 + 0.3 * U(rng)};
        for (int q = 0; q < 3; ++q)
          for (int s = 0; s < 5; ++s) {
            a[0][q][s * 5] = s == 0 ? W[q] : std::ldexp(U(rng), -3 * s);
            a[1][q][s * 5] = std::ldexp(a[0][q][s * 5], er + q * ev);
          }
        for (int v = 0; v < 2; ++v) {
          const double ir = 1.0 / a[v][0][0], u = a[v][1][0] * ir, p = 0.4 * (a[v][2][0] - 0.5 * a[v][1][0] * u);
          const CkLead lead{ir, fx_hi(u) & 0x7fffffff, fx_hi((a[v][2][0] + p) * ir) & 0x7fffffff, fx_hi(std::sqrt(1.4 * p * ir)) & 0x7fffffff};
          ck_fixed<3, 1>(a[v], lead, C, t[v]);
        }
        for (int q = 0; q < 3; ++q)
          for (int k = 1; k < 5; ++k) {
            const double unit = std::ldexp(1.0, er + (q + k) * ev);  // 0 or denormal: out of a double's range
            if (unit > 1e-290 && unit < 1e290) worst = std::fmax(worst, std::fabs(t[1][q][k] / unit - t[0][q][k]));
          }
      }
      std::printf("%d %d %.3e\n", er, ev, worst);
    }
}

int main(int argc, char**) {
  if (argc > 1) {
    units();
    return 0;
  }
  std::mt19937_64 rng(1);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  for (double g : {1.001, 1.02, 1.1, 1.2, 1.4, 5.0 / 3.0, 3.0, 4.0, 7.0, 30.0, 1e3, 1e6}) {
    CkFixed C;
    finalize_ck_fixed(C, 1, 1.0, 1.0, g);
    double lib[3] = {}, fp[3] = {};
    // a density wave of any shape at uniform pressure and Mach 0.05 of c = sqrt(gamma)
    const double vel = 0.05 * std::sqrt(g);
    for (int it = 0; it < 2000; ++it) {
      double a[3][25] = {}, f = 1.0;
      a[0][0] = 1.0 + 0.3 * U(rng);
      for (int s = 1; s < 5; ++s) a[0][s * 5] = (f *= 0.1) * U(rng);
      for (int s = 0; s < 5; ++s) {
        a[1][s * 5] = a[0][s * 5] * vel;
        a[2][s * 5] = 0.5 * a[0][s * 5] * vel * vel + (s == 0 ? 1.0 / (g - 1.0) : 0.0);
      }
      const double ir = 1.0 / a[0][0], u = a[1][0] * ir, p = (g - 1.0) * (a[2][0] - 0.5 * a[1][0] * u);
      const CkLead lead{ir, fx_hi(u) & 0x7fffffff, fx_hi((a[2][0] + p) * ir) & 0x7fffffff, fx_hi(std::sqrt(g * p * ir)) & 0x7fffffff};
      double tl[3][5], td[3][5];
      T tt[3][5];
      ck_fixed<3, 1>(a, lead, C, tl);
      ck_euler1d(a, td, C.gm1);
      recursion(a, g, tt);
      const T tau = 0.5 / std::sqrt(g);
      for (int q = 0; q < 3; ++q) {
        T sl = 0, sd = 0, st = 0;
        for (int k = 4; k > 0; --k) sl = (sl + tl[q][k]) * tau, sd = (sd + td[q][k]) * tau, st = (st + tt[q][k]) * tau;
        const T w = q == 1 ? a[0][0] * std::sqrt(g * p * ir) : a[q][0];
        lib[q] = std::fmax(lib[q], (double)(std::fabs(sl - st) / w));
        fp[q] = std::fmax(fp[q], (double)(std::fabs(sd - st) / w));
      }
    }
    double sl2[3] = {}, sf2[3] = {};
    for (int it = 0; it < 2000; ++it) {
      double a[3][25] = {};
      const double rho = 1.0 + 0.3 * U(rng), p = 1.0 + 0.3 * U(rng), u = 0.7 * std::sqrt(g) * U(rng);
      const double W[3] = {rho, rho * u, p / (g - 1.0) + 0.5 * rho * u * u};
      for (int q = 0; q < 3; ++q)
        for (int s = 0; s < 5; ++s) a[q][s * 5] = s == 0 ? W[q] : U(rng) * (q == 0 ? 1.0 : q == 1 ? std::sqrt(g) : W[2]);
      const double ir = 1.0 / rho, v = W[1] * ir, pp = (g - 1.0) * (W[2] - 0.5 * W[1] * v), c = std::sqrt(g * pp * ir);
      const CkLead lead{ir, fx_hi(v) & 0x7fffffff, fx_hi((W[2] + pp) * ir) & 0x7fffffff, fx_hi(c) & 0x7fffffff};
      double tl[3][5], td[3][5];
      T tt[3][5];
      ck_fixed<3, 1>(a, lead, C, tl);
      ck_euler1d(a, td, C.gm1);
      recursion(a, g, tt);
      const T tau = 0.3 / std::sqrt(g);
      for (int q = 0; q < 3; ++q) {
        T el = 0, ef = 0, sum = 0;
        for (int k = 4; k > 0; --k) {
          el = (el + tl[q][k] - tt[q][k]) * tau;
          ef = (ef + td[q][k] - tt[q][k]) * tau;
          sum = (sum + std::fabs(tt[q][k])) * tau;
        }
        const T w = (q == 1 ? rho * c : std::fabs(W[q])) + sum;
        sl2[q] += (double)(el / w * el / w);
        sf2[q] += (double)(ef / w * ef / w);
      }
    }
    std::printf("%g %.3e %.3e %.3e %.3e %.3e %.3e ", g, lib[0], lib[1], lib[2], fp[0], fp[1], fp[2]);
    for (int q = 0; q < 3; ++q) std::printf("%.3e %.3e%s", std::sqrt(sl2[q] / 2000), std::sqrt(sf2[q] / 2000), q < 2 ? " " : "\n");
  }
}
