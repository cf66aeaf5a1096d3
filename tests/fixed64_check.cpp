// Checks csrc/fixed64.cuh on the host: its collisions against the same
// equations in long double (64 or more significant bits), beside the FP64
// collision written out as the FP64 form evaluates them.  Prints one line per
// setting: kind, largest error in units of 2^(E - 57) less the final rounding,
// rms error of the fixed-point and of the FP64 form (of the largest |d|),
// and the number of cells outside the fixed-point range.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>

#include "fixed64.cuh"
using namespace psm;

static const int CX[9] = {1, 0, 0, 1, 1, 1, 1, 0, 0}, CY[9] = {0, 1, 0, 1, -1, 0, 0, 1, 1},
                 CZ[9] = {0, 0, 1, 0, 0, 1, -1, 1, -1};
template <typename T>
static T wk(int k) { return k < 3 ? T(1) / T(18) : T(1) / T(36); }

// Eqs. 3-8 and 17-21 on deviations, one particle of weight V[3]
template <typename T>
static void collide(const double* din, double wp_, double wm_, const double* f_, const double* V,
                    T* o, T* Fc) {
  const T wp = wp_, wm = wm_, one = 1, two = 2;
  T d[19], f[3], s[9], a[9], R, j[3] = {0, 0, 0}, U[3], v[3];
  for (int q = 0; q < 19; ++q) d[q] = din[q];
  R = d[0];
  for (int k = 0; k < 9; ++k) {
    s[k] = d[2 * k + 1] + d[2 * k + 2];
    a[k] = d[2 * k + 1] - d[2 * k + 2];
    R += s[k];
    j[0] += a[k] * T(CX[k]);
    j[1] += a[k] * T(CY[k]);
    j[2] += a[k] * T(CZ[k]);
  }
  for (int i = 0; i < 3; ++i) {
    f[i] = f_[i];
    v[i] = V[i];
    U[i] = j[i] + f[i] / two;
  }
  const T uu = U[0] * U[0] + U[1] * U[1] + U[2] * U[2];
  const T uf = U[0] * f[0] + U[1] * f[1] + U[2] * f[2];
  const T dU = (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]) - uu;
  const T gp = one - wp / two, gm = one - wm / two, B = V[3];
  const T f0 = d[0] * (one - wp) + wp / T(3) * (R - T(1.5) * uu) - gp * uf;
  o[0] = (one - B) * f0 + B * (d[0] - dU / two);
  for (int k = 0; k < 9; ++k) {
    const T w = wk<T>(k), x = CX[k], y = CY[k], z = CZ[k];
    const T cu = x * U[0] + y * U[1] + z * U[2], cf = x * f[0] + y * f[1] + z * f[2];
    const T cv = x * v[0] + y * v[1] + z * v[2];
    const T S = (one - wp) / two * s[k] + wp * w * (R - T(1.5) * uu + T(4.5) * cu * cu) +
                gp * w * (T(9) * cf * cu - T(3) * uf);
    const T A = (one - wm) / two * a[k] + T(3) * w * (wm * cu + gm * cf);
    const T e = w * (T(4.5) * (cv * cv - cu * cu) - T(1.5) * dU), t = T(3) * w * (cu + cv);
    o[2 * k + 1] = (one - B) * (S + A) + B * (d[2 * k + 2] + e + t);
    o[2 * k + 2] = (one - B) * (S - A) + B * (d[2 * k + 1] + e - t);
  }
  for (int i = 0; i < 3; ++i) Fc[i] = B * (U[i] - v[i] - f[i]);
}

static double rnd() { return 2.0 * drand48() - 1.0; }

int main() {
  // a covered cell of any weight, of weight 1, and none (B = 0), in the part form
  const char* names[] = {"fluid", "mixed", "full", "none"};
  for (int kind = 0; kind < 4; ++kind)
    for (double tau : {0.505, 0.55, 0.6, 1.0, 5.0})
      for (int trt = 0; trt < 2; ++trt)
        for (double um : {1e-12, 1e-5, 1e-3, 2e-2, 0.3})
          for (double fm : {0.0, 1e-6})
            for (int wild = 0; wild < 2; ++wild) {
              const double wp = 1.0 / tau, wm = trt ? 1.0 / (0.5 + 0.1875 / (tau - 0.5)) : wp;
              FxRates c;
              fx_fill(c, wp, wm);
              double worst = 0.0, sn = 0.0, so = 0.0, ferr = 0.0;
              int out = 0, cells = 0;
              for (int n = 0; n < 400; ++n) {
                double f[3] = {fm * rnd(), fm * rnd(), fm * rnd()}, V[4], d[19];
                for (int i = 0; i < 3; ++i) V[i] = um * rnd();
                V[3] = kind == 2 ? 1.0 : (n % 7 == 0 ? 0.0 : drand48());
                if (kind == FX_FLUID || kind == 3) V[0] = V[1] = V[2] = V[3] = 0.0;
                if (wild) {  // any values below um, signs that add up in places
                  for (int q = 0; q < 19; ++q)
                    d[q] = um * (n % 3 == 0 ? (n % 2 ? 1.0 : -1.0) * (0.9 + 0.1 * drand48())
                                            : (n % 3 == 1 ? rnd() : rnd() * std::exp(20.0 * rnd())));
                  for (int q = 0; q < 19; ++q) d[q] = std::max(-um, std::min(um, d[q]));
                  if (n % 9 == 0)
                    for (int k = 0; k < 9; ++k) {  // momentum along (1, 1, 1)
                      const int s = CX[k] + CY[k] + CZ[k];
                      d[2 * k + 1] = um * (s > 0 ? 0.999 : 0.0);
                      d[2 * k + 2] = -d[2 * k + 1];
                    }
                } else {  // near equilibrium
                  const double u[3] = {um * rnd(), um * rnd(), um * rnd()};
                  const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2], dr = 0.1 * um * rnd();
                  d[0] = (dr - 1.5 * uu) / 3.0;
                  for (int k = 0; k < 9; ++k) {
                    const double cu = CX[k] * u[0] + CY[k] * u[1] + CZ[k] * u[2];
                    for (int m = 0; m < 2; ++m)
                      d[2 * k + 1 + m] = wk<double>(k) * (dr + (m ? -3 : 3) * cu + 4.5 * cu * cu -
                                                          1.5 * uu + 0.05 * um * rnd());
                  }
                }
                const int E0 = fx_e0(c, f);
                int top = fx_top(d);
                if (kind != FX_FLUID)
                  top = fx_top_velocity(top, V, FX_VBITS_MIXED);
                const int E = fx_exponent(top, E0) + (kind != FX_FLUID ? 1 : 0);
                ++cells;
                if (E > (kind == FX_FLUID ? FX_EMAX : FX_EMAX_SOLID)) {
                  ++out;
                  continue;
                }
                FxRow row;
                fx_row(c, f, E0, std::min(E - E0, FX_ROWS - 1), row);
                double o[19], Fc[3] = {0, 0, 0};
                auto put = [&](int q, double v) { o[q] = v; };
                auto force = [&](const double* F) {
                  for (int i = 0; i < 3; ++i) Fc[i] = F[i];
                };
                if (kind == FX_FLUID) fx_collide<FX_FLUID>(c, row, E, d, V, force, put);
                else fx_collide<FX_MIXED>(c, row, E, d, V, force, put);
                long double r[19], Fr[3];
                double p[19], Fp[3];
                collide<long double>(d, wp, wm, f, V, r, Fr);
                collide<double>(d, wp, wm, f, V, p, Fp);
                const double unit = std::ldexp(1.0, E - 57);
                double big = 0.0;
                for (int q = 0; q < 19; ++q) big = std::max(big, (double)std::fabs(r[q]));
                if (big == 0.0) continue;
                for (int q = 0; q < 19; ++q) {
                  const double en = (double)((long double)o[q] - r[q]);
                  const double eo = (double)((long double)p[q] - r[q]);
                  worst = std::max(worst, (std::fabs(en) - 0x1p-53 * std::fabs(o[q])) / unit);
                  sn += en * en / (big * big);
                  so += eo * eo / (big * big);
                }
                if (kind != FX_FLUID)
                  for (int i = 0; i < 3; ++i)
                    ferr = std::max(ferr, (std::fabs((double)((long double)Fc[i] - Fr[i])) -
                                           0x1p-53 * std::fabs(Fc[i])) / unit);
              }
              const double m = 19.0 * std::max(1, cells - out);
              std::printf("%s %d %g %d %g %g %.3f %.3f %.4g %.4g %d %d\n", names[kind], wild, tau, trt,
                          um, fm, worst, ferr, std::sqrt(sn / m), std::sqrt(so / m), out, cells);
            }
  return 0;
}
