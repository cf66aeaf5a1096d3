// Checks csrc/fixed64.cuh on the host where the sizes within a cell are far
// apart: its collision and FP64 arithmetic (the operations of the FP64 form,
// csrc/lbm_kernels.cu) against the same equations in 113 bits, each with the
// exponents the kernels take.  One line per setting: kind, relaxation, sizes,
// weight, cells, cells outside the range, and per class of results (rest,
// face and edge directions, mass, momentum, force) the rms error of either
// form and what the inputs carry already, the error of having been stored in
// FP64, all relative to the cell's largest |d| (force: the largest |B (U - V - f)|).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>

#include "fixed64.cuh"
using namespace psm;
#ifdef __SIZEOF_FLOAT128__
typedef __float128 wide;
#else
typedef long double wide;  // 113 bits where there is no __float128
#endif

static const int CX[9] = {1, 0, 0, 1, 1, 1, 1, 0, 0}, CY[9] = {0, 1, 0, 1, -1, 0, 0, 1, 1},
                 CZ[9] = {0, 0, 1, 0, 0, 1, -1, 1, -1};
template <typename T>
static T wk(int k) { return k < 3 ? T(1) / T(18) : T(1) / T(36); }
static double rnd() { return 2.0 * drand48() - 1.0; }
static double absw(wide v) { return (double)(v < 0 ? -v : v); }

// Eqs. 3-8 and 17-21 on deviations, one particle of weight V[3]
static void reference(const double* din, double wp_, double wm_, const double* f_, const double* V,
                      wide* o, wide* Fc) {
  const wide wp = wp_, wm = wm_, one = 1, two = 2;
  wide d[19], f[3], s[9], a[9], R, j[3] = {0, 0, 0}, U[3], v[3];
  for (int q = 0; q < 19; ++q) d[q] = din[q];
  R = d[0];
  for (int k = 0; k < 9; ++k) {
    s[k] = d[2 * k + 1] + d[2 * k + 2];
    a[k] = d[2 * k + 1] - d[2 * k + 2];
    R += s[k];
    j[0] += a[k] * CX[k];
    j[1] += a[k] * CY[k];
    j[2] += a[k] * CZ[k];
  }
  for (int i = 0; i < 3; ++i) {
    f[i] = f_[i];
    v[i] = V[i];
    U[i] = j[i] + f[i] / two;
  }
  const wide uu = U[0] * U[0] + U[1] * U[1] + U[2] * U[2];
  const wide uf = U[0] * f[0] + U[1] * f[1] + U[2] * f[2];
  const wide dU = (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]) - uu;
  const wide gp = one - wp / two, gm = one - wm / two, B = V[3];
  const wide f0 = d[0] * (one - wp) + wp / 3 * (R - uu * 3 / 2) - gp * uf;
  o[0] = (one - B) * f0 + B * (d[0] - dU / two);
  for (int k = 0; k < 9; ++k) {
    const wide w = wk<wide>(k), x = CX[k], y = CY[k], z = CZ[k];
    const wide cu = x * U[0] + y * U[1] + z * U[2], cf = x * f[0] + y * f[1] + z * f[2];
    const wide cv = x * v[0] + y * v[1] + z * v[2];
    const wide S = (one - wp) / two * s[k] + wp * w * (R - uu * 3 / 2 + cu * cu * 9 / 2) +
                   gp * w * (9 * cf * cu - 3 * uf);
    const wide A = (one - wm) / two * a[k] + 3 * w * (wm * cu + gm * cf);
    const wide e = w * ((cv * cv - cu * cu) * 9 / 2 - dU * 3 / 2), t = 3 * w * (cu + cv);
    o[2 * k + 1] = (one - B) * (S + A) + B * (d[2 * k + 2] + e + t);
    o[2 * k + 2] = (one - B) * (S - A) + B * (d[2 * k + 1] + e - t);
  }
  for (int i = 0; i < 3; ++i) Fc[i] = B * (U[i] - v[i] - f[i]);
}

// the FP64 form's operations, products and sums fused as the compiler does
static double dot(int k, const double* u) {
  const double t[9] = {u[0], u[1], u[2], u[0] + u[1], u[0] - u[1], u[0] + u[2], u[0] - u[2],
                       u[1] + u[2], u[1] - u[2]};
  return t[k];
}
static void fp64(int kind, const double* din, double wp, double wm, const double* f,
                 const double* V, double* d, double* Fc) {
  double s[9], a[9];
  for (int k = 0; k < 9; ++k) {
    s[k] = din[2 * k + 1] + din[2 * k + 2];
    a[k] = din[2 * k + 1] - din[2 * k + 2];
  }
  const double drho = ((din[0] + (s[0] + s[1])) + ((s[2] + s[3]) + (s[4] + s[5]))) +
                      ((s[6] + s[7]) + s[8]);
  const double U[3] = {((a[0] + a[3]) + (a[4] + a[5])) + a[6] + 0.5 * f[0],
                       ((a[1] + a[3]) - (a[4] - a[7])) + a[8] + 0.5 * f[1],
                       ((a[2] + a[5]) - (a[6] - a[7])) - a[8] + 0.5 * f[2]};
  auto dot3 = [](const double* x, const double* y) {
    return std::fma(x[2], y[2], std::fma(x[0], y[0], x[1] * y[1]));
  };
  const double gp = 1.0 - 0.5 * wp, gm = 1.0 - 0.5 * wm;
  const double uu = dot3(U, U), uf = dot3(U, f), base = std::fma(-1.5, uu, drho);
  const double W[3] = {1.0 / 3.0, 1.0 / 18.0, 1.0 / 36.0};
  auto C = [&](int c) { return std::fma(wp * W[c], base, (-3.0 * W[c] * gp) * uf); };
  const double C0 = C(1), C1 = C(2);
  if (kind == FX_FLUID) {
    d[0] = std::fma(1.0 - wp, din[0], C(0));
    for (int k = 0; k < 9; ++k) {
      const double w = wk<double>(k), cu = dot(k, U), cf = dot(k, f);
      const double X = std::fma(std::fma(4.5 * w * wp, cu, gp * 9.0 * w * cf), cu, k < 3 ? C0 : C1);
      const double Y = std::fma(3.0 * w * wm, cu, gm * 3.0 * w * cf);
      const double S = std::fma(0.5 * (1.0 - wp), s[k], X), A = std::fma(0.5 * (1.0 - wm), a[k], Y);
      d[2 * k + 1] = S + A;
      d[2 * k + 2] = S - A;
    }
    return;
  }
  const double B = V[3], omB = 1.0 - B, dU2 = dot3(V, V) - uu, BdU = B * dU2;
  d[0] = std::fma((-1.5 * W[0]), BdU, std::fma(omB, std::fma(-wp, din[0], C(0)), din[0]));
  const double as = std::fma(omB, -0.5 * wp, 0.5), aa = std::fma(omB, -0.5 * wm, 0.5 - B);
  for (int k = 0; k < 9; ++k) {
    const double w = wk<double>(k), cu = dot(k, U), cv = dot(k, V), cf = dot(k, f);
    const double c45 = (4.5 * w) * B, c3 = (3.0 * w) * B, cd = (-1.5 * w) * BdU;
    const double al = std::fma(omB, 4.5 * w * wp, -c45), ga = std::fma(omB, k < 3 ? C0 : C1, cd);
    const double de = std::fma(omB, 3.0 * w * wm, c3);
    const double sy = std::fma(std::fma(al, cu, omB * (gp * 9.0 * w * cf)), cu, ga);
    const double S = std::fma(as, s[k], std::fma(c45 * cv, cv, sy));
    const double an = std::fma(de, cu, std::fma(c3, cv, omB * (gm * 3.0 * w * cf)));
    const double A = std::fma(aa, a[k], an);
    d[2 * k + 1] = S + A;
    d[2 * k + 2] = S - A;
  }
  for (int i = 0; i < 3; ++i) Fc[i] = B * ((U[i] - V[i]) - f[i]);
}

// the fixed-point form as the kernels call it; false: outside its range
static bool fixed(int kind, const FxRates& c, const double* d, const double* f, const double* V,
                  double* o, double* Fc) {
  const int E0 = fx_e0(c, f);
  const FxRange r = kind == FX_FLUID ? fx_range<FX_FLUID>(d, V, E0) : fx_range<FX_MIXED>(d, V, E0);
  if (r.slow) return false;
  FxRow re, rm, rp;  // a row for each call, as the kernels' table has
  int calls = 0;
  auto rowE = [&](int E) -> const FxRow& {
    FxRow& r = calls++ ? rm : re;
    fx_row_at(c, f, E0 + std::min(E - E0, FX_ROWS - 1), fx_p0(E0), r);
    return r;
  };
  auto rowP = [&](int P) -> const FxRow& {
    fx_row_at(c, f, E0, fx_p0(E0) + std::min(P - fx_p0(E0), FX_ROWS - 1), rp);
    return rp;
  };
  auto put = [&](int q, double v) { o[q] = v; };
  auto force = [&](const double* F) {
    for (int i = 0; i < 3; ++i) Fc[i] = F[i];
  };
  if (kind == FX_FLUID) fx_cell<FX_FLUID>(c, rowE, rowP, E0, r.E, r.Ps, d, V, force, put);
  else fx_cell<FX_MIXED>(c, rowE, rowP, E0, r.E, r.Ps, d, V, force, put);
  return true;
}

struct Err {
  double e2[6] = {};
  long n[6] = {};
  void add(int c, double v) {
    e2[c] += v * v;
    ++n[c];
  }
  double rms(int c) const { return n[c] ? std::sqrt(e2[c] / (double)n[c]) : 0.0; }
};

// Values of any sign up to the largest that an exponent admits, signs that add
// up in places, forces and velocities up to theirs: per kind the largest error
// of the 18 moving directions in units of 2^(E - 59), of the rest direction in
// units of 2^(E - 53) and of the force in units of 2^-56 of B times the largest
// |d_q|, |U|, |V|, each less the final rounding; and the largest |d_q| taken.
static int wild(int cells) {
  for (int kind = 0; kind < 2; ++kind) {
    double worst = 0.0, rest = 0.0, ferr = 0.0, largest = 0.0;
    int in = 0;
    for (int n = 0; n < cells; ++n) {
      const double tau = 0.5 + std::exp(-6.0 + 8.0 * drand48());
      const double wp = 1.0 / tau, wm = n % 2 ? 1.0 / (0.5 + 0.1875 / (tau - 0.5)) : wp;
      FxRates c;
      fx_fill(c, wp, wm);
      const double um = 0.125 * std::exp2(-(n % 5 < 2 ? 4.0 * drand48() : 40.0 * drand48()));
      const double sg = drand48() < 0.5 ? -1.0 : 1.0, dir[3] = {rnd(), rnd(), rnd()};
      double f[3], V[4], d[19];
      for (int q = 0; q < 19; ++q) {
        const double top = um * (q == 0 ? 8.0 : (q < 7 ? 1.0 : 0.5));
        switch (n % 4) {
          case 0: d[q] = sg * top * (0.999 - 0.1 * drand48()); break;  // density
          case 1: d[q] = top * rnd(); break;
          case 2: d[q] = top * rnd() * std::exp(20.0 * (drand48() - 1.0)); break;
          default: {  // momentum along dir
            const int k = (q - 1) / 2;
            const double c1 = q ? CX[k] * dir[0] + CY[k] * dir[1] + CZ[k] * dir[2] : 0.0;
            d[q] = q == 0 ? 0.0 : (q % 2 ? 1.0 : -1.0) * (c1 > 0 ? 0.999 : -0.999) * top;
          }
        }
      }
      const double fm = n % 3 ? um * std::exp2(-8.0 * drand48()) : 0.0;
      const double vm = um * std::exp2(12.0 * drand48() - 4.0);
      for (int i = 0; i < 3; ++i) {
        f[i] = fm * rnd();
        V[i] = vm < 1.0 ? vm * (n % 5 ? rnd() : 0.999 * sg) : 0.0;
      }
      V[3] = n % 6 == 0 ? 1.0 : (n % 6 == 1 ? 0.0 : std::exp(12.0 * (drand48() - 1.0)));
      if (kind == FX_FLUID) V[0] = V[1] = V[2] = V[3] = 0.0;
      double o[19], F[3] = {0, 0, 0};
      wide r[19], Fr[3];
      if (!fixed(kind, c, d, f, V, o, F)) continue;
      ++in;
      const FxRange g = kind ? fx_range<FX_MIXED>(d, V, fx_e0(c, f))
                             : fx_range<FX_FLUID>(d, V, fx_e0(c, f));
      reference(d, wp, wm, f, V, r, Fr);
      for (int q = 0; q < 19; ++q) {
        const double e = absw((wide)o[q] - r[q]) - 0x1p-53 * std::fabs(o[q]);
        if (q == 0) rest = std::max(rest, std::ldexp(e, 53 - g.E));
        else {
          worst = std::max(worst, std::ldexp(e, 59 - g.E));
          largest = std::max(largest, std::fabs(d[q]));
        }
      }
      if (kind && V[3] > 0.0) {
        double top = um;
        for (int i = 0; i < 3; ++i)
          top = std::max(top, absw(Fr[i]) / V[3] + std::fabs(V[i]) + std::fabs(f[i]));
        for (int i = 0; i < 3; ++i)
          ferr = std::max(ferr, (absw((wide)F[i] - Fr[i]) - 0x1p-53 * std::fabs(F[i])) /
                                    (V[3] * top * 0x1p-56));
      }
    }
    std::printf("%d %d %d %.3f %.3f %.3f %g\n", kind, cells, in, worst, rest, ferr, largest);
  }
  return 0;
}

// variance of the rounding error that FP64 leaves in v
static double stored(double v) {
  int e;
  if (v == 0.0) return 0.0;
  std::frexp(v, &e);
  return std::ldexp(1.0, 2 * (e - 53)) / 12.0;
}

int main(int argc, char** argv) {
  const int cells = argc > 2 ? std::atoi(argv[2]) : 400;
  if (argc > 1 && argv[1][0] == 'w') return wild(cells);
  const double taus[] = {0.505, 0.55, 1.0, 5.0}, vel[] = {1e-5, 2e-2};
  const double dens[] = {0.0, 1e-4, 1e-2, 1.0, 1e2, 1e4};
  const double fu[] = {0.0, 1e-3, 1.0, 1e2}, Vu[] = {0.0, 1.0, 30.0, 1000.0};
  const double Bs[] = {0.0, 1e-5, 2e-3, 0.7, 1.0};
  const double noneq = 0.02;
  for (int kind = 0; kind < 2; ++kind)
    for (double tau : taus)
      for (double um : vel)
        for (double dr : dens)
          for (double fr : fu)
            for (double vr : Vu)
              for (double B : Bs) {
                if (kind == FX_FLUID && (vr != 0.0 || B != 0.0)) continue;
                if (kind == FX_MIXED && fr != 0.0 && vr != 1.0) continue;
                if (um * dr > 0.2 || um * fr > 1e-3 || um * vr > 0.2) continue;
                const bool trt = tau == 0.55 || tau == 5.0;
                const double wp = 1.0 / tau, wm = trt ? 1.0 / (0.5 + 0.1875 / (tau - 0.5)) : wp;
                FxRates c;
                fx_fill(c, wp, wm);
                Err en, eo, st;
                int out = 0;
                for (int n = 0; n < cells; ++n) {
                  double u[3], f[3], V[4], d[19], uu = 0.0;
                  const double rho = um * dr * rnd();
                  for (int i = 0; i < 3; ++i) {
                    u[i] = um * rnd();
                    f[i] = um * fr * rnd();
                    V[i] = um * vr * rnd();
                    uu += u[i] * u[i];
                  }
                  V[3] = B;
                  // near equilibrium: the rest of each pair's sum and
                  // difference relative to the size of that kind
                  const double ns = noneq * std::max(um * dr, uu), na = noneq * um;
                  d[0] = (rho - 1.5 * uu + ns * rnd()) / 3.0;
                  for (int k = 0; k < 9; ++k) {
                    const double cu = dot(k, u), w = wk<double>(k);
                    const double S = rho + 4.5 * cu * cu - 1.5 * uu + ns * rnd();
                    const double A = 3.0 * cu + na * rnd();
                    d[2 * k + 1] = w * (S + A);
                    d[2 * k + 2] = w * (S - A);
                  }
                  double o[19], p[19], Fo[3] = {0, 0, 0}, Fp[3] = {0, 0, 0};
                  wide r[19], Fr[3];
                  if (!fixed(kind, c, d, f, V, o, Fo)) {
                    ++out;
                    continue;
                  }
                  reference(d, wp, wm, f, V, r, Fr);
                  fp64(kind, d, wp, wm, f, V, p, Fp);
                  double big = 0.0, fbig = 0.0;
                  for (int q = 0; q < 19; ++q)
                    big = std::max(big, std::max(absw(r[q]), std::fabs(d[q])));
                  for (int i = 0; i < 3; ++i) fbig = std::max(fbig, absw(Fr[i]));
                  if (big == 0.0) continue;
                  double v[19], vm = 0.0, vj[3] = {0, 0, 0};
                  for (int q = 0; q < 19; ++q) {
                    v[q] = stored(d[q]);
                    vm += v[q];
                    const int k = (q - 1) / 2;
                    if (q) {
                      vj[0] += v[q] * CX[k] * CX[k];
                      vj[1] += v[q] * CY[k] * CY[k];
                      vj[2] += v[q] * CZ[k] * CZ[k];
                    }
                  }
                  for (int q = 0; q < 19; ++q)
                    st.add(q == 0 ? 0 : (q < 7 ? 1 : 2), std::sqrt(q ? v[q] : vm / 9.0) / big);
                  st.add(3, std::sqrt(vm) / big);
                  for (int i = 0; i < 3; ++i) {
                    st.add(4, std::sqrt(vj[i]) / big);
                    if (fbig > 0.0) st.add(5, B * std::sqrt(vj[i]) / fbig);
                  }
                  auto tally = [&](const double* y, const double* F, Err& e) {
                    wide mass = 0, mom[3] = {0, 0, 0};
                    for (int q = 0; q < 19; ++q) {
                      const wide x = (wide)y[q] - r[q];
                      mass += x;
                      if (q) {
                        const int k = (q - 1) / 2, s = q % 2 ? 1 : -1;
                        mom[0] += x * (s * CX[k]);
                        mom[1] += x * (s * CY[k]);
                        mom[2] += x * (s * CZ[k]);
                      }
                      e.add(q == 0 ? 0 : (q < 7 ? 1 : 2), absw(x) / big);
                    }
                    e.add(3, absw(mass) / big);
                    for (int i = 0; i < 3; ++i) {
                      e.add(4, absw(mom[i]) / big);
                      if (fbig > 0.0) e.add(5, absw((wide)F[i] - Fr[i]) / fbig);
                    }
                  };
                  tally(o, Fo, en);
                  tally(p, Fp, eo);
                }
                std::printf("%d %g %g %g %g %g %g %d %d", kind, tau, um, dr, fr, vr, B, cells, out);
                for (int i = 0; i < 6; ++i)
                  std::printf(" %.4g %.4g %.4g", en.rms(i), eo.rms(i), st.rms(i));
                std::printf("\n");
              }
  return 0;
}
