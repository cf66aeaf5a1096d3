// fixed64.cuh -- the collision's linear algebra in per-cell block fixed point:
// 64-bit integers that share one exponent per cell.
//
// GB300 executes an FP64 operation at 1/64 of the FP32 rate (16 clocks of an
// SM per warp, measured), a 64-bit integer addition in 0.75 clocks and a
// 64 x 64 -> 64 high product by a constant in about 4.5.  A cell's PDF
// deviations are therefore brought to a common exponent E (all |d| < 2^E),
// x = round(d 2^(58 - E)), and the collision runs on the integers: sums and
// differences are exact, a product by a coefficient errs by at most 1.75 units,
// and only the conversions (one instruction each way) run on the FP64 pipe.
// One input unit, 2^(E - 58), is at most 2^-57 of the cell's largest
// deviation, a sixteenth of the rounding error of an FP64 sum of that size.
// Results carry one bit less (unit 2^(E - 57)): the coefficients are stored
// halved so that every 32-bit partial product fits.
//
// 64-bit sums may wrap on the way (two's complement); every value that is
// multiplied, shifted or converted fits (the bounds beside each of them are
// in units of M = 2^58, the largest input).
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define FX_FN __host__ __device__ __forceinline__
#else
#define FX_FN inline
#endif

namespace psm {

typedef long long fx;

constexpr int FX_BITS = 58;       // input scale: x = d 2^(FX_BITS - E)
constexpr int FX_EMAX = -3;       // largest exponent the fixed-point form takes
constexpr int FX_EMAX_SOLID = -5; // and for covered cells, whose squares are larger
constexpr int FX_EMIN = -900;     // smallest one (smaller deviations round to 0)

FX_FN int fx_hi(fx a) { return (int)(a >> 32); }
FX_FN uint32_t fx_lo(fx a) { return (uint32_t)a; }

// high 32 bits of the signed product, plus c
FX_FN int fx_madhi(int a, int b, int c) {
#ifdef __CUDA_ARCH__
  int r;
  asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
#else
  return (int)((uint32_t)(((long long)a * b) >> 32) + (uint32_t)c);
#endif
}
FX_FN fx fx_madwide(int a, int b, fx c) {
#ifdef __CUDA_ARCH__
  fx r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (fx)((uint64_t)((long long)a * b) + (uint64_t)c);
#endif
}
FX_FN fx fx_add(fx a, fx b) { return (fx)((uint64_t)a + (uint64_t)b); }
FX_FN fx fx_sub(fx a, fx b) { return (fx)((uint64_t)a - (uint64_t)b); }
FX_FN fx fx_shl(fx a, int n) { return (fx)((uint64_t)a << n); }
// arithmetic right shift by any n >= 0 (63 and more give the sign)
FX_FN fx fx_shr(fx a, int n) {
#ifdef __CUDA_ARCH__
  fx r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(n));
  return r;
#else
  return a >> (n > 63 ? 63 : n);
#endif
}

// A coefficient k, |k| <= 1/3, as hi 2^-32 + lo 2^-64 with both parts signed.
// add holds hi/2 (the low word of the multiplicand enters with its top bit
// flipped, i.e. less 2^31), 1 for the mean of the two truncations and lo/2^33
// for that of the product of the low words, rounded; what the rounding leaves
// (fx_bias, at most half a unit) is known and compensated per cell.
struct alignas(16) FxCoef {
  int hi, lo, add, pad;
};

FX_FN double fx_add_exact(int hi, int lo) { return 0.5 * hi + 1.0 + lo / 8589934592.0; }
// k + r, r the rounding error of k: coefficients are kept to 2^-64, an FP64
// number's own error would be 2^-54 of a sum of 19 values
FX_FN FxCoef fx_coef(double k, double r) {
  FxCoef c;
  const double s = k * 4294967296.0;
  const double h = rint(s);
  c.hi = (int)h;
  const double l = rint(((s - h) + r * 4294967296.0) * 4294967296.0);
  c.lo = l > 2147483647.0 ? 2147483647 : (int)l;
  c.add = (int)rint(fx_add_exact(c.hi, c.lo));
  c.pad = 0;
  return c;
}
// a / b, b exact
FX_FN FxCoef fx_ratio(double a, double b) {
  const double k = a / b;
  return fx_coef(k, fma(-k, b, a) / b);
}
// (1 - w) / 4
FX_FN FxCoef fx_relax(double w) {
  const double d = 1.0 - w, bb = d - 1.0;
  const double r = (1.0 - (d - bb)) + (-w - bb);
  return fx_coef(0.25 * d, 0.25 * r);
}
// mean of (fx_mul - product)
FX_FN double fx_bias(const FxCoef& c) { return c.add - fx_add_exact(c.hi, c.lo); }

// x k: errs by at most 1.75 units
FX_FN fx fx_mul(fx x, const FxCoef& k) {
  const int xh = fx_hi(x);
  const int xl = (int)(fx_lo(x) ^ 0x80000000u);
  const int t = fx_madhi(xh, k.lo, fx_madhi(xl, k.hi, k.add));
  return fx_madwide(xh, k.hi, (fx)t);
}

// x^2 2^-64, |x| < 2^63: errs by at most 1.5 units.  With x = xh 2^32 + xl:
// xh^2 + 2 xh xl 2^-32 and xl = xs + 2^31, so 2 hi(xh xs) + xh + xh^2
FX_FN fx fx_sq(fx x) {
  const int xh = fx_hi(x);
  const int xs = (int)(fx_lo(x) ^ 0x80000000u);
  const fx t = (fx)fx_madhi(xh, xs, 0);
  // 2 hi(..) is below its value by 1 on average (and the dropped xl^2 2^-64
  // is a third)
  return fx_madwide(xh, xh, fx_add(fx_add(t, t), (fx)xh + 1));
}

// Relaxation constants of the fixed-point form (fixed for a context).
// Coefficients of results are halved (results have the unit 2^(E - 57)).
struct FxRates {
  FxCoef kp, km;          // (1 - omega+)/4, (1 - omega-)/4
  FxCoef kd;              // omega+ / 6: the density term of the rest direction
  FxCoef ke;              // omega- / 12: the velocity term of a face pair
  FxCoef third, sixth, twelfth;  // face and edge weights over the rest weight: 1/6, 1/12
  FxCoef sig[2];          // sqrt(omega+ / 8) / 2, and that over sqrt(2)
  double tau, sigma[2];   // tau+, sqrt(omega+ / 8), and that over sqrt(2)
  // mean rounding errors of mass and, per axis, of half the momentum
  double bias0, biasA[3];
  int compS;  // 256 times the mean rounding error of fx_solid's mass, negated
};

// The forcing's constants at the scale of one exponent E, rounded, and the
// compensation of the mean rounding errors (256 times a unit).  The rows of
// E0, E0 + 1, .. are a table that a block forms once; from FX_ROWS - 1
// exponents above E0 on every constant rounds to zero.
struct FxRow {
  fx fs[3], fg[3], fh[3], K[10];  // (2 sigma tau+ f) 2^-t, f / 6, f / 2, see fx_row
  int comp0, compA[3];
  int pad[2];
};
constexpr int FX_ROWS = 64;
// directions whose conversion to an integer runs on the integer pipe: 12 of 19
// balance it against the FP64 pipe (256x128x128 without particles: 707 clocks
// of an SM per warp of cells with none, 645 with six, 600 with twelve, 653
// with sixteen)
FX_FN constexpr bool fx_int_conv(int q) { return q < 12; }

// FP64 words
FX_FN int dbl_hi(double v) {
#ifdef __CUDA_ARCH__
  return __double2hiint(v);
#else
  uint64_t u;
  __builtin_memcpy(&u, &v, 8);
  return (int)(u >> 32);
#endif
}
// v 2^n by an addition to the exponent field (the caller's n keeps it in range;
// zero and denormal v give a number far below 1 for n > 0)
FX_FN double dbl_scale(double v, int n20) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(__double2hiint(v) + n20, __double2loint(v));
#else
  uint64_t u;
  __builtin_memcpy(&u, &v, 8);
  u += (uint64_t)(uint32_t)n20 << 32;
  __builtin_memcpy(&v, &u, 8);
  return v;
#endif
}
FX_FN fx dbl_to_fx(double v) {
#ifdef __CUDA_ARCH__
  return __double2ll_rn(v);
#else
  return __builtin_llrint(v);
#endif
}
// v 2^(FX_BITS - E), rounded, |v| < 2^E, by integer instructions: the FP64
// pipe takes 16 clocks of an SM for a conversion, these 17 instructions about 8
// of the integer pipe.  ef = E + 1022, the exponent field of numbers just
// below 2^E
FX_FN fx dbl_to_fx_int(double v, int ef) {
#ifdef __CUDA_ARCH__
  const int hi = __double2hiint(v);
  const uint32_t lo = (uint32_t)__double2loint(v);
#else
  uint64_t u;
  __builtin_memcpy(&u, &v, 8);
  const int hi = (int)(u >> 32);
  const uint32_t lo = (uint32_t)u;
#endif
  const int n = ef - (int)(((uint32_t)hi << 1) >> 21);  // >= 0
  const uint32_t mh = ((uint32_t)hi & 0xfffffu) | 0x100000u;
  // mantissa 2^6 2^-n, one bit below the unit, then rounded.  Zero and
  // denormal numbers (n > 63: E >= FX_EMIN) come out as 0
  const fx m = fx_shl((fx)(((uint64_t)mh << 32) | lo), 6);
  const fx y = fx_shr(fx_add(fx_shr(m, n), 1), 1);
  const fx sg = (fx)(hi >> 31);
  return fx_sub(y ^ sg, sg);
}
FX_FN double fx_to_dbl(fx x, int n20) {  // x 2^n, rounded to FP64
#ifdef __CUDA_ARCH__
  const double v = __ll2double_rn(x);
  const int hi = __double2hiint(v);  // 0 only for x = 0
  return __hiloint2double(hi != 0 ? hi + n20 : 0, __double2loint(v));
#else
  return x == 0 ? 0.0 : dbl_scale((double)x, n20);
#endif
}

FX_FN void fx_fill(FxRates& c, double wp, double wm) {
  c.tau = 1.0 / wp;
  c.kp = fx_relax(wp);
  c.km = fx_relax(wm);
  c.kd = fx_ratio(wp, 6.0);
  c.ke = fx_ratio(wm, 12.0);
  c.third = fx_ratio(1.0, 3.0);
  c.sixth = fx_ratio(1.0, 6.0);
  c.twelfth = fx_ratio(1.0, 12.0);
  for (int i = 0; i < 2; ++i) {
    const double s2 = wp * (i ? 0.0625 : 0.125);  // 9/2 omega+ w of an edge pair, exact
    const double s = sqrt(s2);
    c.sigma[i] = s;
    c.sig[i] = fx_coef(0.5 * s, 0.5 * (fma(-s, s, s2) / (2.0 * s)));
  }
  // mean rounding errors of fx_collide (a square: -1/3; a halved one 1/2 less
  // again: fx_sq gives odd numbers, xh^2 + xh being even)
  const double bkp = fx_bias(c.kp), bkm = fx_bias(c.km), bke = fx_bias(c.ke);
  const double bb = fx_bias(c.kd) + 1.0;
  const double sf = bb / 6.0 + fx_bias(c.sixth) - 1.0 / 6.0 - 0.5 + bkp;
  const double se = bb / 12.0 + fx_bias(c.twelfth) - 1.0 / 3.0 + bkp;
  c.bias0 = 2.0 * bkp + bb + 6.0 * sf + 12.0 * se;
  c.compS = (int)rint(256.0 * (6.0 * fx_bias(c.third) + 12.0 * fx_bias(c.sixth)));
  // along x: A_0 + A_3 + A_4 + A_5 + A_6, and so on, with G's bias bke
  c.biasA[0] = bkm + bke + 4.0 * bkm + 2.0 * bke;
  c.biasA[1] = bkm + bke + 2.0 * bkm + 2.0 * bke;
  c.biasA[2] = bkm + bke + 2.0 * bke;
}

// smallest exponent for a force density f: f / 4 and 2 sigma tau+ f stay
// below 2^(E0 + 2).  Above FX_EMAX when the form does not apply (a force that
// is not finite or absurdly large)
FX_FN int fx_e0(const FxRates& c, const double* f) {
  double big = 0.0;
  for (int a = 0; a < 3; ++a) {
    const double v = fmax(0.25, 2.0 * c.sigma[0] * c.tau) * fabs(f[a]);
    if (!(v <= 1.0)) return 2000;
    big = v > big ? v : big;
  }
  const int e = ((dbl_hi(big) >> 20) & 0x7ff) - 1022 - 2;  // big < 2^(e + 2)
  return e < FX_EMIN ? FX_EMIN : e;
}

// v 2^n rounded; *err gains w times the rounding error (in units)
FX_FN fx fx_round_err(double v, int n, double w, double* err) {
  const double s = scalbn(v, n);  // exact
  const fx y = dbl_to_fx(s);
  *err += w * ((double)y - s);
  return y;
}

// row of the exponent E0 + i for the force density f (finite)
FX_FN void fx_row(const FxRates& c, const double* f, int E0, int i, FxRow& r) {
  const int E = E0 + i, h = -3 - E, od = h & 1;
  const double g = c.tau - 0.5, s2g = c.sigma[0] * c.sigma[0] * g * g;
  double e0 = 0.0, none = 0.0;
  for (int a = 0; a < 3; ++a) {
    r.fs[a] = fx_round_err(2.0 * c.sigma[od] * c.tau * f[a], FX_BITS - E - (h > 0 ? h >> 1 : 0),
                           0.0, &none);
    r.fh[a] = fx_round_err(0.5 * f[a], FX_BITS - E, 0.0, &none);
    double eg = 0.0;
    r.fg[a] = fx_round_err(f[a] / 6.0, FX_BITS - 1 - E, 1.0, &eg);
    // G enters a face pair once and its half the edge pairs twice net
    r.compA[a] = (int)rint(-256.0 * (c.biasA[a] + 3.0 * eg));
  }
  const double ff = (f[0] * f[0] + f[1] * f[1] + f[2] * f[2]) / 3.0;
  const double cf[6] = {f[0] + f[1], f[0] - f[1], f[0] + f[2],
                        f[0] - f[2], f[1] + f[2], f[1] - f[2]};
  for (int k = 0; k < 3; ++k)
    r.K[k] = fx_round_err(2.0 * s2g * (ff - f[k] * f[k]), FX_BITS - 1 - E, 2.0, &e0);
  for (int k = 0; k < 6; ++k)
    r.K[3 + k] = fx_round_err(s2g * (ff - cf[k] * cf[k]), FX_BITS - 1 - E, 2.0, &e0);
  r.K[9] = fx_round_err(12.0 * s2g * ff, FX_BITS - 1 - E, 1.0, &e0);
  r.comp0 = (int)rint(-256.0 * (c.bias0 + e0));
}

// largest |d| of a cell as the high word of an FP64 number
FX_FN int fx_top(const double* d) {
  int m = 0;
  for (int q = 0; q < 19; ++q) {
    const int h = dbl_hi(d[q]) & 0x7fffffff;
    m = h > m ? h : m;
  }
  return m;
}
// exponent of a cell: all |d| < 2^E, E >= E0 (above FX_EMAX, and for NaN and
// infinities, the fixed-point form does not apply)
FX_FN int fx_exponent(int top, int E0) {
  const int E = (top >> 20) - 1022;
  return E > E0 ? E : E0;
}

// half of x, rounded to the nearest integer, ties to even
FX_FN fx fx_half(fx x) { return fx_shr(fx_add(x, fx_shr(x, 1) & 1), 1); }

// a b 2^-64, |a|, |b| < 2^63: errs by at most 2 units, by nothing on average
FX_FN fx fx_prod(fx a, fx b) {
  const int ah = fx_hi(a), bh = fx_hi(b);
  const int as = (int)(fx_lo(a) ^ 0x80000000u), bs = (int)(fx_lo(b) ^ 0x80000000u);
  // the halves of ah and bh belong to the flipped top bits of the low words;
  // 3 makes up for the truncations and the product of the low words
  const fx t = fx_add((fx)fx_madhi(ah, bs, 0), (fx)fx_madhi(bh, as, 0));
  const fx h = fx_shr(fx_add((fx)ah, (fx)bh + 3), 1);
  return fx_madwide(ah, bh, fx_add(t, h));
}

// a value in [0, 256) from the cell's own bits: the mean rounding errors,
// fractions of a unit, are added as whole units with it
FX_FN int fx_dither(fx R) { return (int)((fx_lo(R) * 0x9E3779B1u) >> 24); }

// c_k . (a0, a1, a2) of an edge pair, k = 3..8
FX_FN fx fx_edge(int k, const fx* a) {
  switch (k) {
    case 3: return fx_add(a[0], a[1]);
    case 4: return fx_sub(a[0], a[1]);
    case 5: return fx_add(a[0], a[2]);
    case 6: return fx_sub(a[0], a[2]);
    case 7: return fx_add(a[1], a[2]);
    default: return fx_sub(a[1], a[2]);
  }
}

// the deviations of a cell at its scale (x <= M), and their moments R = sum d
// (<= 19 M), j (<= 10 M)
struct FxCell {
  fx x[19], R, j[3];
};
FX_FN void fx_load(const double* d, int E, FxCell& C) {
  const int n20 = (FX_BITS - E) << 20;
  fx* x = C.x;
#pragma unroll
  for (int q = 0; q < 19; ++q)
    x[q] = fx_int_conv(q) ? dbl_to_fx_int(d[q], E + 1022) : dbl_to_fx(dbl_scale(d[q], n20));
  fx a[9];
  C.R = x[0];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    C.R = fx_add(C.R, fx_add(x[2 * k + 1], x[2 * k + 2]));
    a[k] = fx_sub(x[2 * k + 1], x[2 * k + 2]);
  }
  C.j[0] = fx_add(fx_add(fx_add(a[0], a[3]), fx_add(a[4], a[5])), a[6]);
  C.j[1] = fx_add(fx_add(fx_sub(a[1], a[4]), fx_add(a[3], a[7])), a[8]);
  C.j[2] = fx_add(fx_sub(fx_sub(a[2], a[6]), a[8]), fx_add(a[5], a[7]));
}

// Fluid collision (Eqs. 3-8, TRT/SRT with forcing) of a cell, exponent E (E0
// <= E <= FX_EMAX), results in units of 2^(E - 57).
// With s_k, a_k the sums and differences of a pair, R = sum d, j = sum a_k c_k:
//   S_k = (1 - omega+)/2 s_k + omega+ w R + 9/2 omega+ w [(c.U')^2 - U'.U'/3] + K_k
//   A_k = (1 - omega-)/2 a_k + 3 omega- w (c.j) + 3 w (c.f)
//   d_q' = S_k + A_k, d_qbar' = S_k - A_k,
// U' = j + tau+ f: completing the squares moves the forcing terms of Eq. 8
// (Guo prefactors) into that velocity and the constants
// K_k = 9/2 omega+ w (tau+ - 1/2)^2 [f.f/3 - (c.f)^2].
// The terms common to the pairs are formed first; the pairs follow one by
// one, so that a cell needs its 19 values and these terms in registers.
struct FxFluid {
  fx F[3], q[3], bf, be, G[3], Ge[3], d0;
};
FX_FN void fx_fluid(const FxRates& c, const FxRow& row, int E, const FxCell& C, int dith,
                    FxFluid& L) {
  // F = 2 sigma U' 2^-t: the square of F, less 64 bits, is 9/2 omega+ w U'^2
  // of an edge pair in result units when 2 t = -3 - E (every other exponent
  // takes sigma / sqrt 2)
  const int h = -3 - E;
  FxCoef sg;
  sg.hi = (h & 1) ? c.sig[1].hi : c.sig[0].hi;
  sg.lo = (h & 1) ? c.sig[1].lo : c.sig[0].lo;
  sg.add = (h & 1) ? c.sig[1].add : c.sig[0].add;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    L.F[i] = fx_add(fx_shr(fx_shl(fx_mul(C.j[i], sg), 2), h >> 1), row.fs[i]);  // <= 14 M
    L.q[i] = fx_sq(fx_add(L.F[i], L.F[i]));
    const fx g = fx_add(fx_mul(C.j[i], c.ke), row.fg[i]);
    L.Ge[i] = fx_half(g);
    L.G[i] = fx_add(g, (row.compA[i] + dith) >> 8);
  }
  // the rest direction's equilibrium; a face pair's is a sixth, an edge
  // pair's a twelfth of it (without the (c.U)^2 terms)
  const fx base = fx_sub(fx_mul(C.R, c.kd), fx_add(fx_add(L.q[0], L.q[1]), L.q[2]));
  L.bf = fx_mul(base, c.sixth);
  L.be = fx_mul(base, c.twelfth);
  const fx r = fx_mul(C.x[0], c.kp);
  L.d0 = fx_add(fx_add(fx_add(r, r), row.K[9]), fx_add(base, (row.comp0 + dith) >> 8));
}
FX_FN void fx_fluid_pair(const FxRates& c, const FxRow& row, const FxCell& C, const FxFluid& L,
                         int k, fx* qa, fx* qb) {
  const fx s = fx_add(C.x[2 * k + 1], C.x[2 * k + 2]), a = fx_sub(C.x[2 * k + 1], C.x[2 * k + 2]);
  const fx eq = k < 3 ? fx_add(L.bf, fx_shr(L.q[k], 1)) : fx_add(L.be, fx_sq(fx_edge(k, L.F)));
  const fx S = fx_add(fx_add(eq, fx_mul(s, c.kp)), row.K[k]);  // s, a <= 2 M
  const fx A = fx_add(k < 3 ? L.G[k] : fx_edge(k, L.Ge), fx_mul(a, c.km));
  *qa = fx_add(S, A);
  *qb = fx_sub(S, A);
}

// Difference of two equilibria and an antisymmetric term: with D = V - U, S =
// V + U and a vector W (each <= 15 M, units of 2^(E - 58)), per direction
//   9/2 w [(c.V)^2 - (c.U)^2] - 3/2 w [V.V - U.U] + 3 w c.W
// in the same units.
struct FxSolid {
  fx D[3], S[3], p[3], t3, t6, G[3], Ge[3], d0;
};
FX_FN void fx_solid(const FxRates& c, int E, const fx* D, const fx* S, const fx* W, int dith,
                    FxSolid& L) {
  // the products' operands are shifted by n = -3 - E in all, so that an edge
  // pair's product less 64 bits is its 9/2 w (..) in units of the result
  const int n = -3 - E, t1 = n >> 1, t2 = n - t1;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    L.G[i] = fx_mul(W[i], c.sixth);
    L.Ge[i] = fx_half(L.G[i]);
    L.D[i] = fx_shr(D[i], t1);
    L.S[i] = fx_shr(S[i], t2);
    L.p[i] = fx_prod(fx_add(L.D[i], L.D[i]), L.S[i]);
  }
  const fx T = fx_add(fx_add(L.p[0], L.p[1]), L.p[2]);
  L.t3 = fx_mul(T, c.third);
  L.t6 = fx_mul(T, c.sixth);
  L.d0 = fx_sub((fx)((c.compS + dith) >> 8), fx_add(T, T));
}
FX_FN void fx_solid_pair(const FxSolid& L, int k, fx* qa, fx* qb) {
  const fx eq = k < 3 ? fx_sub(L.p[k], L.t3)
                      : fx_sub(fx_prod(fx_edge(k, L.D), fx_edge(k, L.S)), L.t6);
  const fx an = k < 3 ? L.G[k] : fx_edge(k, L.Ge);
  *qa = fx_add(eq, an);
  *qb = fx_sub(eq, an);
}

// a weight 0 <= B <= 1 as the coefficient B / 4
FX_FN FxCoef fx_weight(double B) {
  const fx v = dbl_to_fx(dbl_scale(B, 62 << 20));  // B 2^62
  FxCoef c;
  c.hi = fx_hi(fx_add(v, 1ll << 31));
  c.lo = (int)fx_lo(v);
  // rounded to the nearer half; B = 0 gives exact zeros
  c.add = v == 0 ? 0 : ((c.hi + (c.lo > 0 ? 1 : 0)) >> 1) + 1;
  c.pad = 0;
  return c;
}

// a cell's top word with a velocity taken in: |V| < 2^(E + bits)
FX_FN int fx_top_velocity(int top, const double* V, int bits) {
  for (int a = 0; a < 3; ++a) {
    const int h = (dbl_hi(V[a]) & 0x7fffffff) - (bits << 20);
    top = h > top ? h : top;
  }
  return top;
}
constexpr int FX_VBITS_MIXED = 3;

// Collision of one cell of a kind; put(q, value) takes the results.
//  FX_FLUID  no particle.
//  FX_MIXED  one particle of weight B <= 1 and surface velocity V (B = 0:
//            none): d' = F + B (S - F), F the fluid collision and S the solid
//            operator's result (Eq. 19), which swaps each pair and adds the
//            difference of the equilibria, d_q' = d_qbar + E_s(V) - E_s(U) +
//            3 w c.(V + U).  E is one above the cell's exponent (with |V| <
//            2^(E + 2)), so that twice S - F fits.
// V: 4 values, surface velocity and weight.  force(Fc) takes the force
// B (U - V - f) of Eq. 21.
enum { FX_FLUID = 0, FX_MIXED = 1 };
template <int KIND, typename Force, typename Put>
FX_FN void fx_collide(const FxRates& c, const FxRow& row, int E, const double* d, const double* V,
                      Force force, Put put) {
  FxCell C;
  FxFluid L;
  FxSolid M;
  FxCoef w{0, 0, 0, 0};
  fx_load(d, E, C);
  const int o20 = (E - (FX_BITS - 1)) * (1 << 20);
  const int dith = fx_dither(C.R);
  fx_fluid(c, row, E, C, dith, L);
  if constexpr (KIND == FX_MIXED) {
    const int n20 = (FX_BITS - E) << 20;
    double Fc[3];
    fx D[3], S[3];
    w = fx_weight(V[3]);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const fx v = dbl_to_fx(dbl_scale(V[i], n20));
      const fx U = fx_add(C.j[i], row.fh[i]);  // <= 11 M
      D[i] = fx_sub(v, U);
      S[i] = fx_add(v, U);
      // U - V - f
      const fx u = fx_sub(fx_sub(0, D[i]), fx_add(row.fh[i], row.fh[i]));
      Fc[i] = fx_to_dbl(fx_mul(fx_add(u, u), w), o20);
    }
    force(Fc);
    fx_solid(c, E, D, S, S, dith, M);
  }
  // F in units of 2^(E - 57), s in units of 2^(E - 58)
  auto blend = [&](fx F, fx s) {
    const fx b = fx_sub(s, fx_add(F, F));
    return fx_add(F, fx_mul(fx_add(b, b), w));
  };
  if constexpr (KIND == FX_FLUID) put(0, fx_to_dbl(L.d0, o20));
  else put(0, fx_to_dbl(blend(L.d0, fx_add(C.x[0], M.d0)), o20));
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    fx qa, qb, sa, sb;
    fx_fluid_pair(c, row, C, L, k, &qa, &qb);
    if constexpr (KIND == FX_MIXED) {
      fx_solid_pair(M, k, &sa, &sb);
      qa = blend(qa, fx_add(C.x[2 * k + 2], sa));
      qb = blend(qb, fx_add(C.x[2 * k + 1], sb));
    }
    put(2 * k + 1, fx_to_dbl(qa, o20));
    put(2 * k + 2, fx_to_dbl(qb, o20));
  }
}

}  // namespace psm
