// fixed64.cuh -- the collision's linear algebra in per-cell block fixed point:
// 64-bit integers under exponents of the cell's own.
//
// GB300 executes an FP64 operation at 1/64 of the FP32 rate (16 clocks of an
// SM per warp, measured), a 64-bit integer addition in 0.75 clocks and a
// 64 x 64 -> 64 high product by a constant in about 4.5.  A cell's PDF
// deviations are therefore brought to common exponents and the collision runs
// on the integers: sums and differences are exact, a product by a coefficient
// errs by at most 3/4 of a unit, and only the conversions (one instruction each
// way) run on the FP64 pipe.
//
// Exponents.  FP64 rounds every number relative to its own size.  A collision
// keeps numbers whose sizes have little to do with one another: pressure and
// momentum, a particle's velocity and the fluid's, and a weight times either.
// So they do not share one exponent:
//   E  the 18 moving directions: |d| < 2^E of a face, 2^(E - 1) of an edge
//      direction, 2^(E + 3) of the rest direction (a density deviation alone
//      has d_0 = 6 d_face = 12 d_edge); the force's and the particle's share
//      bounded likewise (fx_range).  Values d 2^(60 - E), results 2^(59 - E):
//      an input unit is 2^-58 to 2^-60 of the largest |d_q| (covered cells
//      2^-57 to 2^-59) unless the force or the particle's velocity times its
//      weight is larger than the values themselves.
//   P  the rest direction and the density, which are small beside the others
//      where velocity dominates (d_0 is quadratic in it then).  Values
//      2^(60 - P), results 2^(59 - P).
//   M  covered cells: |U|, |V| <= 2^(M - 1), U the fluid's velocity, small
//      beside the d_q where pressure dominates, and V the particle's.  Values
//      2^(61 - M).  Products with the weight B carry B's own exponent eb,
//      B <= 2^eb; so a fast particle costs a cell of small weight nothing.
// Against FP64 arithmetic on the same inputs (tests/fixed64_classes.cpp, rms
// error over that of FP64, mean over density deviations of 0 to 10^4 times the
// velocity, particles up to 1000 times as fast, weights 0 to 1): cells without
// particles 0.6 rest direction, 0.3 the others, 0.4 mass, 0.25 momentum;
// covered cells 0.7, 0.3, 0.55, 0.25, force 0.55.  (One exponent for all, that
// of the largest value: 10, 0.4, 0.6, 0.4; 25, 0.8 to 1, 2.4, 0.7, force 28.)
//
// 64-bit sums may wrap on the way (two's complement); every value that is
// multiplied, shifted or converted fits (the bounds stand beside them).
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define FX_FN __host__ __device__ __forceinline__
#else
#define FX_FN inline
#endif

namespace psm {

typedef long long fx;

constexpr int FX_BITS = 60;    // input scale, 2^(FX_BITS - exponent)
constexpr int FX_ETOP = -3;    // largest E: (c.U)^2 terms fit
constexpr int FX_EMIN = -440;  // smallest E; smaller values round to 0
constexpr int FX_VMAX = 20;    // largest exponent of a particle's velocity

FX_FN int fx_hi(fx a) { return (int)(a >> 32); }
FX_FN uint32_t fx_lo(fx a) { return (uint32_t)a; }

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
// c rounds the product's middle words: the low word of the multiplicand enters
// with its top bit flipped, i.e. less 2^31, so half of k is due beside the 2^31
// that make the truncation a rounding.
struct alignas(16) FxCoef {
  int hi, lo;
  fx c;
};
FX_FN FxCoef fx_coef_of(int hi, int lo) {
  FxCoef c;
  c.hi = hi;
  c.lo = lo;
  c.c = fx_add(fx_add(fx_shl(hi, 31), lo >> 1), 1ll << 31);
  return c;
}
// k + r, r the rounding error of k: coefficients are kept to 2^-64, an FP64
// number's own error would be 2^-54 of a sum of 19 values
FX_FN FxCoef fx_coef(double k, double r) {
  const double s = k * 4294967296.0;
  const double h = rint(s);
  const double l = rint(((s - h) + r * 4294967296.0) * 4294967296.0);
  return fx_coef_of((int)h, l > 2147483647.0 ? 2147483647 : (int)l);
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
// mean of (fx_mul - product): halves are rounded up, which matters where k has
// few binary places
FX_FN double fx_bias(const FxCoef& c) {
  const uint64_t v = ((uint64_t)(uint32_t)c.hi << 32) + (uint64_t)(int64_t)c.lo;
  return v == 0 ? 0.0 : 0.5 * (double)(v & (0 - v)) * 0x1p-64;
}

// x k: errs by at most 3/4 of a unit, 0 for 0.  |x| < 2^63 for |k| <= 1/4,
// |x| <= 5 2^60 for |k| <= 1/3.  (Products truncated to 32 bits, with the mean
// of the truncations added, err by up to 1.75 and give a unit for zero: a
// momentum that no flow has.)
FX_FN fx fx_mul(fx x, const FxCoef& k) {
  const int xh = fx_hi(x);
  const int xl = (int)(fx_lo(x) ^ 0x80000000u);
  const fx t = fx_madwide(xh, k.lo, fx_madwide(xl, k.hi, k.c));
  return fx_madwide(xh, k.hi, (fx)fx_hi(t));
}

// x^2 2^-64, |x| < 2^63: errs by at most 1.2 units, 0 for 0.  With x = xh 2^32
// + xl, xl = xs + 2^31: xh^2 + xh + 2 (xh xs + 2^30) 2^-32, and a third for the
// mean of xl^2 2^-64
FX_FN fx fx_sq(fx x) {
  const int xh = fx_hi(x);
  const int xs = (int)(fx_lo(x) ^ 0x80000000u);
  const fx t = fx_shr(fx_madwide(xh, xs, (1ll << 30) + (1ll << 31) / 3), 31);
  return fx_madwide(xh, xh, fx_add(t, (fx)xh));
}

// Relaxation constants of the fixed-point form (fixed for a context).
// Coefficients of results are halved (results have twice the unit of inputs).
struct FxRates {
  FxCoef kp, km;          // (1 - omega+)/4, (1 - omega-)/4
  FxCoef kd;              // omega+ / 6: the density term of the rest direction
  FxCoef ke;              // omega- / 12: the velocity term of a face pair
  FxCoef third, sixth, twelfth;  // face and edge weights over the rest weight: 1/6, 1/12
  FxCoef sig[2];          // sqrt(omega+ / 8) / 2, and that over sqrt(2)
  double tau, sigma[2];   // tau+, sqrt(omega+ / 8), and that over sqrt(2)
  // mean rounding errors of the rest direction, of a pair's sum, and per axis
  // of half the momentum (products' halves, fx_bias)
  double bias0, biasS, biasA[3];
};

// The forcing's constants at one exponent, rounded, and the compensation of
// their and the mean rounding errors (256 times a unit).  Row i of a table that
// a block copies to shared memory holds E = E0 + i and P = P0 + i, E0 and P0
// the smallest ones for the force; in the last row every constant of the force
// has rounded to zero.
struct alignas(16) FxRow {
  fx fs[3], fg[3], fh[3], K[9];  // sigma tau+ f, f / 6 (result unit), f / 2, see fx_fluid
  fx K0;                         // the rest direction's, at P
  int compA[3], compF, compD, comp0;
};
static_assert(sizeof(FxRow) % 16 == 0 && alignof(FxRow) == 16, "copied 16 bytes at a time");
constexpr int FX_ROWS = 64;
FX_FN constexpr int fx_p0(int E0) { return 2 * E0 + 2; }
// Directions whose conversion to an integer runs on the integer pipe, to
// balance it against the FP64 pipe: 6 of 19.  Collision of a 256^3 settling box
// 1.64 ms, of a channel at 20% solid fraction 0.98, of 256x128x128 without
// particles 0.290 (none in cells without particles: 2% more, 2% less, 4% more;
// 12 there: 2% and 2% more, 1% less)
FX_FN constexpr bool fx_int_conv(int q) { return q < 6; }

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
// of the integer pipe
FX_FN fx dbl_to_fx_int(double v, int E) {
#ifdef __CUDA_ARCH__
  const int hi = __double2hiint(v);
  const uint32_t lo = (uint32_t)__double2loint(v);
#else
  uint64_t u;
  __builtin_memcpy(&u, &v, 8);
  const int hi = (int)(u >> 32);
  const uint32_t lo = (uint32_t)u;
#endif
  // E + 1022: the exponent field of numbers just below 2^E
  const int n = E + 1022 - (int)(((uint32_t)hi << 1) >> 21);  // >= 0
  const uint32_t mh = ((uint32_t)hi & 0xfffffu) | 0x100000u;
  // mantissa 2^-n, one bit below the unit, then rounded.  Zero and
  // denormal numbers (n > 63) come out as 0
  const fx m = fx_shl((fx)(((uint64_t)mh << 32) | lo), FX_BITS - 52);
  const fx y = fx_shr(fx_add(fx_shr(m, n), 1), 1);
  const fx sg = (fx)(hi >> 31);
  return fx_sub(y ^ sg, sg);
}
FX_FN fx fx_from(double v, int E, bool by_int) {
  return by_int ? dbl_to_fx_int(v, E) : dbl_to_fx(dbl_scale(v, (FX_BITS - E) * (1 << 20)));
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
// |a| <= 2^fx_bits(u), u the OR of one or more fx_abs_hi(a)
FX_FN uint32_t fx_abs_hi(fx a) { return (uint32_t)(fx_hi(a) ^ (fx_hi(a) >> 31)); }
FX_FN int fx_bits(uint32_t u) {
#ifdef __CUDA_ARCH__
  return 64 - __clz((int)u);
#else
  return u == 0 ? 32 : 64 - __builtin_clz(u);
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
  const double bkp = fx_bias(c.kp), bkm = fx_bias(c.km);
  c.bias0 = 2.0 * bkp;
  c.biasS = bkp;
  // along x: A_0 + A_3 + A_4 + A_5 + A_6, and so on
  c.biasA[0] = 5.0 * bkm;
  c.biasA[1] = 3.0 * bkm;
  c.biasA[2] = bkm;
}

// exponent of an FP64 number's high word (sign cleared): v < 2^result
FX_FN int fx_exp(uint32_t top) { return (int)(top >> 20) - 1022; }

// smallest E for a force density f: sigma tau+ |f| and |f| / 8 are below 2^E.
// 2000 when the form does not apply (a force that is not finite or absurdly
// large)
FX_FN int fx_e0(const FxRates& c, const double* f) {
  double big = 0.0;
  for (int a = 0; a < 3; ++a) {
    const double v = fmax(0.125, c.sigma[0] * c.tau) * fabs(f[a]);
    if (!(v <= 1.0)) return 2000;
    big = v > big ? v : big;
  }
  const int e = fx_exp((uint32_t)dbl_hi(big));
  return e < FX_EMIN ? FX_EMIN : e;
}

// v 2^n rounded, |n| < 1000; *err gains w times the rounding error (in units)
FX_FN fx fx_round_err(double v, int n, double w, double* err) {
  const double s = v * dbl_scale(1.0, n * (1 << 20));  // exact
  const fx y = dbl_to_fx(s);
  *err += w * ((double)y - s);
  return y;
}

// constants of the force density f (finite) for the exponents E and P, in
// parts that the threads of step_const_kernel share: an axis, the face pairs
// with the rest direction, the edge pairs
FX_FN void fx_row_axis(const FxRates& c, double fa, int E, int a, FxRow& r) {
  double none = 0.0, eg = 0.0;
  r.fs[a] = fx_round_err(c.sigma[(E + 1) & 1] * c.tau * fa, FX_BITS - E, 0.0, &none);
  r.fh[a] = fx_round_err(0.5 * fa, FX_BITS - E, 0.0, &none);
  r.fg[a] = fx_round_err(fa / 6.0, FX_BITS - 1 - E, 1.0, &eg);
  // G enters a face pair once and its half the edge pairs twice net
  r.compA[a] = (int)rint(-256.0 * (c.biasA[a] + 3.0 * eg));
}
FX_FN double fx_s2g(const FxRates& c) {
  const double g = c.tau - 0.5;
  return c.sigma[0] * c.sigma[0] * g * g;
}
FX_FN double fx_third_of_square(const double* f) {
  return (f[0] * f[0] + f[1] * f[1] + f[2] * f[2]) / 3.0;
}
FX_FN void fx_row_faces(const FxRates& c, const double* f, int E, int P, FxRow& r) {
  const double s2g = fx_s2g(c), ff = fx_third_of_square(f);
  double eF = 0.0, e0 = 0.0;
  for (int k = 0; k < 3; ++k)
    r.K[k] = fx_round_err(2.0 * s2g * (ff - f[k] * f[k]), FX_BITS - 1 - E, 1.0 / 3.0, &eF);
  r.K0 = fx_round_err(12.0 * s2g * ff, FX_BITS - 1 - P, 1.0, &e0);
  r.compF = (int)rint(-256.0 * (c.biasS + eF));
  r.comp0 = (int)rint(-256.0 * (c.bias0 + e0));
}
FX_FN void fx_row_edges(const FxRates& c, const double* f, int E, FxRow& r) {
  const double s2g = fx_s2g(c), ff = fx_third_of_square(f);
  const double cf[6] = {f[0] + f[1], f[0] - f[1], f[0] + f[2],
                        f[0] - f[2], f[1] + f[2], f[1] - f[2]};
  double eD = 0.0;
  for (int k = 0; k < 6; ++k)
    r.K[3 + k] = fx_round_err(s2g * (ff - cf[k] * cf[k]), FX_BITS - 1 - E, 1.0 / 6.0, &eD);
  r.compD = (int)rint(-256.0 * (c.biasS + eD));
}
FX_FN void fx_row_at(const FxRates& c, const double* f, int E, int P, FxRow& r) {
  for (int a = 0; a < 3; ++a) fx_row_axis(c, f[a], E, a, r);
  fx_row_faces(c, f, E, P, r);
  fx_row_edges(c, f, E, r);
}

// half of x, rounded to the nearest integer, ties to even
FX_FN fx fx_half(fx x) { return fx_shr(fx_add(x, fx_shr(x, 1) & 1), 1); }

// a b 2^-64, |a|, |b| <= 2^62: errs by at most 1.25 units, 0 for 0 (a quarter
// for the mean of the low words' product)
FX_FN fx fx_prod(fx a, fx b) {
  const int ah = fx_hi(a), bh = fx_hi(b);
  const int as = (int)(fx_lo(a) ^ 0x80000000u), bs = (int)(fx_lo(b) ^ 0x80000000u);
  // 2^31 times ah + bh belongs to the flipped top bits of the low words
  const fx h = fx_add(fx_shl((fx)ah + bh, 31), (1ll << 31) + (1ll << 30));
  const fx t = fx_madwide(ah, bs, fx_madwide(bh, as, h));
  return fx_madwide(ah, bh, (fx)fx_hi(t));
}

// random bits of the cell's own: the rounding errors of the forcing's
// constants, fractions of a unit, are made up for in whole units with the
// first eight, and the ninth breaks ties
FX_FN uint32_t fx_dither(fx R, fx j) { return (fx_lo(R) + fx_lo(j)) * 0x9E3779B1u; }

// v 2^-n: a left shift (exact) or a right one to the nearest integer, ties
// either way by the cell's bit (half of them up would be a drift where n is small)
struct FxShift {
  int l, r;
  fx half;
};
FX_FN FxShift fx_shift(int n, uint32_t bits) {
  FxShift s;
  s.l = n < 0 ? -n : 0;
  s.r = n > 0 ? (n < 62 ? n : 62) : 0;
  s.half = n > 0 ? fx_shl(1, s.r - 1) - (fx)((bits >> 23) & 1u) : 0;
  return s;
}
FX_FN fx fx_moved(fx v, const FxShift& s) {
  return fx_shr(fx_add(fx_shl(v, s.l), s.half), s.r);
}

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

// Fluid collision (Eqs. 3-8, TRT/SRT with forcing).
// With s_k, a_k the sums and differences of a pair, R = sum d, j = sum a_k c_k:
//   S_k = (1 - omega+)/2 s_k + omega+ w R + 9/2 omega+ w [(c.U')^2 - U'.U'/3] + K_k
//   A_k = (1 - omega-)/2 a_k + 3 omega- w (c.j) + 3 w (c.f)
//   d_q' = S_k + A_k, d_qbar' = S_k - A_k,
// U' = j + tau+ f: completing the squares moves the forcing terms of Eq. 8
// (Guo prefactors) into that velocity and the constants
// K_k = 9/2 omega+ w (tau+ - 1/2)^2 [f.f/3 - (c.f)^2].
// The terms common to the pairs are formed first; the pairs follow one by
// one, so that a cell needs its 19 values and these terms in registers.
// Bounds, E <= FX_ETOP: |j| <= 6, |F| <= 4 and |c.F| <= 7 times 2^60; at P,
// |R| <= 5 times 2^60 and the rest direction's result below 14 times 2^59
// (fx_cell chooses P so); S_k and A_k below 6.3 and 3.3 times 2^59.
struct FxFluid {
  fx F[3], eq[3], be, G[3], Ge[3], d0;
};
FX_FN void fx_fluid(const FxRates& c, const FxRow& re, const FxRow& rp, int E, int P,
                    const fx* j, const fx* F, fx R, fx x0, uint32_t bits, FxFluid& L) {
  const int dith = (int)(bits >> 24);
  // F = sigma U' (odd E: sigma U' / sqrt 2), sigma^2 = 9/2 omega+ w of an edge
  // pair, shifted so that its square, less 64 bits, is sigma^2 U'^2 in result
  // units: at E for the edge pairs, at P (H) for the rest.  P has the parity
  // of E.
  const int h = FX_ETOP - E, hp = (P - 2 * E - 3 - (h & 1)) / 2;
  const FxShift down = fx_shift(E - P, bits);  // results from P to E
  fx q[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    L.F[i] = fx_shr(F[i], h >> 1);
    const fx H = hp < 0 ? fx_shl(F[i], -hp) : fx_shr(F[i], hp);
    q[i] = fx_sq(fx_add(H, H));
    const fx g = fx_add(fx_mul(j[i], c.ke), re.fg[i]);
    L.Ge[i] = fx_half(g);
    L.G[i] = fx_add(g, (re.compA[i] + dith) >> 8);
  }
  // the rest direction's equilibrium; a face pair's is a sixth, an edge
  // pair's a twelfth of it (without the (c.U)^2 terms)
  const fx base = fx_sub(fx_mul(R, c.kd), fx_add(fx_add(q[0], q[1]), q[2]));
  const fx be = fx_moved(base, down);
  const fx bf = fx_add(fx_mul(be, c.sixth), (re.compF + dith) >> 8);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const fx f2 = fx_sq(L.F[k]);
    L.eq[k] = fx_add(fx_add(f2, f2), bf);
  }
  L.be = fx_add(fx_mul(be, c.twelfth), (re.compD + dith) >> 8);
  const fx r = fx_mul(x0, c.kp);
  L.d0 = fx_add(fx_add(fx_add(r, r), rp.K0), fx_add(base, (rp.comp0 + dith) >> 8));
}
// S_k and A_k
FX_FN void fx_fluid_pair(const FxRates& c, const FxRow& re, fx s, fx a, const FxFluid& L, int k,
                         fx* S, fx* A) {
  const fx eq = k < 3 ? L.eq[k] : fx_add(L.be, fx_sq(fx_edge(k, L.F)));
  *S = fx_add(fx_add(eq, fx_mul(s, c.kp)), re.K[k]);
  *A = fx_add(k < 3 ? L.G[k] : fx_edge(k, L.Ge), fx_mul(a, c.km));
}

// A weight 0 <= B <= 1 as the coefficients B / 4 and, with B's exponent eb
// (B <= 2^eb, eb <= 0) taken out, B 2^-eb / 4
struct FxWeight {
  FxCoef w, m;
  int eb;
};
// v 2^-64, halves rounded either way (B = 1 has many)
FX_FN FxCoef fx_weight_coef(fx v, uint32_t bits) {
  FxCoef c;
  c.hi = fx_hi(fx_add(v, 1ll << 31));
  c.lo = (int)fx_lo(v);
  c.c = fx_add(fx_shr(v, 1), (1ll << 31) - (fx)((bits >> 23) & 1u));
  return c;
}
FX_FN int fx_weight_exp(double B) {
  const int eb = fx_exp((uint32_t)dbl_hi(B));
  return eb > 0 ? 0 : (eb < -128 ? -128 : eb);
}
FX_FN FxWeight fx_weight(double B, uint32_t bits) {
  FxWeight W;
  W.eb = fx_weight_exp(B);
  const fx v = dbl_to_fx(dbl_scale(B, (62 - W.eb) << 20));  // B 2^(62 - eb)
  W.m = fx_weight_coef(v, bits);
  W.w = fx_weight_coef(fx_shr(v, -W.eb), bits);
  return W;
}

// B times the solid operator's equilibria (Eq. 19): with D = V - U, S = V + U
// (|D|, |S| <= 2^61 at M), per direction
//   9/2 w B [(c.V)^2 - (c.U)^2] - 3/2 w B [V.V - U.U] + 3 w B c.S
// in result units at E, and the rest direction's at P.
struct FxSolid {
  fx D[3], S[3], eq[3], t6, G[3], Ge[3], d0;
};
FX_FN void fx_solid(const FxRates& c, const FxWeight& W, int E, int P, int M, const fx* D,
                    const fx* S, uint32_t bits, FxSolid& L) {
  // 4 B D and S, shifted by n in all, so that an edge pair's product less 64
  // bits is its 9/2 w (..) in result units
  const int n = P - 2 * M - W.eb + 2, n1 = n >> 1, n2 = n - n1;      // n >= 0
  const int m = E - 2 * M - W.eb + 2, m1 = m >> 1, m2 = m - m1;      // m >= 0
  const FxShift down = fx_shift(E - P, bits), ag = fx_shift(E + 1 - M - W.eb, bits);
  fx p[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    L.G[i] = fx_moved(fx_mul(fx_mul(S[i], W.m), c.third), ag);
    L.Ge[i] = fx_half(L.G[i]);
    const fx B4 = fx_shl(fx_mul(D[i], W.m), 2);
    L.D[i] = fx_shr(B4, m1);
    L.S[i] = fx_shr(S[i], m2);
    const fx H = fx_shr(B4, n1);
    p[i] = fx_prod(fx_add(H, H), fx_shr(S[i], n2));
  }
  const fx T = fx_add(fx_add(p[0], p[1]), p[2]), t3 = fx_mul(T, c.third);
#pragma unroll
  for (int k = 0; k < 3; ++k) L.eq[k] = fx_moved(fx_sub(p[k], t3), down);
  L.t6 = fx_moved(fx_mul(T, c.sixth), down);
  L.d0 = fx_sub(0, fx_add(T, T));
}

// Collision of one cell of a kind, d its deviations, E and Ps from fx_range;
// rowE(E) (E >= E0) and rowP(P) give the forcing's constants; put(q, value)
// takes the results.
//  FX_FLUID  no particle.
//  FX_MIXED  one particle of weight B <= 1 and surface velocity V (B = 0:
//            none): d' = F + B (S - F), F the fluid collision and S the solid
//            operator's result (Eq. 19), which swaps each pair and adds the
//            difference of the equilibria, d_q' = d_qbar + E_s(V) - E_s(U) +
//            3 w c.(V + U): a pair's sum stays, its difference turns round.
//            E and P are one above what the values ask for, so that four
//            times s/4 - S and twice d_0/2 - F_0 fit.
// V: 4 values, surface velocity and weight.  force(Fc) takes the force
// B (U - V - f) of Eq. 21.
enum { FX_FLUID = 0, FX_MIXED = 1 };
template <int KIND, typename RowE, typename RowP, typename Force, typename Put>
FX_FN void fx_cell(const FxRates& c, RowE rowE, RowP rowP, int E0, int E, int Ps, const double* d,
                   const double* V, Force force, Put put) {
  constexpr int up = KIND == FX_MIXED ? 1 : 0;
  fx x[19], j[3], a[9], sf = 0, se = 0;
#pragma unroll
  for (int q = 1; q < 19; ++q) x[q] = fx_from(d[q], E, fx_int_conv(q));
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const fx s = fx_add(x[2 * k + 1], x[2 * k + 2]);
    a[k] = fx_sub(x[2 * k + 1], x[2 * k + 2]);
    if (k < 3) sf = fx_add(sf, s);
    else se = fx_add(se, s);  // both <= 6 2^60
  }
  j[0] = fx_add(fx_add(fx_add(a[0], a[3]), fx_add(a[4], a[5])), a[6]);
  j[1] = fx_add(fx_add(fx_sub(a[1], a[4]), fx_add(a[3], a[7])), a[8]);
  j[2] = fx_add(fx_sub(fx_sub(a[2], a[6]), a[8]), fx_add(a[5], a[7]));
  const FxRow& re = rowE(E);
  const uint32_t bits = fx_dither(fx_add(sf, se), j[0]);
  fx F[3];
  const int od = (E + 1) & 1;
  FxCoef sg;
  sg.hi = od ? c.sig[1].hi : c.sig[0].hi;
  sg.lo = od ? c.sig[1].lo : c.sig[0].lo;
  sg.c = od ? c.sig[1].c : c.sig[0].c;
  uint32_t hF = 0u;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const fx v = fx_mul(j[i], sg);
    F[i] = fx_add(fx_add(v, v), re.fs[i]);
    hF |= fx_abs_hi(F[i]);
  }
  // P: of d_0, of the squares of the velocities (4 sigma^2 U'^2 in all is at
  // most 6 times 2^P, or 3) and of the density
  int P = Ps, M = 0;
  auto at_least = [&](int v) { P = v > P ? v : P; };
  at_least(2 * (E - FX_BITS + fx_bits(hF)) + 1 + od + up);
  at_least(E - FX_BITS - 1 + up + fx_bits(fx_abs_hi(sf) | fx_abs_hi(se)));
  FxWeight W;
  if constexpr (KIND == FX_MIXED) {
    W = fx_weight(V[3], bits);
    uint32_t t = 0u, hj = 0u;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const uint32_t h = (uint32_t)dbl_hi(V[i]) & 0x7fffffffu;
      t = h > t ? h : t;
      hj |= fx_abs_hi(fx_add(j[i], re.fh[i])) | fx_abs_hi(fx_sub(j[i], re.fh[i]));
    }
    const int eu = E - FX_BITS + fx_bits(hj), ev = fx_exp(t);
    M = (eu > ev ? eu : ev) + 1;
    M = M > E0 + 1 ? M : E0 + 1;
    at_least(2 * M + W.eb - 2);
  }
  P += (P + E) & 1;
  const FxRow& rp = rowP(P);
  const fx x0 = fx_from(d[0], P, fx_int_conv(0));
  const FxShift up_p = fx_shift(P - E, bits);
  const fx R = fx_add(x0, fx_add(fx_moved(sf, up_p), fx_moved(se, up_p)));
  FxFluid L;
  fx_fluid(c, re, rp, E, P, j, F, R, x0, bits, L);
  FxSolid H;
  if constexpr (KIND == FX_MIXED) {
    const FxShift um = fx_shift(M - E - 1, bits);  // j from E to M
    const FxRow& rm = rowE(M - 1);                 // whose input unit is M's
    fx D[3], S[3];
    double Fc[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const fx v = dbl_to_fx(dbl_scale(V[i], (FX_BITS + 1 - M) * (1 << 20)));
      const fx jm = fx_moved(j[i], um), U = fx_add(jm, rm.fh[i]);
      D[i] = fx_sub(v, U);
      S[i] = fx_add(v, U);
      // U - V - f
      const fx u = fx_sub(fx_sub(jm, rm.fh[i]), v);
      Fc[i] = fx_to_dbl(fx_mul(u, W.m), (M + W.eb - (FX_BITS - 1)) * (1 << 20));
    }
    force(Fc);
    fx_solid(c, W, E, P, M, D, S, bits, H);
  }
  {
    fx d0 = L.d0;
    if constexpr (KIND == FX_MIXED) {
      const fx b = fx_mul(fx_sub(x0, fx_add(d0, d0)), W.w);
      d0 = fx_add(fx_add(d0, fx_add(b, b)), H.d0);
    }
    put(0, fx_to_dbl(d0, (P - (FX_BITS - 1)) * (1 << 20)));
  }
  const int o20 = (E - (FX_BITS - 1)) * (1 << 20);
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const fx s = fx_add(x[2 * k + 1], x[2 * k + 2]), b = fx_sub(x[2 * k + 1], x[2 * k + 2]);
    fx S, A;
    fx_fluid_pair(c, re, s, b, L, k, &S, &A);
    if constexpr (KIND == FX_MIXED) {
      const fx eq = k < 3 ? H.eq[k]
                          : fx_sub(fx_prod(fx_edge(k, H.D), fx_edge(k, H.S)), H.t6);
      S = fx_add(fx_add(S, eq), fx_mul(fx_sub(s, fx_shl(S, 2)), W.w));
      A = fx_add(fx_sub(A, fx_mul(fx_add(b, fx_shl(A, 2)), W.w)),
                 k < 3 ? H.G[k] : fx_edge(k, H.Ge));
    }
    put(2 * k + 1, fx_to_dbl(fx_add(S, A), o20));
    put(2 * k + 2, fx_to_dbl(fx_sub(S, A), o20));
  }
}

// Exponents of a cell with the deviations d (and, FX_MIXED, velocity and weight
// V), E0 = fx_e0 of the force.  slow: outside the range (the FP64 form takes
// it); quiet: exactly quiescent without forces (the result is zero)
struct FxRange {
  int E, Ps;
  bool slow, quiet;
};
template <int KIND>
FX_FN FxRange fx_range(const double* d, const double* V, int E0) {
  constexpr int up = KIND == FX_MIXED ? 1 : 0;
  uint32_t mf = 0u, me = 0u, t = 0u;
#pragma unroll
  for (int q = 1; q < 19; ++q) {
    const uint32_t h = (uint32_t)dbl_hi(d[q]) & 0x7fffffffu;
    if (q < 7) mf = h > mf ? h : mf;
    else me = h > me ? h : me;
  }
  const uint32_t h0 = (uint32_t)dbl_hi(d[0]) & 0x7fffffffu;
  const uint32_t me2 = me + (1u << 20), m = mf > me2 ? mf : me2;
  const int e0 = fx_exp(h0), e1 = fx_exp(m);
  FxRange r;
  const int raw = e1 > e0 - 3 ? e1 : e0 - 3;
  r.E = raw + up > E0 ? raw + up : E0;
  r.Ps = (e0 > fx_p0(E0) ? e0 : fx_p0(E0)) + up;
  // deviations far below the force, but not zero, would lose bits to it (a
  // flow has left that state after a step from rest)
  r.slow = raw < E0 - 3 && (mf | me | h0) != 0u;
  if constexpr (KIND == FX_MIXED) {
    for (int i = 0; i < 3; ++i) {
      const uint32_t h = (uint32_t)dbl_hi(V[i]) & 0x7fffffffu;
      t = h > t ? h : t;
    }
    // B V, and B times the products of U (|U| < 2^eu) and V, fit beside the d_q
    const int ev = fx_exp(t), eb = fx_weight_exp(V[3]);
    int eu = (raw > E0 ? raw : E0) + 3;
    eu = eu > ev ? eu : ev;
    const int ew = (2 * eu > ev - 3 ? 2 * eu : ev - 3) + eb;
    r.E = r.E > ew ? r.E : ew;
    r.slow = r.slow || ev > FX_VMAX;
  }
  r.slow = r.slow || r.E > FX_ETOP;
  r.quiet = E0 <= FX_EMIN && (mf | me | h0 | t) == 0u;
  if (r.slow) {  // the lane's fixed-point result is not used
    r.E = E0;
    r.Ps = fx_p0(E0);
  }
  return r;
}

// ---- One exponent E for all of a cell: every |d_q| below 2^E (FX_MIXED: below
// 2^(E - 1), and |V| below 2^(E + 2)), with the exponents E + 1, P = E + 3 and
// M = E + 4.  Every unit is then at its largest for the cell's values, and the
// error bounds are checked with it.
constexpr int FX_EMAX = FX_ETOP - 1, FX_EMAX_SOLID = FX_ETOP - 2, FX_VBITS_MIXED = 3;
FX_FN int fx_top(const double* d) {
  uint32_t m = 0u;
  for (int q = 0; q < 19; ++q) {
    const uint32_t h = (uint32_t)dbl_hi(d[q]) & 0x7fffffffu;
    m = h > m ? h : m;
  }
  return (int)m;
}
FX_FN int fx_top_velocity(int top, const double* V, int bits) {
  for (int a = 0; a < 3; ++a) {
    const int h = (dbl_hi(V[a]) & 0x7fffffff) - (bits << 20);
    top = h > top ? h : top;
  }
  return top;
}
FX_FN int fx_exponent(int top, int E0) {
  const int E = fx_exp((uint32_t)top);
  return E > E0 ? E : E0;
}
FX_FN void fx_row(const FxRates& c, const double* f, int E0, int i, FxRow& r) {
  fx_row_at(c, f, E0 + i + 1, E0 + i + 3, r);
}
template <int KIND, typename Force, typename Put>
FX_FN void fx_collide(const FxRates& c, const FxRow& row, int E, const double* d, const double* V,
                      Force force, Put put) {
  FxRow m = row;  // of the exponent M - 1 = E + 3
  for (int a = 0; a < 3; ++a) m.fh[a] = fx_half(fx_half(row.fh[a]));
  fx_cell<KIND>(
      c, [&](int e) -> const FxRow& { return e == E + 1 ? row : m; },
      [&](int) -> const FxRow& { return row; }, E + 3, E + 1, E + 3, d, V, force, put);
}

}  // namespace psm
