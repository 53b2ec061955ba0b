// One design variable's step of the method of moving asymptotes (Svanberg, Int. J. Numer. Meth.
// Eng. 24, 1987; asymptote and move-limit rules of his 2007 course notes) for the design problem
// of eq. topopt, which bounds the densities and has no other constraint, so every variable's
// convex subproblem is solved in closed form.  Host and device: the functions that run in
// k_mma_step also compile for the host, where they are checked against each other and the rules
// (with the host's division and square root).
#pragma once
#include <math.h>
#include <string.h>

#if defined(__CUDACC__)
#define PC_HD __host__ __device__ __forceinline__
#else
#define PC_HD inline
#endif

// Order of doubles on the integer units: the device's FP64 unit is the bound of this update, and a comparison
// costs as much there as a multiply-add.
PC_HD long long mma_bits(double v) {
#if defined(__CUDA_ARCH__)
  return __double_as_longlong(v);
#else
  long long b;
  memcpy(&b, &v, sizeof(b));
  return b;
#endif
}
PC_HD long long mma_key(double v) {  // ascending with v (not NaN)
  const long long b = mma_bits(v);
  return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
PC_HD double mma_min(double a, double b) { return mma_key(a) < mma_key(b) ? a : b; }
PC_HD double mma_max(double a, double b) { return mma_key(a) > mma_key(b) ? a : b; }
PC_HD int mma_exponent(double v) { return (int)((mma_bits(v) >> 52) & 0x7ff) - 1023; }  // infinities, NaN: 1024
PC_HD bool mma_below(double v, int e) { return mma_exponent(v) < e; }                    // |v| < 2^e
PC_HD bool mma_within(double v, int e) { return mma_below(v, e) && mma_exponent(v) >= -e; }
// 1 / v and 1 / sqrt(v) of a normal v > 0 whose result is normal too, to an ulp, from the hardware's approximation y
// of some 20 bits: with the residual e = 1 - v y (1 - v y^2) the result is y (1 - e)^-1 (y (1 - e)^-1/2), and one
// step of third order takes that series to e^2 (Householder, The Numerical Treatment of a Single Nonlinear Equation,
// 1970), e^3 being 2^-57 to 2^-60.
PC_HD double mma_inv(double v) {
#if defined(__CUDA_ARCH__)
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(v));
  const double e = fma(-v, y, 1.0);
  return fma(y, fma(e, e, e), y);
#else
  return 1.0 / v;
#endif
}
PC_HD double mma_rsqrt(double v) {
#if defined(__CUDA_ARCH__)
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(v));
  const double e = fma(-v * y, y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
#else
  return 1.0 / sqrt(v);
#endif
}

// x: current value; df: d(objective)/dx of the objective being MAXIMISED.
// xo1, xo2: the two previous values; low, upp: the previous asymptotes (all four ignored for
// iter < 2).  On return they hold the values for the next call, and *xnew the new value.
// The rules as stated, for any values (infinities and NaN among them).
PC_HD void mma_box_update(double x, double df, int iter, double xmin, double xmax, double* xo1, double* xo2,
                           double* low, double* upp, double* xnew) {
  const double span = xmax - xmin;
  double L, U;
  if (iter < 2) {
    L = x - 0.5 * span;
    U = x + 0.5 * span;
  } else {
    // Shrink the asymptote distances where x oscillates, widen them where it keeps its direction.
    const double trend = (x - *xo1) * (*xo1 - *xo2);
    const double g = trend < 0.0 ? 0.7 : (trend > 0.0 ? 1.2 : 1.0);
    L = x - g * (*xo1 - *low);
    U = x + g * (*upp - *xo1);
    L = fmin(fmax(L, x - 10.0 * span), x - 0.01 * span);
    U = fmin(fmax(U, x + 0.01 * span), x + 10.0 * span);
  }
  const double alpha = fmax(fmax(xmin, L + 0.1 * (x - L)), x - 0.5 * span);
  const double beta = fmin(fmin(xmax, U - 0.1 * (U - x)), x + 0.5 * span);
  // Minimise g = -f through the model p / (U - x) + q / (x - L), whose slope at x is dg.
  const double dg = -df;
  const double pos = fmax(dg, 0.0), neg = fmax(-dg, 0.0), reg = 1e-5 / span;
  const double p = (U - x) * (U - x) * (1.001 * pos + 0.001 * neg + reg);
  const double q = (x - L) * (x - L) * (0.001 * pos + 1.001 * neg + reg);
  const double sp = sqrt(p), sq = sqrt(q);
  const double xs = (sp * L + sq * U) / (sp + sq);
  *xnew = fmin(fmax(xs, alpha), beta);
  *xo2 = *xo1;
  *xo1 = x;
  *low = L;
  *upp = U;
}

// The update of k_mma_step; reg: 1e-5 / (xmax - xmin).  The same rules in the distances a = U - x and b = x - L: the limits on the asymptotes are limits on a and
// b, and with p / a^2 and q / b^2 the slopes of the model and r = sqrt((q / b^2) / (p / a^2)) its minimum
// (sqrt(p) L + sqrt(q) U) / (sqrt(p) + sqrt(q)) is x + a b (r - 1) / (a + b r).  31 FP64 instructions with
// one reciprocal and one reciprocal square root, where the rules as stated take 86 (comparisons among them).
PC_HD void mma_box_step(double x, double df, int iter, double xmin, double xmax, double reg, double* xo1, double* xo2,
                        double* low, double* upp, double* xnew) {
  const double span = xmax - xmin;
  // (a box small against its values is left to the rules: there the order of the roundings shows)
  bool plain = mma_within(span, 200) && mma_exponent(x) < mma_exponent(span) + 16 && mma_below(df, 500);
  if (iter >= 2)
    plain = plain && mma_below(*xo1, 500) && mma_below(*xo2, 500) && mma_below(*low, 500) && mma_below(*upp, 500);
  if (!plain) {
    mma_box_update(x, df, iter, xmin, xmax, xo1, xo2, low, upp, xnew);
    return;
  }
  double a = 0.5 * span, b = a;
  if (iter >= 2) {
    const double trend = (x - *xo1) * (*xo1 - *xo2);
    const long long tb = mma_bits(trend);
    const double g = (tb << 1) == 0 ? 1.0 : (tb < 0 ? 0.7 : 1.2);
    b = mma_min(mma_max(g * (*xo1 - *low), 0.01 * span), 10.0 * span);
    a = mma_min(mma_max(g * (*upp - *xo1), 0.01 * span), 10.0 * span);
  }
  const double alpha = mma_max(xmin, x - mma_min(0.9 * b, 0.5 * span));
  const double beta = mma_min(xmax, x + mma_min(0.9 * a, 0.5 * span));
  const double ad = fabs(df), big = 1.001 * ad + reg, small = 0.001 * ad + reg;
  const double r = (df < 0.0 ? small : big) * mma_rsqrt(big * small);
  const double xs = x + (a * b) * (r - 1.0) * mma_inv(a + b * r);
  *xnew = mma_min(mma_max(xs, alpha), beta);
  *xo2 = *xo1;
  *xo1 = x;
  *low = x - b;
  *upp = x + a;
}
