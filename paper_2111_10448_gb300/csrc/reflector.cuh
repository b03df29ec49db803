// The scalars of a Householder reflector.
#pragma once

namespace tts {

// Reflector of a column with squared norm g over rows i.. and head x0: v = (x0 - alpha,
// rest), R(i, i) = alpha, beta = 2 / (v^T v) = 1 / (g + |x0| sqrt(g)) (0 for a zero
// column and for one with a NaN).  One lane's serial chain in every QR step, so the root and the quotient
// are Newton iterations from the 20-bit approximate instructions (two each: five dependent
// FMAs, where the library's root and division took about 690 and 670 cycles).  The last
// step of each adds the correction from the residual, g - s^2 and 1 - d q, to the iterate
// (Markstein, IBM J. Res. Dev. 34, 1990): with 2^-40 in iterate and slope the sum before its
// rounding is within 2^-25 of a unit in the last place, so that all but one result in some
// 10^7 are the nearest.  (A last step 1/2 - s h, which does not see g, left 22 % of
// the roots one unit off.)
__device__ __forceinline__ void reflector(double g, double x0, double& alpha, double& b, double& v0) {
  alpha = 0.0, b = 0.0, v0 = 0.0;
  if (!(g > 0.0)) return;
  const int e = (__double2hiint(g) >> 20) & 0x7ff;
  double nx;
  if (e > 40 && e < 2000) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(g));
    double s = g * y, h = 0.5 * y;
    const double r = fma(-s, h, 0.5);
    s = fma(s, r, s);
    h = fma(h, r, h);
    nx = fma(fma(-s, s, g), h, s);
    const double d = fma(fabs(x0), nx, g);
    double q;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(q) : "d"(d));
    q = fma(q, fma(-d, q, 1.0), q);
    b = fma(q, fma(-d, q, 1.0), q);
  } else {
    nx = sqrt(g);
    b = 1.0 / fma(fabs(x0), nx, g);
  }
  alpha = -copysign(nx, x0);
  v0 = x0 - alpha;
}

}  // namespace tts
