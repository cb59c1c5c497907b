// mx_kepler_short.cuh -- the Kepler drift of a short step (arXiv 2601.16791,
// Sec. 2) with fewer FP64 instructions, for mx_kepler_drift and for systems of
// light big bodies (SysDev::split).
//
// What bounds the drift is FP64 issue, 64 cycles a warp instruction:
// kepler_drift takes about 105 on a short step.  Here Kepler's equation is
// solved in relative variables, sigma = s r0/h near 1, with
//   a = eta h/r0^2, b = beta (h/r0)^2, m = mu h^2/r0^3, c = m - b,
//   F(sigma) = sigma + a U2 + c U3 - 1 = 0,  U_k = sigma^k c_k(b sigma^2),
// in FP32 first; one FP64 evaluation there gives the last correction d (about
// 1e-7), and U1..U3 are carried to sigma + d by their Taylor steps.  The state
// moves by the differences f - 1 = -m U2, g = h - h m U3, gd - 1 = -m U2/rho,
// fd = -(m/h) U1/rho, rho = r/r0 = 1 + a U1 + c U2.  About 77 FP64
// instructions.  Against 64-bit-mantissa arithmetic over 20,000 orbits (1 to 15
// AU, h = 10 d): position 5.7e-17 rms (kepler_drift 5.7e-17), velocity 6.8e-17
// (7.6e-17).  Measured: mx_kepler_drift of 200,000 bodies 75.4 -> 55.4 us a call;
// k_jump_drift of 64 disks with 2.4 million bodies 481 -> 375 us a launch, three
// steps of them 4.1 -> 3.7 ms.
#pragma once
#include "mx_kepler.cuh"
#include "mx_split.cuh"

namespace mx {

// Advances the state and returns true, or returns false with it untouched:
// |b| above 0.12 (a step of about 0.35 rad of mean motion), |a| or |c| above 0.25,
// a value off FP32's range or not finite, or a correction above 4e-6.  (A warp
// with one such body runs both forms, so the range covers the whole disk of the
// usual step, about a twentieth of the innermost orbit: with |b| to 0.04 an
// embryo disk from 0.5 AU at h = 6 d took 83 us a launch against 68 before.)
__device__ __forceinline__ bool kepler_drift_short(double mu, double h, double& x, double& y,
                                                   double& z, double& u, double& v, double& w) {
  const double r02 = fma(x, x, fma(y, y, z * z));
  const double ir0 = rsqrt_d(r02);
  const double v2 = fma(u, u, fma(v, v, w * w));
  const double eta = fma(x, u, fma(y, v, z * w));
  const double hi = h * ir0, q0 = hi * ir0, p = mu * ir0;
  const double hi2 = hi * hi;
  const double m = p * hi2;
  const double b = fma(-v2, hi2, m + m);
  const double a = eta * q0;
  const double c = m - b;
  // r0 in 2^-40 .. 2^40 and m above 2^-80 (h = 0 goes the general way)
  const int hr = __double2hiint(r02) >> 20;
  if (!(hr > 1023 - 80 && hr < 1023 + 80 && __double2hiint(m) >= (1023 - 80) << 20 &&
        abs_le(b, 0.12) && abs_le(a, 0.25) && abs_le(c, 0.25)))
    return false;
  const float af = ff_of(a).h, bf = ff_of(b).h, cf = ff_of(c).h;
  // FP32: the series inverted to third order, then two Halley corrections
  float s = fmaf(af, fmaf(0.5f, af, -0.5f), fmaf(cf, -1.0f / 6.0f, 1.0f));
  float u0, u1, u2, u3;
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const float s2 = s * s, zf = bf * s2;
    u2 = s2 * fmaf(-zf, fmaf(-zf, 1.0f / 720.0f, 1.0f / 24.0f), 0.5f);
    u3 = s2 * s * fmaf(-zf, fmaf(-zf, 1.0f / 5040.0f, 1.0f / 120.0f), 1.0f / 6.0f);
    u1 = fmaf(-bf, u3, s);
    u0 = fmaf(-bf, u2, 1.0f);
    const float F = fmaf(cf, u3, fmaf(af, u2, s - 1.0f));
    const float Fp = fmaf(cf, u2, fmaf(af, u1, 1.0f)), Fpp = fmaf(cf, u1, af * u0);
    s -= __fdividef(F * Fp, fmaf(Fp, Fp, -0.5f * F * Fpp));
  }
  // FP64 at sigma = s (24 bits, so s - 1 and s^2 are exact): the series with
  // their tails from z^4 on in FP32 (1e-8 of the sum)
  const double sd = bits_to_double(s);
  const double s2 = sd * sd;
  const double zd = b * s2;
  const float zf = ff_of(zd).h;
  const double t2 = bits_to_double(fmaf(-zf, fmaf(-zf, 1.0f / 87178291200.0f, 1.0f / 479001600.0f),
                                        1.0f / 3628800.0f));
  const double t3 = bits_to_double(fmaf(-zf, fmaf(-zf, 1.0f / 1307674368000.0f, 1.0f / 6227020800.0f),
                                        1.0f / 39916800.0f));
  const double c2 =
      fma(-zd, fma(-zd, fma(-zd, fma(-zd, t2, 1.0 / 40320.0), 1.0 / 720.0), 1.0 / 24.0), 0.5);
  const double c3 =
      fma(-zd, fma(-zd, fma(-zd, fma(-zd, t3, 1.0 / 362880.0), 1.0 / 5040.0), 1.0 / 120.0), 1.0 / 6.0);
  const double U2 = s2 * c2, U3 = (s2 * sd) * c3;
  const double U1 = fma(-b, U3, sd);
  const double F = fma(c, U3, fma(a, U2, bits_to_double(s - 1.0f)));
  const double Fp = fma(c, U2, fma(a, U1, 1.0));
  // d = -q (1 + q F''/(2 F')), q = F/F' in a pair of FP32 numbers
  const FF r = ff_rcp(ff_of(Fp)), q = ff_mul(ff_of(F), r);
  if (!(fabsf(q.h) < 4e-6f)) return false;
  const float half = 0.5f * fmaf(cf, u1, af * u0) * r.h * q.h;
  const double d = -(bits_to_double(q.h) + bits_to_double(fmaf(q.h, half, q.l)));
  const double hd = 0.5 * d;
  const double M2 = fma(hd, U1, U2);              // U2, U0, U1 halfway to sigma + d
  const double M0 = fma(-b, M2, 1.0);
  const double M1 = fma(hd, M0, U1);
  const double W1 = fma(d, M0, U1), W2 = fma(d, M1, U2), W3 = fma(d, M2, U3);
  const double ir = rcp_d(fma(c, W2, fma(a, W1, 1.0)));
  const double f1 = -m * W2;
  const double g = fma(-h, m * W3, h);
  const double fd = -(p * q0) * (W1 * ir);
  const double gd1 = f1 * ir;
  const double f = fma(-m, W2, 1.0);
  const double xn = fma(f, x, g * u), yn = fma(f, y, g * v), zn = fma(f, z, g * w);
  u = fma(fd, x, fma(gd1, u, u));
  v = fma(fd, y, fma(gd1, v, v));
  w = fma(fd, z, fma(gd1, w, w));
  x = xn;
  y = yn;
  z = zn;
  return true;
}

// The drift of a system's body: the short form where `light` and it applies.
__device__ __forceinline__ bool kepler_drift_sel(bool light, double mu, double h, int maxit,
                                                 double& x, double& y, double& z, double& u,
                                                 double& v, double& w) {
  // (a cap below ten iterations keeps the solver that counts them; on a short
  // step it takes two or three)
  if (light && maxit >= 10 && kepler_drift_short(mu, h, x, y, z, u, v, w)) return true;
  return kepler_drift(mu, h, maxit, x, y, z, u, v, w);
}

}  // namespace mx
