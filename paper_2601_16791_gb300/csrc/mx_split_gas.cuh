// mx_split_gas.cuh -- the gas drag and the velocity update of a half kick in
// pairs of FP32 numbers (mx_split.cuh; arXiv 2601.16791, Sec. 3.1), shared by
// the step's kick and the catch-up of deferred planetesimals (systems whose
// masses are fixed: no gaps in the gas).
//
// What stays FP64: the state, the gas velocity at the body (g) and so the
// relative velocity dv, which is a small difference of large velocities; the
// pairs inside a changeover shell and the disk's gravity; the impulse h times
// the sum of all accelerations, and its addition to the velocity.
// Held in FP32 pairs (about 45 bits): the far pairs' sum (mx_split.cuh), rho_g,
// 1/c_s, |dv|, Re, Ma, C_D and the drag coef dv.  45 bits are 2.8e-14 of the
// drag, so its share of the velocity's error is 2.8e-14 h/t_stop |dv|: with
// h/t_stop up to 2^-6 and |dv| up to a tenth of the velocity, 4e-17 of it,
// below half a unit of its last place.  A body with a larger h/t_stop, or whose
// Re, Ma or |dv| leaves the range FP32 holds with room, keeps the FP64 drag
// (drag_fp64), as mx_gas_drag and mx_accel, which return the drag itself, do.
#pragma once
#include "mx_physics.cuh"
#include "mx_split.cuh"

namespace mx {

// drag_const in pairs.
struct DragSplit {
  bool in_gas;
  double offu, offv, offw;   // dv = (u + offu, v + offv, w + offw), u barycentric
  FF inv_cs, re_k, coef_k;   // Ma = inv_cs |dv|, Re = re_k |dv|, coef = C_D coef_k |dv|
  double adg[2];             // disk gravity (x, y), zero unless enabled
};

__device__ __forceinline__ DragSplit drag_split(const SysDev& S, double x, double y, double hp0,
                                                double hp1, double hp2, double rp_cm, double kd) {
  DragSplit c;
  double g;
  FF rho;
  c.adg[0] = c.adg[1] = 0.0;
  if (S.flare_quarter && S.gamma_one && S.rc_inf && !S.dg_on) {
    // as gas_at, with g by FP64 rsqrt chains and the rest in pairs
    const double R2 = fma(x, x, y * y);
    const double iR = rsqrt_d(R2);
    const double R = R2 * iR;
    c.in_gas = !(__double_as_longlong(R) < __double_as_longlong(S.r_in));
    const double ih = rsqrt_d(R);                                  // R^-1/2
    const double t = fma(-2.0 * S.c_eta, R * ih, 1.0);             // 1 - 2 eta
    g = (S.sqrt_mu0 * ih) * (t * rsqrt_d(t)) * iR;
    const FF ih2 = ff_of(ih), iR2 = ff_of(iR);
    const FF q = ff_rsqrt(ih2);                                    // R^1/4
    c.inv_cs = ff_mul(q, ff_of(S.inv_c_cs));
    const FF rmh = ff_mul(iR2, ff_mul(q, ih2));                    // R^-5/4
    rho = ff_mul(ff_mul(ff_of(S.c_rho), ff_mul(ff_of(S.sigma1), iR2)), rmh);
  } else {
    const GasAt q = gas_at(S, x, y);
    c.in_gas = q.in_gas;
    g = q.g;
    c.inv_cs = ff_of(q.inv_cs);
    rho = ff_of(q.rho);
    c.adg[0] = q.adg[0];
    c.adg[1] = q.adg[1];
  }
  c.offu = fma(g, y, hp0);
  c.offv = fma(-g, x, hp1);
  c.offw = hp2;
  c.re_k = ff_mul(ff_mul(ff_of(S.c_re), ff_of(rp_cm)), ff_mul(rho, c.inv_cs));
  c.coef_k = ff_mul(ff_mul(ff_of(S.cd_scale), ff_of(kd)), rho);
  return c;
}

// The FP64 drag of the same body (gas_at, drag_const, gas_drag_coef): coef dv.
static __device__ __noinline__ void drag_fp64(const SysDev& S, double x, double y, double hp0,
                                              double hp1, double hp2, double rp_cm, double kd,
                                              double u, double v, double w, double* a, int kb_in,
                                              int* kb_out) {
  const GasAt q = gas_at(S, x, y);
  const double coef = gas_drag_coef(S, drag_const(S, q, x, y, hp0, hp1, hp2, rp_cm, kd), u, v, w, a,
                                    kb_in, kb_out);
  for (int c = 0; c < 3; ++c) a[c] *= coef;
}

// gas_drag_coef in pairs (Eqs. 3, 7) for a half kick of h: coef of -coef dv, dv
// written to d[3]; false where the values leave the range above.
__device__ __forceinline__ bool drag_coef_split(const SysDev& S, const DragSplit& c, float h,
                                                double u, double v, double w, FF (&d)[3], FF& coef,
                                                int kb_in, int* kb_out) {
  d[0] = ff_of(u + c.offu);
  d[1] = ff_of(v + c.offv);
  d[2] = ff_of(w + c.offw);
  const FF d2 = ff_norm2(d[0].h, d[0].l, d[1].h, d[1].l, d[2].h, d[2].l);
  const FF dm = ff_mul(d2, ff_rsqrt(d2));
  const FF Ma = ff_mul(dm, c.inv_cs), Re = ff_mul(dm, c.re_k);
  if (!(d2.h > 1e-28f && d2.h < 1e8f && Ma.h > 1e-12f && Ma.h < 1e4f && Re.h > 1e-10f && Re.h < 1e10f))
    return false;
  const int kb = (kb_in >= 0) ? kb_in : ((Re.h < 1e5f || (Re.h == 1e5f && Re.l < 0.0f)) ? 0 : 1);
  *kb_out = kb;
  const FF k16 = kb ? FF{0x1.47ae14p-2f, 0x1.eb851ep-28f} : FF{0x1.47ae14p-1f, 0x1.eb851ep-27f};
  const FF D = ff_add(FF{240.0f, 0.0f}, ff_scale(Re, 64.0f));
  const FF maD = ff_mul(ff_mul(FF{0x1.d70a3ep-3f, -0x1.1eb852p-28f}, Ma), D);   // 0.23 Ma D
  const FF den1 = ff_add(ff_mul(Re, ff_add(FF{10.0f, 0.0f}, Re)), maD);
  const FF A = ff_add(FF{0x1.99999ap0f, -0x1.99999ap-26f}, Ma);                  // 1.6 + Ma
  const FF r = ff_rcp(ff_mul(den1, A));
  const FF t2 = ff_add(ff_scale(Ma, 2.0f), k16);
  FF cd;
  if (S.cd_mode == 1) {
    const FF first = ff_mul(ff_mul(D, A), r);
    cd = ff_add(ff_mul(first, first), ff_mul(ff_mul(t2, den1), r));
  } else {
    cd = ff_mul(ff_add(ff_mul(t2, den1), ff_mul(D, A)), r);
  }
  coef = ff_mul(ff_mul(cd, c.coef_k), dm);
  return fabsf(h * coef.h) <= 0x1p-6f;
}

// u - h (t - a): t the accelerations held in pairs (sign reversed), a the FP64
// ones.  The impulse is one FP64 product, added with one rounding.
__device__ __forceinline__ double kick_split(double h, FF t, double a, double u) {
  double s = bits_to_double(t.h) + bits_to_double(t.l);
  if (__double_as_longlong(a) != 0) s -= a;   // zero for most bodies
  return fma(-h, s, u);
}

// The half kicks of one body (nkick of h each): the far pairs' sum acc (sign
// reversed), the FP64 acceleration (ax, ay, az; pairs inside a changeover
// shell, disk gravity) and, with drag, the gas at (x, y).  branch(kk) gives the
// k branch of Eq. 7 to take (-1: from Re), keep(kk, kb) receives the one taken.
template <class In, class Out>
__device__ __forceinline__ void split_kicks(const SysDev& S, double h, int nkick,
                                            const SplitAcc& acc, double ax, double ay, double az,
                                            bool drag, const DragSplit& dc, double x, double y,
                                            double hp0, double hp1, double hp2, double rp,
                                            double kd, double& u, double& v, double& w,
                                            In&& branch, Out&& keep) {
  const FF gx{acc.xh, acc.xl}, gy{acc.yh, acc.yl}, gz{acc.zh, acc.zl};
#pragma unroll 1
  for (int kk = 0; kk < nkick; ++kk) {
    FF tx = gx, ty = gy, tz = gz;
    double bx = ax, by = ay, bz = az;
    if (drag && dc.in_gas) {
      const int kin = branch(kk);
      int kout = 0;
      FF d[3], coef;
      if (drag_coef_split(S, dc, ff_of(h).h, u, v, w, d, coef, kin, &kout)) {
        tx = ff_add(tx, ff_mul(coef, d[0]));
        ty = ff_add(ty, ff_mul(coef, d[1]));
        tz = ff_add(tz, ff_mul(coef, d[2]));
      } else {
        double a[3];
        drag_fp64(S, x, y, hp0, hp1, hp2, rp, kd, u, v, w, a, kin, &kout);
        bx -= a[0];
        by -= a[1];
        bz -= a[2];
      }
      keep(kk, kout);
    }
    u = kick_split(h, tx, bx, u);
    v = kick_split(h, ty, by, v);
    w = kick_split(h, tz, bz, w);
  }
}

}  // namespace mx
