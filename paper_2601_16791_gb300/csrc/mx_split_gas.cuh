// mx_split_gas.cuh -- the gas drag and the velocity update of a half kick in
// pairs of FP32 numbers (mx_split.cuh; arXiv 2601.16791, Sec. 3.1), shared by
// the step's kick and the catch-up of deferred planetesimals (systems whose
// masses are fixed: no gaps in the gas).
//
// What stays FP64: the state, the gas velocity at the body (g) and so the
// relative velocity dv, which is a small difference of large velocities.
// Formed in FP32 pairs (about 45 bits): rho_g, 1/c_s, |dv|, Re, Ma, C_D and
// the impulse h (a_grav - coef dv), which then enters the velocity with one
// FP64 rounding.  The drag changes a velocity by h/t_stop times dv, below
// 1e-3 of it for an explicit kick to make sense, so 45 bits of it are finer
// than the velocity's own last place.  mx_gas_drag and mx_accel, which return
// the drag itself, keep FP64 (mx_physics.cuh), and so does a body whose Re, Ma
// or |dv| leave the range FP32 holds with room (drag_coef_fp64).
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

// The FP64 coefficient of the same body (gas_at, drag_const, gas_drag_coef).
static __device__ __noinline__ double drag_coef_fp64(const SysDev& S, double x, double y, double hp0,
                                                     double hp1, double hp2, double rp_cm, double kd,
                                                     double u, double v, double w, int kb_in,
                                                     int* kb_out) {
  const GasAt q = gas_at(S, x, y);
  double dvec[3];
  return gas_drag_coef(S, drag_const(S, q, x, y, hp0, hp1, hp2, rp_cm, kd), u, v, w, dvec, kb_in,
                       kb_out);
}

// gas_drag_coef in pairs (Eqs. 3, 7): coef of -coef dv, dv written to d[3];
// false where the values leave the range above (nothing else written).
__device__ __forceinline__ bool drag_coef_split(const SysDev& S, const DragSplit& c, double u,
                                                double v, double w, FF (&d)[3], FF& coef, int kb_in,
                                                int* kb_out) {
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
  return true;
}

// u - h (acc + coef dv): acc the gravity with its sign reversed.
__device__ __forceinline__ double kick_split(FF h, FF acc, FF coef, FF dv, double u) {
  const FF p = ff_mul(h, ff_add(acc, ff_mul(coef, dv)));
  return u - (bits_to_double(p.h) + bits_to_double(p.l));
}
__device__ __forceinline__ double kick_split(FF h, FF acc, double u) {
  const FF p = ff_mul(h, acc);
  return u - (bits_to_double(p.h) + bits_to_double(p.l));
}

// A body's gravity, sign reversed, from the far pairs' sum and the FP64 one
// (pairs inside a changeover shell, disk gravity; zero for most bodies).
struct SplitGrav {
  FF x, y, z;
};

__device__ __forceinline__ SplitGrav split_gravity(const SplitAcc& acc, double ax, double ay,
                                                   double az) {
  SplitGrav g{{acc.xh, acc.xl}, {acc.yh, acc.yl}, {acc.zh, acc.zl}};
  if (__double_as_longlong(ax) != 0 || __double_as_longlong(ay) != 0 || __double_as_longlong(az) != 0) {
    g.x = ff_add(g.x, ff_neg(ff_of(ax)));
    g.y = ff_add(g.y, ff_neg(ff_of(ay)));
    g.z = ff_add(g.z, ff_neg(ff_of(az)));
  }
  return g;
}

// The half kicks of one body (nkick of h each) with the gravity g and, with drag, the gas at (x, y).  kick_branch(kk) gives the k
// branch of Eq. 7 to take (-1: from Re), keep(kk, kb) receives the one taken.
template <class In, class Out>
__device__ __forceinline__ void split_kicks(const SysDev& S, double kick_h, int nkick,
                                            const SplitGrav& g, bool drag, const DragSplit& dc,
                                            double x, double y, double hp0, double hp1, double hp2,
                                            double rp, double kd, double& u, double& v, double& w,
                                            In&& branch, Out&& keep) {
  const FF h = ff_of(kick_h);
#pragma unroll 1
  for (int kk = 0; kk < nkick; ++kk) {
    FF d[3] = {}, coef{0.0f, 0.0f};
    if (drag && dc.in_gas) {
      const int kin = branch(kk);
      int kout = 0;
      if (!drag_coef_split(S, dc, u, v, w, d, coef, kin, &kout))
        coef = ff_of(drag_coef_fp64(S, x, y, hp0, hp1, hp2, rp, kd, u, v, w, kin, &kout));
      keep(kk, kout);
      u = kick_split(h, g.x, coef, d[0], u);
      v = kick_split(h, g.y, coef, d[1], v);
      w = kick_split(h, g.z, coef, d[2], w);
    } else {
      u = kick_split(h, g.x, u);
      v = kick_split(h, g.y, v);
      w = kick_split(h, g.z, w);
    }
  }
}

}  // namespace mx
