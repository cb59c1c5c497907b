// mx_split.cuh -- the kick's pair sum in pairs of FP32 numbers (arXiv
// 2601.16791, Sec. 2.1.3), for systems of light big bodies (SysDev::split) and
// targets outside a big body's changeover shell.
//
// What bounds the pair sum: FP64 issues one warp instruction per scheduler in
// 64 cycles on sm_103a, FP32 one per cycle (both measured), so the 17 FP64
// instructions of pair_acc take about 1,100 cycles for 32 pairs.  The
// same pair in pairs of FP32 numbers (a value kept as hi + lo, 48 bits) takes
// about 115 instructions.
//
// What the precision is: the state, the jump, the impulse h a and its addition
// to the velocity stay FP64.  In FP32 pairs are a far pair's acceleration
// mu d/s^3, with a relative error of about 1.5e-14 (rms, against 80-bit
// arithmetic; mu itself is held to 48 bits), and the sum of the far pairs, or
// of kSplitSeg of them.  A half kick adds (h/2) a to a velocity; outside the
// changeover shell (3 Hill radii) that is at most a few 1e-4 of the velocity,
// so the split's share of the new velocity's error is below 1e-17 of it, where
// the FP64 rounding of the velocity itself is 1e-16.  A pair inside the shell,
// where the acceleration is largest and K varies, goes through the FP64
// pair_acc and is added in FP64, and so is every pair of a target outside the
// positions' grid below.  mx_accel, which returns accelerations, takes three
// FP32 parts instead (below).
//
// Measured: k_jump_kick with 2,000 big bodies and 200,000 planetesimals 11.8 ->
// 1.61 ms a launch (34 -> 251 G pairs/s, 84% of the issue slots filled); 301 big
// bodies and 20,011 planetesimals 0.43 -> 0.05 ms a launch.  64 gas disks of 2
// to 50 light bodies (2.4 million bodies; with the drag, see mx_split_gas.cuh)
// 2.35 -> 0.41 ms a launch, three steps (with the drift's short form) 12.0 ->
// 3.7 ms.
//
// Positions: each coordinate is cut on one grid for target and sources into
// three FP32 parts, x = x0 + x1 + x2 with x0 a multiple of 2^(k-23), x1 of
// 2^(k-47) and x2 the rest, |x| < 2^k, so that the differences of the first two
// parts are exact.  x2 and its difference round at 2^(k-73) and 2^(k-72): a
// separation is off by at most 2^(k-71), and pairs closer than 2^(k-17) go
// through FP64 (split_near2), so the others' separations keep 54 bits.
// k comes from the positions of the chunk's big bodies (never from the tile),
// so results do not depend on the tiling.  A body 300 AU out (k = 10) sends the
// pairs within 0.008 AU to FP64; the changeover shell of a lunar embryo at
// 0.5 AU has 0.0035 AU.
#pragma once
#include <limits.h>
#include "mx_common.cuh"
#include "mx_physics.cuh"

namespace mx {

constexpr int kSplitRun = 32;     // big bodies summed in FP32 pairs before the low parts are put back below the high ones
constexpr int kSplitMinK = -10;   // positions' grid: 2^k AU above the big bodies' coordinates,
constexpr int kSplitMaxK = 10;    // else the pair sum stays FP64 (FP32 range of mu/s^3)

__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }

// x = o0 + o1 + o2 on the grid of 2^k (|x| < 2^k).  Integer instructions but
// for the conversions.
__device__ __forceinline__ void split3(double x, int k, float& o0, float& o1, float& o2) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7ff;
  const unsigned long long m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
  // |x| = m 2^(e-1075) = v 2^(k-62) + rem 2^(e-1075)
  const int sh = (k - 62) - (e - 1075);
  unsigned long long v;
  if (sh <= 0) v = m << min(-sh, 63);
  else if (sh < 54) v = (m + (1ull << (sh - 1))) >> sh;
  else v = 0;
  const bool neg = (b >> 63) != 0;
  const long long s = neg ? -(long long)v : (long long)v;
  const long long a = (s + (1ll << 38)) >> 39;           // multiples of 2^(k-23)
  const long long r = s - (a << 39);                     // |r| <= 2^38
  const long long c = (r + (1ll << 14)) >> 15;           // multiples of 2^(k-47)
  const int q = (int)(r - (c << 15));                    // |q| <= 2^14
  o0 = __int2float_rn((int)a) * pow2f(k - 23);
  o1 = __int2float_rn((int)c) * pow2f(k - 47);
  o2 = __int2float_rn(q) * pow2f(k - 62);
  if (sh > 0 && e >= 885) {   // below 2^-138 AU nothing is left to keep
    const long long rem = (long long)m - (long long)(sh < 54 ? v << sh : 0);
    // in two factors: 2^(e-1075) itself may be below FP32's range
    const float f = __ll2float_rn(neg ? -rem : rem) * 0x1p-64f * pow2f(max(e - 1075 + 64, -126));
    o2 = __fadd_rn(o2, f);
  }
}

// The grid's k for bodies whose largest coordinate has the high word `hi`
// (sign off): twice the power of two above it.
__device__ __forceinline__ int split_k(int hi) { return max((hi >> 20) - 1022 + 1, kSplitMinK); }

__device__ __forceinline__ int abs_hi(double x) { return __double2hiint(x) & 0x7fffffff; }

// |x|, |y|, |z| < 2^k (false for a NaN)
__device__ __forceinline__ bool split_in_range(double x, double y, double z, int k) {
  const int lim = (k + 1023) << 20;
  return abs_hi(x) < lim && abs_hi(y) < lim && abs_hi(z) < lim;
}

// ------------------------------------------------------- pairs of FP32 numbers
// A value kept as h + l, l at most about an ulp of h: 48 bits.  Only rounding
// intrinsics, so that the compiler contracts nothing and every caller gets the
// same bits.
struct FF {
  float h, l;
};

__device__ __forceinline__ FF ff_fast(float a, float b) {   // |a| >= |b| or a = 0
  const float s = __fadd_rn(a, b);
  return FF{s, __fsub_rn(b, __fsub_rn(s, a))};
}

__device__ __forceinline__ FF ff_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float v = __fsub_rn(s, a);
  return FF{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v))};
}

__device__ __forceinline__ FF ff_add(FF a, FF b) {
  const FF s = ff_two_sum(a.h, b.h);
  return ff_fast(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}

__device__ __forceinline__ FF ff_mul(FF a, FF b) {
  const float p = __fmul_rn(a.h, b.h);
  return ff_fast(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p))));
}

__device__ __forceinline__ FF ff_neg(FF a) { return FF{-a.h, -a.l}; }

// A product with a power of two, exactly.
__device__ __forceinline__ FF ff_scale(FF a, float s) {
  return FF{__fmul_rn(a.h, s), __fmul_rn(a.l, s)};
}

// x^2 + y^2 + z^2 of three pairs.
__device__ __forceinline__ FF ff_norm2(float hx, float mx, float hy, float my, float hz, float mz) {
  const float px = __fmul_rn(hx, hx), py = __fmul_rn(hy, hy), pz = __fmul_rn(hz, hz);
  const float qx = __fmaf_rn(hx, hx, -px), qy = __fmaf_rn(hy, hy, -py),
              qz = __fmaf_rn(hz, hz, -pz);
  const FF s1 = ff_two_sum(px, py);
  const FF s = ff_two_sum(s1.h, pz);
  const float hm = __fmaf_rn(hx, mx, __fmaf_rn(hy, my, __fmul_rn(hz, mz)));
  return FF{s.h, __fmaf_rn(2.0f, hm, __fadd_rn(__fadd_rn(__fadd_rn(qx, qy), qz),
                                               __fadd_rn(s1.l, s.l)))};
}

// 1 - x y^2 = a + c for an estimate y of x^(-1/2), with y^2 = y2 + y2l:
// 1 - x.h y2 exactly as a = 1 - p and p's rounding, then the low parts.
__device__ __forceinline__ void ff_rsqrt_residual(FF x, float y, float& y2, float& y2l, float& a,
                                                  float& c) {
  y2 = __fmul_rn(y, y);
  y2l = __fmaf_rn(y, y, -y2);
  const float p = __fmul_rn(y2, x.h);
  const float pe = __fmaf_rn(y2, x.h, -p);
  a = __fsub_rn(1.0f, p);
  c = -__fmaf_rn(y2, x.l, __fmaf_rn(y2l, x.h, pe));
}

// x^(-1/2) = y (1 + e/2 + 3 e^2/8), x > 0 (x.h normal)
__device__ __forceinline__ FF ff_rsqrt(FF x) {
  const float y = rsqrtf(x.h);
  float y2, y2l, a, c;
  ff_rsqrt_residual(x, y, y2, y2l, a, c);
  const float e = __fadd_rn(a, c);
  const FF g = ff_fast(y, __fmul_rn(__fmul_rn(0.5f, y), a));
  return FF{g.h, __fadd_rn(g.l, __fmul_rn(y, __fmaf_rn(0.5f, c, __fmul_rn(__fmul_rn(0.375f, e), e))))};
}

// 1/x = y (1 + e + e^2)
__device__ __forceinline__ FF ff_rcp(FF x) {
  float y;
  asm("rcp.approx.f32 %0, %1;" : "=f"(y) : "f"(x.h));
  const float e = __fmaf_rn(-x.l, y, __fmaf_rn(-x.h, y, 1.0f));
  return ff_fast(y, __fmul_rn(y, __fmaf_rn(e, e, e)));
}

// A double's leading 48 bits, read off its bit pattern (zero below 2^-126; a
// NaN from 2^127 on, infinities and NaNs among them, so that the kick still
// reports them).  Integer and FP32 instructions only.
__device__ __forceinline__ FF ff_of(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned a = hi & 0x7fffffffu, sg = hi & 0x80000000u;
  if (a < (897u << 20)) return FF{0.0f, 0.0f};
  if (a >= (1150u << 20)) return FF{__uint_as_float(0x7fc00000u), 0.0f};
  const float h = __uint_as_float(sg | ((a - (896u << 20)) << 3) | (lo >> 29));
  const float r = __fmul_rn(__uint2float_rn(lo & 0x1fffffffu), 0x1p-52f);
  const float sc = __uint_as_float(sg | (((a >> 20) - 896u) << 23));
  return FF{h, __fmul_rn(r, sc)};
}

// A float as a double, exactly, by moving its bits (zero for a subnormal, a
// NaN for an infinity).
__device__ __forceinline__ double bits_to_double(float f) {
  const unsigned u = __float_as_uint(f), a = u & 0x7fffffffu;
  if (a < 0x00800000u) return 0.0;
  if (a >= 0x7f800000u) return __hiloint2double(0x7ff80000, 0);
  return __hiloint2double((int)((u & 0x80000000u) | ((a >> 3) + (896u << 20))), (int)(a << 29));
}

// One staged big body: its position in parts, mu as a pair, and the squared
// separation below which the pair belongs to the FP64 path.
struct alignas(16) SplitBig {
  float x0, x1, x2, y0, y1, y2, z0, z1, z2, muh, mul, near2;
};

struct SplitPos {
  float x0, x1, x2, y0, y1, y2, z0, z1, z2;
};

// hi + lo sums of a target's acceleration (sign reversed).
struct SplitAcc {
  float xh, xl, yh, yl, zh, zl;
};

// At least (1e-6 AU)^2: mu/s^3 stays in FP32's range.
__device__ __forceinline__ float near2_of(double rc2) {
  return fmaxf(to_float_bits(rc2) * 1.0001f, 1e-12f);
}

// A source's near2 on the grid of 2^k: its shell, and the pairs whose
// separation the grid does not hold to 54 bits (the positions, above).
__device__ __forceinline__ float split_near2(double rc2, int k) {
  return fmaxf(near2_of(rc2), pow2f(2 * (k - 17)));
}

// Whether the products of mu with powers of a far pair's 1/s keep their parts
// normal FP32 numbers: zero, or between 1e-18 and 1e3 (a body of 1e-14 of the
// Sun has 3e-18 AU^3/d^2); false for a NaN.
__device__ __forceinline__ bool split_mass(double mu) {
  const int hi = abs_hi(mu);
  return (hi >= 0x3c327000 && hi < 0x408f4000) || (hi == 0 && __double2loint(mu) == 0);
}

// A two-sum into the pair (h, l), with the term's low part.
__device__ __forceinline__ void split_add(float& h, float& l, float ph, float pl) {
  const FF s = ff_two_sum(h, ph);
  h = s.h;
  l = __fadd_rn(l, __fadd_rn(s.l, pl));
}

// d = a - b of parts, as hi + lo.
__device__ __forceinline__ void split_sub(float a0, float a1, float a2, float b0, float b1,
                                          float b2, float& h, float& m) {
  const float d0 = __fsub_rn(a0, b0), d1 = __fsub_rn(a1, b1), d2 = __fsub_rn(a2, b2);
  h = __fadd_rn(d0, d1);
  m = __fadd_rn(__fsub_rn(d1, __fsub_rn(h, d0)), d2);
}

// A far pair's mu d/s^3 as hi + lo by component.
struct SplitTerm {
  float xh, xl, yh, yl, zh, zl;
};

// A pair's mu d/s^3; returns false, f zero, for a pair inside near2 (without a
// branch, so that the caller's pairs overlap).
// 1/s^3 = y^3 (1 + 3e/2 + 15e^2/8) from the single-precision estimate y of
// 1/s, e = 1 - s^2 y^2, as in pair_weight.
__device__ __forceinline__ bool split_term(const SplitPos& t, const SplitBig& b, float near2,
                                           SplitTerm& f) {
  float hx, mx, hy, my, hz, mz;
  split_sub(t.x0, t.x1, t.x2, b.x0, b.x1, b.x2, hx, mx);
  split_sub(t.y0, t.y1, t.y2, b.y0, b.y1, b.y2, hy, my);
  split_sub(t.z0, t.z1, t.z2, b.z0, b.z1, b.z2, hz, mz);
  const FF s2 = ff_norm2(hx, mx, hy, my, hz, mz);
  const bool far = !(s2.h < near2);
  const float y = rsqrtf(s2.h);
  float y2, y2l, a, c;
  ff_rsqrt_residual(s2, y, y2, y2l, a, c);
  const float e = __fadd_rn(a, c);
  const float k1 = __fmul_rn(1.5f, a);
  const float k2 = __fmaf_rn(1.5f, c, __fmul_rn(__fmul_rn(1.875f, e), e));
  // w = mu y^3 (1 + k1 + k2) = wh + wl
  const float y3 = __fmul_rn(y2, y);
  const float y3l = __fmaf_rn(y2l, y, __fmaf_rn(y2, y, -y3));
  float wh = __fmul_rn(b.muh, y3);
  float wl = __fmaf_rn(b.muh, y3, -wh);
  wl = __fmaf_rn(b.muh, y3l, wl);
  wl = __fmaf_rn(b.mul, y3, wl);
  wl = __fmaf_rn(wh, k2, wl);
  wl = __fmaf_rn(wh, k1, wl);
  wh = far ? wh : 0.0f;
  wl = far ? wl : 0.0f;
  f.xh = __fmul_rn(wh, hx);
  f.yh = __fmul_rn(wh, hy);
  f.zh = __fmul_rn(wh, hz);
  f.xl = __fmaf_rn(wl, hx, __fmaf_rn(wh, mx, __fmaf_rn(wh, hx, -f.xh)));
  f.yl = __fmaf_rn(wl, hy, __fmaf_rn(wh, my, __fmaf_rn(wh, hy, -f.yh)));
  f.zl = __fmaf_rn(wl, hz, __fmaf_rn(wh, mz, __fmaf_rn(wh, hz, -f.zh)));
  return far;
}

__device__ __forceinline__ void split_sum(SplitAcc& acc, const SplitTerm& f) {
  split_add(acc.xh, acc.xl, f.xh, f.xl);
  split_add(acc.yh, acc.yl, f.yh, f.yl);
  split_add(acc.zh, acc.zl, f.zh, f.zl);
}

// Puts the low parts back below the high ones' last place.
__device__ __forceinline__ void split_renorm(SplitAcc& acc) {
  const FF x = ff_fast(acc.xh, acc.xl), y = ff_fast(acc.yh, acc.yl), z = ff_fast(acc.zh, acc.zl);
  acc = SplitAcc{x.h, x.l, y.h, y.l, z.h, z.l};
}

__device__ __forceinline__ void split_flush(SplitAcc& acc, double& ax, double& ay, double& az) {
  ax -= bits_to_double(acc.xh) + bits_to_double(acc.xl);
  ay -= bits_to_double(acc.yh) + bits_to_double(acc.yl);
  az -= bits_to_double(acc.zh) + bits_to_double(acc.zl);
  acc = SplitAcc{};
}

// ----------------------------------------------- a far pair in three FP32 parts
// The same sum for mx_accel, which returns the acceleration itself: every
// quantity carries a third FP32 part, so that a pair's relative error is 8e-20
// (rms, against 80-bit arithmetic; FP64's is 1.3e-16) where the grid holds the
// whole separation, 2^-54 of it by coordinate at the least; what is left of the
// sum's is its FP64 adds, one in kSplitSeg.  About 340 FP32 instructions a pair
// against pair_acc's 17 of 64 cycles.  Measured: k_accel with 2,000 big bodies
// and 200,000 planetesimals 11.8 -> 4.51 ms (86% of the issue slots filled), and the
// result's error against a 64-bit sum over all pairs 1.6e-15 -> 5.7e-16.
struct FT {
  float h, m, l;
};

struct alignas(16) SplitBig3 {
  SplitBig b;
  float mu2, pad[3];   // the third part of mu
};

struct SplitAcc3 {
  FT x, y, z;
};

__device__ __forceinline__ FT ft_sub(float a0, float a1, float a2, float b0, float b1, float b2) {
  const float d0 = __fsub_rn(a0, b0), d1 = __fsub_rn(a1, b1), d2 = __fsub_rn(a2, b2);
  const FF h = ff_fast(d0, d1), m = ff_fast(h.l, d2);
  return FT{h.h, m.h, m.l};
}

__device__ __forceinline__ FF ff_prod(float a, float b) {   // a b exactly
  const float p = __fmul_rn(a, b);
  return FF{p, __fmaf_rn(a, b, -p)};
}

// w d in three parts added to a.
__device__ __forceinline__ void ft_fma(FT& a, const FT& w, const FT& d) {
  const FF p = ff_prod(w.h, d.h), q = ff_prod(w.h, d.m), r = ff_prod(w.m, d.h);
  const FF s1 = ff_two_sum(p.l, q.h), s2 = ff_two_sum(s1.h, r.h);
  float f2 = __fadd_rn(__fadd_rn(s1.l, s2.l), __fadd_rn(q.l, r.l));
  f2 = __fmaf_rn(w.h, d.l, f2);
  f2 = __fmaf_rn(w.m, d.m, f2);
  f2 = __fmaf_rn(w.l, d.h, f2);
  const FF t0 = ff_two_sum(a.h, p.h), t1 = ff_two_sum(a.m, s2.h), t2 = ff_two_sum(t1.h, t0.l);
  a.h = t0.h;
  a.m = t2.h;
  a.l = __fadd_rn(a.l, __fadd_rn(__fadd_rn(t1.l, t2.l), f2));
}

__device__ __forceinline__ bool split_term3(const SplitPos& t, const SplitBig3& g, float near2,
                                            SplitAcc3& acc) {
  const SplitBig& b = g.b;
  const FT dx = ft_sub(t.x0, t.x1, t.x2, b.x0, b.x1, b.x2);
  const FT dy = ft_sub(t.y0, t.y1, t.y2, b.y0, b.y1, b.y2);
  const FT dz = ft_sub(t.z0, t.z1, t.z2, b.z0, b.z1, b.z2);
  // s^2 = s + l0 + l1
  const FF px = ff_prod(dx.h, dx.h), py = ff_prod(dy.h, dy.h), pz = ff_prod(dz.h, dz.h);
  const FF s1 = ff_two_sum(px.h, py.h), s2 = ff_two_sum(s1.h, pz.h);
  const float s = s2.h;
  if (s < near2) return false;
  const FF tx = ff_prod(dx.h, __fmul_rn(2.0f, dx.m)), ty = ff_prod(dy.h, __fmul_rn(2.0f, dy.m)),
           tz = ff_prod(dz.h, __fmul_rn(2.0f, dz.m));
  const FF a1 = ff_two_sum(tx.h, ty.h), a2 = ff_two_sum(a1.h, tz.h);
  const FF a3 = ff_two_sum(px.l, py.l), a4 = ff_two_sum(a3.h, pz.l);
  const FF a5 = ff_two_sum(s1.l, s2.l), a6 = ff_two_sum(a2.h, a4.h), a7 = ff_two_sum(a6.h, a5.h);
  const float l0 = a7.h;
  float l1 = __fadd_rn(__fadd_rn(__fadd_rn(a1.l, a2.l), __fadd_rn(a3.l, a4.l)),
                       __fadd_rn(__fadd_rn(a5.l, a6.l), a7.l));
  l1 = __fadd_rn(l1, __fadd_rn(__fadd_rn(tx.l, ty.l), tz.l));
  l1 = __fmaf_rn(dx.m, dx.m, __fmaf_rn(dy.m, dy.m, __fmaf_rn(dz.m, dz.m, l1)));
  const float hl = __fmaf_rn(dx.h, dx.l, __fmaf_rn(dy.h, dy.l, __fmul_rn(dz.h, dz.l)));
  l1 = __fmaf_rn(2.0f, hl, l1);
  // e = 1 - s^2 y^2 = e0 + e1
  const float y = rsqrtf(s);
  const FF y2 = ff_prod(y, y);
  const FF p = ff_prod(y2.h, s), t1 = ff_prod(y2.l, s), t2 = ff_prod(y2.h, l0);
  const FF u = ff_two_sum(p.l, t1.h), v = ff_two_sum(u.h, t2.h);
  float c = __fadd_rn(__fadd_rn(u.l, v.l), __fadd_rn(t1.l, t2.l));
  c = __fmaf_rn(y2.l, l0, c);
  c = __fmaf_rn(y2.h, l1, c);
  const FF e = ff_two_sum(__fsub_rn(1.0f, p.h), -v.h);
  // k = (1 - e)^(-3/2) - 1 = 3e/2 + 15e^2/8 = k0 + k1
  const FF k = ff_prod(1.5f, e.h);
  const float k1 = __fmaf_rn(__fmul_rn(1.875f, e.h), e.h, __fmaf_rn(1.5f, __fsub_rn(e.l, c), k.l));
  // mu y^3
  const FF g0 = ff_prod(y2.h, y), h0 = ff_prod(y2.l, y), q0 = ff_two_sum(g0.l, h0.h);
  const float q1 = __fadd_rn(q0.l, h0.l);
  const FF m0 = ff_prod(b.muh, g0.h), ma = ff_prod(b.muh, q0.h), mb = ff_prod(b.mul, g0.h);
  const FF n1 = ff_two_sum(m0.l, ma.h), n2 = ff_two_sum(n1.h, mb.h);
  float m2 = __fadd_rn(__fadd_rn(n1.l, n2.l), __fadd_rn(ma.l, mb.l));
  m2 = __fmaf_rn(b.muh, q1, m2);
  m2 = __fmaf_rn(b.mul, q0.h, m2);
  m2 = __fmaf_rn(g.mu2, g0.h, m2);
  // w = mu y^3 (1 + k)
  const FF mk = ff_prod(m0.h, k.h);
  const FF w0 = ff_fast(m0.h, mk.h), w1 = ff_two_sum(w0.l, n2.h);
  float w2 = __fadd_rn(__fadd_rn(m2, mk.l), w1.l);
  w2 = __fmaf_rn(m0.h, k1, w2);
  w2 = __fmaf_rn(n2.h, k.h, w2);
  const FT w{w0.h, w1.h, w2};
  ft_fma(acc.x, w, dx);
  ft_fma(acc.y, w, dy);
  ft_fma(acc.z, w, dz);
  return true;
}

// How gravity_split sums its far pairs: in pairs (the kick), or in three parts
// (mx_accel).  make: the staged record of a big body; term: adds a far pair,
// false for a near one; flush: the sums into the FP64 acceleration.
struct PairSum {
  using Big = SplitBig;
  using Acc = SplitAcc;
  static __device__ __forceinline__ Big make(const SplitBig& b, double) { return b; }
  static __device__ __forceinline__ float near2(const Big& b) { return b.near2; }
  static __device__ __forceinline__ bool term(const SplitPos& t, const Big& b, float near2, Acc& a) {
    SplitTerm f;
    if (!split_term(t, b, near2, f)) return false;
    split_sum(a, f);
    return true;
  }
  static __device__ __forceinline__ void flush(Acc& a, double& ax, double& ay, double& az) {
    split_flush(a, ax, ay, az);
  }
  static __device__ __forceinline__ void renorm(Acc& a) { split_renorm(a); }
};

struct TripleSum {
  using Big = SplitBig3;
  using Acc = SplitAcc3;
  static __device__ __forceinline__ Big make(const SplitBig& b, double mu) {
    Big g{b, 0.0f, {0.0f, 0.0f, 0.0f}};
    // mu = muh + mul + mu2: ff_of cuts mul at 24 bits of its own
    g.mu2 = (float)((mu - (double)b.muh) - (double)b.mul);
    return g;
  }
  static __device__ __forceinline__ float near2(const Big& b) { return b.b.near2; }
  static __device__ __forceinline__ bool term(const SplitPos& t, const Big& b, float near2, Acc& a) {
    return split_term3(t, b, near2, a);
  }
  static __device__ __forceinline__ void flush(Acc& a, double& ax, double& ay, double& az) {
    ax -= bits_to_double(a.x.h) + (bits_to_double(a.x.m) + bits_to_double(a.x.l));
    ay -= bits_to_double(a.y.h) + (bits_to_double(a.y.m) + bits_to_double(a.y.l));
    az -= bits_to_double(a.z.h) + (bits_to_double(a.z.m) + bits_to_double(a.z.l));
    a = Acc{};
  }
  static __device__ __forceinline__ void renorm(Acc&) {}
};

}  // namespace mx
