// mx_split.cuh -- the kick's pair sum in FP32 pairs (arXiv 2601.16791,
// Sec. 2.1.3), for targets outside a big body's changeover shell.
//
// What bounds the pair sum: FP64 issues one warp instruction per scheduler in
// 64 cycles on sm_103a, FP32 one per cycle (both measured), so the 17 FP64
// instructions of pair_acc take about 1,100 cycles for 32 pairs.  The
// same pair in pairs of FP32 numbers (a value kept as hi + lo, 48 bits) takes
// about 115 instructions.
//
// What the precision is: the state, the jump, the velocity update and the sum
// over blocks of kSplitRun big bodies stay FP64; only a far pair's
// acceleration mu d/s^3 is formed in FP32 pairs, with a relative error of
// about 1.5e-14 (rms, against 80-bit arithmetic).  A half kick adds
// (h/2) a to a velocity; for a body outside the changeover shell (3 Hill
// radii) that is at most a few 1e-4 of the velocity, so the split's share of
// the new velocity's error is below 1e-17 of it, where the FP64 rounding of
// the velocity itself is 1e-16.  A pair inside the shell, where the
// acceleration is largest and K varies, goes through the FP64 pair_acc, and
// so does a target outside the positions' grid below.  mx_accel, which returns
// accelerations, keeps FP64 throughout.
//
// Measured: k_jump_kick with 2,000 big bodies and 200,000 planetesimals 11.8 ->
// 1.73 ms a launch (34 -> 233 G pairs/s), two steps of that disk 40.2 -> 9.9 ms;
// 301 big bodies and 20,011 planetesimals 0.43 -> 0.068 ms a launch.
//
// Positions: each coordinate is cut on one grid for target and sources into
// three FP32 parts, x = x0 + x1 + x2 with x0 a multiple of 2^(k-23), x1 of
// 2^(k-47), |x| < 2^k, so that the differences of the parts are exact and a
// separation keeps the bits of the FP64 positions however close the pair.
// k comes from the positions of the chunk's big bodies (never from the tile),
// so results do not depend on the tiling.
#pragma once
#include <limits.h>
#include "mx_common.cuh"
#include "mx_physics.cuh"

namespace mx {

constexpr int kSplitRun = 32;     // big bodies summed in FP32 pairs between FP64 adds
constexpr int kSplitMinK = -10;   // positions' grid: 2^k AU above the big bodies' coordinates,
constexpr int kSplitMaxK = 10;    // else the pair sum stays FP64 (FP32 range of mu/s^3)

__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }

// x = o[0] + o[1] + o[2] on the grid of 2^k (|x| < 2^k); bits of x below
// 2^(k-62) are rounded off.  Integer instructions only.
__device__ __forceinline__ void split3(double x, int k, float& o0, float& o1, float& o2) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7ff;
  const unsigned long long m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
  // x = m 2^(e-1075); v = x / 2^(k-62)
  const int sh = (k - 62) - (e - 1075);
  unsigned long long v;
  if (sh <= 0) v = m << min(-sh, 63);
  else if (sh < 54) v = (m + (1ull << (sh - 1))) >> sh;
  else v = 0;
  const long long s = (b >> 63) ? -(long long)v : (long long)v;
  const long long a = (s + (1ll << 38)) >> 39;           // multiples of 2^(k-23)
  const long long r = s - (a << 39);                     // |r| <= 2^38
  const long long c = (r + (1ll << 14)) >> 15;           // multiples of 2^(k-47)
  const int q = (int)(r - (c << 15));                    // |q| <= 2^14
  o0 = __int2float_rn((int)a) * pow2f(k - 23);
  o1 = __int2float_rn((int)c) * pow2f(k - 47);
  o2 = __int2float_rn(q) * pow2f(k - 62);
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

__device__ __forceinline__ float near2_of(double rc2) {
  return fmaxf(to_float_bits(rc2) * 1.0001f, 1e-30f);
}

// s + c + (error): a two-sum into the pair (h, l), with the product's low part.
__device__ __forceinline__ void split_add(float& h, float& l, float ph, float pl) {
  const float s = __fadd_rn(h, ph);
  const float b = __fsub_rn(s, h);
  const float er = __fadd_rn(__fsub_rn(h, __fsub_rn(s, b)), __fsub_rn(ph, b));
  h = s;
  l = __fadd_rn(l, __fadd_rn(er, pl));
}

// d = a - b of parts, as hi + lo.
__device__ __forceinline__ void split_sub(float a0, float a1, float a2, float b0, float b1,
                                          float b2, float& h, float& m) {
  const float d0 = __fsub_rn(a0, b0), d1 = __fsub_rn(a1, b1), d2 = __fsub_rn(a2, b2);
  h = __fadd_rn(d0, d1);
  m = __fadd_rn(__fsub_rn(d1, __fsub_rn(h, d0)), d2);
}

// A pair's mu d/s^3 added to acc; returns false, with nothing added, for a
// pair inside near2.  1/s^3 = y^3 (1 + 3e/2 + 15e^2/8) from the single-
// precision estimate y of 1/s, e = 1 - s^2 y^2, as in pair_weight.
__device__ __forceinline__ bool split_pair(const SplitPos& t, const SplitBig& b, float near2,
                                           SplitAcc& acc) {
  float hx, mx, hy, my, hz, mz;
  split_sub(t.x0, t.x1, t.x2, b.x0, b.x1, b.x2, hx, mx);
  split_sub(t.y0, t.y1, t.y2, b.y0, b.y1, b.y2, hy, my);
  split_sub(t.z0, t.z1, t.z2, b.z0, b.z1, b.z2, hz, mz);
  // s^2 = s + l
  const float px = __fmul_rn(hx, hx), py = __fmul_rn(hy, hy), pz = __fmul_rn(hz, hz);
  const float qx = __fmaf_rn(hx, hx, -px), qy = __fmaf_rn(hy, hy, -py),
              qz = __fmaf_rn(hz, hz, -pz);
  const float s1 = __fadd_rn(px, py);
  const float b1 = __fsub_rn(s1, px);
  const float e1 = __fadd_rn(__fsub_rn(px, __fsub_rn(s1, b1)), __fsub_rn(py, b1));
  const float s = __fadd_rn(s1, pz);
  const float b2 = __fsub_rn(s, s1);
  const float e2 = __fadd_rn(__fsub_rn(s1, __fsub_rn(s, b2)), __fsub_rn(pz, b2));
  if (s < near2) return false;
  const float hm = __fmaf_rn(hx, mx, __fmaf_rn(hy, my, __fmul_rn(hz, mz)));
  const float l = __fmaf_rn(2.0f, hm, __fadd_rn(__fadd_rn(__fadd_rn(qx, qy), qz),
                                                __fadd_rn(e1, e2)));
  const float y = rsqrtf(s);
  const float y2 = __fmul_rn(y, y);
  const float y2l = __fmaf_rn(y, y, -y2);
  // e = a + c: 1 - y2 s exactly as 1 - p (exact) - pe, then the low parts
  const float p = __fmul_rn(y2, s);
  const float pe = __fmaf_rn(y2, s, -p);
  const float a = __fsub_rn(1.0f, p);
  const float c = -__fmaf_rn(y2, l, __fmaf_rn(y2l, s, pe));
  const float e = __fadd_rn(a, c);
  const float k1 = __fmul_rn(1.5f, a);
  const float k2 = __fmaf_rn(1.5f, c, __fmul_rn(__fmul_rn(1.875f, e), e));
  // w = mu y^3 (1 + k1 + k2) = wh + wl
  const float y3 = __fmul_rn(y2, y);
  const float y3l = __fmaf_rn(y2l, y, __fmaf_rn(y2, y, -y3));
  const float wh = __fmul_rn(b.muh, y3);
  float wl = __fmaf_rn(b.muh, y3, -wh);
  wl = __fmaf_rn(b.muh, y3l, wl);
  wl = __fmaf_rn(b.mul, y3, wl);
  wl = __fmaf_rn(wh, k2, wl);
  wl = __fmaf_rn(wh, k1, wl);
  const float fx = __fmul_rn(wh, hx), fy = __fmul_rn(wh, hy), fz = __fmul_rn(wh, hz);
  split_add(acc.xh, acc.xl, fx, __fmaf_rn(wl, hx, __fmaf_rn(wh, mx, __fmaf_rn(wh, hx, -fx))));
  split_add(acc.yh, acc.yl, fy, __fmaf_rn(wl, hy, __fmaf_rn(wh, my, __fmaf_rn(wh, hy, -fy))));
  split_add(acc.zh, acc.zl, fz, __fmaf_rn(wl, hz, __fmaf_rn(wh, mz, __fmaf_rn(wh, hz, -fz))));
  return true;
}

__device__ __forceinline__ void split_flush(SplitAcc& acc, double& ax, double& ay, double& az) {
  ax -= (double)acc.xh + (double)acc.xl;
  ay -= (double)acc.yh + (double)acc.yl;
  az -= (double)acc.zh + (double)acc.zl;
  acc = SplitAcc{};
}

}  // namespace mx
