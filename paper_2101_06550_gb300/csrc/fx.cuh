// Fixed-point arithmetic on the integer pipes, for the FP64 path of the 2D step.
//
// GB300 issues FP64 at 2 lanes per clock and SM, 1/64 of its FP32 and 1/32 of its
// integer rate: an FP64 multiply-add holds an SM sub-partition's FP64 unit for 64
// cycles per warp.  A circulant sweep (circulant.cuh) multiplies a state by two
// constants only, so its values can share one exponent: held as 64-bit integers
// they carry more bits than an FP64 significand (59 below the largest value,
// against 53), and a row's two multiply-adds are six 32 x 32 + 64-bit integer
// multiply-adds and seven additions and shifts.
//
// A constant k, |k| < 2, is the integer k 2^62 in two signed halves
// (x 2^32 + y, |y| <= 2^31), a state g, |g| < 2^60, likewise, so that every partial
// product is one signed wide multiply-add.  The product of the two low halves
// (at most 1 unit, of either sign) is left out; the rest is rounded to nearest.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace chx {

constexpr int kFxLevels = 7;  // up to 128 segments

// One direction's operator 1 + a delta^4 = kappa L L^T for one simulation.
struct FxDir {
  int2 k1, k2;          // -l1, -l2
  // state transfer over 2^k segments, and over as many with the last (short) one among
  // them, / 2^qs; the same over the segments of the lower bits of `count`
  int2 step[kFxLevels][2][4], rest[kFxLevels][2][4];
  int2 close[4];        // (1 - transfer over the system)^{-1}, / 2^qc
  int qs, qc;
  int W;                // rows after which a state has decayed below 2^-62
  int count;            // segments put together: as many as a state reaches, or all P of them
  int round;            // (through `close`)
  int eb;               // bits the sum over segments of the states they leave can grow by
  // |h_{r+1} g1 - l2 h_r g2| <= a1 |g1 - g2| + a2 |g2|
  float a1, a2;
  double scale;         // 1 / kappa
};
static_assert(sizeof(FxDir) % 8 == 0, "copied in 8-byte words");

// gamma / dx^2 and gamma / dy^2, both over 2^q, their sum below 1/2, for one simulation.
struct FxGl {
  int2 gx, gy;
  int q, pad;
};
FxGl fx_gl_host(double gx, double gy);

#ifdef __CUDACC__
__device__ __forceinline__ long long fx_wide(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}

// A state and its signed halves.
struct FxVal {
  int h, l;
};
__device__ __forceinline__ FxVal fx_halves(long long g) {
  FxVal v;
  v.l = (int)g;
  v.h = (int)(g >> 32) + (int)((unsigned)v.l >> 31);
  return v;
}

// k1 g1 + k2 g2
__device__ __forceinline__ long long fx_mul2(int2 k1, FxVal g1, int2 k2, FxVal g2) {
  long long c = fx_wide(k2.y, g2.h, 1ll << 29);
  c = fx_wide(k2.x, g2.l, c);
  c = fx_wide(k1.x, g1.l, c);
  c = fx_wide(k1.y, g1.h, c);
  long long p = fx_wide(k2.x, g2.h, 0);
  p = fx_wide(k1.x, g1.h, p);
  return (p << 2) + (c >> 30);
}

// f 2^-t + k1 g1 + k2 g2, with up = 2^(30 - t), 1 <= t <= 30: the shift is a product too,
// rounded with the others (|f| < 2^60).
__device__ __forceinline__ long long fx_step(long long f, int up, int2 k1, FxVal g1, int2 k2, FxVal g2) {
  const FxVal v = fx_halves(f);
  long long c = fx_wide(up, v.l, 1ll << 29);
  long long p = fx_wide(up, v.h, 0);
  c = fx_wide(k2.y, g2.h, c);
  c = fx_wide(k2.x, g2.l, c);
  p = fx_wide(k2.x, g2.h, p);
  c = fx_wide(k1.x, g1.l, c);
  c = fx_wide(k1.y, g1.h, c);
  p = fx_wide(k1.x, g1.h, p);
  return (p << 2) + (c >> 30);
}

// a 2^-ta + b 2^-tb + k1 g1 + k2 g2, ua = 2^(30 - ta), ub = 2^(30 - tb), rounded once.
__device__ __forceinline__ long long fx_step2(FxVal a, int ua, FxVal b, int ub, int2 k1, FxVal g1, int2 k2, FxVal g2) {
  long long c = fx_wide(ua, a.l, 1ll << 29);
  long long p = fx_wide(ua, a.h, 0);
  c = fx_wide(ub, b.l, c);
  p = fx_wide(ub, b.h, p);
  c = fx_wide(k2.y, g2.h, c);
  c = fx_wide(k2.x, g2.l, c);
  p = fx_wide(k2.x, g2.h, p);
  c = fx_wide(k1.x, g1.l, c);
  c = fx_wide(k1.y, g1.h, c);
  p = fx_wide(k1.x, g1.h, p);
  return (p << 2) + (c >> 30);
}

// f + (k1 g1 + k2 g2) 2^q to half a unit, 0 <= q < 30, |k1| + |k2| <= 2: low products and
// the bits below the unit are kept until the scaling.
__device__ __forceinline__ long long fx_dot2(long long f, int2 k1, FxVal g1, int2 k2, FxVal g2, int q) {
  long long c = (long long)__mulhi(k1.y, g1.l) + __mulhi(k2.y, g2.l) + (1ll << (29 - q));
  c = fx_wide(k2.y, g2.h, c);
  c = fx_wide(k2.x, g2.l, c);
  c = fx_wide(k1.x, g1.l, c);
  c = fx_wide(k1.y, g1.h, c);
  long long p = fx_wide(k2.x, g2.h, 0);
  p = fx_wide(k1.x, g1.h, p);
  return f + (p << (2 + q)) + (c >> (30 - q));
}

// k g
__device__ __forceinline__ long long fx_mul(int2 k, FxVal g) {
  long long c = fx_wide(k.y, g.h, 1ll << 29);
  c = fx_wide(k.x, g.l, c);
  return (fx_wide(k.x, g.h, 0) << 2) + (c >> 30);
}

// v 2^(B - (E - 1022)) rounded, E >= 128 at least v's biased exponent (|v| < 2^(E - 1022)),
// B <= 59.  Values below 2^-895 count as zero.
__device__ __forceinline__ long long fx_from_double(double v, int E, int B) {
  const unsigned hi = (unsigned)__double2hiint(v);
  const unsigned e = (hi >> 20) & 0x7ffu;
  const unsigned long long mant =
      ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32 | (unsigned)__double2loint(v)) << 9;
  int t = 61 - B + E - (int)e;
  t = t > 63 ? 63 : t;
  const long long x = (long long)(((mant >> t) + 1) >> 1);
  const long long s = (long long)((int)hi >> 31);
  return (x ^ s) - s;
}

// f 2^-t, 0 <= t < 32, rounded to nearest even: rounding the ties up would shift the
// mean, by 1/4 of a unit at t = 1, and the sweeps pass a mean on with the gain of L^{-1}
// (4096^2, rough state: 3e-11 of the mean of |C| per step).
__device__ __forceinline__ long long fx_shift(long long f, int t) {
  const int any = t > 0;
  const unsigned odd = ((unsigned)f >> t) & any;
  f += (unsigned)((1u << t) >> 1) - any + odd;
  return (long long)(((unsigned long long)(unsigned)((int)(f >> 32) >> t) << 32) |
                     __funnelshift_r((unsigned)f, (unsigned)(f >> 32), t));
}

// x 2^S as FP64, rounded to nearest (0 and infinity outside its range).  24 integer
// instructions where a conversion instruction takes the FP64 unit for 64 cycles per warp.
__device__ __forceinline__ double fx_to_double(long long x, int S) {
  const long long s = x >> 63;
  const unsigned long long a = (unsigned long long)((x ^ s) - s);
  const int lz = __clzll((long long)a);
  const unsigned long long n = a << (lz & 63);
  const int e = 1023 + 63 - lz + S;
  unsigned long long b = (n >> 11) + ((n >> 10) & 1);  // 53 bits, or 2^53
  b += (unsigned long long)(unsigned)(e - 1) << 52;
  if (a == 0 || e <= 0) b = 0;
  if (e >= 2047) b = 0x7ff0000000000000ull;
  return __longlong_as_double((long long)(b | ((unsigned long long)s & 0x8000000000000000ull)));
}

// High word of |g|, within one unit.
__device__ __forceinline__ int fx_mag(long long g) {
  const int h = (int)(g >> 32);
  return h ^ (h >> 31);
}

__device__ __forceinline__ int fx_bits(int v) { return 32 - __clz(v); }

// 2^k for k in [-1022, 1023].
__device__ __forceinline__ double fx_pow2(int k) { return __hiloint2double((k + 1023) << 20, 0); }
#endif  // __CUDACC__

// Tables of 1 + a delta^4 over n rows in P segments of m; false when a is next to 0 or stiffer than
// kFxStiff, or the factorisation or the fixed-point range does not serve (the caller keeps
// the FP64 solves).  At a = 3e5 (4096^2, a rough state) the circulant factors lose the field's
// mean to 1.5e-12 of |C|'s per step, the LU factors with pivots 8e-13; at 1.9e4 (2048^2) it is
// 3e-15 against 2e-13.
constexpr double kFxStiff = 5e4;
bool fx_dir_host(int n, int P, int m, double a, FxDir* out);

}  // namespace chx
