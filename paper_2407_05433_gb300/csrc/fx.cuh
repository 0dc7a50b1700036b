// fx.cuh -- scaled integer arithmetic of 57 and 114 fractional bits.
//
// Why.  On sm_103a an FP64 warp instruction occupies its SM sub-partition for
// about 76 cycles, and nothing overlaps it there: measured, a chain of
// dependent DFMAs runs at 64 cycles each and four independent chains at 76,
// from 1 to 16 warps per SM.  A 32 x 32 + 64 bit integer multiply-add issues
// every 2.3 cycles (3.6 dependent).  A product of a 114-bit number (four
// 29-bit limbs) with a 57-bit one (two limbs) takes seven of them, 16 cycles,
// and their 64-bit sums carry a whole dot product of 33 terms without a carry
// in between, so a multiply-add with twice the bits of FP64 costs a fifth of a
// DFMA.
//
// Number format.  A matrix keeps one binary exponent per row and one per column;
// an entry is an integer times 2^(r_i + e_j - 57) or 2^(r_i + e_j - 114).
// Limbs are balanced: x = sum_k w_k 2^(29 k) with w_k in [-2^28, 2^28) except
// the highest (int2: x = high, y = low; int4: x = lowest ... w = highest).
#pragma once
#include <stdint.h>

namespace eclqr {

typedef __int128 i128;

// single-precision approximations (PTX rsqrt.approx / rcp.approx, relative
// error about 2^-22), used only as seeds and for small integer quotients
__device__ __forceinline__ float rsqrt_seed(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_seed(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

constexpr int kFxA = 57;          // fractional bits of a two-limb entry
constexpr int kFxP = 114;         // fractional bits of a four-limb entry
constexpr int kFxB = 29;          // bits of a limb
constexpr int kFxNone = -100000;  // exponent of zero

// a b + c, one instruction (written out: the compiler takes (long long)a * b + c for a 64-bit product)
__device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}

__device__ __forceinline__ int2 fx_split(long long x) {
  const long long h = (x + (1ll << (kFxB - 1))) >> kFxB;
  return make_int2((int)h, (int)x - ((int)h << kFxB));
}
// |x| < 2^118
__device__ __forceinline__ int4 fx_split4(i128 x) {
  constexpr unsigned kMask = (1u << kFxB) - 1;
  constexpr int kHalf = 1 << (kFxB - 1);
  x += ((i128)kHalf << (2 * kFxB)) + ((i128)kHalf << kFxB) + kHalf;
  const unsigned x0 = (unsigned)x, x1 = (unsigned)(x >> 32), x2 = (unsigned)(x >> 64), x3 = (unsigned)(x >> 96);
  return make_int4((int)(x0 & kMask) - kHalf, (int)(__funnelshift_r(x0, x1, 29) & kMask) - kHalf,
                   (int)(__funnelshift_r(x1, x2, 26) & kMask) - kHalf, (int)__funnelshift_r(x2, x3, 23));
}
__device__ __forceinline__ i128 fx_join4(int4 a) {
  const long long lo = fx_mad(a.y, 1 << kFxB, (long long)a.x), hi = fx_mad(a.w, 1 << kFxB, (long long)a.z);
  return ((i128)hi << (2 * kFxB)) + lo;
}

// smallest b with |x| < 2^b (0 for zero)
__device__ __forceinline__ int fx_bits(long long x) { return 64 - __clzll(x < 0 ? -x : x); }
__device__ __forceinline__ int fx_bits(i128 x) {
  if (x < 0) x = -x;
  const long long hi = (long long)(x >> 64);
  return hi ? 128 - __clzll(hi) : 64 - __clzll((long long)x);
}

// x 2^s (0 or -1 where every bit falls away); the caller knows that a left shift fits.  64-bit
// values are rounded to nearest, 128-bit ones down: half a unit of their 2^-114
__device__ __forceinline__ long long fx_shift(long long x, int s) {
  if (s >= 0) return x << s;
  return -s > 62 ? 0ll : ((x >> (-s - 1)) + 1) >> 1;
}
__device__ __forceinline__ i128 fx_shift(i128 x, int s) { return s >= 0 ? x << s : x >> min(-s, 127); }

// smallest e with |x| < 2^e; kFxNone for zero (and for subnormal x, taken as zero)
__device__ __forceinline__ int fx_expo(double x) {
  const int ex = (__double2hiint(x) >> 20) & 0x7ff;
  return ex == 0 ? kFxNone : ex - 1022;
}
__device__ __forceinline__ bool fx_nonfinite(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) == 0x7ff; }

// the signed 53-bit significand of x (0 for zero and subnormals): x = this 2^(fx_expo(x) - 53)
__device__ __forceinline__ long long fx_significand(double x) {
  const int hi = __double2hiint(x);
  if (((hi >> 20) & 0x7ff) == 0) return 0;
  const long long v = ((long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(x);
  return hi < 0 ? -v : v;
}
// x 2^(57 - e), rounded to nearest, for |x| <= 2^e
__device__ __forceinline__ long long fx_from(double x, int e) {
  return fx_shift(fx_significand(x), min(fx_expo(x) - 53 + kFxA - e, 10));
}
// x 2^(114 - e), rounded to nearest, for |x| <= 2^e
__device__ __forceinline__ i128 fx_from4(double x, int e) {
  return fx_shift((i128)fx_significand(x), min(fx_expo(x) - 53 + kFxP - e, 70));
}

// x 2^s as a double, rounded to nearest (overflow to infinity, below the normal range to zero)
__device__ __forceinline__ double fx_to(long long x, int s) {
  if (x == 0) return 0.0;
  const unsigned long long a = x < 0 ? -(unsigned long long)x : (unsigned long long)x;
  const int z = __clzll((long long)a);
  const unsigned long long n = a << z;  // the leading bit at position 63; 53 kept
  unsigned long long m = (n >> 11) + ((n >> 10) & 1);
  int ex = 63 - z + s + 1023 + (int)(m >> 53);  // rounded up to the next power of two: m's low bits are 0
  if (ex >= 0x7ff) m = 0, ex = 0x7ff;
  if (ex <= 0) return 0.0;
  const unsigned long long b = ((unsigned long long)ex << 52) | (m & 0xfffffffffffffull);
  return __longlong_as_double((long long)(b | (x < 0 ? 0x8000000000000000ull : 0ull)));
}
// the leading 62 bits of x and the exponent that goes with them
__device__ __forceinline__ long long fx_lead(i128 x, int &s) {
  s = max(fx_bits(x) - 62, 0);
  return (long long)(x >> s);
}

// m^(-1/2) 2^62 for m = s 2^(-62) in [1, 4): a single-precision seed y0 and one
// third-order step y0 (1 + e/2 + 3 e^2 / 8), e = 1 - m y0^2, in integers; relative
// error below 2^-59
__device__ __forceinline__ unsigned long long fx_rsqrt(unsigned long long s) {
  const float mf = (float)(unsigned)(s >> 32) * 0x1p-30f;
  const unsigned y0 = (unsigned)min(rsqrt_seed(mf) * 0x1p32f, 4294967040.0f);
  const unsigned long long t = (unsigned long long)y0 * y0;  // y0^2 2^64
  const long long e = (long long)(1ull << 62) - (long long)__umul64hi(s, t);
  const long long eh = e >> 20;
  const long long corr = (e >> 1) + ((3 * ((eh * eh) >> 22)) >> 3);
  return ((unsigned long long)y0 << 30) + (unsigned long long)__mul64hi(corr << 18, (long long)y0 << 14);
}
// 2^55 / m for m = u 2^(-64) in [1/4, 1): seed r0 and r0 (1 + e + e^2), e = 1 - m r0
__device__ __forceinline__ long long fx_rcp(unsigned long long u) {
  const float mf = (float)(unsigned)(u >> 32) * 0x1p-32f;
  const unsigned r0 = (unsigned)(rcp_seed(mf) * 0x1p29f);
  const long long e = (long long)(1ull << 61) - (long long)__umul64hi(u, (unsigned long long)r0 << 32);
  const long long eh = e >> 20;
  const long long corr = e + ((eh * eh) >> 21);
  return ((long long)r0 << 26) + __mul64hi(corr << 20, (long long)r0 << 9);
}

// The scalars of FP64 factorizations on the integer pipe: the dozen dependent FP64 instructions of a
// seeded FP64 step occupy the sub-partition for 64 to 76 cycles each.  A positive normal d is
// 2^(2 h) s 2^-62 with s in [2^62, 2^64); ok is false, with the results unusable, unless d is positive
// and within [2^-1000, 2^1001).
__device__ __forceinline__ unsigned long long fx_even(double d, int &h, bool &ok) {
  const int hi = __double2hiint(d), ex = ((hi >> 20) & 0x7ff) - 1023, odd = ex & 1;
  h = (ex - odd) >> 1;
  ok = hi > 0 && ex >= -1000 && ex <= 1000;
  return ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)__double2loint(d)) << (10 + odd);
}
// d^(-1/2): relative error below 2^-59 before the rounding to FP64
__device__ __forceinline__ double fx_rsqrt_f64(double d, bool &ok) {
  int h;
  const unsigned long long s = fx_even(d, h, ok);
  return fx_to((long long)fx_rsqrt(s), -62 - h);
}

// sums of products of four-limb by two-limb entries: c[3] 2^116 + c[2] 2^87 + c[1] 2^58 + c[0] 2^29,
// the product of the lowest limbs left out (below 2^-167 of the unit product)
struct FxAcc {
  long long c[4];
  __device__ __forceinline__ void zero() { c[0] = c[1] = c[2] = c[3] = 0; }
  __device__ __forceinline__ void mad(int4 p, int2 a) {
    c[3] = fx_mad(p.w, a.x, c[3]);
    c[2] = fx_mad(p.w, a.y, fx_mad(p.z, a.x, c[2]));
    c[1] = fx_mad(p.z, a.y, fx_mad(p.y, a.x, c[1]));
    c[0] = fx_mad(p.y, a.y, fx_mad(p.x, a.x, c[0]));
  }
  // the sum 2^(-S), S = 54 .. 58 or 60
  template <int S>
  __device__ __forceinline__ i128 value() const {
    const i128 hi = ((i128)c[3] << (116 - S)) + ((i128)c[2] << (87 - S));
    if (S == 60) return hi + ((c[1] + (c[0] >> kFxB) + 2) >> 2);
    return hi + ((i128)c[1] << (S <= 58 ? 58 - S : 0)) + (c[0] >> (S - 29));
  }
};
// sums of products of four-limb entries, from the 2^87 of the limbs up: the error is below 2^-110
// of the unit product
struct FxAcc4 {
  long long c[4];
  __device__ __forceinline__ void zero() { c[0] = c[1] = c[2] = c[3] = 0; }
  __device__ __forceinline__ void mad(int4 a, int4 b) {
    c[3] = fx_mad(a.w, b.w, c[3]);
    c[2] = fx_mad(a.w, b.z, fx_mad(a.z, b.w, c[2]));
    c[1] = fx_mad(a.w, b.y, fx_mad(a.z, b.z, fx_mad(a.y, b.w, c[1])));
    c[0] = fx_mad(a.w, b.x, fx_mad(a.z, b.y, fx_mad(a.y, b.z, fx_mad(a.x, b.w, c[0]))));
  }
  __device__ __forceinline__ i128 value() const {  // the sum 2^(-112)
    return ((i128)c[3] << 62) + ((i128)c[2] << 33) + ((i128)c[1] << 4) + (c[0] >> 25);
  }
};

}  // namespace eclqr
