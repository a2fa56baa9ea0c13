// Block fixed-point arithmetic of the transforms: a complex value of one transform is a pair of 64-bit
// integers X = x 2^k with one exponent k per transform.
//
// Why integers: GB300 retires 1.68 binary64 additions per clock per SM, but 60 64-bit integer additions and 30
// 32 x 32 + 64 -> 64 bit multiply-adds (measured, 8 independent chains per thread), so a transform in 64-bit
// fixed point issues its arithmetic several times faster than one in binary64, and in fewer instructions than
// one in double-float.
// Why it is as accurate: the additions are exact, a twiddle product rounds to one unit, and k is as large as
// the sum S = sum (|re| + |im|) of the transform's inputs allows: no partial sum of a transform exceeds S, so
// with S 2^k <= 2^61.7 nothing overflows. The unit is then at most 2^-60.7 S <= 2^-60.7 sqrt(2 n) ||x||, that
// is 2^-51.2 of the inputs' rms at n = 512, and rounding errors enter the result as noise of about half a
// unit times sqrt(n), where binary64 rounds every addition of every stage: measured against a transform in
// extended precision, the error is below the binary64 transform's up to 768 points, and with guard bits beyond
// (figures in fft.cu).
#pragma once
#include "df64.h"
#include "lmvd_internal.h"

namespace lmvd {

struct __align__(16) cfx {
  long long re, im;
};
__device__ __forceinline__ cfx operator+(cfx a, cfx b) { return cfx{a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ cfx operator-(cfx a, cfx b) { return cfx{a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ cfx fx_ti(cfx a) { return cfx{-a.im, a.re}; }  // i a

// c + a b as one 64-bit multiply-add: written as a low / high pair, which the assembler fuses (the C expression
// becomes a multiply and two additions: a complex product then takes 68 instructions instead of 26)
__device__ __forceinline__ long long madw(int a, int b, long long c) {
  long long r;
  asm("{\n\t.reg .s32 l, h;\n\tmov.b64 {l, h}, %3;\n\tmad.lo.cc.s32 l, %1, %2, l;\n\tmadc.hi.s32 h, %1, %2, h;\n\t"
      "mov.b64 %0, {l, h};\n\t}"
      : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

// A factor w in [-1, 1] as two signed limbs: w = hi 2^-31 + lo 2^-62, |lo| <= 2^30 (twiddles: (re.hi, re.lo,
// im.hi, im.lo) in an int4). A value is split at bit 32 with a signed low word, X = (h2 / 2) 2^32 + l, so that
// every partial product is signed and the one left out, l lo 2^-62 (at most half a unit), has mean zero:
// X w = h2 hi + (h2 lo + l hi) 2^-31. With |X| <= 2^61.7 and |w| <= 1 the sum of the four middle products of a
// complex product stays below 2^63.
constexpr long long kFxHalf = 1ll << 30;  // rounds the middle products
__device__ __forceinline__ int fx_high2(long long x) { return (int)(x >> 31) + (int)((unsigned)x >> 31); }

template <int SIGN>
__device__ __forceinline__ cfx fx_mulw(cfx v, int4 w) {  // v (w.re + SIGN i w.im)
  const int rh = fx_high2(v.re), ih = fx_high2(v.im), rl = (int)v.re, il = (int)v.im;
  const int ph = SIGN > 0 ? w.z : -w.z, pl = SIGN > 0 ? w.w : -w.w, nh = SIGN > 0 ? -w.z : w.z, nl = SIGN > 0 ? -w.w : w.w;
  const long long mr = madw(il, nh, madw(ih, nl, madw(rl, w.x, madw(rh, w.y, kFxHalf))));
  const long long mi = madw(il, w.x, madw(ih, w.y, madw(rl, ph, madw(rh, pl, kFxHalf))));
  return cfx{madw(ih, nh, madw(rh, w.x, mr >> 31)), madw(ih, w.x, madw(rh, ph, mi >> 31))};
}
__device__ __forceinline__ long long fx_mulr(long long x, int2 w) {  // x (w.x 2^-31 + w.y 2^-62)
  const int h = fx_high2(x), l = (int)x;
  return madw(h, w.x, madw(l, w.x, madw(h, w.y, kFxHalf)) >> 31);
}

// limbs of w in [-1, 1]; |hi| <= 2^31 - 1, so that both parts can be negated (+-1 becomes +-(1 - 2^-62))
template <class F>
__host__ __device__ inline void fx_limbs(F w, int& hi, int& lo) {
  const F a = (w < 0 ? -w : w) * (F)2147483648.0;
  F h = (F)(long long)(a + (F)0.5);
  if (h > (F)2147483647.0) h = (F)2147483647.0;
  F l = (a - h) * (F)2147483648.0;
  l = l >= 0 ? (F)(long long)(l + (F)0.5) : -(F)(long long)((F)0.5 - l);
  if (l > (F)2147483647.0) l = (F)2147483647.0;
  hi = w < 0 ? -(int)(long long)h : (int)(long long)h;
  lo = w < 0 ? -(int)(long long)l : (int)(long long)l;
}

// ------------------------------------------------------------------ magnitudes
// The sums S are formed in FP32 from the high words of the doubles: |x| with its mantissa truncated to 20 bits
// (a magnitude below 2^-126 counts as zero, one above 2^128 sets the flag below). A thread accumulates the sum
// and the largest high word.
struct FxMag {
  float sum = 0.f;
  int top = 0;  // largest |high word|
  __device__ __forceinline__ void add(double x, double y) {
    const int t = __double2hiint(x) & 0x7fffffff, u = __double2hiint(y) & 0x7fffffff;
    top = __vimax3_s32(top, t, u);
    sum += __int_as_float(__viaddmax_s32(t, -0x38000000, 0) << 3);
    sum += __int_as_float(__viaddmax_s32(u, -0x38000000, 0) << 3);
  }
  __device__ __forceinline__ void add(df x, df y) {
    const float a = fabsf(x.hi), b = fabsf(y.hi);
    top = __vimax3_s32(top, __float_as_int(a), __float_as_int(b));
    sum += a;
    sum += b;
  }
};
// Sums in [kFxTiny, kFxHuge) (or all-zero inputs) need no rescaling; outside, or with inf / nan, the slow path
// first divides the inputs by a power of two (fx_rescale).
constexpr float kFxTiny = 0x1p-100f, kFxHuge = 0x1p60f;
__device__ __forceinline__ bool fx_out_of_range(const FxMag& m, bool df_in) {
  return !(m.sum < kFxHuge) || (m.sum < kFxTiny && m.top != 0) || (!df_in && m.top >= 0x47000000);
}

// k for the sum S: S 2^k <= 2^61.7 (sums truncate by < 2^-18); at most 161
constexpr int kFxZeroK = 162;  // a transform of zeros: it has no exponent of its own (fx_stored_exponent)
__device__ __forceinline__ int fx_exponent(float S) {
  S = fmaxf(S, kFxTiny);
  const int b = __float_as_int(S), e = (b >> 23) - 127;
  return (b & 0x7fffff) <= 0x4ff000 ? 61 - e : 60 - e;  // mantissa 1.6245 < 2^0.7
}

// ------------------------------------------------------------------ conversions (integer operations)
__device__ __forceinline__ unsigned long long shr64(unsigned long long a, int n) {
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(n));  // 0 for n > 63
  return r;
}
__device__ __forceinline__ long long sar64(long long a, int n) {
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(n));  // the sign for n > 63
  return r;
}
__device__ __forceinline__ unsigned shl32(unsigned a, int n) {
  unsigned r;
  asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(n));  // 0 for n > 31
  return r;
}
__device__ __forceinline__ unsigned long long shl64(unsigned long long a, int n) {
  unsigned long long r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(n));
  return r;
}
// x 2^k (|x| 2^k < 2^62), rounded to nearest; a magnitude below 2^-33 of the largest possible one is truncated toward
// zero. A subnormal x becomes 0: where a transform consists of such values fx_rescale has scaled them.
__device__ __forceinline__ long long fx_from(double x, int k) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  const unsigned long long m = ((unsigned long long)mh << 32 | (unsigned)lo) << 10;  // leading bit 62
  const int n = 1085 - k - e;
  const long long s = hi >> 31;
  return (long long)(shr64(m + shl32(1u, n - 1), n) ^ (unsigned long long)s) - s;
}
// (hi + lo) 2^k: 20-bit limbs split off on the FP32 pipe by adding 1.5 2^23 (the integer is then the low
// mantissa bits), exactly; sa = 2^(k - 40). The last limb rounds.
__device__ __forceinline__ long long fx_from(df x, float sa) {
  constexpr float M = 12582912.0f;
  constexpr unsigned Mi = 0x4B400000u;
  const float t1 = __fmaf_rn(x.hi, sa, M), r1 = __fmaf_rn(x.hi, sa, -__fsub_rn(t1, M));
  const float t2 = __fmaf_rn(r1, 0x1p20f, M), r2 = __fmaf_rn(r1, 0x1p20f, -__fsub_rn(t2, M));
  const float t3 = __fmaf_rn(r2, 0x1p20f, M);
  const float l = __fmul_rn(x.lo, sa);
  const float t4 = __fmaf_rn(l, 0x1p20f, M), r4 = __fmaf_rn(l, 0x1p20f, -__fsub_rn(t4, M));
  const float t5 = __fmaf_rn(r4, 0x1p20f, M);
  const int i1 = (int)(__float_as_uint(t1) - Mi), i2 = (int)(__float_as_uint(t2) + __float_as_uint(t4) - 2u * Mi),
            i3 = (int)(__float_as_uint(t3) + __float_as_uint(t5) - 2u * Mi);
  return ((long long)i1 << 40) + madw(i2, 1 << 20, i3);
}
// X 2^-k rounded to a double with integer operations: the position of the leading bit from an FP32 conversion
// (rounded toward zero), the mantissa shifted there and rounded to nearest
__device__ __forceinline__ double fx_to(long long X, int k) {
  const int s = (int)(X >> 63);
  const unsigned long long a = ((unsigned long long)X ^ (unsigned long long)(long long)s) - (long long)s;
  const float f = __fmaf_rz(__uint2float_rz((unsigned)(a >> 32)), 0x1p32f, __uint2float_rz((unsigned)a));
  const int ef = __float_as_int(f) >> 23;  // 127 + position of the leading bit
  const unsigned long long m = (shl64(a, 189 - ef) + 512) >> 10;
  const int hi = (int)(m >> 32) + ((ef + 895 - k) << 20);
  return __hiloint2double(ef == 0 ? 0 : (hi | (s & 0x80000000)), (int)(unsigned)m);
}
// The same through two binary64 additions (the otherwise idle FP64 pipe): (2^84 + (xh + 2^31) 2^32) - (2^84 +
// 2^63 + 2^52) is exact, and adding (2^52 + xl) rounds once. kx = k << 20.
__device__ __forceinline__ double fx_to_fp(long long X, int kx) {
  const double c = __hiloint2double(0x45300000 - kx, (int)0x80100000u);  // (2^84 + 2^63 + 2^52) 2^-k
  const double dh = __hiloint2double(0x45300000 - kx, (int)(X >> 32) ^ (int)0x80000000u);
  const double dl = __hiloint2double(0x43300000 - kx, (int)X);
  return __dadd_rn(__dsub_rn(dh, c), dl);
}

}  // namespace lmvd
