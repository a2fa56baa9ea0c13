// Batched Fourier transforms in the periodic directions with the 3/2 rule (paper Eq. disc_f and
// Sec. 4.4: products are formed in physical space on a grid padded to 3N/2 points, so that
// quadratic products of retained modes do not alias; coefficients are truncated back to
// |kx| < nx/2, |kz| < nz/2 with the Nyquist slots zero).
//
// Each field transform runs in two passes through an intermediate array T[y][z][kx]
// (kx < nx/2 only -- the padded kx range carries zeros and is never stored):
//   inverse: z-pass (complex, length pz, zero-padded in kz) then x-pass (complex-to-real, length px,
//            two real rows packed into one complex transform);
//   forward: x-pass (real-to-complex, two rows per complex transform, split by Hermitian symmetry; the
//            split's factor 1/2 is left to the z-pass) then z-pass (complex, truncated, scaled by
//            1/(2 px pz)).
// Synthesis is unnormalised: f(x, z) = sum_k fhat_k exp(i (k1 x + k3 z)).
// A pass is one CTA per (plane, field, batch of columns / row pairs); every 1D transform is a
// Stockham autosort FFT in shared memory with radix-4/2/3 stages, a last stage of radix 12 (or 6) and a
// precomputed twiddle table. The z-passes fetch their columns with TMA tile copies
// (cp.async.bulk.tensor), the inverse x-pass its rows with bulk copies.
//
// Arithmetic: 64-bit fixed point with one exponent per 1D transform (fx.cuh), in both precisions. The
// FP64 pipe retires 1.68 additions per clock per SM here, and transforms in complex double were bound by
// it (85% busy); in fixed point the same passes run on the integer pipes (ALU 45-52%, multiply pipe
// 50-60% busy), 5.4 times faster than in complex double and 1.4 times faster than in the double-float
// arithmetic of the former precision path: at 512 x 65 x 512, per substage, 100.1 ms (complex double) and
// 25.2 ms (double-float) -> 18.4 ms. Spectral fields are complex double (the precision path's inputs
// double-float pairs) and physical fields double; T is fixed point with an array of exponents, so the
// conversions are at the ends only.
// Accuracy (rms error over rms result against a transform in extended precision; 2D transforms of white noise, the
// least and the most over amplitudes 1 .. 2, which the unit follows in one step; in parentheses complex double):
//   modes           32^2              128^2             512^2             768^2             1024^2
//   inverse   4.7-5.1e-17 (2.1e-16)  6.5-8.4e-17 (2.5)  1.4-2.5e-16 (2.8)  1.0-1.5e-16 (3.0)  1.3-1.7e-16 (3.0)
//   forward   8.4-9.2e-17 (2.4e-16)  1.0-1.2e-16 (2.6)  1.9-2.8e-16 (2.9)  1.5-1.8e-16 (3.1)  1.6-2.2e-16 (3.0)
// k^-2 spectra, inverse: 4.8e-17 (1.8e-16) at 32^2, 6.1e-17 (2.4e-16) at 512^2, 7.3e-17 (2.7e-16) at 1024^2.
// Inputs whose sums leave the range of single precision (fx_out_of_range) or lie near its low end take a slow path: 4
// fields of 512 x 65 x 512 at 1e-34 2.41 / 2.23 ms instead of 1.43 / 1.38 (complex double 7.8 / 8.6).
#include <cuda.h>  // CUtensorMap and its enums (the encoder is reached through the runtime, no libcuda link)

#include <climits>
#include <cmath>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "fx.cuh"

namespace lmvd {

LMVD_DEFINE_OOB_TAKE(fft)

struct FieldsC {
  const cd* p[10];
};
struct FieldsW {
  cd* p[10];
};
struct FieldsRC {
  const void* p[10];
};
struct FieldsRW {
  void* p[10];
};

// ------------------------------------------------------------------ Stockham stages
// A transform of length n is shared by tpt = n / EPT threads, EPT = 12 or (n an odd multiple of 6) 6. Its last
// stage has radix EPT, computed in a thread's registers; the stages before it have radices 4, 2 and 3, in place
// in shared memory: thread tt owns the butterflies tt, tt + tpt, ... (EPT / R of them), loads all their inputs
// into registers, waits for the whole block, then writes the outputs back to the same buffer.
// S: distance in elements between consecutive points of a transform in shared memory (1: contiguous; the
// z-passes interleave their columns, point i of column c at (i S + c)).
template <int SIGN>
__device__ __forceinline__ void fx_bfly4(cfx& v0, cfx& v1, cfx& v2, cfx& v3) {
  // the outputs as sums of three terms: one 64-bit addition of three operands takes the same two instructions as
  // one of two
  const cfx s = v1 + v3, d = v1 - v3, t = SIGN > 0 ? fx_ti(d) : cfx{d.im, -d.re};  // t = (SIGN i) (v1 - v3)
  const cfx a = v0, c = v2;
  v0 = (a + s) + c;
  v1 = (a + t) - c;
  v2 = (a - s) + c;
  v3 = (a - t) - c;
}
// FAIR: the half of an odd t rounds up or down as v0 is odd or even, so that its error has no direction of its own (rounded
// down, the three or four radix-3 stages of 432 to 648 modes put errors of 14 to 26 times the rms into a few outputs); an
// even t stays exact. 4 fields of 216 x 65 x 108, six such stages in its two passes: 171.7 -> 174.8 us. The last stage of
// lengths without guard bits rounds down: that moves an output by 1.5 units on average, a tenth of the noise, and the
// rounding would cost registers there: 3 fields of 256 x 129 x 256 forward 498.2 -> 505.0 us.
template <int SIGN, bool FAIR>
__device__ __forceinline__ void fx_bfly3(cfx& v0, cfx& v1, cfx& v2, int2 s3) {
  const cfx t = v1 + v2, d = v1 - v2;
  const cfx m = FAIR ? cfx{v0.re - ((t.re + (v0.re & 1)) >> 1), v0.im - ((t.im + (v0.im & 1)) >> 1)}
                     : cfx{v0.re - (t.re >> 1), v0.im - (t.im >> 1)};
  const long long ur = fx_mulr(d.re, s3), ui = fx_mulr(d.im, s3);
  const cfx u = SIGN > 0 ? cfx{-ui, ur} : cfx{ui, -ur};  // (SIGN i sin(2 pi / 3)) (v1 - v2)
  v0 = v0 + t;
  v1 = m + u;
  v2 = m - u;
}
template <int SIGN, int R>
__device__ __forceinline__ void fx_butterfly(cfx (&v)[R], const FFTPlan& pl) {
  if constexpr (R == 4) {
    fx_bfly4<SIGN>(v[0], v[1], v[2], v[3]);
  } else if constexpr (R == 3) {
    fx_bfly3<SIGN, true>(v[0], v[1], v[2], pl.s3);
  } else {
    const cfx t = v[0];
    v[0] = t + v[1];
    v[1] = t - v[1];
  }
}

// A twiddle. The passes with 6 elements a thread use plain loads, so that a launch may overlap the kernel that wrote the
// table (the allocation-free transform, 20.5 -> 18.5 us at 64 x 33 x 64). With 12 elements the choice is which spills less
// (bytes, read-only / plain: forward x-pass 136 / 120, inverse z-pass 124 / 140, forward z-pass 116 / 124, inverse x-pass
// 64 / 64), a difference of half a percent: plain in the forward x-pass (3-field 256 x 129 x 256 analysis 500.0 -> 497.2
// us), the read-only path in the others (4-field 216 x 65 x 108 synthesis 170.9, plain 171.5 us).
template <int SIGN, int EPT, int S>
__device__ __forceinline__ int4 fx_tw(const int4* p) {
  if constexpr (EPT == 12 && (S > 1 || SIGN > 0)) return __ldg(p);
  else return *p;
}

// Guard bits (GUARD, lengths above kFxGuardLength). The unit follows the sum S of a transform's inputs, which grows like n
// for a white input, while binary64's error hardly grows: above 768 points the noise, most of it from the rounding of the
// inputs, would exceed it. But the first two stages add up at most 16 inputs, so their values carry e <= 2 more bits where
// 16 times the largest input allows (white inputs; with a few large ones S is small already), and the third stage's
// twiddles are 2^-e as large, so that its products round back to the unit. The noise of a 1536-point transform falls from
// 17.5 units to 6.3, the error at 1024 x 1024 modes from 3.9-5.8e-16 to 1.3-1.7e-16 (inverse) and from 3.6-5.3e-16 to
// 1.6-2.2e-16 (forward; complex double 3.0e-16). It costs registers and a tenth of the time: 4 fields of 768 x 33 x 768
// 1.99 / 1.93 -> 2.18 / 2.07 ms (inverse / forward; complex double 9.9 / 10.8). Shorter lengths are as accurate without.
constexpr int kFxGuardLength = 768, kFxGuardBits = 2, kFxGuardStage = 2;
__device__ __forceinline__ int fx_guard(int most, int emin, int k) {  // most: see the callers
  return max(0, min(min(most, emin - k), kFxGuardBits));
}
// the limbs of w 2^-e, e > 0; the low one toward zero, so that those of 1 and -1, whose products may end in a half, round
// that toward zero and not always up
__device__ __forceinline__ int2 fx_limbs_shift(int hi, int lo, int e) {
  const int h = (hi >> e) + ((hi >> (e - 1)) & 1), rem = (int)((unsigned)hi - ((unsigned)h << e));
  return make_int2(h, (int)((unsigned)rem << (31 - e)) + ((lo + (lo >> 31 & (1 << e) - 1)) >> e));
}
// x 2^-e, e > 0, rounded to nearest; a half goes up or down by a bit that the result does not hold (to even would favour
// even results, whose lowest bits steer fx_bfly3)
__device__ __forceinline__ long long fx_round(long long x, int e) {
  return (x + ((1ll << (e - 1)) - 1 + ((x >> (e + 1)) & 1))) >> e;
}

// The sub-length L divides tpt (the radices before the last multiply to tpt), so a thread's butterflies share k = tt mod
// L and their twiddles, which are fetched before the barrier. SHIFT: the stage takes off e guard bits.
template <int SIGN, int R, int EPT, int S, bool SHIFT>
__device__ __forceinline__ void fx_stage(cfx* x, const FFTPlan& pl, int L, int tt, int tpt, int e) {
  constexpr int NBT = EPT / R;
  const int n = pl.n;
  const int nb = n / R;
  const int k = (L & (L - 1)) == 0 ? (tt & (L - 1)) : (tt % L);
  const int kt = k * (n / (L * R));
  int4 w[R];
#pragma unroll
  for (int q = 1; q < R; ++q) w[q] = fx_tw<SIGN, EPT, S>(pl.tw + q * kt);
  if (SHIFT && e)
#pragma unroll
    for (int q = 1; q < R; ++q) {
      const int2 c = fx_limbs_shift(w[q].x, w[q].y, e), s = fx_limbs_shift(w[q].z, w[q].w, e);
      w[q] = make_int4(c.x, c.y, s.x, s.y);
    }
  cfx v[NBT][R];
#pragma unroll
  for (int j = 0; j < NBT; ++j)
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int i = tt + j * tpt + q * nb;
      v[j][q] = LMVD_IN(i, n) ? x[i * S] : cfx{0, 0};
    }
  __syncthreads();
  cfx* y = x + ((tt - k) * R + k) * S;
#pragma unroll
  for (int j = 0; j < NBT; ++j) {
    if (!LMVD_IN((tt - k) * R + k + j * tpt * R + (R - 1) * L, n)) continue;
    if (k || SHIFT && e)  // (a product with w = 1 would not be exact)
#pragma unroll
      for (int q = 1; q < R; ++q) v[j][q] = fx_mulw<SIGN>(v[j][q], w[q]);
    if (SHIFT && e) v[j][0] = cfx{fx_round(v[j][0].re, e), fx_round(v[j][0].im, e)};
    fx_butterfly<SIGN, R>(v[j], pl);
#pragma unroll
    for (int q = 0; q < R; ++q) y[(j * tpt * R + q * L) * S] = v[j][q];
  }
  __syncthreads();
}

// First stage of radix 4 (L = 1, no twiddles) from registers: v[4 j + q] is input point tt + j tpt + q n / 4. The
// caller has waited for every thread's reads.
template <int SIGN, int S>
__device__ __forceinline__ void fx_first4(cfx (&v)[12], cfx* x, const FFTPlan& pl, int tt, int tpt) {
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    fx_bfly4<SIGN>(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
    const int base = (tt + j * tpt) * 4;
    if (!LMVD_IN(base + 3, pl.n)) continue;
#pragma unroll
    for (int q = 0; q < 4; ++q) x[(base + q) * S] = v[4 * j + q];
  }
  __syncthreads();
}

// Stages s0 .. nst - 2; returns when every point of the last stage's input is in x. e: the inputs' guard bits (a length
// above kFxGuardLength has four of these stages).
template <int SIGN, int EPT, int S, bool GUARD>
__device__ __forceinline__ void fx_middle(cfx* x, const FFTPlan& pl, int s0, int tt, int tpt, int e) {
  int L = 1;
  unsigned code = pl.code;
  if (s0) {
    L = 4;
    code >>= 2;
  }
  auto stage = [&](auto shift) {
    constexpr bool SHIFT = decltype(shift)::value;
    const unsigned r2 = code & 3u;
    if (EPT == 12 && r2 == 0) {
      fx_stage<SIGN, 4, EPT, S, SHIFT>(x, pl, L, tt, tpt, e);
      L *= 4;
    } else if (r2 == 1) {
      fx_stage<SIGN, 2, EPT, S, SHIFT>(x, pl, L, tt, tpt, e);
      L *= 2;
    } else {
      fx_stage<SIGN, 3, EPT, S, SHIFT>(x, pl, L, tt, tpt, e);
      L *= 3;
    }
    code >>= 2;
  };
  int s = s0;
  if constexpr (GUARD) {
    for (; s < kFxGuardStage; ++s) stage(std::false_type{});
    stage(std::true_type{});
    ++s;
  }
  for (; s < pl.nst - 1; ++s) stage(std::false_type{});
}

// Last stage: radix EPT, L = n / EPT = tpt; thread tt's butterfly reads and produces the points tt + q L. The EPT-point
// transform is a prime-factor one (3 x 4 or 3 x 2): input q = (EPT / 3) a + 3 b, output q = 4 a' + s b' mod EPT
// with s = 9 (EPT 12) or 3 (EPT 6), and no twiddles between its two parts. Against a radix-4 and a radix-3 stage
// it saves an exchange through shared memory and a third of the two stages' twiddle products.
template <int SIGN, int EPT, int S, bool GUARD>
__device__ __forceinline__ void fx_last(const cfx* x, const FFTPlan& pl, int tt, cfx (&v)[EPT]) {
  constexpr int R = EPT / 3;
  const int L = pl.tpt;
  cfx u[EPT];
#pragma unroll
  for (int q = 0; q < EPT; ++q) u[q] = LMVD_IN(tt + q * L, pl.n) ? x[(tt + q * L) * S] : cfx{0, 0};
  if (tt)
#pragma unroll
    for (int q = 1; q < EPT; ++q) u[q] = fx_mulw<SIGN>(u[q], fx_tw<SIGN, EPT, S>(pl.tw + q * tt));
#pragma unroll
  for (int b = 0; b < R; ++b) fx_bfly3<SIGN, GUARD>(u[3 * b], u[(R + 3 * b) % EPT], u[(2 * R + 3 * b) % EPT], pl.s3);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    // u[(R a + 3 b) mod EPT] now holds (a', b) = (a, b)
    cfx w[R];
#pragma unroll
    for (int b = 0; b < R; ++b) w[b] = u[(R * a + 3 * b) % EPT];
    if constexpr (R == 4) fx_bfly4<SIGN>(w[0], w[1], w[2], w[3]);
    else fx_butterfly<SIGN, R>(w, pl);
#pragma unroll
    for (int b = 0; b < R; ++b) v[(4 * a + (R == 4 ? 9 : 3) * b) % EPT] = w[b];
  }
}

// ------------------------------------------------------------------ the exponent of a transform
// red: partial sums of the CTA (one float per group of g threads of a transform), top: its largest high word
// (for the slow path), emin: its warps' smallest E (fx_scale_t). Thread tt of a transform whose threads are S lanes
// apart; g is the largest power of two dividing tpt with g S <= 32, so a group lies in one warp.
constexpr int FX_RED = 256;
struct FxShared {
  float red[FX_RED];
  int emin[8];
  int top;
  int wtop[8];  // (GUARD) the warps' largest magnitudes
};

__device__ __forceinline__ unsigned warp_lanes() {  // the lanes of this warp (the last one may be partial)
  const unsigned lanes = blockDim.x - (threadIdx.x & ~31u);
  return lanes >= 32 ? 0xffffffffu : (1u << lanes) - 1u;
}
__device__ __forceinline__ float group_sum(float v, int g, int S) {
  const unsigned mask = warp_lanes();
  for (int o = S; o < g * S; o <<= 1) v += __shfl_xor_sync(mask, v, o);
  return v;
}

// The slow path of inputs outside the range of the FP32 sums: divides them by 2^xe, the exponent of the CTA's
// largest magnitude; INT_MIN if one of them is inf or nan (the results are then nan).
constexpr int kFxPoison = INT_MIN;
__device__ __noinline__ double fx_scale2(double x, int e) { return scalbn(x, e); }
__device__ __noinline__ float fx_scale2f(float x, int e) { return scalbnf(x, e); }
__device__ __forceinline__ cd fx_scaled(cd x, int e) { return cd{fx_scale2(x.re, e), fx_scale2(x.im, e)}; }
__device__ __forceinline__ df fx_scaled(df x, int e) { return df{fx_scale2f(x.hi, e), fx_scale2f(x.lo, e)}; }
__device__ __forceinline__ cdf fx_scaled(cdf x, int e) { return cdf{fx_scaled(x.re, e), fx_scaled(x.im, e)}; }
template <class RAW, int N>
__device__ __forceinline__ int fx_rescale(RAW (&raw)[N], int top, FxShared& sh) {
  constexpr bool d = std::is_same<RAW, cd>::value;
  atomicMax(&sh.top, top);
  __syncthreads();
  const int m = sh.top;
  if (m >= (d ? 0x7ff00000 : 0x7f800000)) return kFxPoison;
  const int xe = d ? max(m >> 20, 1) - 1023 : max(m >> 23, 1) - 127;
#pragma unroll
  for (int i = 0; i < N; ++i) raw[i] = fx_scaled(raw[i], -xe);
  return xe;
}
__device__ __noinline__ double fx_unscale(double d, int xe) {
  return xe == kFxPoison ? __longlong_as_double(0x7ff8000000000000ll) : scalbn(d, xe);
}

__device__ __forceinline__ void mag_add(FxMag& m, cd x) { m.add(x.re, x.im); }
__device__ __forceinline__ void mag_add(FxMag& m, cdf x) { m.add(x.re, x.im); }
template <class RAW>
constexpr bool kIsDf = std::is_same<RAW, cdf>::value;
template <int N>
__device__ __forceinline__ int fx_any_bits(const cd (&raw)[N]) {
  int any = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) any |= __double2loint(raw[i].re) | __double2loint(raw[i].im);
  return any != 0;
}
template <int N>
__device__ __forceinline__ int fx_any_bits(const cdf (&)[N]) { return 0; }

// the CTA's largest of the threads' non-negative integers m, in two parts around a barrier
__device__ __forceinline__ void fx_max_put(int m, FxShared& sh) {
  m = __reduce_max_sync(warp_lanes(), m);
  if ((threadIdx.x & 31) == 0) sh.wtop[threadIdx.x >> 5] = m;
}
__device__ __forceinline__ int fx_max_get(const FxShared& sh) {
  int m = 0;
  for (int w = 0; w < (int)(blockDim.x + 31) >> 5; ++w) m = max(m, sh.wtop[w]);
  return m;
}

// k of this thread's transform from the RAW values its threads hold, all threads of the CTA together; xe: see fx_rescale
// (0 on the usual path); e: the guard bits the inputs may carry beyond k (0 without GUARD): a magnitude with the high word
// `top` is below 2^(t + 1), so 16 inputs' |re| + |im| stay below 2^(t + 6) and 2^(t + 6 + k + e) <= 2^61. One barrier.
template <bool GUARD, class RAW, int N>
__device__ __forceinline__ int fx_scale(RAW (&raw)[N], FxShared& sh, int slot, int np, int stride, int g, int S, int tt,
                                        int& xe, int& e) {
  FxMag m;
#pragma unroll
  for (int i = 0; i < N; ++i) mag_add(m, raw[i]);
  if (m.top == 0) m.top = fx_any_bits(raw);  // magnitudes below 2^-1042 have an empty high word
  float v = group_sum(m.sum, g, S);
  if ((tt & (g - 1)) == 0 && LMVD_IN(slot + (tt / g) * stride, FX_RED)) sh.red[slot + (tt / g) * stride] = v;
  if (GUARD) fx_max_put(m.top, sh);
  xe = 0;
  if (__syncthreads_or(fx_out_of_range(m, kIsDf<RAW>))) {
    xe = fx_rescale(raw, m.top, sh);
    FxMag r;
#pragma unroll
    for (int i = 0; i < N; ++i) mag_add(r, raw[i]);
    v = group_sum(r.sum, g, S);
    if ((tt & (g - 1)) == 0 && LMVD_IN(slot + (tt / g) * stride, FX_RED)) sh.red[slot + (tt / g) * stride] = v;
    if (GUARD) fx_max_put(r.top, sh);
    __syncthreads();
  }
  float s = 0.f;
  for (int i = 0; i < np; ++i) s += sh.red[slot + i * stride];
  const int k = s == 0.f ? kFxZeroK : fx_exponent(s);
  e = 0;
  if (GUARD) e = fx_guard(55 - (kIsDf<RAW> ? (fx_max_get(sh) >> 23) - 127 : (fx_max_get(sh) >> 20) - 1023) - k, INT_MAX, k);
  return k;
}
// The intermediate T between the two passes of a transform stays in fixed point: 16 bytes per element and one
// exponent E per transform of the first pass (a kx column of the inverse, a row pair of the forward one; the value is
// X 2^-E), so neither side converts; kFxNan marks a transform with inf or nan in it, kFxZero one of zeros (or of values
// below 2^-126 of the largest one of its CTA). The second pass's exponent k is at most the smallest E of its inputs
// (their own unit: a smaller one holds no information), so that its inputs only shift right; zeros have no unit and are
// above every E, so that an empty column does not limit the others of its plane. Sums are formed from the high words in
// FP32, E in the range that the usual path gives (up to 161, where fx_exponent ends too).
constexpr int kFxNan = INT_MIN, kFxZero = 1 << 20, kFxMinE = -40, kFxMaxE = 161;
__device__ __forceinline__ float fx_abs_hi(long long x) { return fabsf(__int2float_rn((int)(x >> 32))); }
__device__ __forceinline__ float fx_mag_hi(cfx x) { return fx_abs_hi(x.re) + fx_abs_hi(x.im); }
__device__ __forceinline__ float fx_pow2(int e) { return __int_as_float((e + 127) << 23); }  // -126 <= e <= 127
// sum |X| 2^-E of inputs that share E (kFxMinE <= E; a sum at an E beyond kFxMaxE may read too large, never too small)
__device__ __forceinline__ float fx_mag(float hi_sum, int E) { return hi_sum * 0x1p-32f * fx_pow2(max(64 - E, -126)); }

// As fx_scale, for fixed-point inputs: per thread the sum `mag` of its inputs' magnitudes (each |re| + |im|), the largest of
// them `big` and the smallest E. On the slow path E is first counted from the CTA's smallest (remag recomputes mag and big
// for the shifted E's).
template <bool GUARD, class Remag>
__device__ __forceinline__ int fx_scale_t(float mag, float big, int& emin, FxShared& sh, int slot, int np, int stride, int g,
                                          int S, int tt, int& xe, int& e, Remag&& remag) {
  float v = group_sum(mag, g, S);
  if ((tt & (g - 1)) == 0 && LMVD_IN(slot + (tt / g) * stride, FX_RED)) sh.red[slot + (tt / g) * stride] = v;
  emin = __reduce_min_sync(warp_lanes(), emin);
  if ((threadIdx.x & 31) == 0) sh.emin[threadIdx.x >> 5] = emin;
  if (GUARD) fx_max_put(__float_as_int(big), sh);
  xe = 0;
  const bool slow = __syncthreads_or(emin < kFxMinE || emin > kFxMaxE && emin != kFxZero);
  const int nw = (blockDim.x + 31) >> 5;
  for (int w = 0; w < nw; ++w) emin = min(emin, sh.emin[w]);
  if (slow) {
    if (emin == kFxNan) {
      xe = kFxPoison;
    } else {
      xe = 61 - emin;  // E' = E + xe: the largest inputs are of the order of one
      v = group_sum(remag(xe, big), g, S);
      __syncthreads();
      if ((tt & (g - 1)) == 0 && LMVD_IN(slot + (tt / g) * stride, FX_RED)) sh.red[slot + (tt / g) * stride] = v;
      if (GUARD) fx_max_put(__float_as_int(big), sh);
      __syncthreads();
      emin = 61;
    }
  }
  float s = 0.f;
  for (int i = 0; i < np; ++i) s += sh.red[slot + i * stride];
  const int k = min(fx_exponent(s), emin);
  e = 0;
  if (GUARD) e = fx_guard(56 - ((fx_max_get(sh) >> 23) - 127) - k, emin, k);  // (as in fx_scale: `big` is a sum already)
  return k;
}
// X 2^(k - E), rounded to nearest; d = E - k >= 0. Beyond 62 places a magnitude of up to 2^62 becomes 0; the forward
// pass's row sums may reach 2^62.7, which then become -1, an error below two units. (Without the rounding above 32 places
// the columns of a decaying spectrum were off by half a unit on average, all in the same direction.)
__device__ __forceinline__ cfx fx_align(cfx x, int d) {
  const long long h = (long long)((unsigned long long)shl32(1u, min(d, 63) - 33) << 32 | shl32(1u, d - 1));
  return cfx{sar64(x.re + h, d), sar64(x.im + h, d)};
}
__device__ __forceinline__ cfx fx_convert(cd x, int k, float) { return cfx{fx_from(x.re, k), fx_from(x.im, k)}; }
__device__ __forceinline__ cfx fx_convert(cdf x, int, float sa) { return cfx{fx_from(x.re, sa), fx_from(x.im, sa)}; }
__device__ __forceinline__ float fx_sa(int k) { return __int_as_float((k - 40 + 127) << 23); }

// A result as a complex double: the two parts take different routes, so that the FP64 pipe does half of the
// conversions beside the integer pipes.
__device__ __forceinline__ cd fx_result(cfx v, int k, int xe) {
  cd r{fx_to_fp(v.re, k << 20), fx_to(v.im, k)};
  if (xe) r = cd{fx_unscale(r.re, xe), fx_unscale(r.im, xe)};
  return r;
}

// CTAs: the x-passes run small ones (128 threads), so that the load, compute and store phases of different CTAs
// (separated by barriers) overlap; the z-passes take 4 kx columns per CTA (2 when 4 transforms do not fit
// FFT_CTA_Z threads).
constexpr int FFT_CTA_X = 128, FFT_CTA_Z = 256;
// CTAs per SM each pass is compiled for, i.e. its register cap (80). A thread holds 12 elements of 4 registers; at
// 512 x 65 x 512 the inverse x-passes take 7.06 / 6.95 / 7.05 ms per substage at 5 / 6 / 7 CTAs, the forward ones
// 4.97 / 4.91 / 5.21, the z-passes 8.22 / 7.11 at 2 / 3 (4: 5% slower than 3).
constexpr int FFT_MIN_X = 6, FFT_MIN_Z = 3;

// ---------------------------------------------------------------- tile loads (TMA)
// The z-passes read columns of a row-major plane: batch consecutive kx (16-byte elements) of every z-row. A
// tensor-map tile copy (cp.async.bulk.tensor) fetches such a box (2 batch doubles x rows) into shared
// memory as one asynchronous operation completing on an mbarrier, instead of one 16-byte load per thread
// and element. The box lands row-major, i.e. as the interleaved layout the z-pass transforms work in.
struct ZMaps {
  CUtensorMap m[TBUF_MAX];  // the spectral inputs, one per field of the launch
};

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// box of the 3D map at (x, y, z) (x in doubles) into dst; completes tx bytes on bar
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z,
                                            unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(smem_addr(dst)), "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_addr(bar))
      : "memory");
}

// bytes (a multiple of 16, both addresses 16-byte aligned) from src to dst; completes them on bar
__device__ __forceinline__ void bulk_load(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}

// Every thread waits for phase 0 of bar, for at most ~1 s of SM clock; false (and bit 2 of the context's
// status word, when there is one) if the copies did not complete by then.
__device__ __forceinline__ bool mbar_wait_bounded(unsigned long long* bar, unsigned* flags) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, 0)) {
    if (clock64() - t0 > 2000000000ll) {
      if (flags && threadIdx.x == 0) atomicOr(flags, 4u);
      return false;
    }
  }
  return true;
}

// The exponent a transform's fixed-point results are stored with (xe: fx_rescale's)
__device__ __forceinline__ int fx_stored_exponent(int k, int xe) {
  return xe == kFxPoison ? kFxNan : (k == kFxZeroK ? kFxZero : k - xe);
}

// Fixed-point inputs v of a transform in shared memory: through a first radix-4 stage in registers (v in the order of
// fx_first4), or, for a plan without one, to the points tt + u tpt (v in that order), then the middle stages.
template <int SIGN, int EPT, int S, bool GUARD>
__device__ __forceinline__ void fx_run(cfx (&v)[EPT], cfx* x, const FFTPlan& pl, bool first4, int tt, int e) {
  if constexpr (EPT == 12) {
    if (first4) {
      fx_first4<SIGN, S>(v, x, pl, tt, pl.tpt);
      fx_middle<SIGN, EPT, S, GUARD>(x, pl, 1, tt, pl.tpt, e);
      return;
    }
  }
#pragma unroll
  for (int u = 0; u < EPT; ++u)
    if (LMVD_IN(tt + u * pl.tpt, pl.n)) x[(tt + u * pl.tpt) * S] = v[u];
  __syncthreads();
  fx_middle<SIGN, EPT, S, GUARD>(x, pl, 0, tt, pl.tpt, e);
}
// input point u of a thread, in the order fx_run expects (step: n / 4 with a first radix-4 stage)
__device__ __forceinline__ int fx_point(int u, bool first4, int tt, int tpt, int step) {
  return first4 ? tt + (u >> 2) * tpt + (u & 3) * step : tt + u * tpt;
}

// ---------------------------------------------------------------- inverse z-pass
// in: spectral value fields [ny][nz][nxh] of RAW (complex double, or the double-float pairs that the precision
// path's evaluations store in the same 16 bytes); T: [f][ny][pz][nx/2] fixed-point, te: [f][ny][nx/2] its exponents.
// A CTA transforms COLS kx columns of one plane. Shared layout: point z of column c at a[z COLS + c]; two
// tile loads per row block put the kz >= 0 rows at the top and the kz < 0 rows at the bottom of the padded
// column (the Nyquist row lands inside the zero band, which is never read).
template <class RAW, int EPT, int COLS>
__global__ void __launch_bounds__(FFT_CTA_Z, FFT_MIN_Z)
    k_fft_z_inv(FFTPlan pl, Grid g, const __grid_constant__ ZMaps maps, cfx* T, size_t tstride, int* te, unsigned* flags) {
  grid_wait();
  extern __shared__ __align__(128) unsigned char sm_raw[];
  __shared__ FxShared sh;
  cfx* a = reinterpret_cast<cfx*>(sm_raw);
  const int pz = g.pz, nz = g.nz, h = g.nx / 2, n2 = nz / 2, H = pl.rows_in, tpt = pl.tpt;
  const int kx0 = blockIdx.x * COLS, j = blockIdx.y, f = blockIdx.z;
  const int c = threadIdx.x % COLS, tt = threadIdx.x / COLS, kx = kx0 + c;
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(sm_raw + (size_t)pz * COLS * sizeof(cfx));
  if (threadIdx.x == 0) {
    mbar_init(bar);
    sh.top = 0;
  }
  __syncthreads();
  if (threadIdx.x == 0 && LMVD_IN(f, TBUF_MAX)) {
    mbar_expect_tx(bar, (unsigned)(nz * COLS * sizeof(cfx)));
    for (int r = 0; r < nz; r += H) {
      const int pos = r < n2 ? r : pz - nz + r;
      if (LMVD_IN((pos + H) * COLS - 1, pz * COLS)) tma_load_3d(a + (size_t)pos * COLS, &maps.m[f], 2 * kx0, r, j, bar);
    }
  }
  if (!mbar_wait_bounded(bar, flags)) return;
  const bool first4 = EPT == 12 && pl.first4;
  RAW raw[EPT];
  const int lo = n2, hi = pz - n2 + 1;  // kz padding: zero
#pragma unroll
  for (int u = 0; u < EPT; ++u) {
    const int i = fx_point(u, first4, tt, tpt, pz >> 2);
    raw[u] = kx < h && LMVD_IN(i, pz) && (i < lo || i >= hi) ? reinterpret_cast<const RAW*>(a)[i * COLS + c] : RAW{};
  }
  constexpr bool GUARD = COLS == 2;  // (the lengths of which 4 columns do not fit in a CTA)
  static_assert(4 * kFxGuardLength == 12 * FFT_CTA_Z, "2 columns: above kFxGuardLength");
  int xe, e;
  const int gz = pl.red_g, k = fx_scale<GUARD>(raw, sh, c, tpt / gz, COLS, gz, COLS, tt, xe, e);
  {
    cfx v[EPT];
    const float sa = fx_sa(k + e);
#pragma unroll
    for (int u = 0; u < EPT; ++u) {
      const int i = fx_point(u, first4, tt, tpt, pz >> 2);
      v[u] = cfx{0, 0};
      if (i < lo || i >= hi) v[u] = fx_convert(raw[u], k + e, sa);  // (whole warps skip the padding)
    }
    fx_run<1, EPT, COLS, GUARD>(v, a + c, pl, first4, tt, e);
  }
  cfx v[EPT];
  fx_last<1, EPT, COLS, GUARD>(a + c, pl, tt, v);
  if (kx >= h) return;
  if (tt == 0) te[((size_t)f * g.ny + j) * h + kx] = fx_stored_exponent(k, xe);
  cfx* dst = T + f * tstride + (size_t)j * pz * h + kx;
#pragma unroll
  for (int q = 0; q < EPT; ++q)
    if (LMVD_IN((size_t)(tt + q * tpt) * h + kx, (size_t)pz * h)) dst[(size_t)(tt + q * tpt) * h] = v[q];
}

// ---------------------------------------------------------------- inverse x-pass (c2r, 2 rows per transform)
// With MUL the epilogue stores w * phys instead of phys (w: a physical field of the same layout, one for all
// fields of the launch): the product f'(z) dz/dt of the fixed point (Sec. 4.3) formed as the transform is
// written, so neither dz/dt on the grid nor a separate product pass is needed. (pz is even: 6 divides it.)
template <int EPT, bool GUARD, bool MUL>
__device__ __forceinline__ void x_inv_body(const FFTPlan& pl, const Grid& g, const cfx* T, size_t tstride, const int* te,
                                           const FieldsRW& out, const double* wmul, unsigned* flags) {
  extern __shared__ __align__(128) unsigned char sm_raw[];
  __shared__ FxShared sh;
  cfx* a = reinterpret_cast<cfx*>(sm_raw);
  const int batch = pl.batch, ld = pl.n + pl.pad, px = g.px, pz = g.pz, h = g.nx / 2, tpt = pl.tpt;
  const int pr0 = blockIdx.x * batch, j = blockIdx.y, f = blockIdx.z;
  const int bt = threadIdx.x / tpt, tt = threadIdx.x - bt * tpt;
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(sm_raw + (size_t)batch * ld * sizeof(cfx));
  if (threadIdx.x == 0) mbar_init(bar);
  __syncthreads();
  // A transform's rows za = 2 (pr0 + bt) and za + 1 of T are contiguous (2 h elements): one bulk copy each
  // (TMA, cp.async.bulk) into the upper part [h, 3 h) = [h, px) of its buffer, completing on the mbarrier
  if (threadIdx.x == 0) {
    const cfx* src = T + f * tstride + (size_t)j * pz * h;
    int nb = 0;
    while (nb < batch && 2 * (pr0 + nb) < pz) ++nb;
    mbar_expect_tx(bar, (unsigned)(nb * 2 * h * sizeof(cfx)));
    for (int bb = 0; bb < nb; ++bb) {
      const int za = 2 * (pr0 + bb);
      if (LMVD_IN(bb * ld + px - 1, batch * ld) && LMVD_IN((size_t)(za + 2) * h - 1, (size_t)pz * h))
        bulk_load(a + bb * ld + h, src + (size_t)za * h, (unsigned)(2 * h * sizeof(cfx)), bar);
    }
  }
  // two real rows into one complex transform: y[k] = Xa[k] + i Xb[k], y[px - k] = conj(Xa[k]) + i conj(Xb[k]).
  // A thread takes the EPT / 3 pairs k = tt, tt + tpt, ... < h; the scale's barrier precedes every write of a
  // y[px - k] over the copied rows.
  constexpr int NP = EPT / 3;
  const int za = 2 * (pr0 + bt);
  const bool live = za < pz;
  cfx* y = a + bt * ld;
  int E[NP], emin = INT_MAX;
  const int* ej = te + ((size_t)f * g.ny + j) * h;
#pragma unroll
  for (int u = 0; u < NP; ++u) {
    E[u] = LMVD_IN(tt + u * tpt, h) ? ej[tt + u * tpt] : kFxZero;
    emin = min(emin, E[u]);
  }
  if (!mbar_wait_bounded(bar, flags)) return;
  cfx raw[2 * NP];
  // |re| + |im| of y[k] and y[px - k] add up to 2 (max(|Xa.re|, |Xb.im|) + max(|Xa.im|, |Xb.re|)); the sum of the four
  // magnitudes is half a bit more (rms error of a white 1024 x 16 inverse at an unlucky amplitude: 5.3e-16)
  float hs[NP], mag = 0.f, big = 0.f;
#pragma unroll
  for (int u = 0; u < NP; ++u) {
    const int kk = tt + u * tpt;
    const bool in = live && LMVD_IN(bt * ld + 2 * h + kk, batch * ld);
    raw[2 * u] = in ? y[h + kk] : cfx{0, 0};
    raw[2 * u + 1] = in ? y[2 * h + kk] : cfx{0, 0};
    if (kk == 0) raw[2 * u].im = raw[2 * u + 1].im = 0;  // the kx = 0 coefficient of a real row is real
    hs[u] = 2.f * (fmaxf(fx_abs_hi(raw[2 * u].re), fx_abs_hi(raw[2 * u + 1].im)) +
                   fmaxf(fx_abs_hi(raw[2 * u].im), fx_abs_hi(raw[2 * u + 1].re)));
    const float y2 = fx_mag(hs[u], E[u]);
    mag += y2;
    big = fmaxf(big, y2);
  }
  int xe, e;
  const int gx = pl.red_g, np = tpt / gx;
  const int k = fx_scale_t<GUARD>(mag, big, emin, sh, bt * np, np, 1, gx, 1, tt, xe, e, [&](int s, float& b) {
    float m = b = 0.f;
#pragma unroll
    for (int u = 0; u < NP; ++u) {
      const float y2 = fx_mag(hs[u], E[u] += s);
      m += y2;
      b = fmaxf(b, y2);
    }
    return m;
  });
#pragma unroll
  for (int u = 0; u < NP; ++u) {
    const int kk = tt + u * tpt;
    const cfx xa = fx_align(raw[2 * u], E[u] - k - e), xb = fx_align(raw[2 * u + 1], E[u] - k - e);
    if (!LMVD_IN(kk, h)) continue;
    if (kk == 0) {
      y[0] = cfx{xa.re, xb.re};
    } else {
      y[kk] = cfx{xa.re - xb.im, xa.im + xb.re};       // Xa[k] + i Xb[k]
      y[px - kk] = cfx{xa.re + xb.im, xb.re - xa.im};  // conj(Xa[k]) + i conj(Xb[k])
    }
  }
  // the kx padding [h, 2 h] (a first stage of its own that skips it instead was 3% slower: instruction cache)
#pragma unroll
  for (int u = 0; u < NP; ++u)
    if (LMVD_IN(h + tt + u * tpt, px)) y[h + tt + u * tpt] = cfx{0, 0};
  if (tt == 0 && LMVD_IN(2 * h, px)) y[2 * h] = cfx{0, 0};
  __syncthreads();
  fx_middle<1, EPT, 1, GUARD>(y, pl, 0, tt, tpt, e);
  double* dst = reinterpret_cast<double*>(pick(out.p, f)) + (size_t)j * g.P + (size_t)za * px;
  const double* w = MUL ? wmul + (size_t)j * g.P + (size_t)za * px : nullptr;
  cfx v[EPT];
  fx_last<1, EPT, 1, GUARD>(y, pl, tt, v);
  if (!live) return;
#pragma unroll
  for (int q = 0; q < EPT; ++q) {
    const int x = tt + q * tpt;
    if (!LMVD_IN((size_t)(za + 1) * px + x, g.P)) continue;
    const cd r = fx_result(v[q], k, xe);
    dst[x] = MUL ? w[x] * r.re : r.re;
    dst[px + x] = MUL ? w[px + x] * r.im : r.im;
  }
}
template <int EPT, bool GUARD>
__global__ void __launch_bounds__(FFT_CTA_X, FFT_MIN_X) k_fft_x_inv(FFTPlan pl, Grid g, const cfx* T, size_t tstride,
                                                                    const int* te, FieldsRW out, unsigned* flags) {
  grid_wait();
  x_inv_body<EPT, GUARD, false>(pl, g, T, tstride, te, out, nullptr, flags);
}
template <int EPT, bool GUARD>
__global__ void __launch_bounds__(FFT_CTA_X, FFT_MIN_X) k_fft_x_inv_mul(FFTPlan pl, Grid g, const cfx* T, size_t tstride,
                                                                        const int* te, FieldsRW out, const double* wmul,
                                                                        unsigned* flags) {
  grid_wait();
  x_inv_body<EPT, GUARD, true>(pl, g, T, tstride, te, out, wmul, flags);
}

// ---------------------------------------------------------------- forward x-pass (r2c, 2 rows per transform)
// With DOT3 the loads form -(w1 m1 + w2 m2 + w3 m3) from six physical fields instead of reading one (d: w[0..2],
// m[0..2]; one launch, one field): the tail -(1/rho) grad z . m^c of L (Sec. 4.3) formed as the transform reads
// it, so no product pass and no product field are needed.
// The loads are the first stage's inputs: they go from global memory to registers. te: [f][ny][pz/2] exponents of T.
struct Dot3 {
  const double* w[3];
  const double* m[3];
};
template <int EPT, bool GUARD, bool DOT3>
__device__ __forceinline__ void x_fwd_body(const FFTPlan& pl, const Grid& g, const FieldsRC& in, cfx* T, size_t tstride,
                                           int* te, const Dot3& d) {
  extern __shared__ __align__(128) unsigned char sm_raw[];
  __shared__ FxShared sh;
  cfx* a = reinterpret_cast<cfx*>(sm_raw);
  const int batch = pl.batch, ld = pl.n + pl.pad, px = g.px, pz = g.pz, h = g.nx / 2, tpt = pl.tpt;
  const int pr0 = blockIdx.x * batch, j = blockIdx.y, f = blockIdx.z;
  const int bt = threadIdx.x / tpt, tt = threadIdx.x - bt * tpt;
  const int za = 2 * (pr0 + bt);
  const bool live = za < pz;
  cfx* y = a + bt * ld;
  if (threadIdx.x == 0) sh.top = 0;
  const bool first4 = EPT == 12 && pl.first4;
  cd raw[EPT];
  const size_t row = (size_t)j * g.P + (size_t)za * px;
  const double* src = DOT3 ? nullptr : reinterpret_cast<const double*>(pick(in.p, f)) + row;
#pragma unroll
  for (int u = 0; u < EPT; ++u) {
    const int x = fx_point(u, first4, tt, tpt, px >> 2);
    cd v{};
    if (live && LMVD_IN((size_t)(za + 1) * px + x, g.P)) {
      if (DOT3) {
        const size_t o = row + x;
        v.re = -(d.w[0][o] * d.m[0][o] + d.w[1][o] * d.m[1][o] + d.w[2][o] * d.m[2][o]);
        const size_t o2 = o + px;
        v.im = -(d.w[0][o2] * d.m[0][o2] + d.w[1][o2] * d.m[1][o2] + d.w[2][o2] * d.m[2][o2]);
      } else {
        v = cd{src[x], src[px + x]};
      }
    }
    raw[u] = v;
  }
  __syncthreads();  // sh.top
  int xe, e;
  // (the sums p + conj(m) = twice a row's coefficient formed at the end may reach 2^62.7: no product follows)
  const int gx = pl.red_g, np = tpt / gx, k = fx_scale<GUARD>(raw, sh, bt * np, np, 1, gx, 1, tt, xe, e);
  {
    cfx v[EPT];
#pragma unroll
    for (int u = 0; u < EPT; ++u) v[u] = fx_convert(raw[u], k + e, 0.f);
    fx_run<-1, EPT, 1, GUARD>(v, y, pl, first4, tt, e);
  }
  // last stage: the retained kx are the outputs q < NP (kx = tt + q tpt) and q >= 2 NP (px - kx); a thread keeps the
  // first and stores the others for the thread that pairs them
  constexpr int NP = EPT / 3;
  cfx v[EPT];
  fx_last<-1, EPT, 1, GUARD>(y, pl, tt, v);
#pragma unroll
  for (int q = 2 * NP; q < EPT; ++q)
    if (LMVD_IN(tt + q * tpt, px)) y[tt + q * tpt] = v[q];  // this thread's own inputs
  __syncthreads();
  if (!live) return;
  if (tt == 0) te[((size_t)f * g.ny + j) * (pz / 2) + pr0 + bt] = fx_stored_exponent(k, xe);
  cfx* dst = T + f * tstride + (size_t)j * pz * h + (size_t)za * h;
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    const int kk = tt + q * tpt;
    if (!LMVD_IN((size_t)(za + 1) * h + kk, (size_t)pz * h)) continue;
    const cfx p = v[q], m = kk == 0 ? p : y[px - kk];
    // twice the two rows' spectra (the 1/2 is in the z-pass's scale): p + conj(m) and (p - conj(m)) / i
    dst[kk] = cfx{p.re + m.re, p.im - m.im};
    dst[h + kk] = cfx{p.im + m.im, m.re - p.re};
  }
}
template <int EPT, bool GUARD>
__global__ void __launch_bounds__(FFT_CTA_X, FFT_MIN_X) k_fft_x_fwd(FFTPlan pl, Grid g, FieldsRC in, cfx* T, size_t tstride,
                                                                    int* te) {
  grid_wait();
  x_fwd_body<EPT, GUARD, false>(pl, g, in, T, tstride, te, Dot3{});
}
template <int EPT, bool GUARD>
__global__ void __launch_bounds__(FFT_CTA_X, FFT_MIN_X) k_fft_x_fwd_dot3(FFTPlan pl, Grid g, cfx* T, size_t tstride, int* te,
                                                                         Dot3 d) {
  grid_wait();
  x_fwd_body<EPT, GUARD, true>(pl, g, FieldsRC{}, T, tstride, te, d);
}

// ---------------------------------------------------------------- forward z-pass (truncate, scale)
// T: [f][ny][pz][nx/2], read through the tensor map (all fields of the launch: planes f ny + j), its exponents te [f][ny]
// [pz/2]; out: spectral fields [ny][nz][nxh]. Same interleaved layout as the inverse z-pass; kx = nx/2 and the kz
// Nyquist row are written as zero. The last stage's middle outputs are the truncated kz. add (may be null, one field):
// a spectral field added to the result.
template <int EPT, int COLS>
__global__ void __launch_bounds__(FFT_CTA_Z, FFT_MIN_Z)
    k_fft_z_fwd(FFTPlan pl, Grid g, const __grid_constant__ CUtensorMap map, const int* te, FieldsW out, const cd* add,
                unsigned* flags) {
  grid_wait();
  extern __shared__ __align__(128) unsigned char sm_raw[];
  __shared__ FxShared sh;
  cfx* a = reinterpret_cast<cfx*>(sm_raw);
  const int pz = g.pz, h = g.nx / 2, n2 = g.nz / 2, H = pl.rows_t, tpt = pl.tpt;
  const int kx0 = blockIdx.x * COLS, j = blockIdx.y, f = blockIdx.z;
  const int c = threadIdx.x % COLS, tt = threadIdx.x / COLS, kx = kx0 + c;
  unsigned long long* bar = reinterpret_cast<unsigned long long*>(sm_raw + (size_t)pz * COLS * sizeof(cfx));
  if (threadIdx.x == 0) mbar_init(bar);
  __syncthreads();
  if (threadIdx.x == 0) {
    mbar_expect_tx(bar, (unsigned)(pz * COLS * sizeof(cfx)));
    for (int r = 0; r < pz; r += H)
      if (LMVD_IN((r + H) * COLS - 1, pz * COLS)) tma_load_3d(a + (size_t)r * COLS, &map, 2 * kx0, r, f * g.ny + j, bar);
  }
  const bool first4 = EPT == 12 && pl.first4;
  int E[EPT], emin = INT_MAX;
  const int* ej = te + ((size_t)f * g.ny + j) * (pz / 2);
#pragma unroll
  for (int u = 0; u < EPT; ++u) {
    const int i = fx_point(u, first4, tt, tpt, pz >> 2);
    E[u] = LMVD_IN(i, pz) ? ej[i >> 1] : kFxZero;
    emin = min(emin, E[u]);
  }
  if (!mbar_wait_bounded(bar, flags)) return;
  cfx v[EPT];
  float mag = 0.f, big = 0.f;
#pragma unroll
  for (int u = 0; u < EPT; ++u) {
    const int i = fx_point(u, first4, tt, tpt, pz >> 2);
    v[u] = LMVD_IN(i, pz) ? a[i * COLS + c] : cfx{0, 0};
    const float z = fx_mag(fx_mag_hi(v[u]), E[u]);
    mag += z;
    big = fmaxf(big, z);
  }
  constexpr bool GUARD = COLS == 2;  // (as in the inverse z-pass)
  int xe, e;
  const int gz = pl.red_g;
  const int k = fx_scale_t<GUARD>(mag, big, emin, sh, c, tpt / gz, COLS, gz, COLS, tt, xe, e, [&](int s, float& b) {
    float m = b = 0.f;
#pragma unroll
    for (int u = 0; u < EPT; ++u) {
      const float z = fx_mag(fx_mag_hi(v[u]), E[u] += s);
      m += z;
      b = fmaxf(b, z);
    }
    return m;
  });
#pragma unroll
  for (int u = 0; u < EPT; ++u) v[u] = fx_align(v[u], E[u] - k - e);
  fx_run<-1, EPT, COLS, GUARD>(v, a + c, pl, first4, tt, e);
  fx_last<-1, EPT, COLS, GUARD>(a + c, pl, tt, v);
  if (kx > h) return;
  cd* dst = pick(out.p, f) + (size_t)j * g.M + kx;
  // outputs q < NP (kz = tt + q tpt) and q >= 2 NP (kz = i - n2, row n2 + i; i = 0 is the Nyquist row)
  constexpr int NP = EPT / 3;
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    const int b = tt + q * tpt;
    if (!LMVD_IN((size_t)(n2 + b) * g.nxh + kx, g.M)) continue;
    cd p = pl.scale_d * fx_result(v[q], k, xe), m = pl.scale_d * fx_result(v[2 * NP + q], k, xe);
    if (kx == h) p = m = mk(0, 0);
    if (b == 0) m = mk(0, 0);
    const size_t op = (size_t)b * g.nxh, om = (size_t)(n2 + b) * g.nxh;
    if (add) {
      const cd* q0 = add + (size_t)j * g.M + kx;
      if (kx < h) p = p + q0[op];
      if (kx < h && b != 0) m = m + q0[om];
    }
    dst[op] = p;
    dst[om] = m;
  }
}

// ---------------------------------------------------------------- host side
// Radix order 4s, 2s, 3s, then the last stage's 12 (6 when n has a single factor 2): the sub-length L is a power of
// two in every radix-4/2 stage (mask arithmetic). 12 (6) elements per thread; at most cta threads per
// CTA (so n <= 12 cta); one shared buffer of batch transforms with leading dimension n + pad.
static bool make_plan(int n, int cta, FFTPlan& p, int ept = 0) {
  p.n = n;
  p.nst = 0;
  p.ept = ept ? ept : (n % 12 == 0) ? 12 : ((n % 6 == 0) ? 6 : 0);
  if (!p.ept || n % p.ept) return false;
  p.tpt = n / p.ept;
  p.code = 0;
  int m = p.tpt;
  for (int r : {4, 2, 3})  // (6 elements per thread hold no radix-4 butterflies)
    for (; m % r == 0 && !(r == 4 && p.ept == 6); m /= r) p.code |= (unsigned)(r == 4 ? 0 : (r == 2 ? 1 : 2)) << (2 * p.nst++);
  if (m != 1 || p.nst > 15) return false;
  ++p.nst;  // the last stage, radix ept
  p.first4 = p.ept == 12 && p.tpt % 4 == 0;
  if (p.tpt > cta) return false;
  for (p.red_g = 1; p.tpt % (2 * p.red_g) == 0 && p.red_g < (cta == FFT_CTA_Z ? 8 : 32);) p.red_g *= 2;
  const long double s3 = sqrtl(3.0L) / 2.0L;
  fx_limbs(s3, p.s3.x, p.s3.y);
  p.batch = cta / p.tpt;
  p.pad = 1;  // the x-passes: leading dimension n + 1 keeps the transforms of a batch in different banks
  if (cta == FFT_CTA_Z) {
    // the z-passes: 4 interleaved columns per CTA (2 when 4 transforms of n do not fit in cta threads; the
    // 6-element plans exist only for 4), and tile copies whose rows divide their range and start on 128-byte
    // boundaries in shared memory (rows x batch x 16 bytes a multiple of 128)
    p.batch = 4 * p.tpt <= cta ? 4 : (p.ept == 12 && 2 * p.tpt <= cta ? 2 : 0);
    if (!p.batch || n % 3) return false;
    p.pad = 0;
    auto rows = [&](int total) {
      for (int r = total < 256 ? total : 256; r > 0; --r)
        if (total % r == 0 && (r * p.batch) % 8 == 0) return r;
      return 0;
    };
    p.rows_in = rows(n / 3);  // nz / 2 = pz / 3
    p.rows_t = rows(n);
    if (!p.rows_in || !p.rows_t) return false;
  }
  return true;
}

// A launch with few transforms is a chain of one thread's instructions (about 250 per element, one or two warps per
// SM), so it takes the plan with 6 elements per thread where there is one (twice the threads, radix-2 stages for radix-4
// ones). 32 x 33 x 32, per substage: the four passes 0.128 / 0.167 / 0.150 / 0.143 -> 0.119 / 0.141 / 0.137 / 0.133 ms,
// 72 x 61 x 48: 0.187 / 0.244 / 0.220 / 0.200 -> 0.155 / 0.218 / 0.184 / 0.169. The line: fewer than 384 threads per SM
// with 12 elements each (128: 72 x 61 x 48 loses 4%, 512: 64 x 65 x 64 loses 1%).
constexpr double FFT_SMALL_THREADS = 152 * 384;
static const FFTPlan& pick_plan(const FFTPlan& full, const FFTPlan& small, double transforms) {
  return small.n && transforms * full.tpt < FFT_SMALL_THREADS ? small : full;
}
static void make_small_plan(const FFTPlan& full, int cta, FFTPlan& p) {
  if (full.ept != 12 || !make_plan(full.n, cta, p, 6)) p.n = 0;
  p.tw = full.tw;
  p.scale_d = full.scale_d;
}

// a pass's buffer is followed by its mbarrier (the z-passes' and the inverse x-pass's copies)
static size_t smem_bytes(const FFTPlan& p) { return (size_t)p.batch * (p.n + p.pad) * sizeof(cfx) + 16; }

// Tensor maps for the z-passes' tile copies. cuTensorMapEncodeTiled is a driver function; the runtime hands
// out its address, so the library needs no link to the driver library.
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_tiled() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

// A map over planes x rows x cols 16-byte elements at base (row-major, contiguous), addressed in doubles:
// boxes of (2 bcols doubles, brows rows, 1 plane); out-of-range parts of a box read as zero.
static bool tile_map(CUtensorMap* m, const void* base, size_t cols, size_t rows, size_t planes, int bcols, int brows) {
  const EncodeTiledFn fn = encode_tiled();
  if (!fn || !base || ((uintptr_t)base & 15)) return false;
  const cuuint64_t dims[3] = {2 * (cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)planes};
  const cuuint64_t strides[2] = {16 * (cuuint64_t)cols, 16 * (cuuint64_t)cols * rows};
  const cuuint32_t box[3] = {(cuuint32_t)(2 * bcols), (cuuint32_t)brows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 3, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// the instantiation of an x-pass a plan runs (6 elements per thread: at most 768 points)
#define FX_X_KERNEL(K, P) ((P).ept == 6 ? K<6, false> : (P).n > kFxGuardLength ? K<12, true> : K<12, false>)
static unsigned threads(const FFTPlan& p) { return (unsigned)(p.batch * p.tpt); }

// Every pass may take up to kFftSmemMax bytes of dynamic shared memory. The limit is a property of the
// kernel, shared by all contexts and the allocation-free path in the process: setting it to one grid's size
// would break the launches of another context with a larger grid, so it is set once, to the maximum a plan
// may ask for (fft_prepare rejects larger plans).
constexpr int kFftSmemMax = 200 * 1024;

template <class K>
static bool smem_limit(K kernel) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFftSmemMax) == cudaSuccess;
}
template <int EPT, int COLS>
static bool smem_limit_z() {
  return smem_limit(k_fft_z_inv<cd, EPT, COLS>) && smem_limit(k_fft_z_inv<cdf, EPT, COLS>) &&
         smem_limit(k_fft_z_fwd<EPT, COLS>);
}
template <int EPT, bool GUARD>
static bool smem_limit_x() {
  return smem_limit(k_fft_x_inv<EPT, GUARD>) && smem_limit(k_fft_x_inv_mul<EPT, GUARD>) &&
         smem_limit(k_fft_x_fwd<EPT, GUARD>) && smem_limit(k_fft_x_fwd_dot3<EPT, GUARD>);
}
static int set_smem() {
  return smem_limit_z<12, 4>() && smem_limit_z<12, 2>() && smem_limit_z<6, 4>() && smem_limit_x<12, false>() &&
                 smem_limit_x<12, true>() && smem_limit_x<6, false>()
             ? LMVD_OK
             : LMVD_ERR_CUDA;
}

int fft_prepare(Ctx& c) {
  if (!make_plan(c.g.px, FFT_CTA_X, c.fx) || !make_plan(c.g.pz, FFT_CTA_Z, c.fz)) return LMVD_ERR_UNSUPPORTED;
  const long double scale = 1.0L / ((long double)c.g.px * (long double)c.g.pz);
  const long double pi = 3.141592653589793238462643383279502884L;
  for (FFTPlan* p : {&c.fx, &c.fz}) {
    if (smem_bytes(*p) > kFftSmemMax) return LMVD_ERR_UNSUPPORTED;
    std::vector<int4> tw(p->n);
    for (int m = 0; m < p->n; ++m) {
      const long double ang = 2.0L * pi * (long double)m / (long double)p->n;
      fx_limbs(cosl(ang), tw[m].x, tw[m].y);
      fx_limbs(sinl(ang), tw[m].z, tw[m].w);
    }
    int4* d = nullptr;
    if (cudaMalloc(&d, sizeof(int4) * p->n) != cudaSuccess) return LMVD_ERR_OOM;
    c.small_allocs.push_back(d);
    c.small_bytes += sizeof(int4) * p->n;
    if (cudaMemcpy(d, tw.data(), sizeof(int4) * p->n, cudaMemcpyHostToDevice) != cudaSuccess) return LMVD_ERR_CUDA;
    p->tw = d;
    p->scale_d = (double)(scale / 2);  // used by the forward z-pass (see the file head)
  }
  make_small_plan(c.fx, FFT_CTA_X, c.fx6);
  make_small_plan(c.fz, FFT_CTA_Z, c.fz6);
  return set_smem();
}

static inline unsigned cdiv(unsigned a, unsigned b) { return (a + b - 1) / b; }
// conventional algorithmic flop count of one complex transform of length n: 5 n log2 n
static inline double fft_flops(double n) { return 5.0 * n * std::log2(n); }

// A tensor map that could not be encoded: the context's status becomes LMVD_ERR_CUDA (unless one is set).
static void map_failed(Ctx& c) {
  if (c.status == LMVD_OK) c.status = LMVD_ERR_CUDA;
}

// The inverse z-pass of n fields (spectral inputs fi) into T, and the forward z-pass of n fields of T into
// fo: tensor maps for their tile copies, then one launch of the instantiation the plan selects.
template <class RAW>
static void z_inv_launch(Ctx& c, const FieldsC& fi, int n, size_t tstride, double fl, double by) {
  const Grid& g = c.g;
  const FFTPlan& p = pick_plan(c.fz, c.fz6, (double)(g.nx / 2) * g.ny * n);
  ZMaps maps;
  for (int f = 0; f < n; ++f)
    if (!tile_map(&maps.m[f], fi.p[f], g.nxh, g.nz, g.ny, p.batch, p.rows_in)) {
      map_failed(c);
      return;
    }
  const dim3 gz(cdiv(g.nx / 2, p.batch), g.ny, n);
  if (p.ept == 12 && p.batch == 4)
    LMVD_LAUNCH(c, KC_FFT_Z_INV, fl, by, (k_fft_z_inv<RAW, 12, 4>), gz, threads(p), smem_bytes(p), p, g, maps,
                c.tbuf, tstride, c.texp, c.dflags);
  else if (p.ept == 12)
    LMVD_LAUNCH(c, KC_FFT_Z_INV, fl, by, (k_fft_z_inv<RAW, 12, 2>), gz, threads(p), smem_bytes(p), p, g, maps,
                c.tbuf, tstride, c.texp, c.dflags);
  else
    LMVD_LAUNCH(c, KC_FFT_Z_INV, fl, by, (k_fft_z_inv<RAW, 6, 4>), gz, threads(p), smem_bytes(p), p, g, maps,
                c.tbuf, tstride, c.texp, c.dflags);
}

static void z_fwd_launch(Ctx& c, int n, const FieldsW& fo, double fl, double by, const cd* add = nullptr) {
  const Grid& g = c.g;
  const FFTPlan& p = pick_plan(c.fz, c.fz6, (double)(g.nx / 2 + 1) * g.ny * n);
  CUtensorMap map;
  if (!tile_map(&map, c.tbuf, g.nx / 2, g.pz, (size_t)n * g.ny, p.batch, p.rows_t)) {
    map_failed(c);
    return;
  }
  const dim3 gz(cdiv(g.nx / 2 + 1, p.batch), g.ny, n);
  if (p.ept == 12 && p.batch == 4)
    LMVD_LAUNCH(c, KC_FFT_Z_FWD, fl, by, (k_fft_z_fwd<12, 4>), gz, threads(p), smem_bytes(p), p, g, map, c.texp, fo, add,
                c.dflags);
  else if (p.ept == 12)
    LMVD_LAUNCH(c, KC_FFT_Z_FWD, fl, by, (k_fft_z_fwd<12, 2>), gz, threads(p), smem_bytes(p), p, g, map, c.texp, fo, add,
                c.dflags);
  else
    LMVD_LAUNCH(c, KC_FFT_Z_FWD, fl, by, (k_fft_z_fwd<6, 4>), gz, threads(p), smem_bytes(p), p, g, map, c.texp, fo, add,
                c.dflags);
}

// df_in: the spectral inputs are double-float pairs (the precision path's evaluations)
static void inverse(Ctx& c, cd* const* in, double* const* out, int nf, bool df_in, const double* wmul = nullptr) {
  const Grid& g = c.g;
  const size_t tstride = (size_t)g.ny * g.pz * (g.nx / 2);
  for (int f0 = 0; f0 < nf; f0 += c.tbuf_n) {
    const int n = nf - f0 < c.tbuf_n ? nf - f0 : c.tbuf_n;
    FieldsC fi{};
    FieldsRW fo{};
    for (int f = 0; f < n; ++f) {
      fi.p[f] = in[f0 + f];
      fo.p[f] = out[f0 + f];
    }
    const double h = g.nx / 2, ny = g.ny, pz = g.pz, px = g.px;
    const double zfl = n * ny * h * fft_flops(pz), zby = n * ny * h * 16.0 * ((g.nz - 1) + pz);
    if (df_in) z_inv_launch<cdf>(c, fi, n, tstride, zfl, zby);
    else z_inv_launch<cd>(c, fi, n, tstride, zfl, zby);
    const FFTPlan& p = pick_plan(c.fx, c.fx6, 0.5 * g.pz * g.ny * n);
    dim3 gx(cdiv(cdiv(g.pz, 2), p.batch), g.ny, n);
    const double xfl = n * ny * ((g.pz + 1) / 2) * fft_flops(px), xby = n * ny * pz * (16.0 * h + 8.0 * px);
    if (wmul)  // the product with w in the epilogue: one more physical field read, one multiply per point
      LMVD_LAUNCH(c, KC_FFT_X_INV, xfl + n * ny * pz * px, xby + n * ny * pz * 8.0 * px, FX_X_KERNEL(k_fft_x_inv_mul, p), gx,
                  threads(p), smem_bytes(p), p, g, c.tbuf, tstride, c.texp, fo, wmul, c.dflags);
    else
      LMVD_LAUNCH(c, KC_FFT_X_INV, xfl, xby, FX_X_KERNEL(k_fft_x_inv, p), gx, threads(p), smem_bytes(p), p, g, c.tbuf,
                  tstride, c.texp, fo, c.dflags);
  }
}

void fft_forward(Ctx& c, double* const* in, cd* const* out, int nf) {
  const Grid& g = c.g;
  const size_t tstride = (size_t)g.ny * g.pz * (g.nx / 2);
  for (int f0 = 0; f0 < nf; f0 += c.tbuf_n) {
    const int n = nf - f0 < c.tbuf_n ? nf - f0 : c.tbuf_n;
    FieldsRC fi{};
    FieldsW fo{};
    for (int f = 0; f < n; ++f) {
      fi.p[f] = in[f0 + f];
      fo.p[f] = out[f0 + f];
    }
    const double h = g.nx / 2, ny = g.ny, pz = g.pz, px = g.px;
    const FFTPlan& p = pick_plan(c.fx, c.fx6, 0.5 * g.pz * g.ny * n);
    dim3 gx(cdiv(cdiv(g.pz, 2), p.batch), g.ny, n);
    LMVD_LAUNCH(c, KC_FFT_X_FWD, n * ny * ((g.pz + 1) / 2) * fft_flops(px), n * ny * pz * (16.0 * h + 8.0 * px),
                FX_X_KERNEL(k_fft_x_fwd, p), gx, threads(p), smem_bytes(p), p, g, fi, c.tbuf, tstride, c.texp);
    z_fwd_launch(c, n, fo, n * ny * h * fft_flops(pz), n * ny * 16.0 * (pz * h + (double)g.nz * g.nxh));
  }
}

// add + the forward transform of -(w1 m1 + w2 m2 + w3 m3), formed in the x-pass prologue, into one spectral field
void fft_forward_dot3(Ctx& c, const double* const* w, const double* const* m, const cd* add, cd* out) {
  const Grid& g = c.g;
  const size_t tstride = (size_t)g.ny * g.pz * (g.nx / 2);
  Dot3 d{};
  for (int f = 0; f < 3; ++f) {
    d.w[f] = w[f];
    d.m[f] = m[f];
  }
  FieldsW fo{};
  fo.p[0] = out;
  const double h = g.nx / 2, ny = g.ny, pz = g.pz, px = g.px;
  const FFTPlan& p = pick_plan(c.fx, c.fx6, 0.5 * g.pz * g.ny * 1);
  const dim3 gx(cdiv(cdiv(g.pz, 2), p.batch), g.ny, 1);
  const double xfl = ny * ((g.pz + 1) / 2) * fft_flops(px) + 6.0 * ny * pz * px, xby = ny * pz * (16.0 * h + 48.0 * px);
  LMVD_LAUNCH(c, KC_FFT_X_FWD, xfl, xby, FX_X_KERNEL(k_fft_x_fwd_dot3, p), gx, threads(p), smem_bytes(p), p, g, c.tbuf,
              tstride, c.texp, d);
  z_fwd_launch(c, 1, fo, ny * h * fft_flops(pz), ny * 16.0 * (pz * h + 2.0 * g.nz * g.nxh), add);
}

// the substage's inputs come from the double-float evaluations in the precision path
void fft_inverse(Ctx& c, cd* const* in, double* const* out, int nf) { inverse(c, in, out, nf, c.cfg.precision == 1); }
void fft_inverse_d(Ctx& c, cd* const* in, double* const* out, int nf) { inverse(c, in, out, nf, false); }
void fft_inverse_mul(Ctx& c, cd* in, double* out, const double* w, bool df_in) {
  cd* i[1] = {in};
  double* o[1] = {out};
  inverse(c, i, o, 1, df_in, w);
}

// The bounded wait of the z-passes, on its own (lmvd_tile_wait_probe): one CTA expects 128 + extra bytes on
// an mbarrier and copies 128 of them; with extra > 0 the phase never completes and the wait gives up.
__global__ void k_tile_wait_probe(const double* src, int extra, unsigned* status) {
  __shared__ __align__(128) double buf[16];
  __shared__ __align__(8) unsigned long long bar;
  if (threadIdx.x == 0) mbar_init(&bar);
  __syncthreads();
  if (threadIdx.x == 0) {
    mbar_expect_tx(&bar, 128u + (unsigned)extra);
    bulk_load(buf, src, 128u, &bar);
  }
  if (!mbar_wait_bounded(&bar, status)) return;
  if (threadIdx.x < 16 && buf[threadIdx.x] != src[threadIdx.x]) atomicOr(status, 8u);
}

}  // namespace lmvd

// ====================================================================== allocation-free inverse transform
// lmvd_inverse_transform_noalloc: the same synthesis as lmvd_inverse_transform, for callers that cannot
// allocate device memory (no context exists, so nothing of lmvd_create is needed). Its only working
// memory is the file-scope array below, which the CUDA module reserves on every device that loads the
// library and keeps until the process exits. All calls on a device share it: the twiddle tables and
// the intermediate array are rewritten by each call before they are read (nothing has to start at
// zero), and calls whose work overlaps on the GPU (other streams, other host threads) race on it.
namespace lmvd {
namespace {

constexpr size_t kNoAllocScratchBytes = size_t(32) << 20;  // 32 MiB per device
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mu;
void* g_noalloc_ptr[kNoAllocMaxDevices] = {};
// exponents of T: one per kx column and plane, for the shortest columns (pz = 6) that fill the scratch
static __device__ int g_noalloc_exp[kNoAllocScratchBytes / sizeof(cd) / 6];
int* g_noalloc_exp_ptr[kNoAllocMaxDevices] = {};

// twiddle table tw[m] = limbs of (cos 2 pi m / n, sin 2 pi m / n) computed on the device
__global__ void k_twiddles(int4* tx, int nx, int4* tz, int nz) {
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < nx + nz; m += gridDim.x * blockDim.x) {
    const int i = m < nx ? m : m - nx, n = m < nx ? nx : nz;
    double s, c;
    sincospi(2.0 * (double)i / (double)n, &s, &c);
    int4 w;
    fx_limbs(c, w.x, w.y);
    fx_limbs(s, w.z, w.w);
    (m < nx ? tx : tz)[i] = w;
  }
}

// Once per device, with that device current: the device address of the scratch array (in host code
// the array's name is only a stand-in) and the shared-memory limits of the two kernels.
int noalloc_setup(int dev, void** ptr, int** te) {
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (g_noalloc_ptr[dev]) {
    *ptr = g_noalloc_ptr[dev];
    *te = g_noalloc_exp_ptr[dev];
    return LMVD_OK;
  }
  void* p = nullptr;
  if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return LMVD_ERR_CUDA;
  if (set_smem())
    return LMVD_ERR_CUDA;
  void* e = nullptr;
  if (cudaGetSymbolAddress(&e, g_noalloc_exp) != cudaSuccess || !e) return LMVD_ERR_CUDA;
  *te = g_noalloc_exp_ptr[dev] = (int*)e;
  g_noalloc_ptr[dev] = p;
  *ptr = p;
  return LMVD_OK;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

}  // namespace lmvd

extern "C" int lmvd_inverse_transform_noalloc(int nx, int ny, int nz, const void* spec, double* phys, int nfields,
                                              void* cuda_stream) {
  using namespace lmvd;
  if (!spec || !phys || nfields < 0 || ny < 1 || nx < 4 || nz < 4 || (nx % 2) || (nz % 2) || ((uintptr_t)spec & 15))
    return LMVD_ERR_INVALID_ARG;
  if (ny > 65535) return LMVD_ERR_INVALID_ARG;  // ny is the grid's y-dimension (at most 65535 CTAs)
  Grid g{};
  g.nx = nx;
  g.ny = ny;
  g.nz = nz;
  g.nxh = nx / 2 + 1;
  g.px = 3 * nx / 2;
  g.pz = 3 * nz / 2;
  g.M = (size_t)nz * g.nxh;
  g.P = (size_t)g.px * g.pz;
  FFTPlan fx, fz;
  if (!make_plan(g.px, FFT_CTA_X, fx) || !make_plan(g.pz, FFT_CTA_Z, fz)) return LMVD_ERR_UNSUPPORTED;
  for (FFTPlan* p : {&fx, &fz})
    if (smem_bytes(*p) > kFftSmemMax) return LMVD_ERR_UNSUPPORTED;
  // scratch layout: x twiddles | z twiddles | one field's intermediate T[ny][pz][nx/2]
  const size_t off_tz = align256(sizeof(int4) * g.px);
  const size_t off_tb = off_tz + align256(sizeof(int4) * g.pz);
  const size_t tbytes = sizeof(cfx) * (size_t)ny * g.pz * (nx / 2);
  if (off_tb + tbytes > kNoAllocScratchBytes) return LMVD_ERR_INVALID_ARG;  // grid too large for the scratch
  // a launch error left pending on this host thread by earlier work is not this call's to report
  (void)cudaGetLastError();
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoAllocMaxDevices) return LMVD_ERR_CUDA;
  void* base = nullptr;
  int* te = nullptr;
  int err = noalloc_setup(dev, &base, &te);
  if (err) return err;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  char* sb = (char*)base;
  fx.tw = (const int4*)sb;
  fz.tw = (const int4*)(sb + off_tz);
  cfx* T = (cfx*)(sb + off_tb);
  k_twiddles<<<cdiv(g.px + g.pz, 128), 128, 0, st>>>((int4*)sb, g.px, (int4*)(sb + off_tz), g.pz);
  if (cudaGetLastError() != cudaSuccess) return LMVD_ERR_CUDA;
  const size_t S = (size_t)ny * g.M, P = (size_t)ny * g.P;
  FFTPlan fx6, fz6;
  make_small_plan(fx, FFT_CTA_X, fx6);
  make_small_plan(fz, FFT_CTA_Z, fz6);
  fx = pick_plan(fx, fx6, 0.5 * g.pz * ny);
  fz = pick_plan(fz, fz6, (double)(nx / 2) * ny);
  for (int f = 0; f < nfields; ++f) {
    FieldsC fi{};
    FieldsRW fo{};
    fi.p[0] = (const cd*)spec + (size_t)f * S;
    fo.p[0] = phys + (size_t)f * P;
    ZMaps maps;
    if (!tile_map(&maps.m[0], fi.p[0], g.nxh, nz, ny, fz.batch, fz.rows_in)) return LMVD_ERR_CUDA;
    dim3 gz(cdiv(nx / 2, fz.batch), ny, 1);
    // an ordinary launch where the twiddles, which the kernel ahead may have written, come through the read-only path
    if (fz.ept == 12 && fz.batch == 4) k_fft_z_inv<cd, 12, 4><<<gz, threads(fz), smem_bytes(fz), st>>>(fz, g, maps, T, 0, te, nullptr);
    else if (fz.ept == 12) k_fft_z_inv<cd, 12, 2><<<gz, threads(fz), smem_bytes(fz), st>>>(fz, g, maps, T, 0, te, nullptr);
    else launch_next(k_fft_z_inv<cd, 6, 4>, gz, threads(fz), smem_bytes(fz), st, fz, g, maps, T, 0, te, nullptr);
    if (cudaGetLastError() != cudaSuccess) return LMVD_ERR_CUDA;
    dim3 gx(cdiv(cdiv(g.pz, 2), fx.batch), ny, 1);
    launch_next(FX_X_KERNEL(k_fft_x_inv, fx), gx, threads(fx), smem_bytes(fx), st, fx, g, T, 0, te, fo, nullptr);
    if (cudaGetLastError() != cudaSuccess) return LMVD_ERR_CUDA;
  }
  return LMVD_OK;
}

extern "C" int lmvd_tile_wait_probe(const double* src, int extra_bytes, unsigned* status, void* cuda_stream) {
  using namespace lmvd;
  if (!src || !status || ((uintptr_t)src & 15) || extra_bytes < 0 || extra_bytes > 1024 || (extra_bytes & 15))
    return LMVD_ERR_INVALID_ARG;
  (void)cudaGetLastError();
  k_tile_wait_probe<<<1, 32, 0, (cudaStream_t)cuda_stream>>>(src, extra_bytes, status);
  return cudaGetLastError() == cudaSuccess ? LMVD_OK : LMVD_ERR_CUDA;
}
