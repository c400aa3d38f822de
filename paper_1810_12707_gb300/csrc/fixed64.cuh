// fixed64.cuh -- the arithmetic of the FP64 transforms: a pencil (one transform's N complex values)
// is carried as 64-bit fixed-point numbers with one common exponent.
//
// GB300 executes 1.7 FP64 fused multiply-adds per clock and SM, but 116 32-bit integer additions
// and 60 32-bit integer multiplications (measured); an FP64 radix-8 butterfly costs 72 FP64
// instructions, about 5800 cycles of a scheduler's FP64 pipe per warp.  A discrete Fourier
// transform is linear, so its butterflies need no exponents: in fixed point an addition is two
// integer instructions and exact, a real product with a twiddle three 32 x 32 -> 64-bit
// multiplications, and a butterfly about 700 issue cycles.
//
// Accuracy.  The common exponent comes from the pencil itself: the first stage's butterfly sums
// are bounded by A, the largest sum of |re| + |im| over one butterfly's inputs, the transform by
// T, the sum over the whole pencil.  The inputs are converted so that A fills 60 bits, and the
// stages after the first shift right only as far as T / A demands (the shift rides on the
// twiddles), so the unit of the fixed-point numbers is at most 2^-59 T.  T is at most sqrt(2 N) of the
// result's RMS (Parseval; all magnitudes equal): the unit is at most 2^-56 of the RMS at 32 points,
// 2^-54 at 512, 2^-53.5 at 1024, and far less for spectra with a few large modes; an FP64
// butterfly rounds every value of every stage at 2^-53.  Values more than 2^60 below the largest
// first-stage sum round to zero; in FP64 they are lost in the same butterflies' rounding errors.
//
// A pencil with a NaN or an infinity transforms to NaN everywhere.  The conversions that every pencil
// takes hold for largest magnitudes from 2^-959 to 2^977; any other takes the paths of FxScale::bad,
// which hold over the whole range of doubles (but a pencil below 2^-1042 altogether is taken as zeros).
#pragma once

#include <stdint.h>
#include <string.h>

#include "mhd_internal.h"

namespace mhd {

#ifdef __CUDACC__
#define FX_FN __host__ __device__ __forceinline__
#else
#define FX_FN inline
#endif

// Complex fixed-point value (16 bytes, in place of a cplx64 in shared memory).
struct alignas(16) cfx {
  using value_type = int64_t;
  int64_t re, im;
};

// Twiddles are TwFx (mhd_internal.h).  A table holds kFxShifts copies, copy s scaled by 2^-s: a
// stage that has to shift its inputs right by s reads copy s.

// ---- 32-bit pieces ----
FX_FN int64_t fx_mad(int32_t a, int32_t b, int64_t c) {
#ifdef __CUDA_ARCH__
  int64_t r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (int64_t)a * b + c;
#endif
}
// Shifts by any amount (32 and more give 0; the funnel shift stops at 32).
FX_FN uint32_t fx_shr(uint32_t x, uint32_t s) {
#ifdef __CUDA_ARCH__
  uint32_t r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(s));
  return r;
#else
  return s >= 32 ? 0u : x >> s;
#endif
}
FX_FN uint32_t fx_shl(uint32_t x, uint32_t s) {
#ifdef __CUDA_ARCH__
  uint32_t r;
  asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(s));
  return r;
#else
  return s >= 32 ? 0u : x << s;
#endif
}
FX_FN uint32_t fx_funnel_r(uint32_t lo, uint32_t hi, uint32_t s) {  // low word of (hi:lo) >> min(s, 32)
#ifdef __CUDA_ARCH__
  return __funnelshift_rc(lo, hi, s);
#else
  return s >= 32 ? hi : (uint32_t)((((uint64_t)hi << 32) | lo) >> s);
#endif
}
FX_FN uint32_t fx_funnel_l(uint32_t lo, uint32_t hi, uint32_t s) {  // high word of (hi:lo) << min(s, 32)
#ifdef __CUDA_ARCH__
  return __funnelshift_lc(lo, hi, s);
#else
  return s >= 32 ? lo : (uint32_t)(((((uint64_t)hi << 32) | lo) << s) >> 32);
#endif
}
FX_FN int fx_clz(uint32_t x) {
#ifdef __CUDA_ARCH__
  return __clz((int)x);
#else
  return x ? __builtin_clz(x) : 32;
#endif
}
FX_FN int64_t fx_join(uint32_t hi, uint32_t lo) { return (int64_t)(((uint64_t)hi << 32) | lo); }
FX_FN uint32_t fx_hi(double x) {
  uint64_t b;
  memcpy(&b, &x, 8);
  return (uint32_t)(b >> 32);
}
FX_FN uint32_t fx_lo(double x) {
  uint64_t b;
  memcpy(&b, &x, 8);
  return (uint32_t)b;
}
FX_FN double fx_double(uint32_t hi, uint32_t lo) {
  const uint64_t b = ((uint64_t)hi << 32) | lo;
  double x;
  memcpy(&x, &b, 8);
  return x;
}

// ---- the pencil's exponent ----
// Magnitudes are measured in units of 2^(M - 1043), M the largest biased exponent among the values
// seen: a value of biased exponent e is below fx_size(its high word, M) of them.
FX_FN uint32_t fx_exp(uint32_t hi) { return (hi >> 20) & 0x7ffu; }
FX_FN uint32_t fx_size(uint32_t hi, uint32_t m) {
  return fx_shr((hi & 0xfffffu) | 0x100000u, m - fx_exp(hi)) + 1u;
}
// The biased exponent of the largest of some magnitudes, from the largest of their high words: 1 if
// they are all subnormal, 0 if all zero.
FX_FN uint32_t fx_max_exp(uint32_t hi) {
  const uint32_t e = hi >> 20, any = hi < 1u ? hi : 1u;
  return e > any ? e : any;
}
// What some of a pencil's values say: the largest biased exponent m, the largest first-stage sum a
// and the whole sum t / 8, both in units of 2^(m - 1043).
struct FxPart {
  uint32_t m, a, t;
};
FX_FN FxPart fx_merge(FxPart x, FxPart y) {
  const uint32_t m = x.m > y.m ? x.m : y.m;
  const uint32_t xa = fx_shr(x.a, m - x.m) + 1u, ya = fx_shr(y.a, m - y.m) + 1u;
  return FxPart{m, xa > ya ? xa : ya, fx_shr(x.t, m - x.m) + fx_shr(y.t, m - y.m) + 2u};
}
// A value of biased exponent e is its 63-bit significand (leading one at bit 62) >> (ek - e) in
// fixed point, so a fixed-point x stands for x 2^(ek - 1085); `shift` is what the later stages
// have to shift right in all, and x 2^(ek + shift - 1085) what their results stand for.
struct FxScale {
  uint32_t ek;
  int shift;
  bool bad;
};
FX_FN FxScale fx_scale(FxPart p, int log2_groups) {
  int ca = 11 - fx_clz(p.a - 1u);  // a <= 2^(21 + ca)
  int ct = 14 - fx_clz(p.t - 1u);  // t <= 2^(18 + ct)
  if (ca < 0) ca = 0;
  if (ct < ca) ct = ca;
  int sh = ct - ca;
  if (sh > log2_groups) sh = log2_groups;  // T is at most (groups) A
  FxScale s;
  s.ek = p.m < 64u ? 200u : p.m + 3u + (uint32_t)ca;  // A < 2^60
  s.shift = sh;
  s.bad = p.m >= 2000u;
  return s;
}
// The scale of any pencil.  `bad`: outside the range of the conversions that the transforms use (and
// not all zeros, which those handle).  Such a pencil's `ek` is moved by 256 towards the middle: its
// values are converted by fx_from_any with fx_bad_ek, its results as ever and then multiplied by
// fx_bad_factor, 2^-256, 2^256 or NaN.  Both sit behind branches that a whole group takes or not, the
// multiplications in loops: as predicated instructions in line they held the FP64 pipe in every pencil
// (256^3 FP64 run 140 -> 159 ms; so, 138 ms).
FX_FN FxScale fx_scale_any(FxPart p, int log2_groups) {
  const bool low = p.m - 1u < 63u, out = low || p.m >= 2000u;
  FxPart q = p;
  if (out) q.m = low ? p.m + 256u : p.m == 2047u ? 4096u : p.m - 256u;
  FxScale s = fx_scale(q, log2_groups);
  s.bad = out;
  return s;
}
FX_FN uint32_t fx_bad_ek(uint32_t ek) { return ek < 1024u ? ek - 256u : ek + 256u; }
FX_FN double fx_bad_factor(uint32_t ek) {
  return fx_double(ek >= 4096u ? 0x7ff80000u : ek < 1024u ? 0x2ff00000u : 0x4ff00000u, 0u);
}

// ---- conversions ----
FX_FN int64_t fx_from_double(uint32_t hi, uint32_t lo, uint32_t ek) {
  const uint32_t s = ek - fx_exp(hi);
  const uint32_t mh = (hi & 0xfffffu) | 0x100000u;
  const uint32_t h = (mh << 10) | (lo >> 22), l = lo << 10;
  const uint32_t s2 = s > 32u ? s - 32u : 0u;
  const int64_t v = fx_join(fx_shr(h, s), fx_shr(fx_funnel_r(l, h, s), s2));
  return (int32_t)hi < 0 ? -v : v;
}
// The same for every exponent: subnormal numbers have no leading one, and zero is zero.
FX_FN int64_t fx_from_any(uint32_t hi, uint32_t lo, uint32_t ek) {
  const uint32_t e = fx_exp(hi), s = ek - (e ? e : 1u);
  const uint32_t mh = (hi & 0xfffffu) | (e ? 0x100000u : 0u);
  const uint64_t m = (((uint64_t)mh << 32) | lo) << 10;
  const int64_t v = s > 63u ? 0 : (int64_t)(m >> s);
  return (int32_t)hi < 0 ? -v : v;
}
// v 2^(be - 1086), rounded to nearest (`be`: the biased exponent of a value whose leading one is
// at bit 63).
FX_FN double fx_to_double(int64_t v, uint32_t be) {
  const uint64_t a = (uint64_t)(v < 0 ? -v : v);
  uint32_t hi = (uint32_t)(a >> 32), lo = (uint32_t)a;
  if (hi == 0u) {
    hi = lo;
    lo = 0u;
    be -= 32u;
  }
  const uint32_t n = (uint32_t)fx_clz(hi);
  const bool zero = hi == 0u;
  hi = fx_funnel_l(lo, hi, n);
  lo = fx_shl(lo, n);
  // the leading one adds 1 to the exponent field, as does a carry out of the rounding
  const uint64_t r = (((uint64_t)(hi >> 11) << 32) | fx_funnel_r(lo, hi, 11)) + ((lo >> 10) & 1u) +
                     ((uint64_t)((be - n - 1u) << 20) << 32);
  const uint32_t sign = (uint32_t)(v >> 32) & 0x80000000u;
  return zero ? 0.0 : fx_double((uint32_t)(r >> 32) | sign, (uint32_t)r);
}

// The same on the FP64 pipe: v = h 2^32 + l read into the significands of 2^84 + (h + 2^31) 2^32
// and 2^52 + l, whose difference and sum with the offsets' total is v, rounded once (to even).  Two
// additions of the FP64 pipe and one integer instruction instead of about 20 integer ones: for
// kernels that leave the FP64 pipe idle (the column passes and the set and get passes).  A result
// below 2^-1022 is rounded as FP64 rounds it.
FX_FN double fx_to_double_dp(int64_t v, uint32_t be) {
  const uint32_t eh = (be + 21u) << 20, el = (be - 11u) << 20;
  const double h = fx_double(eh, (uint32_t)(v >> 32) ^ 0x80000000u), l = fx_double(el, (uint32_t)v);
  return (h - fx_double(eh, 0x80100000u)) + l;
}

// ---- butterflies ----
FX_FN int32_t fx_low(int64_t x) { return (int32_t)x; }
FX_FN int32_t fx_high(int64_t x) { return (int32_t)((x + 0x80000000ll) >> 32); }  // with the signed low word

// x W (forward) or x conj(W) (inverse), the twiddle's scale 2^-s included.  The product of the low
// words (a quarter of the result's unit) is left out.
template <int DIR>
FX_FN cfx fx_mul(cfx x, TwFx w) {
  const int32_t rl = fx_low(x.re), rh = fx_high(x.re), il = fx_low(x.im), ih = fx_high(x.im);
  constexpr int64_t half = -(1ll << 29);  // rounds, negated with the sum it is in
  const int64_t rc = fx_mad(rh, w.cl, fx_mad(rl, w.ch, half)), is = fx_mad(ih, w.sl, fx_mad(il, w.sh, 0));
  const int64_t ic = fx_mad(ih, w.cl, fx_mad(il, w.ch, half)), rs = fx_mad(rh, w.sl, fx_mad(rl, w.sh, 0));
  const int32_t r4 = rh * 4, i4 = ih * 4;
  // c = -Re W:  forward re = -re c - im s, im = re s - im c;  inverse re = im s - re c, im = -im c - re s
  if (DIR < 0)
    return cfx{fx_mad(-i4, w.sh, fx_mad(-r4, w.ch, (-rc - is) >> 30)), fx_mad(r4, w.sh, fx_mad(-i4, w.ch, (rs - ic) >> 30))};
  return cfx{fx_mad(i4, w.sh, fx_mad(-r4, w.ch, (is - rc) >> 30)), fx_mad(-r4, w.sh, fx_mad(-i4, w.ch, (-ic - rs) >> 30))};
}

// x sqrt(1/2): sqrt(1/2) 2^62 = h 2^32 + l
FX_FN int64_t fx_mul_h(int64_t x) {
  constexpr int32_t h = 759250125, l = -25716447;
  const int32_t xl = fx_low(x), xh = fx_high(x);
  return fx_mad(xh * 4, h, fx_mad(xl, h, fx_mad(xh, l, 1ll << 29)) >> 30);
}

FX_FN cfx fx_add(cfx a, cfx b) { return cfx{a.re + b.re, a.im + b.im}; }
FX_FN cfx fx_sub(cfx a, cfx b) { return cfx{a.re - b.re, a.im - b.im}; }
template <int DIR>
FX_FN cfx fx_mul_i(cfx a) {
  return DIR > 0 ? cfx{-a.im, a.re} : cfx{a.im, -a.re};
}
FX_FN cfx fx_shift(cfx a, int s) {  // arithmetic right shift by 0 <= s < 32, rounded down
  return cfx{a.re >> s, a.im >> s};
}

template <int DIR>
FX_FN void fx_dft4(cfx *v) {
  const cfx s0 = fx_add(v[0], v[2]), d0 = fx_sub(v[0], v[2]);
  const cfx s1 = fx_add(v[1], v[3]), d1 = fx_mul_i<DIR>(fx_sub(v[1], v[3]));
  v[0] = fx_add(s0, s1);
  v[2] = fx_sub(s0, s1);
  v[1] = fx_add(d0, d1);
  v[3] = fx_sub(d0, d1);
}

// Length 8 by one decimation-in-frequency split; ZP: inputs 3 and 4 are zeros (the zero-padded
// first stage of an inverse transform).
template <int DIR, bool ZP>
FX_FN void fx_dft8(cfx *v) {
  cfx b[4], c[4];
  if (ZP) {
    b[0] = c[0] = v[0];
    b[3] = v[7];
    c[3] = cfx{-v[7].re, -v[7].im};
  } else {
    b[0] = fx_add(v[0], v[4]);
    c[0] = fx_sub(v[0], v[4]);
    b[3] = fx_add(v[3], v[7]);
    c[3] = fx_sub(v[3], v[7]);
  }
  b[1] = fx_add(v[1], v[5]);
  c[1] = fx_sub(v[1], v[5]);
  b[2] = fx_add(v[2], v[6]);
  c[2] = fx_sub(v[2], v[6]);
  // W8 = h (1 + DIR i), W8^2 = DIR i, W8^3 = h (-1 + DIR i)
  if (DIR > 0) {
    c[1] = cfx{fx_mul_h(c[1].re - c[1].im), fx_mul_h(c[1].im + c[1].re)};
    c[3] = cfx{fx_mul_h(-c[3].re - c[3].im), fx_mul_h(c[3].re - c[3].im)};
  } else {
    c[1] = cfx{fx_mul_h(c[1].re + c[1].im), fx_mul_h(c[1].im - c[1].re)};
    c[3] = cfx{fx_mul_h(c[3].im - c[3].re), fx_mul_h(-c[3].im - c[3].re)};
  }
  c[2] = fx_mul_i<DIR>(c[2]);
  fx_dft4<DIR>(b);
  fx_dft4<DIR>(c);
  for (int m = 0; m < 4; ++m) {
    v[2 * m] = b[m];
    v[2 * m + 1] = c[m];
  }
}

template <int R, int DIR>
FX_FN void fx_dft(cfx *v) {
  if (R == 8) {
    fx_dft8<DIR, false>(v);
  } else if (R == 4) {
    fx_dft4<DIR>(v);
  } else {
    const cfx a = v[0], b = v[1];
    v[0] = fx_add(a, b);
    v[1] = fx_sub(a, b);
  }
}

}  // namespace mhd
