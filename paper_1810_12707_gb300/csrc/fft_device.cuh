// fft_device.cuh -- device building blocks: complex arithmetic, small DFTs in registers, and the
// Stockham pencil FFT executed by a group of N/VPT threads (VPT = 8, or 16 in FP32) on a pencil
// held in shared memory.
//
// Transform convention (both directions unscaled):  X[k] = sum_j x[j] exp(DIR * 2 pi i j k / N)
// with DIR = -1 for the forward and +1 for the inverse transform.
#pragma once

#include "dfloat.cuh"
#include "fixed64.cuh"
#include "mhd_internal.h"

#include <type_traits>

namespace mhd {

template <typename C>
__device__ __forceinline__ C c_add(C a, C b) { return {a.re + b.re, a.im + b.im}; }
template <typename C>
__device__ __forceinline__ C c_sub(C a, C b) { return {a.re - b.re, a.im - b.im}; }
template <typename C>
__device__ __forceinline__ C c_scale(C a, typename C::value_type s) { return {a.re * s, a.im * s}; }
// a * w
template <typename C>
__device__ __forceinline__ C c_mul(C a, C w) {
  return {a.re * w.re - a.im * w.im, a.re * w.im + a.im * w.re};
}
// a * conj(w)
template <typename C>
__device__ __forceinline__ C c_mulc(C a, C w) {
  return {a.re * w.re + a.im * w.im, a.im * w.re - a.re * w.im};
}
// a * (DIR i)
template <int DIR, typename C>
__device__ __forceinline__ C c_mul_i(C a) {
  return DIR > 0 ? C{-a.im, a.re} : C{a.im, -a.re};
}
// precision conversion
template <typename CT, typename CF>
__device__ __forceinline__ CT c_cvt(CF a) {
  using R = typename CT::value_type;
  return CT{(R)a.re, (R)a.im};
}

// Double-float complex values use the generic forms above through the dfr operators (lazy sums
// and products).  A pass scales its output by a power of two only, given as an FP32 number.
__device__ __forceinline__ cdf c_scale(cdf a, float s) { return cdf{s * a.re, s * a.im}; }

// What a pass stores to global memory: double-float values renormalised, others as they are.
template <typename C>
__device__ __forceinline__ C c_store(C a) { return a; }
__device__ __forceinline__ cdf c_store(cdf a) { return cdf_norm(a); }

// NaN-propagating maximum (a non-finite CFL speed must reach the step-size kernel).
__device__ __forceinline__ double nan_max(double a, double b) {
  if (a != a) return a;
  if (b != b) return b;
  return a > b ? a : b;
}

// ---- DFTs of length 2, 4, 8 on registers, natural order in and out ----

template <int DIR, typename C>
__device__ __forceinline__ void dft2(C *v) {
  const C a = v[0], b = v[1];
  v[0] = c_add(a, b);
  v[1] = c_sub(a, b);
}

template <int DIR, typename C>
__device__ __forceinline__ void dft4(C *v) {
  const C s0 = c_add(v[0], v[2]), d0 = c_sub(v[0], v[2]);
  const C s1 = c_add(v[1], v[3]), d1 = c_mul_i<DIR>(c_sub(v[1], v[3]));
  v[0] = c_add(s0, s1);
  v[2] = c_sub(s0, s1);
  v[1] = c_add(d0, d1);
  v[3] = c_sub(d0, d1);
}

// Length 8 by one decimation-in-frequency split: b_j = a_j + a_{j+4} feeds the even outputs,
// c_j = (a_j - a_{j+4}) W8^j the odd ones, each through a length-4 DFT.
template <int DIR, typename C>
__device__ __forceinline__ void dft8(C *v) {
  using R = typename C::value_type;
  constexpr R h = (R)0.70710678118654752440;  // sqrt(2) / 2
  C b[4], c[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    b[j] = c_add(v[j], v[j + 4]);
    c[j] = c_sub(v[j], v[j + 4]);
  }
  // W8^1 = h (1 + DIR i), W8^2 = DIR i, W8^3 = h (-1 + DIR i)
  c[1] = C{h * (c[1].re - DIR * c[1].im), h * (c[1].im + DIR * c[1].re)};
  c[2] = c_mul_i<DIR>(c[2]);
  c[3] = C{h * (-c[3].re - DIR * c[3].im), h * (-c[3].im + DIR * c[3].re)};
  dft4<DIR>(b);
  dft4<DIR>(c);
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    v[2 * m] = b[m];
    v[2 * m + 1] = c[m];
  }
}

// Length 16 as 4 x 4: n = 4 n1 + n2, k = k1 + 4 k2.  Length-4 DFTs over n1 for each n2, the
// twiddles W16^(n2 k1), then length-4 DFTs over n2 for each k1 (W16 = exp(DIR 2 pi i / 16)).
// ZP: inputs 6..9 are zeros (zero-padded first stage; see pencil_fft): each first-layer length-4
// DFT then has one zero input and loses a butterfly.
template <int DIR, typename C, bool ZP = false>
__device__ __forceinline__ void dft16(C *v) {
  using R = typename C::value_type;
  constexpr R c1 = (R)0.92387953251128675613;  // cos(pi/8)
  constexpr R s1 = (R)0.38268343236508977173;  // sin(pi/8)
  constexpr R h = (R)0.70710678118654752440;   // cos(pi/4)
  C a[4][4];
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) {
    C t[4] = {v[n2], v[n2 + 4], v[n2 + 8], v[n2 + 12]};
    if constexpr (ZP) {
      if (n2 < 2) {  // t[2] = v8 or v9 = 0: (t0 + t2, t0 - t2) = (t0, t0)
        const C s1 = c_add(t[1], t[3]), d1 = c_mul_i<DIR>(c_sub(t[1], t[3]));
        t[2] = c_sub(t[0], s1);
        t[1] = c_add(t[0], d1);
        t[3] = c_sub(t[0], d1);
        t[0] = c_add(t[0], s1);
      } else {  // t[1] = v6 or v7 = 0: (t1 + t3, t1 - t3) = (t3, -t3)
        const C s0 = c_add(t[0], t[2]), d0 = c_sub(t[0], t[2]);
        const C d1 = c_mul_i<DIR>(C{-t[3].re, -t[3].im});
        t[0] = c_add(s0, t[3]);
        t[2] = c_sub(s0, t[3]);
        t[1] = c_add(d0, d1);
        t[3] = c_sub(d0, d1);
      }
    } else {
      dft4<DIR>(t);
    }
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) a[n2][k1] = t[k1];
  }
  const C w1 = {c1, DIR * s1}, w2 = {h, DIR * h}, w3 = {s1, DIR * c1};
  const C w6 = {-h, DIR * h}, w9 = {-c1, -DIR * s1};
  a[1][1] = c_mul(a[1][1], w1);
  a[1][2] = c_mul(a[1][2], w2);
  a[1][3] = c_mul(a[1][3], w3);
  a[2][1] = c_mul(a[2][1], w2);
  a[2][2] = c_mul_i<DIR>(a[2][2]);  // W16^4 = DIR i
  a[2][3] = c_mul(a[2][3], w6);
  a[3][1] = c_mul(a[3][1], w3);
  a[3][2] = c_mul(a[3][2], w6);
  a[3][3] = c_mul(a[3][3], w9);
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
    C t[4] = {a[0][k1], a[1][k1], a[2][k1], a[3][k1]};
    dft4<DIR>(t);
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = t[k2];
  }
}

// Length 8 in double-float: the same split as above; W8 = h (1 + DIR i) with h = sqrt(2)/2 in
// double-float.
template <int DIR>
__device__ __forceinline__ void dft8(cdf *v) {
  constexpr dfr h = dfr_const(0.70710678118654752440);
  cdf b[4], c[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    b[j] = c_add(v[j], v[j + 4]);
    c[j] = c_sub(v[j], v[j + 4]);
  }
  if constexpr (DIR > 0) {
    c[1] = cdf{h * (c[1].re - c[1].im), h * (c[1].im + c[1].re)};
    c[3] = cdf{h * (-c[3].re - c[3].im), h * (c[3].re - c[3].im)};
  } else {
    c[1] = cdf{h * (c[1].re + c[1].im), h * (c[1].im - c[1].re)};
    c[3] = cdf{h * (c[3].im - c[3].re), h * (-c[3].im - c[3].re)};
  }
  c[2] = c_mul_i<DIR>(c[2]);
  dft4<DIR>(b);
  dft4<DIR>(c);
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    v[2 * m] = b[m];
    v[2 * m + 1] = c[m];
  }
}

// The same with inputs 3 and 4 known zeros (the zero-padded first stage): the first layer's
// pairs (v0, v4) and (v3, v7) need no arithmetic, (v0, v0) and (v7, -v7).  The other inputs
// take the operations of dft8, so the results are dft8's.
template <int DIR>
__device__ __forceinline__ void dft8_zp(cdf *v) {
  constexpr dfr h = dfr_const(0.70710678118654752440);
  cdf b[4], c[4];
  b[0] = v[0];
  c[0] = v[0];
  b[3] = v[7];
  c[3] = cdf{-v[7].re, -v[7].im};
#pragma unroll
  for (int j = 1; j < 3; ++j) {
    b[j] = c_add(v[j], v[j + 4]);
    c[j] = c_sub(v[j], v[j + 4]);
  }
  if constexpr (DIR > 0) {
    c[1] = cdf{h * (c[1].re - c[1].im), h * (c[1].im + c[1].re)};
    c[3] = cdf{h * (-c[3].re - c[3].im), h * (c[3].re - c[3].im)};
  } else {
    c[1] = cdf{h * (c[1].re + c[1].im), h * (c[1].im - c[1].re)};
    c[3] = cdf{h * (c[3].im - c[3].re), h * (-c[3].im - c[3].re)};
  }
  c[2] = c_mul_i<DIR>(c[2]);
  dft4<DIR>(b);
  dft4<DIR>(c);
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    v[2 * m] = b[m];
    v[2 * m + 1] = c[m];
  }
}

template <int R, int DIR, typename C>
__device__ __forceinline__ void dft_small(C *v) {
  if constexpr (R == 16) dft16<DIR>(v);
  else if constexpr (R == 8) dft8<DIR>(v);
  else if constexpr (R == 4) dft4<DIR>(v);
  else dft2<DIR>(v);
}

// Twiddle load that the compiler may not hoist out of loops: kernels that transform many pencils
// in a loop would otherwise keep every stage's twiddles live in registers across the loop.
__device__ __forceinline__ cdf tw_load(const cdf *p) {
  cdf v;
  asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.re.hi), "=f"(v.re.lo), "=f"(v.im.hi), "=f"(v.im.lo)
               : "l"(p));
  return v;
}
// The same from a table that a block has staged in shared memory: element i.
__device__ __forceinline__ cdf tw_load_shared(const cdf *table, unsigned i) {
  cdf v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.re.hi), "=f"(v.re.lo), "=f"(v.im.hi), "=f"(v.im.lo)
               : "r"((unsigned)__cvta_generic_to_shared(table) + i * (unsigned)sizeof(cdf)));
  return v;
}
// table + kt r.  N >= 512: as one multiply-add (512^3 flux pass, FP32 5.35 -> 5.05 ms, double-float
// 17.17 -> 17.07); below, left to the compiler (256^3 flux pass 0.559 -> 0.547 and 1.948 -> 1.912 ms,
// the other way round).
template <int N, typename W>
__device__ __forceinline__ const W *tw_at(const W *table, unsigned kt, int r) {
  if constexpr (N >= 512) {
    const W *p;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(p) : "r"(kt), "r"((unsigned)(r * (int)sizeof(W))), "l"(table));
    return p;
  } else {
    return table + kt * (unsigned)r;
  }
}

__device__ __forceinline__ cplx64 tw_load(const cplx64 *p) {
  cplx64 v;
  asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(v.re), "=d"(v.im) : "l"(p));
  return v;
}
__device__ __forceinline__ TwFx tw_load(const TwFx *p) {
  TwFx v;
  asm volatile("ld.global.nc.v4.s32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.ch), "=r"(v.cl), "=r"(v.sh), "=r"(v.sl)
               : "l"(p));
  return v;
}
__device__ __forceinline__ cplx32 tw_load(const cplx32 *p) {
  cplx32 v;
  asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(v.re), "=f"(v.im) : "l"(p));
  return v;
}

// The value of x, opaque to the optimiser: index arithmetic derived from it cannot be hoisted out
// of a persistent loop and kept live (in registers or spilled) across iterations.
__device__ __forceinline__ int launder(int x) {
  int y;
  asm volatile("mov.b32 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}

// ---- shared-memory pencil layout ----
// A pencil element e lives at sm_idx<C>(e) = e + e / (128 / sizeof(C)): one pad element per 128
// bytes.  The first Stockham stage writes with a stride of 8 elements; without the pad every lane
// of a wavefront would hit the same banks.  Pencils are `pencil_pitch` apart, an odd number of
// elements, so that lanes walking across pencils (the column loads) also spread over the banks.
template <typename C>
__host__ __device__ constexpr int sm_pad() { return (int)(128 / sizeof(C)); }
template <typename C>
__host__ __device__ constexpr int sm_idx(int e) { return e + e / sm_pad<C>(); }
template <typename C>
__host__ __device__ constexpr int pencil_pitch(int n) { return sm_idx<C>(n) | 1; }
// The same of an unsigned element index (a shift, where the signed division also handles negatives).
// sm_at(e) + sm_idx(d) = sm_at(e + d) when d is a multiple of sm_pad, or when no carry leaves the low
// log2(sm_pad) bits of e + d: the stages below address a butterfly's elements at constant offsets
// from its first one.
template <typename C>
__device__ __forceinline__ unsigned sm_at(unsigned e) { return e + e / (unsigned)sm_pad<C>(); }

// ---- barrier of one pencil's thread group ----
// A pencil is transformed by the TPP = N/VPT consecutive threads of its group and nobody else
// touches it meanwhile, so the stages only need that group to synchronise: within a warp
// (TPP <= 32) a warp barrier over the lanes that exist, otherwise a named barrier per group
// (ids 1..15; id 0 is __syncthreads), falling back to the block barrier when there are more groups.
__device__ __forceinline__ unsigned existing_lanes() {
  const int left = (int)blockDim.x - (int)(threadIdx.x & ~31u);
  return left >= 32 ? 0xffffffffu : ((1u << left) - 1u);
}

template <int TPP>
__device__ __forceinline__ void group_sync() {
  if constexpr (TPP <= 32) {
    __syncwarp(existing_lanes());
  } else {
    if (blockDim.x / TPP <= 15) {
      asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)(threadIdx.x / TPP)), "r"(TPP) : "memory");
    } else {
      __syncthreads();
    }
  }
}

// ---- IEEE FP64 transforms: twiddles in FMA form ----
// Only the transform of a mixed-precision initial state still runs in IEEE FP64 arithmetic (tables
// of cplx64; every other FP64 transform takes a TwFx table and runs in fixed point, 2.5 to 3.1
// times faster).  The mixed mode's FP32 steps turn a difference of 1e-17 in the state's smallest
// modes into FP32 rounding noise within a step, so a faster transform here would change every
// mixed trajectory by about 4e-8 (measured: 3.8e-8 after 60 steps at 32^3), no less exactly but
// not reproducibly.  Its cost is FP64 instructions, so the twiddled stages use few: every twiddle is
// kept as W = i^q c (1 + i t) with |t| <= 1, and a radix-2 butterfly (a + W x, a - W x) costs six fused
// multiply-adds: z = x + i t x (two), z' = i^q z (an exact swap and sign change done with integer
// operations), a +- c z' (four).  Only forward transforms run so.  The table follows the classic one
// in the same allocation: tw[0..N) classic W_N^m, then N pairs (c, t), then N bytes q
// (ieee_twiddle_bytes).
struct TwF {
  double c, t;
  int q;
};

template <int N>
__device__ __forceinline__ TwF twf_load(const cplx64 *__restrict__ tw, int m) {
  const double *ct = reinterpret_cast<const double *>(tw + N) + 2 * m;
  const unsigned char *qt = reinterpret_cast<const unsigned char *>(tw + 2 * N) + m;
  TwF w;
  unsigned short qq;
  asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(w.c), "=d"(w.t) : "l"(ct));
  asm volatile("ld.global.nc.u8 %0, [%1];" : "=h"(qq) : "l"(qt));
  w.q = qq;
  return w;
}

// The same twiddle turned by a quarter -i (the factor omega_4 of the DIF split).
__device__ __forceinline__ TwF twf_quarter(TwF w) {
  w.q = (w.q + 3) & 3;
  return w;
}

__device__ __forceinline__ double flip_sign(double x, unsigned s) {
  return __hiloint2double(__double2hiint(x) ^ (int)s, __double2loint(x));
}

// i^q z, exactly, with integer selects and sign flips.
__device__ __forceinline__ cplx64 rot_quarter(cplx64 z, int q) {
  const bool sw = q & 1;
  const double a = sw ? z.im : z.re, b = sw ? z.re : z.im;
  const unsigned s_re = (unsigned)((q ^ (q >> 1)) & 1) << 31, s_im = (unsigned)((q >> 1) & 1) << 31;
  return cplx64{flip_sign(a, s_re), flip_sign(b, s_im)};
}

// (x0, x1) <- (x0 + W x1, x0 - W x1)
__device__ __forceinline__ void bfly_fma(cplx64 &x0, cplx64 &x1, const TwF &w) {
  const cplx64 z = rot_quarter(cplx64{fma(-w.t, x1.im, x1.re), fma(w.t, x1.re, x1.im)}, w.q);
  const cplx64 a = x0;
  x0 = cplx64{fma(w.c, z.re, a.re), fma(w.c, z.im, a.im)};
  x1 = cplx64{fma(-w.c, z.re, a.re), fma(-w.c, z.im, a.im)};
}

// Length-R DFT of (W^r x_r)_r, r < R, for R = 8, 4, 2, W = W_N^m, as radix-2
// layers of the decimation-in-frequency split with every twiddle carried into the butterflies:
//   R = 8: layer 1 W^4 (x4); layer 2 W^2 (x2) and (W w8)^2 = W^2 w4 (x2); layer 3 W, W w4, W w8,
//          W w8 w4, with w8 = W_N^(N/8) and w4 = w8^2 a quarter turn.
// Results in natural order in v.
template <int N, int R>
__device__ __forceinline__ void dft_twiddled_fma(cplx64 *v, int m, const cplx64 *__restrict__ tw) {
  if constexpr (R == 8) {
    const TwF w1 = twf_load<N>(tw, m), w2 = twf_load<N>(tw, 2 * m), w4 = twf_load<N>(tw, 4 * m);
    const TwF w18 = twf_load<N>(tw, m + N / 8);  // W w8
#pragma unroll
    for (int j = 0; j < 4; ++j) bfly_fma(v[j], v[j + 4], w4);  // P'_j = v_j, Q'_j = v_j+4
    const TwF w2q = twf_quarter(w2);
    bfly_fma(v[0], v[2], w2);   // PP'_0, PQ'_0
    bfly_fma(v[1], v[3], w2);   // PP'_1, PQ'_1
    bfly_fma(v[4], v[6], w2q);  // QP'_0, QQ'_0
    bfly_fma(v[5], v[7], w2q);  // QP'_1, QQ'_1
    bfly_fma(v[0], v[1], w1);                     // X0, X4
    bfly_fma(v[2], v[3], twf_quarter(w1));   // X2, X6
    bfly_fma(v[4], v[5], w18);                    // X1, X5
    bfly_fma(v[6], v[7], twf_quarter(w18));  // X3, X7
    const cplx64 x0 = v[0], x4 = v[1], x2 = v[2], x6 = v[3], x1 = v[4], x5 = v[5], x3 = v[6], x7 = v[7];
    v[0] = x0; v[1] = x1; v[2] = x2; v[3] = x3; v[4] = x4; v[5] = x5; v[6] = x6; v[7] = x7;
  } else if constexpr (R == 4) {
    const TwF w1 = twf_load<N>(tw, m), w2 = twf_load<N>(tw, 2 * m);
    bfly_fma(v[0], v[2], w2);  // P'_0, Q'_0
    bfly_fma(v[1], v[3], w2);  // P'_1, Q'_1
    bfly_fma(v[0], v[1], w1);                    // X0, X2
    bfly_fma(v[2], v[3], twf_quarter(w1));  // X1, X3
    const cplx64 x0 = v[0], x2 = v[1], x1 = v[2], x3 = v[3];
    v[0] = x0; v[1] = x1; v[2] = x2; v[3] = x3;
  } else {
    bfly_fma(v[0], v[1], twf_load<N>(tw, m));
  }
}

// The first (untwiddled) radix-8 stage as radix-2 layers: twiddle 1 everywhere except the quarter
// turns (free) and w8 = c (1 + i DIR), c = sqrt(2)/2, on two butterflies of layer 3 (two additions
// and four FMAs each).  With ZP the inputs 3 and 4 are known zeros (zero-padded inverse
// transforms: the 2/3-rule gap K+1 .. N-K-1 always covers them, see pencil_fft) and layer 1 loses
// two butterflies.
template <int DIR, bool ZP, typename C>
__device__ __forceinline__ void dft8_first_fma(C *v) {
  using R = typename C::value_type;
  constexpr R c = (R)0.70710678118654752440;  // cos(pi/4)
  // layer 1 (twiddle 1): (v_j, v_j+4) <- (v_j + v_j+4, v_j - v_j+4)
  if constexpr (ZP) {  // j = 0 with v4 = 0, j = 3 with v3 = 0
    v[4] = v[0];
    v[3] = v[7];
    v[7] = C{-v[7].re, -v[7].im};
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (ZP && (j == 0 || j == 3)) continue;
    const C a = v[j], b = v[j + 4];
    v[j] = c_add(a, b);
    v[j + 4] = c_sub(a, b);
  }
  // layer 2: twiddle 1 on (0,2), (1,3); w4 on (4,6), (5,7)
  {
    const C a0 = v[0], a2 = v[2], a1 = v[1], a3 = v[3];
    v[0] = c_add(a0, a2);
    v[2] = c_sub(a0, a2);
    v[1] = c_add(a1, a3);
    v[3] = c_sub(a1, a3);
    const C q6 = c_mul_i<DIR>(v[6]), q7 = c_mul_i<DIR>(v[7]);
    const C a4 = v[4], a5 = v[5];
    v[4] = c_add(a4, q6);
    v[6] = c_sub(a4, q6);
    v[5] = c_add(a5, q7);
    v[7] = c_sub(a5, q7);
  }
  // layer 3: 1 on (0,1), w4 on (2,3), w8 on (4,5), w8 w4 on (6,7)
  {
    const C a0 = v[0], a1 = v[1];
    v[0] = c_add(a0, a1);
    v[1] = c_sub(a0, a1);
    const C a2 = v[2], r3 = c_mul_i<DIR>(v[3]);
    v[2] = c_add(a2, r3);
    v[3] = c_sub(a2, r3);
    const C z5 = {v[5].re - DIR * v[5].im, v[5].im + DIR * v[5].re};  // (1 + i DIR) v5
    const C a4 = v[4];
    v[4] = C{fma(c, z5.re, a4.re), fma(c, z5.im, a4.im)};
    v[5] = C{fma(-c, z5.re, a4.re), fma(-c, z5.im, a4.im)};
    const C z7 = c_mul_i<DIR>(C{v[7].re - DIR * v[7].im, v[7].im + DIR * v[7].re});
    const C a6 = v[6];
    v[6] = C{fma(c, z7.re, a6.re), fma(c, z7.im, a6.im)};
    v[7] = C{fma(-c, z7.re, a6.re), fma(-c, z7.im, a6.im)};
  }
  // (X0, X4, X2, X6, X1, X5, X3, X7) -> natural order
  const C x0 = v[0], x4 = v[1], x2 = v[2], x6 = v[3], x1 = v[4], x5 = v[5], x3 = v[6], x7 = v[7];
  v[0] = x0; v[1] = x1; v[2] = x2; v[3] = x3; v[4] = x4; v[5] = x5; v[6] = x6; v[7] = x7;
}

// The first radix-8 stage in double-float: the plain length-8 DFT, or with the zero-padded
// pencil's inputs 3 and 4 (not loaded) left out of the arithmetic.
template <int DIR, bool ZP>
__device__ __forceinline__ void dft8_first_fma(cdf *v) {
  if constexpr (ZP) dft8_zp<DIR>(v);
  else dft8<DIR>(v);
}

// ---- values per thread ----
// FP32 pencils: 16 values per thread (radix 16: two shared-memory stages at N = 256 where radix 8
// needs three; the FP32 passes are bound by instruction issue).  FP64 and double-float: 8 (their
// 16-byte values fill the registers).  A pencil is transformed by N / VPT threads.
// Kernels may choose 8 or 16 for FP32 (the radix that suits a pass depends on N and on the pass;
// the column passes let the autotuner pick); FP64 always uses 8.
template <typename C>
__host__ __device__ constexpr int fft_vpt() { return sizeof(C) == 8 ? 16 : 8; }
template <int N, int VPT>
__host__ __device__ constexpr int tpp_for() { return N / VPT > 0 ? N / VPT : 1; }
template <int N, typename C>
__host__ __device__ constexpr int fft_tpp() { return tpp_for<N, fft_vpt<C>()>(); }

// ---- Stockham pencil FFT ----
//
// The transform of length N = product of radices (VPT = 16 or 8 while that many points remain,
// then the rest) runs as a sequence of stages.  Before a stage, sub-transforms of length NS are complete;
// butterfly j (0 <= j < N/R) gathers x[j + r N/R] (r < R), multiplies element r by the twiddle
// W_{NS R}^{r (j mod NS)}, applies a length-R DFT and scatters the results to
// (j div NS) NS R + (j mod NS) + r NS.  After the last stage the pencil holds X in natural order
// (the auto-sorting formulation of Cooley-Tukey by Stockham).  Each of the N/VPT threads of a
// group owns VPT / R butterflies per stage, so it always holds VPT values.  `tw[m]` = W_N^m =
// exp(-2 pi i m / N); the inverse uses its conjugate.
//
// Every thread of the block must call this (it contains group barriers); threads with
// `active == false` only take part in the barriers.  The caller separates the transform from the
// preceding writes and the following reads of the pencil with a block barrier.
// TWG: `tw` points to shared memory (double-float only).
// REG: the last stage leaves its results in `out` instead of the pencil: out[q] = X[t + q N/VPT].
template <int N, int DIR, int NS, typename C, int VPT, bool ZP, bool TWG = false, bool REG = false>
__device__ __forceinline__ void stockham_stages(C *buf, int t, bool active, const C *__restrict__ tw,
                                                C *out = nullptr) {
  if constexpr (NS < N) {
    static_assert(VPT == 8 || (VPT == 16 && sizeof(C) == 8), "radix 16 is an FP32 option");
    constexpr int R = (N / NS >= VPT) ? VPT : N / NS;
    constexpr int NB = VPT / R;
    constexpr int TPP = tpp_for<N, VPT>();
    constexpr int TWSTEP = N / (NS * R);
    // IEEE FP64 stages with twiddles take them inside the butterflies (FMA form, fewer FP64
    // instructions); the others multiply on load.
    constexpr bool kFma = std::is_same<C, cplx64>::value && NS > 1;
    // The first radix-8 stage: FMA layers, and with ZP the zero inputs 3 and 4 skipped; the first
    // radix-16 stage with ZP skips its zero inputs 6..9.
    constexpr bool kFirst = NS == 1 && R == 8;
    constexpr bool kFirst16 = NS == 1 && R == 16 && ZP;
    constexpr int K = (N - 1) / 3;
    static_assert(!(ZP && kFirst) || (3 * (N / 8) > K && 5 * (N / 8) - 1 < N - K),
                  "inputs 3 and 4 of the first radix-8 stage must lie in the 2/3-rule gap");
    static_assert(!kFirst16 || (6 * (N / 16) > K && 10 * (N / 16) - 1 < N - K),
                  "inputs 6..9 of the first radix-16 stage must lie in the 2/3-rule gap");
    // reads at constant offsets from the butterfly's first element (see sm_at); the smallest grids'
    // strides are not multiples of the pad's period
    constexpr bool kConst = (N / R) % sm_pad<C>() == 0;
    C v[VPT];
    if (active) {
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        const unsigned j = (unsigned)(t + b * TPP);
        const unsigned kt = (j % (unsigned)NS) * (unsigned)TWSTEP;
        const C *rp = buf + sm_at<C>(j);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (kFirst && ZP && (r == 3 || r == 4)) continue;  // zeros, never read
          if (kFirst16 && r >= 6 && r <= 9) continue;
          C x = kConst ? rp[sm_idx<C>(r * (N / R))] : buf[sm_at<C>(j + r * (N / R))];
          if (!kFma && NS > 1 && r > 0) {
            C w;
            if constexpr (TWG) w = tw_load_shared(tw, kt * (unsigned)r);
            else w = tw_load(tw_at<N>(tw, kt, r));
            x = DIR < 0 ? c_mul(x, w) : c_mulc(x, w);
          }
          v[b * R + r] = x;
        }
      }
    }
    group_sync<TPP>();
    if (active) {
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        const unsigned j = (unsigned)(t + b * TPP);
        const unsigned k = j % (unsigned)NS;
        if constexpr (kFma) {
          static_assert(DIR < 0, "IEEE FP64 transforms are forward ones");
          dft_twiddled_fma<N, R>(reinterpret_cast<cplx64 *>(v) + b * R, (int)(k * TWSTEP),
                                      reinterpret_cast<const cplx64 *>(tw));
        } else if constexpr (kFirst) {
          dft8_first_fma<DIR, ZP>(v + b * R);
        } else if constexpr (kFirst16) {
          dft16<DIR, C, true>(v + b * R);
        } else {
          dft_small<R, DIR, C>(v + b * R);
        }
        if constexpr (REG && NS * R == N) {
#pragma unroll
          for (int r = 0; r < R; ++r) out[b + NB * r] = v[b * R + r];
        } else {
          C *wp = buf + sm_at<C>((j - k) * R + k);
#pragma unroll
          for (int r = 0; r < R; ++r) wp[sm_idx<C>(r * NS)] = v[b * R + r];
        }
      }
    }
    if constexpr (!(REG && NS * R == N)) group_sync<TPP>();
    stockham_stages<N, DIR, NS * R, C, VPT, false, TWG, REG>(buf, t, active, tw, out);
  }
}

// The rest of a `bad` pencil's result.
__device__ __forceinline__ void fx_bad_out(cplx64 &x, const FxScale &sc) { x = c_scale(x, fx_bad_factor(sc.ek)); }

// ---- The FP64 pencil FFT (fixed64.cuh) ----
// The same Stockham stages on a pencil of doubles.  The first stage reads doubles, finds the
// pencil's common exponent and converts; the pencil is fixed-point complex values between the
// stages; the last stage writes doubles.  Against the IEEE FP64 stages this replaced (FP64 pipe 92 %
// busy), ms per pass: 512^3 inverse y 12.4 -> 3.98, forward y 23.8 -> 6.60, flux 65.6 -> 21.1;
// 256^3 step 14.75 -> 4.97.  The exponent's reduction adds no barrier: a group of
// more than a warp leaves its warps' parts in shared memory before the barrier that the first
// stage has between its reads and its writes anyway.  It depends on the group's threads only, so
// a pencil's results are the same bits in every kernel with the same DP and at every tile width.
// DP: the results' conversion runs on the FP64 pipe; `scale2`: they are scaled by 2^scale2.
// REG: the last stage leaves its fixed-point results in `out`, as in stockham_stages.
template <int N, int DIR, int NS, bool DP, bool REG = false>
__device__ __forceinline__ void fx_stages(cfx *buf, int t, bool active, const TwFx *__restrict__ tw, const FxScale &sc,
                                          int left, int scale2, cfx *out = nullptr) {
  constexpr int R = N / NS >= 8 ? 8 : N / NS;
  constexpr int NB = 8 / R;
  constexpr int TPP = tpp_for<N, 8>();
  constexpr int TWSTEP = N / (NS * R);
  constexpr int LOG2R = R == 8 ? 3 : R == 4 ? 2 : 1;
  const int s = left < LOG2R ? left : LOG2R;  // this stage's right shift
  cfx v[8];
  if (active) {
    const TwFx *ts = tw + s * N;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const unsigned j = (unsigned)(t + b * TPP);
      const unsigned kt = (j % (unsigned)NS) * (unsigned)TWSTEP;
      static_assert((N / R) % sm_pad<cplx64>() == 0, "constant read offsets");
      const cfx *rp = buf + sm_at<cplx64>(j);
      v[b * R] = fx_shift(rp[0], s);
#pragma unroll
      for (int r = 1; r < R; ++r)
        v[b * R + r] = fx_mul<DIR>(rp[sm_idx<cplx64>(r * (N / R))], tw_load(tw_at<N>(ts, kt, r)));
      fx_dft<R, DIR>(v + b * R);
    }
  }
  group_sync<TPP>();
  if constexpr (REG && NS * R == N) {
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int r = 0; r < R; ++r) out[b + NB * r] = v[b * R + r];
    return;
  }
  if (active) {
    const uint32_t be = sc.ek + (uint32_t)(sc.shift + scale2) + 1u;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const unsigned j = (unsigned)(t + b * TPP);
      const unsigned k = j % (unsigned)NS;
      cfx *wp = buf + sm_at<cplx64>((j - k) * R + k);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const cfx x = v[b * R + r];
        cfx *p = wp + sm_idx<cplx64>(r * NS);
        if constexpr (NS * R < N) {
          *p = x;
        } else {
          cplx64 d;
          if constexpr (DP) d = cplx64{fx_to_double_dp(x.re, be), fx_to_double_dp(x.im, be)};
          else d = cplx64{fx_to_double(x.re, be), fx_to_double(x.im, be)};
          *reinterpret_cast<cplx64 *>(p) = d;
        }
      }
    }
    if (NS * R == N && sc.bad) {
      cplx64 *pen = reinterpret_cast<cplx64 *>(buf);
#pragma unroll 1
      for (int i = t; i < N; i += TPP) fx_bad_out(pen[sm_at<cplx64>((unsigned)i)], sc);
    }
  }
  group_sync<TPP>();
  if constexpr (NS * R < N) fx_stages<N, DIR, NS * R, DP, REG>(buf, t, active, tw, sc, left - s, scale2, out);
}

// The pencil's scale from every thread's share of its values: `size(m)` is the thread's sum of their
// sizes in units of 2^(m - 1043) (fx_size), `m` its largest biased exponent.  Holds one group barrier
// if SYNC or if the group is more than a warp.
template <int N, bool SYNC, typename Size>
__device__ __forceinline__ FxScale fx_group_scale(uint32_t m, Size size) {
  constexpr int TPP = tpp_for<N, 8>();
  constexpr int LOG2G = TPP == 128 ? 7 : TPP == 64 ? 6 : TPP == 32 ? 5 : TPP == 16 ? 4 : TPP == 8 ? 3 : TPP == 4 ? 2 : 1;
  __shared__ FxPart part[32];  // one entry per warp, for groups of more than one
  if constexpr (TPP >= 32) {
    m = __reduce_max_sync(0xffffffffu, m);
  } else {
#pragma unroll
    for (int o = TPP / 2; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(existing_lanes(), m, o));
  }
  FxPart p = {m, size(m), 0u};
  p.t = (p.a >> 3) + 1u;
  if constexpr (TPP >= 32) {
    p.a = __reduce_max_sync(0xffffffffu, p.a);
    p.t = __reduce_add_sync(0xffffffffu, p.t);
  } else {
#pragma unroll
    for (int o = TPP / 2; o > 0; o >>= 1) {
      p.a = max(p.a, __shfl_xor_sync(existing_lanes(), p.a, o));
      p.t += __shfl_xor_sync(existing_lanes(), p.t, o);
    }
  }
  if constexpr (TPP > 32) {
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = p;
  }
  if constexpr (SYNC || TPP > 32) group_sync<TPP>();
  if constexpr (TPP > 32) {
    const int w0 = (threadIdx.x / TPP) * (TPP / 32);
    p = part[w0];
#pragma unroll
    for (int i = 1; i < TPP / 32; ++i) p = fx_merge(p, part[w0 + i]);
  }
  return fx_scale_any(p, LOG2G);
}

// The transform of the doubles x[r] = element t + r N/8 of each thread of the group: results in the
// pencil `buf` as doubles, or (REG) in `out` as fixed-point values of scale `sc`.  Nothing is read
// from `buf` before the group's first barrier.
template <int N, int DIR, bool ZP, bool DP = false, bool REG = false>
__device__ __forceinline__ void fx_fft_from(const cplx64 *x, cplx64 *buf, int t, bool active,
                                            const TwFx *__restrict__ tw, int scale2 = 0, cfx *out = nullptr,
                                            FxScale *out_scale = nullptr) {
  constexpr int TPP = tpp_for<N, 8>();
  constexpr int K = (N - 1) / 3;
  static_assert(!ZP || (3 * (N / 8) > K && 5 * (N / 8) - 1 < N - K),
                "inputs 3 and 4 of the first stage must lie in the 2/3-rule gap");
  uint32_t m = 0u;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    if (ZP && (r == 3 || r == 4)) continue;
    m = max(m, max(fx_hi(x[r].re) & 0x7fffffffu, fx_hi(x[r].im) & 0x7fffffffu));
  }
  const FxScale sc = fx_group_scale<N, true>(fx_max_exp(m), [&](uint32_t mm) {
    uint32_t a = 0u;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      if (ZP && (r == 3 || r == 4)) continue;
      a += fx_size(fx_hi(x[r].re), mm) + fx_size(fx_hi(x[r].im), mm);
    }
    return a;
  });
  cfx *fb = reinterpret_cast<cfx *>(buf);
  if (active) {
    cfx v[8];
    if (!sc.bad) {
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        if (ZP && (r == 3 || r == 4)) continue;
        v[r] = cfx{fx_from_double(fx_hi(x[r].re), fx_lo(x[r].re), sc.ek),
                   fx_from_double(fx_hi(x[r].im), fx_lo(x[r].im), sc.ek)};
      }
    } else {
      const uint32_t ek = fx_bad_ek(sc.ek);
#pragma unroll
      for (int r = 0; r < 8; ++r)
        v[r] = cfx{fx_from_any(fx_hi(x[r].re), fx_lo(x[r].re), ek), fx_from_any(fx_hi(x[r].im), fx_lo(x[r].im), ek)};
    }
    fx_dft8<DIR, ZP>(v);
#pragma unroll
    for (int r = 0; r < 8; ++r) fb[9u * (unsigned)t + r] = v[r];
  }
  group_sync<TPP>();
  fx_stages<N, DIR, 8, DP, REG>(fb, t, active, tw, sc, sc.shift, scale2, out);
  if constexpr (REG) *out_scale = sc;
}

// The same of the doubles in the pencil `buf`.
template <int N, int DIR, bool ZP, bool DP = false, bool REG = false>
__device__ __forceinline__ void fx_pencil_fft(cplx64 *buf, int t, bool active, const TwFx *__restrict__ tw,
                                              int scale2 = 0, cfx *out = nullptr, FxScale *out_scale = nullptr) {
  constexpr int TPP = tpp_for<N, 8>();
  cplx64 x[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    x[r] = cplx64{0.0, 0.0};
    if (!(ZP && (r == 3 || r == 4)) && active)
      x[r] = TPP % sm_pad<cplx64>() == 0 ? buf[sm_at<cplx64>((unsigned)t) + sm_idx<cplx64>(r * TPP)]
                                         : buf[sm_at<cplx64>((unsigned)(t + r * TPP))];
  }
  fx_fft_from<N, DIR, ZP, DP, REG>(x, buf, t, active, tw, scale2, out, out_scale);
}

// `t` in [0, N / VPT): the thread's index within its pencil's group.  ZP: the pencil is
// zero-padded by the 2/3 rule (elements K+1 .. N-K-1 are zero, K = (N-1)/3), as every inverse
// transform of a truncated spectrum is; the first stage then skips the inputs it knows are zero,
// elements 3N/8 .. 5N/8 - 1, which need not be written (pencil_zero_count, pencil_zero).
// The zeros that do have to be written into a zero-padded pencil: elements K+1 .. 3N/8 - 1 and
// 5N/8 .. N-K-1; zero number i of pencil_zero_count is element pencil_zero(i).
template <int N>
__host__ __device__ constexpr int pencil_zero_count() { return 2 * (3 * (N / 8) - (N - 1) / 3 - 1) + 1; }
template <int N>
__device__ __forceinline__ unsigned pencil_zero(unsigned i) {
  constexpr unsigned K = (N - 1) / 3, A = 3 * (N / 8) - K - 1;  // N-K - 5N/8 = A + 1
  return i < A ? K + 1 + i : 5 * (N / 8) + (i - A);
}
// TW: the twiddle table's type; a TwFx table runs an FP64 pencil in fixed point, with its results
// converted on the FP64 pipe if DP and scaled by 2^scale2.
template <int N, int DIR, typename C, int VPT = fft_vpt<C>(), bool ZP = false, bool TWG = false, bool DP = false,
          typename TW>
__device__ __forceinline__ void pencil_fft(C *buf, int t, bool active, const TW *__restrict__ tw, int scale2 = 0) {
  if constexpr (std::is_same<TW, TwFx>::value) {
    static_assert(std::is_same<C, cplx64>::value && VPT == 8, "fixed-point transforms are FP64's, radix 8");
    fx_pencil_fft<N, DIR, ZP, DP>(buf, t, active, tw, scale2);
  } else {
    stockham_stages<N, DIR, 1, C, VPT, ZP, TWG>(buf, t, active, tw);
  }
}

// ---- x passes: two real rows as one pencil, straight from and to their half spectra ----
// Thread t of a group owns the half-spectrum values k = t + i TPP, i < row_vals: in the pencil
// Z[k] = X0[k] + i X1[k] they are inputs i of its first-stage butterfly, and after a forward
// transform the last stage leaves Z[k] in its registers.  Only the mirrored values Z[N-k], which
// belong to thread TPP - t, cross through shared memory: 3 of a butterfly's 8 values (6 of 16)
// instead of all of them twice, with no zeros to write and no index arithmetic per value.
template <int N, int VPT>
__host__ __device__ constexpr int row_vals() {
  return ((N - 1) / 3 + tpp_for<N, VPT>()) / tpp_for<N, VPT>();  // ceil(NX / TPP)
}
template <int N, typename C, int VPT>
struct RowPair {
  static constexpr int NI = row_vals<N, VPT>(), TPP = tpp_for<N, VPT>(), NX = (N - 1) / 3 + 1;
  static_assert((VPT == 8 && NI == 3) || (VPT == 16 && NI == 6), "the kept values are a butterfly's outer inputs");
  static constexpr bool kConst = TPP % sm_pad<C>() == 0;
  C x0[NI], x1[NI];

  __device__ __forceinline__ static bool kept(int t, int i) { return (i + 1) * TPP <= NX || t + i * TPP < NX; }
  // rows at src and src + NX (zeros beyond K and for an inactive group)
  __device__ __forceinline__ void load(const C *__restrict__ src, int t, bool active) {
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      x0[i] = x1[i] = C{0, 0};
      if (active && kept(t, i)) {
        x0[i] = src[t + i * TPP];
        x1[i] = src[NX + t + i * TPP];
      }
    }
  }
  // pencil element N - (t + i TPP)
  template <typename E>
  __device__ __forceinline__ static E *mirror(E *buf, int t, int i) {
    if constexpr (kConst) return buf + sm_at<C>((unsigned)(N - t)) - sm_idx<C>(i * TPP);
    else return buf + sm_at<C>((unsigned)(N - t - i * TPP));
  }
  // pencil element t + r TPP
  template <typename E>
  __device__ __forceinline__ static E *own(E *buf, int t, int r) {
    if constexpr (kConst) return buf + sm_at<C>((unsigned)t) + sm_idx<C>(r * TPP);
    else return buf + sm_at<C>((unsigned)(t + r * TPP));
  }
  // whether element t + r TPP, r >= VPT - NI, is a mirrored kept value
  __device__ __forceinline__ static bool mirrored(int t, int r) { return N - t - r * TPP < NX; }
};

// What a transform leaves in registers: fixed-point values and their scale in FP64 (a TwFx table).
template <typename C, typename TW>
using reg_of = typename std::conditional<std::is_same<TW, TwFx>::value, cfx, C>::type;

// Inverse transform of a row pair (real part: row 0, imaginary part: row 1) into the pencil `buf`,
// or (REG) into `out`: out[q] = element t + q TPP.  DP as in pencil_fft.
template <int N, typename C, int VPT, bool DP, bool REG = false, typename TW>
__device__ __forceinline__ void rows_inverse(C *buf, int t, bool active, RowPair<N, C, VPT> &x,
                                             const TW *__restrict__ tw, reg_of<C, TW> *out = nullptr,
                                             FxScale *out_scale = nullptr) {
  using RP = RowPair<N, C, VPT>;
  constexpr int NI = RP::NI, TPP = RP::TPP;
  if constexpr (std::is_same<TW, TwFx>::value) {
    if (t == 0) x.x0[0].im = x.x1[0].im = 0.0;  // k = 0: the Hermitian part
    uint32_t m = 0u;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      m = max(m, max(fx_hi(x.x0[i].re) & 0x7fffffffu, fx_hi(x.x0[i].im) & 0x7fffffffu));
      m = max(m, max(fx_hi(x.x1[i].re) & 0x7fffffffu, fx_hi(x.x1[i].im) & 0x7fffffffu));
    }
    // a thread's values bound its own inputs of the first stage and their mirror images alike
    const FxScale sc = fx_group_scale<N, false>(fx_max_exp(m), [&](uint32_t mm) {
      uint32_t a = 0u;
#pragma unroll
      for (int i = 0; i < NI; ++i)
        a += fx_size(fx_hi(x.x0[i].re), mm) + fx_size(fx_hi(x.x0[i].im), mm) + fx_size(fx_hi(x.x1[i].re), mm) +
             fx_size(fx_hi(x.x1[i].im), mm);
      return 2u * a;
    });
    cfx *fb = reinterpret_cast<cfx *>(buf);
    cfx v[8];
    auto pack = [&](int i, int64_t a, int64_t b, int64_t c, int64_t d) {
      v[i] = cfx{a - d, b + c};
      if (active && RP::kept(t, i) && (i > 0 || t > 0)) *RP::mirror(fb, t, i) = cfx{a + d, c - b};
    };
    if (!sc.bad) {
      auto fx = [&](double y) { return fx_from_double(fx_hi(y), fx_lo(y), sc.ek); };
#pragma unroll
      for (int i = 0; i < NI; ++i) pack(i, fx(x.x0[i].re), fx(x.x0[i].im), fx(x.x1[i].re), fx(x.x1[i].im));
    } else {
      const uint32_t ek = fx_bad_ek(sc.ek);
      auto fx = [&](double y) { return fx_from_any(fx_hi(y), fx_lo(y), ek); };
#pragma unroll
      for (int i = 0; i < NI; ++i) pack(i, fx(x.x0[i].re), fx(x.x0[i].im), fx(x.x1[i].re), fx(x.x1[i].im));
    }
    group_sync<TPP>();
    if (active) {
#pragma unroll
      for (int r = 8 - NI; r < 8; ++r) {
        v[r] = cfx{0, 0};
        if (RP::mirrored(t, r)) v[r] = *RP::own(fb, t, r);
      }
      fx_dft8<+1, true>(v);
    }
    group_sync<TPP>();
    if (active) {
#pragma unroll
      for (int r = 0; r < 8; ++r) fb[9u * (unsigned)t + r] = v[r];
    }
    group_sync<TPP>();
    fx_stages<N, +1, 8, DP, REG>(fb, t, active, tw, sc, sc.shift, 0, out);
    if constexpr (REG) *out_scale = sc;
  } else {
    C v[VPT];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const C x0 = x.x0[i], x1 = x.x1[i];
      v[i] = C{x0.re - x1.im, x0.im + x1.re};
      if (i == 0 && t == 0) v[0] = C{x0.re, x1.re};  // k = 0: the Hermitian part
      if (active && RP::kept(t, i) && (i > 0 || t > 0)) *RP::mirror(buf, t, i) = C{x0.re + x1.im, x1.re - x0.im};
    }
    group_sync<TPP>();
    if (active) {
#pragma unroll
      for (int r = NI; r < VPT; ++r) {
        v[r] = C{0, 0};
        if (r >= VPT - NI && RP::mirrored(t, r)) v[r] = *RP::own(buf, t, r);
      }
      if constexpr (VPT == 16) dft16<+1, C, true>(v);
      else dft8_first_fma<+1, true>(v);
    }
    group_sync<TPP>();
    if (active) {
      C *wp = buf + sm_at<C>((unsigned)(t * VPT));
#pragma unroll
      for (int r = 0; r < VPT; ++r) wp[sm_idx<C>(r)] = v[r];
    }
    group_sync<TPP>();
    stockham_stages<N, +1, VPT, C, VPT, false, false, REG>(buf, t, active, tw, out);
  }
}

// The half spectra of the two rows of a forward-transformed pencil, from the values its last stage
// left in registers: doubled (the split's factor 1/2 is left out; fixed point: scaled by 2^scale2),
// through `post`, to dst and dst + NX.
template <int N, typename C, int VPT, bool DP, typename E, typename Post>
__device__ __forceinline__ void rows_split(E *z, const FxScale &sc, C *buf, int t, bool active, C *__restrict__ dst,
                                           int scale2, Post post) {
  using RP = RowPair<N, C, VPT>;
  constexpr int NI = RP::NI, TPP = RP::TPP, NX = RP::NX;
  constexpr bool kFx = std::is_same<E, cfx>::value;
  E *eb = reinterpret_cast<E *>(buf);
  // (the last stage has a barrier after its reads)
  if (active) {
#pragma unroll
    for (int r = VPT - NI; r < VPT; ++r)
      if (RP::mirrored(t, r)) *RP::own(eb, t, r) = z[r];
  }
  group_sync<TPP>();
  if (active) {
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      if (!RP::kept(t, i)) continue;
      E zc = z[0];
      if (i > 0 || t > 0) zc = *RP::mirror(eb, t, i);
      const E r0 = {z[i].re + zc.re, z[i].im - zc.im}, r1 = {z[i].im + zc.im, zc.re - z[i].re};
      C y0, y1;
      if constexpr (kFx) {
        const uint32_t be = sc.ek + (uint32_t)(sc.shift + scale2) + 1u;
        auto out = [&](int64_t v) { return DP ? fx_to_double_dp(v, be) : fx_to_double(v, be); };
        y0 = C{out(r0.re), out(r0.im)};
        y1 = C{out(r1.re), out(r1.im)};
      } else {
        y0 = post(r0);
        y1 = post(r1);
      }
      dst[t + i * TPP] = y0;
      dst[NX + t + i * TPP] = y1;
    }
    if constexpr (kFx) {
      if (sc.bad) {
#pragma unroll 1
        for (int k = t; k < NX; k += TPP) {
          fx_bad_out(dst[k], sc);
          fx_bad_out(dst[NX + k], sc);
        }
      }
    }
  }
}

// Forward transform of the pencil `buf` and the half spectra of its two rows (rows_split).
template <int N, typename C, int VPT, bool DP, typename TW, typename Post>
__device__ __forceinline__ void rows_forward(C *buf, int t, bool active, C *__restrict__ dst,
                                             const TW *__restrict__ tw, int scale2, Post post) {
  reg_of<C, TW> z[VPT];
  FxScale sc{};
  if constexpr (std::is_same<TW, TwFx>::value) fx_pencil_fft<N, -1, false, DP, true>(buf, t, active, tw, 0, z, &sc);
  else stockham_stages<N, -1, 1, C, VPT, false, false, true>(buf, t, active, tw, z);
  rows_split<N, C, VPT, DP>(z, sc, buf, t, active, dst, scale2, post);
}

// The same of the values x[r] = element t + r N/8 that the group's threads hold (radix 8).
template <int N, typename C, bool DP, typename TW, typename Post>
__device__ __forceinline__ void rows_forward_from(C *x, C *buf, int t, bool active, C *__restrict__ dst,
                                                  const TW *__restrict__ tw, int scale2, Post post) {
  constexpr int TPP = tpp_for<N, 8>();
  reg_of<C, TW> z[8];
  FxScale sc{};
  if constexpr (std::is_same<TW, TwFx>::value) {
    fx_fft_from<N, -1, false, DP, true>(x, buf, t, active, tw, 0, z, &sc);
  } else {
    if (active) {
      dft8_first_fma<-1, false>(x);
      C *wp = buf + sm_at<C>((unsigned)(t * 8));
#pragma unroll
      for (int r = 0; r < 8; ++r) wp[sm_idx<C>(r)] = x[r];
    }
    group_sync<TPP>();
    stockham_stages<N, -1, 8, C, 8, false, false, true>(buf, t, active, tw, z);
  }
  rows_split<N, C, 8, DP>(z, sc, buf, t, active, dst, scale2, post);
}

// FFT index of kept index j (0..2K) along a truncated axis: j for j <= K, else j - (2K+1) + N.
__device__ __forceinline__ int kept_to_fft(int j, int K, int n) { return j <= K ? j : j - (2 * K + 1) + n; }
// Signed wavenumber of kept index j.
__device__ __forceinline__ int kept_wave(int j, int K) { return j <= K ? j : j - (2 * K + 1); }

// Block-wide reductions with a fixed combination order (deterministic for a fixed block size).
// `red` must hold blockDim.x / 32 doubles; the result is valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    for (int i = 0; i < nw; ++i) s += red[i];
  }
  return s;
}

// The same in the data's precision: FP32 kernels keep the reduction off the FP64 pipe, which on
// GB300 runs at 1/64 of the FP32 rate (widening the result is exact and monotonic, so the maximum
// is the one an FP64 reduction of the widened values would give).
__device__ __forceinline__ float nan_max(float a, float b) {
  if (a != a) return a;
  if (b != b) return b;
  return a > b ? a : b;
}

__device__ __forceinline__ float block_nan_max(float v, float *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = nan_max(v, __shfl_down_sync(0xffffffffu, v, o));
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  float s = 0.0f;
  if (threadIdx.x == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    s = red[0];
    for (int i = 1; i < nw; ++i) s = nan_max(s, red[i]);
  }
  return s;
}

__device__ __forceinline__ double block_nan_max(double v, double *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = nan_max(v, __shfl_down_sync(0xffffffffu, v, o));
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    s = red[0];
    for (int i = 1; i < nw; ++i) s = nan_max(s, red[i]);
  }
  return s;
}

}  // namespace mhd
