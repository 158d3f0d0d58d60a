// fixed.cuh -- FP64-accurate sums of products on the integer multiply-add units.
//
// GB300 issues 2 FP64 multiply-adds per clock and SM but 30 exact 32 x 32 + 64-bit integer ones (both
// measured over every SM).  A number x with |x| < 2^e is therefore held as two limbs,
//   x ~ (h 2^28 + l) 2^(e - 56),   |h| <= 2^28,  0 <= l < 2^28,
// rounded to nearest (fx_round) or truncated with a one below the last bit (fx_limbs), and a product is
// four exact multiply-adds into three 64-bit sums
//   H += h h',  M += h l' + l h',  L += l l'      (weights 2^56, 2^28, 1).
// 64 products fit before a sum can overflow (|M| <= 64 * 2 * 2^28 * (2^28 - 1) < 2^63), and so do the
// differences of two sums that share them.  The sum itself
// is exact: against the rounding of FP64 partial sums (about 2^-53 of their size at each step) only the
// limbs' 2^-57 of the largest entry is left.  7.5 products a clock and SM, about 4 times the FP64 rate.
//
// The Krylov basis is stored in the same scale, 60 bits a number: x = F 2^(e - 60), F a 64-bit integer
// rounded to nearest, e one exponent per column (the largest entry's).  That is exact for every FP64
// entry within 2^-8 of the column's largest and off by 2^-61 of the largest below; an entry costs three
// integer instructions to become limbs, against about 19 from FP64.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace jtr {

struct fx2 {
  int h, l;
};

// Exponent field of |x| (0 for zero and subnormals): |x| < 2^(field + 1 - 1023).
__device__ __forceinline__ int fx_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// Limbs of x for K = 1023 + e, |x| < 2^e.  Subnormals count as zero.  MinusZero: x may be -0.0.
template <bool MinusZero>
__device__ __forceinline__ fx2 fx_limbs(double x, int K) {
  const int hi = __double2hiint(x);
  const int ex = (hi >> 20) & 0x7ff;
  const uint32_t nz = (uint32_t)min(ex, 1), live = 0u - nz;
  const uint32_t lo = (uint32_t)__double2loint(x) & live;
  const uint32_t mh = (((uint32_t)hi & 0xfffffu) | 0x100000u) & live;   // K may be as low as 1
  const uint32_t th = __funnelshift_l(lo, mh, 11), tl = lo << 11;   // mantissa, left-aligned in 64 bits
  const uint32_t s = (uint32_t)(K - ex + 7);                        // >= 8; (th, tl) >> s is 2 floor(|x| 2^(55-e)) + a bit
  uint32_t h, g;
  asm("shr.u32 %0, %1, %2;" : "=r"(h) : "r"(th), "r"(s - 4u));      // clamps: 0 from 32 on
  asm("shf.r.clamp.b32 %0, %1, %2, %3;" : "=r"(g) : "r"(tl), "r"(th), "r"(s));
  asm("shr.u32 %0, %0, %1;" : "+r"(g) : "r"((uint32_t)max((int)s - 32, 0)));
  int sm = hi >> 31;
  if (MinusZero) sm &= -(int)nz;
  fx2 r;
  r.h = (int)(h ^ (uint32_t)sm);
  r.l = (int)(((g ^ (uint32_t)sm) & 0x0ffffffeu) | nz);   // -F = ~F | 1 for the odd F
  return r;
}

// One complex number of the basis.
struct alignas(16) fxc {
  long long re, im;
};
// x 2^(60 - e) rounded to nearest, for K = 1023 + e, |x| < 2^e
__device__ __forceinline__ long long fx_store(double x, int K) {
  const long long b = __double_as_longlong(x);
  const int ex = (int)(b >> 52) & 0x7ff;
  const int s = K - ex - 1;                                        // right shift of the mantissa at bit 59
  if (ex == 0 || s > 61) return 0;
  unsigned long long t = ((unsigned long long)b & 0xfffffffffffffull) | 0x10000000000000ull;
  t <<= 7;
  if (s > 0) t = (t + (1ull << (s - 1))) >> s;
  return b < 0 ? -(long long)t : (long long)t;
}
__device__ __forceinline__ double fx_load(long long F, int K);     // the FP64 number nearest F 2^(e - 60)
// Limbs of a stored number, rounded to nearest.
__device__ __forceinline__ fx2 fx_round(long long F) {
  F += 8;
  return fx2{(int)(F >> 32), (int)((unsigned)F >> 4)};
}

struct FxAcc {   // one sum
  long long H, M, L;
};
__device__ __forceinline__ void fx_zero(FxAcc& a) { a.H = a.M = a.L = 0; }
// s += x y, exact.  Written as its two halves, which become one wide multiply-add; mad.wide.s32 becomes a
// multiply and a separate 64-bit add.
__device__ __forceinline__ void fx_mad(long long& s, int x, int y) {
  asm("{\n\t.reg .u32 l, h;\n\tmov.b64 {l, h}, %0;\n\tmad.lo.cc.s32 l, %1, %2, l;\n\tmadc.hi.s32 h, %1, %2, h;\n\t"
      "mov.b64 %0, {l, h};\n\t}"
      : "+l"(s)
      : "r"(x), "r"(y));
}
__device__ __forceinline__ void fx_mac(FxAcc& a, fx2 x, fx2 y) {
  fx_mad(a.H, x.h, y.h);
  fx_mad(a.M, x.h, y.l);
  fx_mad(a.M, x.l, y.h);
  fx_mad(a.L, x.l, y.l);
}
__device__ __forceinline__ FxAcc fx_sum(const FxAcc& a, const FxAcc& b) { return FxAcc{a.H + b.H, a.M + b.M, a.L + b.L}; }
__device__ __forceinline__ FxAcc fx_scale(const FxAcc& a, int sign) { return sign > 0 ? a : FxAcc{-a.H, -a.M, -a.L}; }
__device__ __forceinline__ FxAcc fx_diff(const FxAcc& a, const FxAcc& b) { return FxAcc{a.H - b.H, a.M - b.M, a.L - b.L}; }
__device__ __forceinline__ fx2 fx_neg(fx2 a) { return fx2{-a.h, -a.l}; }

// Warp sum of an accumulator as four exact pieces, the same in every lane:
// total = p0 + 2^26 p1 + 2^52 p2 + 2^-26 p3 in units of 2^56 (p3 drops the last two of 28 bits a lane).
__device__ __forceinline__ int4 fx_warp_sum(const FxAcc& a) {
  const long long t = a.M + (a.L >> 28);
  const long long H = a.H + (t >> 28);
  int4 p;
  p.w = (int)__reduce_add_sync(0xffffffffu, ((unsigned)t & 0x0fffffffu) >> 2);
  p.x = (int)__reduce_add_sync(0xffffffffu, (unsigned)H & 0x3ffffffu);
  p.y = (int)__reduce_add_sync(0xffffffffu, (unsigned)(H >> 26) & 0x3ffffffu);
  p.z = __reduce_add_sync(0xffffffffu, (int)(H >> 52));
  return p;
}
// The double nearest (hi 2^64 + lo) 2^k (ties away; 0 below the normal range), by integer operations: an
// FP64 instruction holds its pipe for 64 clocks whatever it does.
__device__ __forceinline__ double fx_to_double(long long hi, unsigned long long lo, int k) {
  const unsigned long long sign = hi < 0 ? 0x8000000000000000ull : 0ull;
  if (hi < 0) {
    lo = ~lo + 1ull;
    hi = ~hi + (lo == 0 ? 1 : 0);
  }
  unsigned long long t = (unsigned long long)hi;
  int lz;
  if (t) {
    lz = __clzll((long long)t);
    if (lz) t = (t << lz) | (lo >> (64 - lz));
  } else {
    if (!lo) return 0.0;
    const int z = __clzll((long long)lo);
    lz = 64 + z;
    t = lo << z;
  }
  const int e = 127 - lz + k + 1023;        // biased exponent of the leading bit
  if (e < 1) return 0.0;
  if (e > 2046) return __longlong_as_double((long long)(sign | 0x7ff0000000000000ull));
  const unsigned long long m = (t >> 11) + ((t >> 10) & 1ull);
  return __longlong_as_double((long long)(sign | ((((unsigned long long)(e - 1)) << 52) + m)));
}
// The warp sum's value for factors |x| < 2^(Kx - 1023), |y| < 2^(Ky - 1023).
__device__ __forceinline__ double fx_value(int4 p, int Kx, int Ky) {
  unsigned long long lo = (unsigned long long)(unsigned)p.w + ((unsigned long long)(unsigned)p.x << 26);
  const unsigned long long add = (unsigned long long)(unsigned)p.y << 52;
  lo += add;
  const long long hi = ((long long)(unsigned)p.y >> 12) + ((long long)p.z << 14) + (lo < add ? 1 : 0);
  return fx_to_double(hi, lo, (Kx - 1023) + (Ky - 1023) - 56 - 26);
}

// One lane's exact sum as FP64, factors below 1 and 2^(K - 1023).
__device__ __forceinline__ double fx_lane_value(const FxAcc& a, int K) {
  const long long t = a.M + (a.L >> 28), H = a.H + (t >> 28);
  return fx_to_double(H >> 36, ((unsigned long long)H << 28) | ((unsigned long long)t & 0x0fffffffull), K - 1023 - 84);
}

// Sum of the cnt doubles src[0], src[stride], ... over a warp, as limbs on the scale of the largest one (the
// power of two above it): off from the exact sum by at most 2^-56 of the scale a term (its limbs) and a lane (the
// bit that the 32 low limbs lose to fit their sum into 32 bits), before it is rounded once.  Every lane gets the
// result.
__device__ __forceinline__ double fx_warp_dsum(const double* src, int stride, int first, int cnt, int step) {
  int ex = 0;
  for (int i = first; i < cnt; i += step) ex = max(ex, fx_field(src[(int64_t)i * stride]));
  ex = __reduce_max_sync(0xffffffffu, ex);
  if (ex == 0x7ff) {   // infinities and NaN go their FP64 way
    double t = 0.0;
    for (int i = first; i < cnt; i += step) t += src[(int64_t)i * stride];
    return warp_sum(t);
  }
  const int K = ex + 1;
  long long sh = 0, sl = 0;
  for (int i = first; i < cnt; i += step) {
    const fx2 v = fx_limbs<true>(src[(int64_t)i * stride], K);
    sh += v.h;
    sl += v.l;
  }
  sh += sl >> 28;                                            // value (sh 2^28 + sl) 2^(K - 1023 - 56)
  const unsigned l = (unsigned)sl & 0x0fffffffu;
  const unsigned w = __reduce_add_sync(0xffffffffu, l >> 1);
  const unsigned a0 = __reduce_add_sync(0xffffffffu, (unsigned)sh & 0x3ffffffu);
  const int a1 = __reduce_add_sync(0xffffffffu, (int)(sh >> 26));
  const long long t = ((long long)a1 << 26) + (long long)a0;   // units 2^28; w in units 2^1
  const unsigned long long lo = ((unsigned long long)t << 27) + w;
  const long long hi = (t >> 37) + (lo < (unsigned long long)w ? 1 : 0);
  return fx_to_double(hi, lo, K - 1023 - 56 + 1);
}

// Sum of one double a lane, as fx_warp_dsum; every lane gets it.
__device__ __forceinline__ double fx_warp_total(double v) {
  const int ex = __reduce_max_sync(0xffffffffu, fx_field(v));
  if (ex == 0x7ff) return warp_sum(v);
  const int K = ex + 1;
  const fx2 t = fx_limbs<true>(v, K);
  const unsigned w = __reduce_add_sync(0xffffffffu, (unsigned)t.l >> 1);          // units 2^1
  const int a = __reduce_add_sync(0xffffffffu, t.h >> 14), b = __reduce_add_sync(0xffffffffu, t.h & 0x3fff);
  const long long hs = ((long long)a << 14) + b;                                  // units 2^28
  const unsigned long long lo = ((unsigned long long)hs << 27) + w;
  const long long hi = (hs >> 37) + (lo < (unsigned long long)w ? 1 : 0);
  return fx_to_double(hi, lo, K - 1023 - 56 + 1);
}

// The high word of 2^-30 ynorm / ((j+1)(j+4)), the line between small and large coefficients of an update
// (UpdFx in gsfx.cu).  A coefficient is compared by its own high word, fx_high: no FP64 instruction, and the
// whole range of FP64 (as FP32 numbers both sides became infinite above 3.4e38, and every column small).  An
// infinite or NaN ynorm gives 0, so that every nonzero coefficient is large.
__device__ __forceinline__ int fx_high(double x) { return __double2hiint(x) & 0x7fffffff; }
__device__ __forceinline__ int fx_line(double ynorm, int j) {
  const int y = fx_high(ynorm), f = y >> 20;
  if (f == 0x7ff) return 0;
  const float t = __int_as_float(0x3f800000 | ((y & 0xfffff) << 3)) *   // the mantissa, in [1, 2)
                  (9.3132257e-10f / ((float)(j + 1) * (float)(j + 4)));
  const int b = __float_as_int(t), e = (b >> 23) - 127 + f;
  return e < 1 ? 0 : (e << 20) | ((b >> 3) & 0xfffff);
}
// Is a coefficient of high word m large in a column whose exponent is `spread` >= 0 above the least?
__device__ __forceinline__ bool fx_large(int m, int spread, int line) {
  return m != 0 && (unsigned)m + ((unsigned)spread << 20) > (unsigned)line;   // both below 2^31
}

__device__ __forceinline__ double fx_load(long long F, int K) { return fx_to_double(F >> 63, (unsigned long long)F, K - 1023 - 60); }

}  // namespace jtr
