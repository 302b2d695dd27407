// Complex helpers shared by the device code of this library (double2 / float2).
#pragma once
#include <cuda_runtime.h>

namespace dks {

template <typename V> struct RealOf;
template <> struct RealOf<double2> { using T = double; };
template <> struct RealOf<float2> { using T = float; };

template <typename V>
__device__ __host__ __forceinline__ V cadd(V a, V b) { return V{a.x + b.x, a.y + b.y}; }
template <typename V>
__device__ __host__ __forceinline__ V csub(V a, V b) { return V{a.x - b.x, a.y - b.y}; }
template <typename V>
__device__ __host__ __forceinline__ V cmul(V a, V b) {
  return V{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
// conj(a) * b
template <typename V>
__device__ __host__ __forceinline__ V cmulc(V a, V b) {
  return V{a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x};
}
// c + a b and c + conj(a) b as four fused multiply-adds
__device__ __forceinline__ float2 cfma(float2 a, float2 b, float2 c) {
  return float2{fmaf(-a.y, b.y, fmaf(a.x, b.x, c.x)), fmaf(a.y, b.x, fmaf(a.x, b.y, c.y))};
}
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 c) {
  return double2{fma(-a.y, b.y, fma(a.x, b.x, c.x)), fma(a.y, b.x, fma(a.x, b.y, c.y))};
}
__device__ __forceinline__ float2 cfmac(float2 a, float2 b, float2 c) {
  return float2{fmaf(a.y, b.y, fmaf(a.x, b.x, c.x)), fmaf(-a.y, b.x, fmaf(a.x, b.y, c.y))};
}
__device__ __forceinline__ double2 cfmac(double2 a, double2 b, double2 c) {
  return double2{fma(a.y, b.y, fma(a.x, b.x, c.x)), fma(-a.y, b.x, fma(a.x, b.y, c.y))};
}
// c + a b, given ib = i b, as two packed FP32 multiply-adds: the products, their order and
// their roundings of cfma, in half the issue slots
__device__ __forceinline__ float2 cfma2(float2 a, float2 b, float2 ib, float2 c) {
  return __ffma2_rn(float2{a.y, a.y}, ib, __ffma2_rn(float2{a.x, a.x}, b, c));
}
template <typename V>
__device__ __forceinline__ V mul_i(V a) { return V{-a.y, a.x}; }
template <typename V, typename T>
__device__ __forceinline__ V cscale(V a, T s) { return V{a.x * s, a.y * s}; }

__device__ __forceinline__ double2 to_d2(double2 v) { return v; }
__device__ __forceinline__ double2 to_d2(float2 v) { return double2{(double)v.x, (double)v.y}; }
template <typename V> __device__ __forceinline__ V from_d2(double2 v);
template <> __device__ __forceinline__ double2 from_d2<double2>(double2 v) { return v; }
template <> __device__ __forceinline__ float2 from_d2<float2>(double2 v) {
  return float2{(float)v.x, (float)v.y};
}

}  // namespace dks

namespace dks {

// ---------------------------------------------------------------- double-float arithmetic
// A value is the unevaluated sum h + l of two floats (about 48 significant bits).  Sums use
// Knuth's two-sum and products Dekker's exact product via fma, each followed by a fast
// renormalisation; all of it runs on the FP32 units.
struct dfl {
  float h, l;
};
__device__ __forceinline__ dfl df_from(double x) {
  const float h = (float)x;
  return dfl{h, (float)(x - (double)h)};
}
__device__ __forceinline__ double df_val(dfl a) { return (double)a.h + (double)a.l; }
// double -> (h, l) with integer operations (no FP64 unit): h = x with the mantissa truncated to
// 24 bits, l = the remaining 29 bits converted to FP32 (rounded), h + l = x to 2^-47 relative.
// Zero and magnitudes outside [2^-74, 2^127) take the FP64 conversions.  For bulk splits
// (k_split_df, shared-memory staging).
__device__ __forceinline__ dfl df_from_bits(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const unsigned hi32 = (unsigned)(u >> 32), lo32 = (unsigned)u;
  const int e = (int)((hi32 >> 20) & 0x7ffu);
  if (e < 949 || e > 1149) return df_from(x);
  const unsigned sign = hi32 & 0x80000000u;
  const float h = __uint_as_float(sign | ((unsigned)(e - 896) << 23) | ((hi32 & 0xfffffu) << 3) | (lo32 >> 29));
  const float lv = __uint2float_rn(lo32 & 0x1fffffffu) * __uint_as_float((unsigned)(e - 948) << 23);
  return dfl{h, sign ? -lv : lv};
}
// out of line, so that the FP64 instructions are not if-converted into the callers' main path (a
// predicated-off FP64 instruction still takes its slot of that unit)
static __device__ __noinline__ dfl df_from_call(double x) { return df_from(x); }
// the same with h rounded to nearest (ties away from zero) instead of truncated, so that l keeps 24
// of the remaining bits: h + l = x to 2^-49 relative.  (A conversion through the FP64 unit costs
// four of its instructions, each worth some 75 FP32 ones on this part.)
__device__ __forceinline__ dfl df_split_rn(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((unsigned)(u >> 52) & 0x7ffu);
  if (e < 949 || e > 1149) return df_from_call(x);
  const unsigned long long t = u + 0x10000000ull;            // a carry into the exponent is right
  const unsigned sign = (unsigned)(u >> 32) & 0x80000000u;
  const unsigned hb = (unsigned)((t & 0x7fffffffffffffffull) >> 29) - (896u << 23);
  const int r = (int)((unsigned)t & 0x1fffffffu) - 0x10000000;   // |x| - |h| in units of 2^(e - 1075)
  const float lv = __int2float_rn(r) * __uint_as_float((unsigned)(e - 948) << 23);
  return dfl{__uint_as_float(hb | sign), __uint_as_float(__float_as_uint(lv) ^ sign)};
}
__device__ __forceinline__ dfl df_add(dfl a, dfl b) {
  const float s = a.h + b.h;
  const float bb = s - a.h;
  float e = (a.h - (s - bb)) + (b.h - bb);
  e += a.l + b.l;
  const float h = s + e;
  return dfl{h, e - (h - s)};
}
__device__ __forceinline__ dfl df_neg(dfl a) { return dfl{-a.h, -a.l}; }
// a + x for a float x (two-sum of the leading parts, then a fast renormalisation)
__device__ __forceinline__ dfl df_add_f(dfl a, float x) {
  const float s = a.h + x;
  const float bb = s - a.h;
  const float e = ((a.h - (s - bb)) + (x - bb)) + a.l;
  const float h = s + e;
  return dfl{h, e - (h - s)};
}
__device__ __forceinline__ dfl df_mul(dfl a, dfl b) {
  const float p = a.h * b.h;
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  const float h = p + e;
  return dfl{h, e - (h - p)};
}

// (h + l) 2^k as a double, from a normalised double-float pair (|l| <= ulp(h) / 2), with integer
// operations only (FP64 instructions, conversions included, are slow on this part): the
// significands are aligned in a 64-bit integer; exact up to a truncation below 2^-52 of h.
// The caller keeps the result's exponent in range (|k| <= 60 and h a normal FP32 number).
__device__ __forceinline__ double df_to_double(float h, float l, int k) {
  const unsigned hb = __float_as_uint(h), lb = __float_as_uint(l);
  const int eh = (int)((hb >> 23) & 255u);
  if (eh == 0) return 0.0;
  if (eh == 255) return __longlong_as_double(0x7FF8000000000000LL);   // NaN or infinity
  long long m = (long long)((hb & 0x7FFFFFu) | 0x800000u) << 29;   // implicit bit at position 52
  const int el = (int)((lb >> 23) & 255u);
  if (el) {
    const int d = eh - el;                                          // >= 24 for a normalised pair
    if (d < 53) {
      const long long ml = ((long long)((lb & 0x7FFFFFu) | 0x800000u) << 29) >> d;
      m += ((hb ^ lb) >> 31) ? -ml : ml;
    }
  }
  long long e = (long long)(eh - 127 + 1023 + k);
  if (m < (1LL << 52)) {   // a borrow took the leading bit
    m <<= 1;
    --e;
  }
  return __longlong_as_double(((long long)(hb >> 31) << 63) | (e << 52) | (m & ((1LL << 52) - 1)));
}

// the same for any pair: below 2^-63 (where the integer form drops a trailing part under 2^-126, and then
// a leading part that is a subnormal number) and for infinities and NaN the sum is formed by the FP64
// unit, out of line as in df_from_call
static __device__ __noinline__ double df_val_call(float h, float l) { return (double)h + (double)l; }
__device__ __forceinline__ double df_to_double_any(float h, float l) {
  const unsigned hb = __float_as_uint(h);
  const unsigned eh = (hb >> 23) & 255u;
  if (eh >= 64u && eh < 255u) return df_to_double(h, l, 0);
  return hb << 1 ? df_val_call(h, l) : 0.0;   // zero pairs are common (a zero block): no call
}

// complex double-float (16 bytes, the size of a double2)
struct cdf {
  dfl re, im;
};
__device__ __forceinline__ cdf cadd(cdf a, cdf b) { return cdf{df_add(a.re, b.re), df_add(a.im, b.im)}; }
__device__ __forceinline__ cdf csub(cdf a, cdf b) {
  return cdf{df_add(a.re, df_neg(b.re)), df_add(a.im, df_neg(b.im))};
}
__device__ __forceinline__ cdf cmul(cdf a, cdf b) {
  return cdf{df_add(df_mul(a.re, b.re), df_neg(df_mul(a.im, b.im))), df_add(df_mul(a.re, b.im), df_mul(a.im, b.re))};
}

// Index checks of the debug build (-DDKS_DEBUG, libdks_debug.so): a failed check records its code
// in its translation unit's status word (the first failure is kept) and the caller skips the
// access.  In the product build the check is `true` and the comparisons compile away.
#ifdef DKS_DEBUG
static __device__ unsigned int g_dks_check = 0u;
__device__ __forceinline__ bool dks_ok(bool ok, unsigned code) {
  if (!ok) atomicCAS(&g_dks_check, 0u, code);
  return ok;
}
#else
__device__ __forceinline__ bool dks_ok(bool, unsigned) { return true; }
#endif
// check codes: kernel in the top byte, the failing item's low 24 bits below it
constexpr unsigned kChkStickInverse = 1u << 24, kChkStickForward = 2u << 24, kChkStickForwardKs = 3u << 24,
                   kChkPlane = 4u << 24, kChkPlaneDensity = 5u << 24, kChkUnpermute = 6u << 24;

}  // namespace dks
