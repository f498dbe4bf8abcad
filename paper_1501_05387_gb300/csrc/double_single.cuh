// Double-single arithmetic: FP64-like precision from FP32 instructions, for
// the per-vertex work of kernels that would otherwise wait on the FP64 pipe.
#pragma once

#include <stdint.h>

namespace gr {

// Double-single numbers: an unevaluated sum hi + lo of two floats with
// |lo| <= ulp(hi) / 2, about 48 significant bits (Dekker's extended
// precision arithmetic; Knuth's TwoSum for exact sums, the product's error
// from one FMA). FP32 instructions issue many times faster than FP64 on this
// GPU, so BC's per-vertex finish (a reciprocal, a product and sums per lane)
// runs in this form (uint64 path counts keep every value within FP32's
// exponent range): on R-MAT s23 x 64 sources it took the finalize from
// 16.2 to 10.8 ms. The backward's per-edge sums stay in FP64: in this form
// its warp-serial loop became issue-bound (75.7 against 53.5 ms). The _rn
// intrinsics keep the compiler from contracting or reassociating the error
// terms.
struct DS {
  float hi, lo;
};

__device__ __forceinline__ DS ds_two_sum(float a, float b) {  // exact: hi + lo = a + b
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, err};
}

__device__ __forceinline__ DS ds_fast_two_sum(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

__device__ __forceinline__ DS ds_add(DS a, DS b) {
  DS s = ds_two_sum(a.hi, b.hi);
  const DS t = ds_two_sum(a.lo, b.lo);
  s = ds_fast_two_sum(s.hi, __fadd_rn(s.lo, t.hi));
  return ds_fast_two_sum(s.hi, __fadd_rn(s.lo, t.lo));
}

__device__ __forceinline__ DS ds_add_f(DS a, float b) {
  const DS s = ds_two_sum(a.hi, b);
  return ds_fast_two_sum(s.hi, __fadd_rn(s.lo, a.lo));
}

__device__ __forceinline__ DS ds_mul(DS a, DS b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);  // the product's rounding error, exactly
  e = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, e));
  return ds_fast_two_sum(p, e);
}

// 1 / a: the FP32 reciprocal refined by one Newton step in double-single,
// r + r (1 - a r), which squares its relative error (2^-24 -> about 2^-48).
__device__ __forceinline__ DS ds_rcp(DS a) {
  const float r = __frcp_rn(a.hi);
  const DS ar = ds_mul(a, DS{r, 0.f});
  const DS res = ds_add(DS{1.f, 0.f}, DS{-ar.hi, -ar.lo});
  return ds_add_f(ds_mul(DS{r, 0.f}, res), r);
}

// A 16-bit integer as a float without a conversion instruction: 2^23 + p
// is a float whose low mantissa bits are p.
__device__ __forceinline__ float u16_to_float(uint32_t p) {
  return __fsub_rn(__int_as_float(0x4B000000 | (int)p), 8388608.f);
}

// A uint64 path count as double-single (its four 16-bit pieces, each exact
// as a float, summed without losing more than the last of 64 bits' worth).
__device__ __forceinline__ DS ds_from_u64(unsigned long long c) {
  if (c >> 32 == 0ull)  // the same sum without the pieces that are 0
    return ds_fast_two_sum(__fmul_rn(u16_to_float((uint32_t)c >> 16), 65536.f),
                           u16_to_float((uint32_t)c & 0xFFFFu));
  DS r{__fmul_rn(u16_to_float((uint32_t)(c >> 48)), 281474976710656.f), 0.f};  // 2^48
  r = ds_add_f(r, __fmul_rn(u16_to_float((uint32_t)(c >> 32) & 0xFFFFu), 4294967296.f));
  r = ds_add_f(r, __fmul_rn(u16_to_float((uint32_t)(c >> 16) & 0xFFFFu), 65536.f));
  return ds_add_f(r, u16_to_float((uint32_t)c & 0xFFFFu));
}

// Conversions between FP64 and double-single take their turn in the FP64
// pipe like arithmetic, three for each direction; for positive values well
// inside FP32's exponent range the bits are moved with integers instead
// (to_double keeps one FP64 addition). The high part is rounded to nearest,
// the rest, a signed 29-bit integer, to FP32: as the conversions do it.
__device__ __forceinline__ DS ds_from_double(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(b >> 52) - 1023;  // above 1023 for a negative x
  if (b == 0ull) return {0.f, 0.f};     // a vertex without children, often
  if (e < -70 || e > 120) {  // very small, very large, negative, not finite
    const float hi = __double2float_rn(x);
    return {hi, __double2float_rn(x - (double)hi)};
  }
  const unsigned long long up = (b + (1ull << 28)) >> 29;  // rounded to FP32's 23 bits
  const int rest = (int)(b & 0x1FFFFFFFull) - (up != (b >> 29) ? 1 << 29 : 0);
  const float hi = __uint_as_float((uint32_t)(up - ((unsigned long long)(1023 - 127) << 23)));
  return {hi, __fmul_rn(__int2float_rn(rest), __uint_as_float((uint32_t)(e - 52 + 127) << 23))};
}

__device__ __forceinline__ double ds_to_double(DS a) {
  const uint32_t h = __float_as_uint(a.hi), l = __float_as_uint(a.lo);
  const uint32_t eh = (h >> 23) & 0xFFu, el = (l >> 23) & 0xFFu;
  if (eh - 1u >= 0xFEu) return (double)a.hi + (double)a.lo;  // 0, subnormal, not finite
  const double dh = __longlong_as_double(
      (long long)(((unsigned long long)(h & 0x80000000u) << 32) |
                  (((unsigned long long)(h & 0x7FFFFFFFu) << 29) + ((unsigned long long)(1023 - 127) << 52))));
  // a subnormal low part is below 2^-126: next to nothing beside hi
  const double dl = el == 0u ? 0.0
                             : __longlong_as_double((long long)(
                                   ((unsigned long long)(l & 0x80000000u) << 32) |
                                   (((unsigned long long)(l & 0x7FFFFFFFu) << 29) +
                                    ((unsigned long long)(1023 - 127) << 52))));
  return dh + dl;
}

__device__ __forceinline__ DS shfl_xor_ds(DS a, int o) {
  return {__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}

// |a - b| exactly, as hi + lo.
__device__ __forceinline__ DS ds_abs_diff(float a, float b) {
  const DS d = ds_two_sum(a, -b);
  return d.hi < 0.f ? DS{-d.hi, -d.lo} : d;
}

// A sum of floats as three floats: what an addition rounds off at one goes to
// the next, so only the last one rounds, below 2^-72 of the sum (FP64: 2^-53).
struct TripleSum {
  float a, b, c;
};

__device__ __forceinline__ void ts_add(TripleSum &s, float x) {
  const DS p = ds_two_sum(s.a, x), q = ds_two_sum(s.b, p.lo);
  s.a = p.hi;
  s.b = q.hi;
  s.c = __fadd_rn(s.c, q.lo);
}

// Rare cases in FP64 are calls: inlined, their few instructions are issued for
// every warp, predicated off, and hold the FP64 pipe all the same (87 cycles a
// vertex in PageRank's update, 27-90 us of it instead of 17 at R-MAT 2^21).
static __device__ __noinline__ double add_f32_to_f64(double r, float c) { return r + (double)c; }
static __device__ __noinline__ float fma_rounded_once_more(double x, float d, float s) {
  return __double2float_rn(fma((double)d, (double)s, x));
}

__device__ __forceinline__ double ts_to_double(const TripleSum &s) {
  const double r = ds_to_double({s.a, s.b});
  return s.c != 0.f ? add_f32_to_f64(r, s.c) : r;
}

// (float)(x + d * s) as FP64 arithmetic gives it, for x = xh + xl to 48 bits
// and finite, non-negative values. The product and the sums are taken apart
// into exact parts; what is rounded off on the way, under 2^-47 of the result,
// matters only where the exact sum lies as near to the middle of two floats,
// and there (2^-20 of half a unit on either side, once in 200,000) FP64 decides.
__device__ __forceinline__ float fma_f64_to_f32(double x, float xh, float xl, float d, float s) {
  const float p = __fmul_rn(d, s);  // p + e = d * s exactly
  const float e = __fmaf_rn(d, s, -p);
  const DS t = ds_two_sum(xh, p);
  const DS r = ds_two_sum(t.hi, __fadd_rn(t.lo, __fadd_rn(e, xl)));
  if (__fadd_rn(r.hi, __fmul_rn(r.lo, 1.f + 0x1p-20f)) != r.hi)
    return fma_rounded_once_more(x, d, s);
  return r.hi;
}

}  // namespace gr
