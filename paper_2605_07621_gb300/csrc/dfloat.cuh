// Float-float arithmetic: a value as hi + lo of two FP32 numbers (48
// significant bits), with error-free products (FMA) and sums (Knuth's TwoSum)
// on the FP32 pipe, which this GPU runs about 70 times faster than FP64.
#pragma once

namespace edk {

// a * 2^sh as hi + lo: hi = the leading 24 significant bits (truncated), lo =
// the next 29 rounded to 24, so hi + lo is within 2^-48 |a 2^sh|; built from
// the FP64 bit fields on the integer pipe.  Magnitudes below 2^-126 (after
// scaling) become zero; the caller keeps the scaled magnitude below 2^127.
__device__ __forceinline__ float2 split_scaled(double a, int sh) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(a);
  const unsigned s = (unsigned)(u >> 63) << 31;
  const int E = (int)((u >> 52) & 0x7ffu);
  if (E == 0) return make_float2(0.f, 0.f);  // zero or FP64 subnormal
  const int e = E - 1023 + sh;
  if (e < -126) return make_float2(0.f, 0.f);
  const unsigned long long M = u & 0xFFFFFFFFFFFFFull;
  const float hi = __uint_as_float(s | ((unsigned)(e + 127) << 23) | (unsigned)(M >> 29));
  const unsigned long long R = M & 0x1FFFFFFFull;  // the remaining 29 bits, unit 2^(e - 52)
  if (R == 0) return make_float2(hi, 0.f);
  const int nb = 64 - __clzll((long long)R);  // bit length, 1..29
  int el = e - 53 + nb;                       // exponent of R's leading bit
  unsigned frac;
  if (nb > 24) {
    const int d = nb - 24;
    unsigned long long q = (R + (1ull << (d - 1))) >> d;
    if (q >> 24) {
      q >>= 1;
      ++el;
    }
    frac = (unsigned)q & 0x7FFFFFu;
  } else {
    frac = (unsigned)(R << (24 - nb)) & 0x7FFFFFu;
  }
  if (el < -126) return make_float2(hi, 0.f);
  return make_float2(hi, __uint_as_float(s | ((unsigned)(el + 127) << 23) | frac));
}

// float-float value as FP64 (exact for a normalised pair)
__device__ __forceinline__ double df_to_d(float2 a) { return (double)a.x + (double)a.y; }

// (sh, sl) += (ah + al)(bh + bl): ah bh split exactly into p + e (FMA), p
// added to sh by TwoSum, the rounding error, e and the cross terms into sl
// (al bl, below 2^-48 of the product, is dropped).  The _rn intrinsics keep
// the compiler from contracting or reordering the error-free steps.
__device__ __forceinline__ void df_fma(float& sh, float& sl, float ah, float al, float bh, float bl) {
  const float p = __fmul_rn(ah, bh);
  const float e = fmaf(ah, bh, -p);
  const float s = __fadd_rn(sh, p);
  const float z = __fsub_rn(s, sh);
  const float err = __fadd_rn(__fsub_rn(sh, __fsub_rn(s, z)), __fsub_rn(p, z));
  sh = s;
  sl = __fadd_rn(sl, __fadd_rn(err, fmaf(ah, bl, fmaf(al, bh, e))));
}
__device__ __forceinline__ void df_fma(float2& s, float2 a, float2 b) { df_fma(s.x, s.y, a.x, a.y, b.x, b.y); }

// (sh, sl) += (bh, bl) for two float-float sums (TwoSum of the leading parts)
__device__ __forceinline__ void df_add(float& sh, float& sl, float bh, float bl) {
  const float s = __fadd_rn(sh, bh);
  const float z = __fsub_rn(s, sh);
  const float err = __fadd_rn(__fsub_rn(sh, __fsub_rn(s, z)), __fsub_rn(bh, z));
  sh = s;
  sl = __fadd_rn(sl, __fadd_rn(err, bl));
}
__device__ __forceinline__ void df_add(float2& s, float2 b) { df_add(s.x, s.y, b.x, b.y); }
// the pair renormalised (|lo| at most half an ulp of hi)
__device__ __forceinline__ float2 df_norm(float2 a) {
  const float s = __fadd_rn(a.x, a.y);
  return make_float2(s, __fsub_rn(a.y, __fsub_rn(s, a.x)));
}
__device__ __forceinline__ float2 df_neg(float2 a) { return make_float2(-a.x, -a.y); }
// a b as a normalised pair
__device__ __forceinline__ float2 df_mul(float2 a, float2 b) {
  float2 s = make_float2(0.f, 0.f);
  df_fma(s, a, b);
  return df_norm(s);
}
// warp-wide float-float sum; lane 0's result is the one to use (the low
// parts of the other lanes may differ in their last bits)
__device__ __forceinline__ float2 df_warp_sum(float2 a) {
  for (int o = 16; o > 0; o >>= 1) {
    const float bh = __shfl_xor_sync(0xffffffffu, a.x, o), bl = __shfl_xor_sync(0xffffffffu, a.y, o);
    df_add(a.x, a.y, bh, bl);
  }
  return a;
}

}  // namespace edk
