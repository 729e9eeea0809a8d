// Update x += scale e of one site of the mixed solver's iterate, in integer limbs.
#pragma once

#include "fx64.cuh"

namespace lqcd {

__host__ __device__ __forceinline__ int fx_bits(float v) {
#ifdef __CUDA_ARCH__
  return __float_as_int(v);
#else
  int u;
  __builtin_memcpy(&u, &v, 4);
  return u;
#endif
}
__host__ __device__ __forceinline__ int fx_clz(unsigned long long v) {  // v > 0
#ifdef __CUDA_ARCH__
  return __clzll((long long)v);
#else
  return __builtin_clzll(v);
#endif
}
__host__ __device__ __forceinline__ long long fx_shift(long long v, int d) {  // v 2^-d, rounded; d <= 62
  return (v + ((1ll << d) >> 1)) >> d;
}

// A scale > 0 as (sh 2^29 + sl) 2^(es - 1080).
struct FxScale {
  int sh, sl, es;
};
__host__ __device__ __forceinline__ FxScale fx_scale(double scale) {
  unsigned long long w;
#ifdef __CUDA_ARCH__
  w = (unsigned long long)__double_as_longlong(scale);
#else
  __builtin_memcpy(&w, &scale, 8);
#endif
  FxScale s;
  s.es = (int)(w >> 52);
  fx_split((long long)((w & 0xfffffffffffffull) | 0x10000000000000ull) << 5, s.sh, s.sl);
  return s;
}

// x += scale e: x[24] in units of 2^(old - 1079), below 2^57 in size (old <= 0: zeros, or
// FX_BAD); the result likewise at the returned exponent.  Each product is rounded to a unit
// of the larger of the two exponents, and the sum normalised once, so that the largest
// component has its 57 bits whatever the number of updates.
__host__ __device__ __forceinline__ int fx_accum_site(const float e[24], const FxScale &s, int old, long long x[24]) {
  constexpr int BAD = -1;
  int m = 0;
#pragma unroll
  for (int k = 0; k < 24; ++k) {
    const int a = fx_bits(e[k]) & 0x7fffffff;
    m = a > m ? a : m;
  }
  const int ee = m >> 23;
  // |scale e| < 2^(E - 1022)
  int E = ee + s.es - 126;
  if (old < 0 || ee == 0xff || s.es >= 0x7ff || E > FX_EMAX) return BAD;
  if (ee == 0 || E < FX_EMIN) return old;
  int Em = E > old ? E : old;
  const int d_new = Em - E, d_old = old > 0 ? (Em - old < 62 ? Em - old : 62) : 0;
  unsigned long long any = 0;
#pragma unroll
  for (int k = 0; k < 24; ++k) {
    // (mantissa 2^4) scale: 57 bits in units of 2^(E' - 1079), E' by the component's own exponent
    const int u = fx_bits(e[k]), ex = (u >> 23) & 0xff, d = ee - ex + d_new;
    int q = ex ? ((u & 0x7fffff) | 0x800000) << 4 : 0;
    q = u < 0 ? -q : q;
    const long long p = (long long)q * s.sh + (((long long)q * s.sl + (1ll << 28)) >> 29);
    x[k] = fx_shift(x[k], d_old) + fx_shift(p, d < 62 ? d : 62);
    any |= (unsigned long long)(x[k] ^ (x[k] >> 63));
  }
  if (any == 0) return 0;
  int up = fx_clz(any) - (64 - 57);  // leading bits that are free; -1: the sum has 58
  if (up > Em - FX_EMIN) up = Em - FX_EMIN;
#pragma unroll
  for (int k = 0; k < 24; ++k) x[k] = up < 0 ? fx_shift(x[k], -up) : x[k] << up;
  Em -= up;
  return Em > FX_EMAX ? BAD : Em;
}

}  // namespace lqcd
