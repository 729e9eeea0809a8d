// Products of FP64 colour vectors with SU(3) links on the integer units.
//
// GB300's FP64 pipe takes 64 cycles per warp-wide fused multiply-add; a 32 x 32 -> 64
// bit integer multiply-add (mad.wide) takes 2 (own probe: 0.60 and 16.9 T lane
// operations/s).  A link entry, |u| <= 1, is held as the integer u 2^58 in two
// balanced 29-bit limbs, and the components of a neighbour spinor as integers below
// 2^(53 + SH) relative to the power of two above the largest of them, split the same
// way (SH: what the sums over all neighbours leave free of the 63 bits).
// Then one real multiply-add is three integer ones (high x high into one 64-bit sum,
// the two mixed products into another; low x low is below the last bit), and the
// rounding errors, a few 2^-57 of the neighbour's largest component, stay below those
// of FP64 arithmetic (2^-53 of each partial sum).  Contributions of neighbours with
// different exponents are aligned by shifts as they are added up.
//
// Range: a contribution whose largest component lies outside [2^-923, 2^877), or is
// not finite, sets `bad`, and the caller evaluates that site in FP64.
#pragma once

#include <cuda_runtime.h>

namespace lqcd {

constexpr int FX_EMIN = 100, FX_EMAX = 1900;  // biased exponents of the largest component

// u in [-1, 1] (a little above is fine) -> (high, low) limbs of rint-free u 2^58
__host__ __device__ __forceinline__ long long fx_link(double u) {
#ifdef __CUDA_ARCH__
  const unsigned long long w = (unsigned long long)__double_as_longlong(u);
#else
  unsigned long long w;
  __builtin_memcpy(&w, &u, 8);
#endif
  const int ex = (int)((w >> 52) & 0x7ff);
  const int s = 1023 - ex < 0 ? 0 : (1023 - ex > 63 ? 63 : 1023 - ex);
  const unsigned long long m = (((w & 0xfffffffffffffull) | 0x10000000000000ull) << 6) >> s;
  return (w >> 63) ? -(long long)m : (long long)m;
}
__host__ __device__ __forceinline__ void fx_split(long long v, int &h, int &l) {  // v = h 2^29 + l, |l| <= 2^28
  l = (int)((unsigned)v << 3) >> 3;
  h = (int)((v + (1ll << 28)) >> 29);
}
__host__ __device__ __forceinline__ int4 fx_link_entry(double re, double im) {
  int4 r;
  fx_split(fx_link(re), r.x, r.y);
  fx_split(fx_link(im), r.z, r.w);
  return r;
}

// the larger of m and |v| as high words of the bit patterns (their exponents decide)
__device__ __forceinline__ int fx_max(int m, double2 v) {
  return max(m, max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff));
}
// v 2^(1075 + SH - E) for |v| < 2^(E - 1022), towards zero
template <int SH> __device__ __forceinline__ long long fx_int(double v, int E) {
  const int hi = __double2hiint(v), lo = __double2loint(v);
  const int s = min(E - ((hi >> 20) & 0x7ff), 63);
  const unsigned mh = (hi & 0xfffff) | 0x100000;
  const unsigned long long m = (((unsigned long long)__funnelshift_l(lo, mh, SH)) << 32) | ((unsigned)lo << SH);
  const long long neg = hi >> 31;
  return ((long long)(m >> s) ^ neg) - neg;
}
__device__ __forceinline__ long long fx_mad(int a, int b, long long c) { return c + (long long)a * b; }

// X = U h (FWD) or U^+ h for a colour vector h in limbs (rh, rl the real, ih, il the
// imaginary parts): 108 integer multiply-adds
template <bool FWD>
__device__ __forceinline__ void fx_su3(const int4 u[9], const int rh[3], const int rl[3], const int ih[3],
                                       const int il[3], long long X[6]) {
  int nh[3], nl[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    nh[k] = FWD ? -ih[k] : -rh[k];  // the part that enters with a minus sign
    nl[k] = FWD ? -il[k] : -rl[k];
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    long long ar = 0, br = 1ll << 28, ai = 0, bi = 1ll << 28;  // b: rounded when shifted
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int4 m = FWD ? u[a * 3 + b] : u[b * 3 + a];  // U, or U^+ = conj of the transpose
      const int ph = FWD ? nh[b] : ih[b], pl = FWD ? nl[b] : il[b];
      const int qh = FWD ? rh[b] : nh[b], ql = FWD ? rl[b] : nl[b];
      ar = fx_mad(m.x, rh[b], ar);
      br = fx_mad(m.x, rl[b], br);
      br = fx_mad(m.y, rh[b], br);
      ar = fx_mad(m.z, ph, ar);
      br = fx_mad(m.z, pl, br);
      br = fx_mad(m.w, ph, br);
      ai = fx_mad(m.x, ih[b], ai);
      bi = fx_mad(m.x, il[b], bi);
      bi = fx_mad(m.y, ih[b], bi);
      ai = fx_mad(m.z, qh, ai);
      bi = fx_mad(m.z, ql, bi);
      bi = fx_mad(m.w, qh, bi);
    }
    X[2 * a] = ar + (br >> 29);
    X[2 * a + 1] = ai + (bi >> 29);
  }
}
__device__ __forceinline__ long long fx_negif(long long v, long long mask) { return (v ^ mask) - mask; }

// acc 2^(Ea - 1075 - SH) as FP64
template <int SH> __device__ __forceinline__ double fx_double(long long acc, int Ea) {
  const double v = __ll2double_rn(acc);
  return acc == 0 ? 0.0 : __hiloint2double(__double2hiint(v) + ((Ea - 1075 - SH) << 20), __double2loint(v));
}

}  // namespace lqcd
