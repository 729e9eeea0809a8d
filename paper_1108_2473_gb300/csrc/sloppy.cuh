// Types shared by the mixed-precision kernels (sloppy.cu).
#pragma once

#include "internal.cuh"

namespace lqcd {

constexpr int ST = 128;  // threads per block of the site-tiled kernels (one site each)

enum { EPI_PLAIN = 0, EPI_AXPY = 1, EPI_DOTR = 2, EPI_TS = 3, EPI_RES = 4 };
enum { FLAG_ACTIVE = 1, FLAG_RU = 2 };

struct D4S {
  double a, b, c, d;
};

// FP32 parity field, one right-hand side per slot: [rhs][6][vh] float4
struct F32F {
  float4 *d;
  int vh;
  __device__ void load(int r, int i, float2 v[12]) const;
  __device__ void store(int r, int i, const float2 v[12]) const;
};

// A complex number for the two right-hand sides of a pair: re = (re_even, re_odd).
struct CP {
  float2 re, im;
};

// Reduced-precision parity field storing right-hand sides in pairs: for pair
// P = rhs / 2 and site i, the 24 reals of both members are 24 16-bit pairs
// (even member in the low half) in 6 uint4: [P][6][vh] uint4.  FP16 fields also
// keep one FP32 norm per member and site, [P][vh] float2: the stored halves are
// the values divided by the largest |real| of that member's site spinor.
struct F16P {
  uint4 *d;
  float2 *n;
  int vh;
};
struct BF16P {
  uint4 *d;
  int vh;
};

// The mixed solver's iterate as integer limbs (layout in fxfield.cuh): both parities,
// cap right-hand sides each.
struct FxIterate {
  int4 *d = nullptr;  // [2 parity] fields of cap right-hand sides
  int *e = nullptr;   // their exponents
  int cap = 0;
};
// x = scale e (first) or x += scale e (even and odd parts) for the listed right-hand sides
int fx_accum(lqcd_ctx *ctx, const FxIterate &x, const F32F &e, const F32F &o, const double *scale, bool first,
             const int *list, const int *count, int G, cudaStream_t st);
// r[parity] = 2^shift (b - D x) in FP32 for the right-hand sides list[0..n) (host list, with
// their shifts); rr (host, indexed by right-hand side) receives |b - D x|^2.  Synchronises st.
int fx_residual(lqcd_ctx *ctx, const FxIterate &x, const double2 *b, const F32F r[2], const int *list,
                const int *shift, int n, double *rr, cudaStream_t st);
// canonical FP64 x (device array have: 0 for right-hand sides whose x is zero)
int fx_join(lqcd_ctx *ctx, const FxIterate &x, const double *have, double2 *out, int nrhs, cudaStream_t st);

// per-RHS state of the inner (sloppy) BiCGstab
struct SState {
  double2 rho, alpha, omega, beta;
  double rr, rmax, rr_ru, target2;
  int iters, status, restart, ru_count, stall, pad0;
};

}  // namespace lqcd
