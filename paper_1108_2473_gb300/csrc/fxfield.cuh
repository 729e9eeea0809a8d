// Spinor fields and links as integer limbs (fx64.cuh) in coalesced layouts, and the
// hopping term on them.
//
// Parity-local sites go in blocks of 32 (the last one padded), so that a warp reads 512
// consecutive bytes per component at constant offsets from one address:
//   field of one parity: [rhs][block][12][32] int4, complex k = 3 spin + colour of a
//     site as (re.h, re.l, im.h, im.l), and [rhs][block][32] int, its biased exponent
//     E: a component is (h 2^29 + l) 2^(E - 1075 - FXF_SH), below 2^(53 + FXF_SH) in
//     size.  E = 0 marks a site of zeros, FX_BAD one that is not finite or out of range.
//     A field that FP64 arithmetic is to be matched on (k_fx_from64) has above the
//     exponent's 11 bits how far each spin row's largest component lies below it, 5 bits
//     a row (FX_ROW_ZERO: a row of zeros);
//   links: [2 parity][4 mu][block][9][32] int4, the sign of the time boundary folded in.
//
// A site is converted once, not by each of its eight neighbours; the hopping term
// then only adds limbs, multiplies and shifts.
#pragma once

#include <type_traits>

#include "internal.cuh"
#include "fx64.cuh"

namespace lqcd {

constexpr int FXF_SH = 4;  // eight directions of |X| < 2.45 * 2 * 2^57 stay below 2^63
constexpr int FX_BAD = -1;
constexpr int FX_ROW_ZERO = 31;
// Output rows whose largest contribution lies more than 2^FX_ROW_BITS below the stencil's
// largest component, to which all limbs are aligned, are evaluated in FP64: rows 0 and 1 do
// not mix, so FP64 arithmetic rounds relative to each.  The limbs' rounding is about
// 2^-55.5 of the stencil's largest component, that of FP64 arithmetic 2^-52.5 of the row's.
// Error of H against quadruple precision in row 1 of a Gaussian field on 8^4 whose rows 1
// to 3 are 1, 2^-2, 2^-3, 2^-4 of row 0: 0.7, 0.9, 1.3, 1.5e-16 (2.4e-16 for the last with
// limbs alone); in FP64 arithmetic 1.55e-16 for all.
constexpr int FX_ROW_BITS = 3;

__host__ __device__ inline int fx_blocks(int vh) { return (vh + 31) / 32; }

struct FxF {
  int4 *d;
  int *e;
  int vb;  // blocks of 32 sites
  __device__ FxF at(size_t rhs) const { return FxF{d + rhs * vb * 384, e + rhs * vb * 32, vb}; }
  __device__ int4 *site(int i) const { return d + (size_t)(i >> 5) * 384 + (i & 31); }  // + 32 k
};

// first entry of the link of parity-local site i; the others follow 32 apart
__host__ __device__ inline size_t fx_link_index(int p, int mu, int vh, int i) {
  return ((size_t)(p * 4 + mu) * fx_blocks(vh) + (i >> 5)) * 288 + (i & 31);
}

// The exponent of a site: FX_BAD out of range, 0 for zeros.  m: fx_max over its
// components, low: OR of their low words.
__device__ __forceinline__ int fx_site_exp(int m, unsigned low) {
  const int E = m >> 20;
  if (m == 0 && low == 0u) return 0;
  return (E < FX_EMIN || E > FX_EMAX) ? FX_BAD : E;
}
// E > 0 with its rows, m[a]: high word of the largest component of row a, low[a]: OR of its low words
__device__ __forceinline__ int fx_with_rows(int E, const int m[4], const unsigned low[4]) {
  int w = E;
#pragma unroll
  for (int a = 0; a < 4; ++a)
    w |= (m[a] == 0 && low[a] == 0u ? FX_ROW_ZERO : min(E - (m[a] >> 20), FX_ROW_ZERO - 1)) << (11 + 5 * a);
  return w;
}
__device__ __forceinline__ int fx_row_exp(int w, int E, int a) {  // 0 for a row of zeros
  const int d = (w >> (11 + 5 * a)) & 31;
  return d == FX_ROW_ZERO ? 0 : E - d;
}
__device__ __forceinline__ int4 fx_split_c(long long re, long long im) {
  int4 q;
  fx_split(re, q.x, q.y);
  fx_split(im, q.z, q.w);
  return q;
}
__device__ __forceinline__ long long fx_value(int h, int l) { return (long long)h * (1 << 29) + l; }

// Contribution of one neighbour (parity-local n, exponent En) to the rows HS (up) and
// the lower row it is paired with (lo), at exponent Em.  Direction mu = 2 j for an
// imaginary spin phase, 2 j + 1 for a real one; the phase of row HS is
//   SG i (x), -+SG (y), +-SG i (z), SG (t) for HS = 0, 1.
template <bool IMAG, bool DAG, bool FWD, int HS>
__device__ __forceinline__ void fxf_dir(int j, int n, const int4 *__restrict__ w, int En, int Em, const FxF &in,
                                        long long up[6], long long lo[6]) {
  if (En <= 0) return;
  constexpr int SG0 = (FWD != DAG) ? -1 : 1;  // projector (1 + SG0 gamma_mu)
  // the sign depends on j for (real, HS = 0: -, +) and (IMAG, HS = 1: +, -)
  constexpr bool VAR = IMAG ? HS == 1 : HS == 0;
  constexpr int SG = SG0;
  const int eps = !VAR ? 1 : (IMAG ? (j ? -1 : 1) : (j ? 1 : -1));
  const int low = j ? 2 + HS : 3 - HS;
  const long long neg = eps >> 31;
  const int4 *q = in.site(n);
  int4 u[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) u[k] = w[32 * k];
  int rh[3], rl[3], ih[3], il[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int4 a = q[32 * (3 * HS + k)];
    int4 b = q[32 * (3 * low + k)];
    if (VAR) b = make_int4(b.x * eps, b.y * eps, b.z * eps, b.w * eps);
    if (IMAG) {  // + SG i b
      rh[k] = SG > 0 ? a.x - b.z : a.x + b.z;
      rl[k] = SG > 0 ? a.y - b.w : a.y + b.w;
      ih[k] = SG > 0 ? a.z + b.x : a.z - b.x;
      il[k] = SG > 0 ? a.w + b.y : a.w - b.y;
    } else {  // + SG b
      rh[k] = SG > 0 ? a.x + b.x : a.x - b.x;
      rl[k] = SG > 0 ? a.y + b.y : a.y - b.y;
      ih[k] = SG > 0 ? a.z + b.z : a.z - b.z;
      il[k] = SG > 0 ? a.w + b.w : a.w - b.w;
    }
  }
  const int d = min(Em - En, 63);
  long long X[6];
  fx_su3<FWD>(u, rh, rl, ih, il, X);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const long long xr = X[2 * a] >> d, xi = X[2 * a + 1] >> d;
    up[2 * a] += xr;
    up[2 * a + 1] += xi;
    const long long yr = VAR ? fx_negif(xr, neg) : xr, yi = VAR ? fx_negif(xi, neg) : xi;
    if (IMAG) {  // the conjugate phase: - SG i x
      lo[2 * a] += SG > 0 ? yi : -yi;
      lo[2 * a + 1] += SG > 0 ? -yr : yr;
    } else {  // + SG x
      lo[2 * a] += SG > 0 ? yr : -yr;
      lo[2 * a + 1] += SG > 0 ? yi : -yi;
    }
  }
}

// one warp's half: rows HS and its shares of the two lower rows
template <bool DAG, int HS>
__device__ __forceinline__ void fxf_half(int p_out, int i, int vh, const int n[8], const int En[8], int Em,
                                         const FxF &in, const int4 *__restrict__ U, long long up[6], long long lo[6],
                                         long long (*share)[32]) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int j = 0; j < 2; ++j) {
    if (j == 1) {
#pragma unroll
      for (int k = 0; k < 6; ++k) {  // mu = x, y: the other half's lower row
        share[k][lane] = lo[k];
        lo[k] = 0;
      }
    }
    auto dir = [&](auto imag, auto fwd, int q) {  // q: neighbour 2 mu + (0 forward, 1 backward) for j = 0
      constexpr bool IM = decltype(imag)::value, FW = decltype(fwd)::value;
      const int nq = j ? n[4 + q] : n[q], eq = j ? En[4 + q] : En[q];
      fxf_dir<IM, DAG, FW, HS>(j, nq, U + fx_link_index(FW ? p_out : 1 - p_out, 2 * j + q / 2, vh, FW ? i : nq), eq,
                               Em, in, up, lo);
    };
    dir(std::true_type{}, std::true_type{}, 0);
    dir(std::true_type{}, std::false_type{}, 1);
    dir(std::false_type{}, std::true_type{}, 2);
    dir(std::false_type{}, std::false_type{}, 3);
  }
}

// H in at site i of parity p_out, rows hs (up) and 2 + hs (low) at exponent Em (0:
// all neighbours zero), in a block of 128 threads: warps 0, 1 take hs = 0, 1 of 32
// sites, warps 2, 3 of the next 32 (so hs is a compile-time constant of each warp's
// code, which an SM sub-partition sees only one half of; the directions are a loop of
// two to keep that code small).  Every thread takes part.
// bad: a neighbour has no integer form, or (ROWS) one of the two rows lies too far below
// Em for the limbs (FX_ROW_BITS); the rows that enter them are those of the projections,
// 0 with 3 and 1 with 2 for mu = x, y, 0 with 2 and 1 with 3 for z, t.
// Per direction 108 multiply-adds on one integer pipe and about 130 adds and shifts on
// the other, half of whose rate it reaches; 16, 20 or 24 resident warps per SM, rolled
// or unrolled directions all took within 4% of the same time.
template <bool DAG, bool ROWS>
__device__ __forceinline__ void fxf_hop(const Geom &g, int p_out, int i, int hs, const FxF &in,
                                        const int4 *__restrict__ U, long long up[6], long long low[6], int &Em,
                                        bool &bad) {
  __shared__ long long share[4][6][32];
  int c[4];
  coords_of(g, p_out, i, c);
  const int s = site_of(g, c);
  int n[8], En[8];  // neighbours 2 mu + (0 forward, 1 backward)
  int stride = 1;
  Em = 0;
  bad = false;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    const int L = g.L[mu];
    n[2 * mu] = (s + (c[mu] + 1 == L ? stride * (1 - L) : stride)) >> 1;
    n[2 * mu + 1] = (s + (c[mu] == 0 ? stride * (L - 1) : -stride)) >> 1;
    stride *= L;
  }
  int xy[2] = {0, 0}, zt[2] = {0, 0};  // largest exponents of the projections' two rows
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int w = in.e[n[q]];
    En[q] = ROWS && w > 0 ? w & 0x7ff : w;
    Em = max(Em, En[q]);
    bad = bad || w < 0;
    if (ROWS) {
      int *m = q < 4 ? xy : zt;
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const int h = q < 4 ? (a == 1 || a == 2) : a & 1;
        m[h] = max(m[h], fx_row_exp(w, En[q], a));
      }
    }
  }
  if (ROWS) {
    const int r0 = max(hs ? xy[1] : xy[0], hs ? zt[1] : zt[0]), r1 = max(hs ? xy[0] : xy[1], hs ? zt[1] : zt[0]);
    bad = bad || (r0 > 0 && r0 < Em - FX_ROW_BITS) || (r1 > 0 && r1 < Em - FX_ROW_BITS);
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) up[k] = low[k] = 0;
  const int warp = threadIdx.x >> 5;
  if (hs) fxf_half<DAG, 1>(p_out, i, g.Vh, n, En, Em, in, U, up, low, share[warp]);
  else fxf_half<DAG, 0>(p_out, i, g.Vh, n, En, Em, in, U, up, low, share[warp]);
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 6; ++k) low[k] += share[warp ^ 1][k][threadIdx.x & 31];
}

}  // namespace lqcd
