// Gaussian quark smearing and APE link smearing (Sec. III, smearing of the
// interpolating fields): link products in 58-bit integers for SU(3) links, else in
// FP64, the SU(3) projection in FP64.  These act on the sources of connected
// correlators; the loops themselves are computed without smearing.
//
// Gaussian:  F = (1 + alpha H)^n within each time slice,
//   (H q)(x) = sum_{i = x, y, z} [ U_i(x) q(x + i) + U_i(x - i)^+ q(x - i) ],
// colour only (all four spins alike), optionally divided by (1 + 6 alpha) per step.
// APE:  U_i'(x) = P[ U_i(x) + alpha sum_{j != i spatial} S_ij(x) ] with the four
// spatial staples S_ij; P = unitary polar factor (scaled Newton iteration,
// Higham) divided by the principal cube root of its determinant; temporal links
// are copied unchanged.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "internal.cuh"
#include "fxfield.cuh"
#include "fpconv.cuh"

namespace lqcd {

struct M3 {
  double2 m[3][3];
};

__device__ __forceinline__ M3 load_m3(const double2 *p) {
  M3 r;
#pragma unroll
  for (int k = 0; k < 9; ++k) r.m[k / 3][k % 3] = p[k];
  return r;
}
__device__ __forceinline__ void store_m3(double2 *p, const M3 &a) {
#pragma unroll
  for (int k = 0; k < 9; ++k) p[k] = a.m[k / 3][k % 3];
}
// a b, a^+ b, a b^+
template <bool DA, bool DB>
__device__ __forceinline__ M3 mm(const M3 &a, const M3 &b) {
  M3 r;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      double2 acc = make_double2(0.0, 0.0);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double2 x = DA ? make_double2(a.m[k][i].x, -a.m[k][i].y) : a.m[i][k];
        const double2 y = DB ? make_double2(b.m[j][k].x, -b.m[j][k].y) : b.m[k][j];
        acc = cmac(acc, x, y);
      }
      r.m[i][j] = acc;
    }
  return r;
}
// a b - c d
__device__ __forceinline__ double2 cminor(double2 a, double2 b, double2 c, double2 d) {
  return cmac(cmul(a, b), make_double2(-c.x, -c.y), d);
}
__device__ __forceinline__ double2 det3(const M3 &a) {
  const double2 c0 = cminor(a.m[1][1], a.m[2][2], a.m[1][2], a.m[2][1]);
  const double2 c1 = cminor(a.m[1][2], a.m[2][0], a.m[1][0], a.m[2][2]);
  const double2 c2 = cminor(a.m[1][0], a.m[2][1], a.m[1][1], a.m[2][0]);
  return cmac(cmac(cmul(a.m[0][0], c0), a.m[0][1], c1), a.m[0][2], c2);
}
// (a^{-1})^+ = conj(cofactor matrix) / conj(det)
__device__ __forceinline__ M3 inv_dag(const M3 &a, double2 det) {
  M3 cof;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int i1 = (i + 1) % 3, i2 = (i + 2) % 3, j1 = (j + 1) % 3, j2 = (j + 2) % 3;
      cof.m[i][j] = cminor(a.m[i1][j1], a.m[i2][j2], a.m[i1][j2], a.m[i2][j1]);
    }
  // a^{-1} = cof^T / det, so (a^{-1})^+ = conj(cof) / conj(det)
  const double n = det.x * det.x + det.y * det.y;
  const double ni = 1.0 / n;
  const double2 inv_cdet = make_double2(det.x * ni, det.y * ni);  // 1 / conj(det)
  M3 r;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) r.m[i][j] = cmul(make_double2(cof.m[i][j].x, -cof.m[i][j].y), inv_cdet);
  return r;
}

// projection onto SU(3): unitary polar factor by the Newton iteration
// X <- (z X + X^{-+} / z) / 2, then the det phase removed.  z = |det X|^{-1/3} speeds
// up the first steps and does not change the limit: it is formed in FP32, from the
// determinant divided by a power of two where its square leaves the range of FP32, and is
// 1 once |det X| is within 2^-10 of 1.
// Bound by the FP64 pipe, so the iteration is written for few FP64 operations: one
// reciprocal per step, the size of a step read off the high words of its differences
// by integer maxima, and no iteration after one that moved X by less than 2^-27: the
// error is squared by each, so that one has already reached rounding.  The cube root
// of the determinant's phase starts from FP32 and takes two Newton steps.
// An APE step on 16^3 x 32 (FP64 staples): 3.1 ms before, 2.1 ms with this.
__device__ M3 project_su3(M3 x) {
  for (int it = 0; it < 30; ++it) {
    const double2 d = det3(x);
    const float ad = sqrtf((float)d.x * (float)d.x + (float)d.y * (float)d.y);
    double hz = 0.5, hzi = 0.5;
    if (!(fabsf(ad - 1.f) <= 0x1p-10f)) {
      const int e = (max(__double2hiint(d.x) & 0x7fffffff, __double2hiint(d.y) & 0x7fffffff) >> 20) - 1023;
      if (ad > 0x1p-60f && ad < 0x1p60f) {
        const float z = cbrtf(1.f / ad);
        hz = 0.5 * z;
        hzi = 0.5f / z;
      } else if (e > -1023 && e < 1024) {  // det = (x0 + i y0) 2^(3 q), of size 1 to 12
        const int q = (e + 1023) / 3 - 341;
        const double f = __hiloint2double((1023 - q) << 20, 0);
        const float x0 = (float)(d.x * f * f * f), y0 = (float)(d.y * f * f * f), z = cbrtf(rsqrtf(x0 * x0 + y0 * y0));
        hz = z * __hiloint2double((1022 - q) << 20, 0);
        hzi = __hiloint2double((1022 + q) << 20, 0) / z;
      }
    }
    const M3 y = inv_dag(x, d);
    int diff = 0;  // high word of the largest |component| of the step
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const double2 nv = make_double2(fma(hz, x.m[i][j].x, hzi * y.m[i][j].x), fma(hz, x.m[i][j].y, hzi * y.m[i][j].y));
        diff = max(diff, max(__double2hiint(nv.x - x.m[i][j].x) & 0x7fffffff, __double2hiint(nv.y - x.m[i][j].y) & 0x7fffffff));
        x.m[i][j] = nv;
      }
    if (diff < (1023 - 27) << 20 && it > 0) break;
  }
  const double2 d = det3(x);  // e^{i phi}; ph = e^{-i phi / 3}, the principal root
  float sn, cs;
  sincosf(atan2f((float)d.y, (float)d.x) / 3.f, &sn, &cs);
  double2 ph = make_double2(cs, -sn);
#pragma unroll
  for (int k = 0; k < 2; ++k) {  // ph <- ph + ph (1 - d ph^3) / 3
    const double2 w = cmul(d, cmul(cmul(ph, ph), ph));
    ph = cmac(ph, ph, make_double2((1.0 - w.x) * (1.0 / 3.0), w.y * (-1.0 / 3.0)));
  }
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) x.m[i][j] = cmul(x.m[i][j], ph);
  return x;
}

__device__ __forceinline__ int shift_site(const Geom &g, const int c[4], int mu, int step) {
  int cn[4] = {c[0], c[1], c[2], c[3]};
  cn[mu] = (c[mu] + step + g.L[mu]) % g.L[mu];
  return site_of(g, cn);
}
__device__ __forceinline__ void coords_full(const Geom &g, int s, int c[4]) {
  c[0] = s % g.L[0];
  int r = s / g.L[0];
  c[1] = r % g.L[1];
  r /= g.L[1];
  c[2] = r % g.L[2];
  c[3] = r / g.L[2];
}

// One APE step, thread per (site, mu): spatial links smeared, temporal copied.  only: null,
// or nothing is done unless *only is set.
__global__ void k_ape_step(Geom g, const double2 *__restrict__ Uin, double2 *Uout, double alpha, const int *only) {
  if (only && !*only) return;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < g.V * 4; idx += gridDim.x * blockDim.x) {
    const int s = idx >> 2, i = idx & 3;
    const double2 *ui = Uin + (size_t)idx * 9;
    double2 *uo = Uout + (size_t)idx * 9;
    if (i == 3) {
#pragma unroll
      for (int k = 0; k < 9; ++k) uo[k] = ui[k];
      continue;
    }
    int c[4];
    coords_full(g, s, c);
    const M3 U = load_m3(ui);
    M3 S;
#pragma unroll
    for (int k = 0; k < 9; ++k) S.m[k / 3][k % 3] = make_double2(0.0, 0.0);
    for (int j = 0; j < 3; ++j) {
      if (j == i) continue;
      const int s_j = shift_site(g, c, j, 1), s_i = shift_site(g, c, i, 1), s_mj = shift_site(g, c, j, -1);
      int cmj[4] = {c[0], c[1], c[2], c[3]};
      cmj[j] = (c[j] - 1 + g.L[j]) % g.L[j];
      const int s_mj_i = shift_site(g, cmj, i, 1);
      const M3 Uj = load_m3(Uin + ((size_t)s * 4 + j) * 9);
      const M3 Ui_j = load_m3(Uin + ((size_t)s_j * 4 + i) * 9);
      const M3 Uj_i = load_m3(Uin + ((size_t)s_i * 4 + j) * 9);
      const M3 up = mm<false, true>(mm<false, false>(Uj, Ui_j), Uj_i);  // U_j(x) U_i(x+j) U_j(x+i)^+
      const M3 Uj_mj = load_m3(Uin + ((size_t)s_mj * 4 + j) * 9);
      const M3 Ui_mj = load_m3(Uin + ((size_t)s_mj * 4 + i) * 9);
      const M3 Uj_mji = load_m3(Uin + ((size_t)s_mj_i * 4 + j) * 9);
      const M3 dn = mm<false, false>(mm<true, false>(Uj_mj, Ui_mj), Uj_mji);  // U_j(x-j)^+ U_i(x-j) U_j(x-j+i)
#pragma unroll
      for (int k = 0; k < 9; ++k) S.m[k / 3][k % 3] = cadd(S.m[k / 3][k % 3], cadd(up.m[k / 3][k % 3], dn.m[k / 3][k % 3]));
    }
    M3 V;
#pragma unroll
    for (int k = 0; k < 9; ++k) V.m[k / 3][k % 3] = make_double2(fma(alpha, S.m[k / 3][k % 3].x, U.m[k / 3][k % 3].x), fma(alpha, S.m[k / 3][k % 3].y, U.m[k / 3][k % 3].y));
    store_m3(uo, project_su3(V));
  }
}

// integer limbs of the spatial links, [3 directions][block of 32 sites][9][32] int4;
// thread per (site, mu).  *bad is set where a link has none: its rows and columns are not
// of length 1, as after the projection of a singular matrix, which is NaN.  FP64 arithmetic
// is then taken everywhere.
__global__ void k_spatial_links(Geom g, const double2 *__restrict__ U, int4 *out, int vb, int *bad) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  const int s = idx >> 2, mu = idx & 3;
  if (s >= g.V || mu == 3) return;
  int4 *o = out + ((size_t)mu * vb + (s >> 5)) * 288 + (s & 31);
  float row[3] = {0.f, 0.f, 0.f}, col[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const double2 u = U[(size_t)idx * 9 + k];
    o[32 * k] = fx_link_entry(u.x, u.y);
    const float re = f64_to_f32_bits(u.x), im = f64_to_f32_bits(u.y), n = fmaf(re, re, im * im);
    row[k / 3] += n;
    col[k % 3] += n;
  }
#pragma unroll
  for (int k = 0; k < 3; ++k)
    if (!(fabsf(row[k] - 1.f) < 0x1p-8f && fabsf(col[k] - 1.f) < 0x1p-8f)) *bad = 1;  // (also NaN)
}

// One APE step for SU(3) links: the staples, columns of three-link products, on the
// integer units (fx64.cuh: 24 matrix-vector products a link), the projection in FP64.
// Lanes are 32 consecutive sites, grid.y the direction; temporal links are copied.
// With the staples in FP64 too (k_ape_step, for any links) a step took 3.1 ms on 16^3 x 32
// before the projection was rewritten, 2.1 after, and takes 0.69 ms here.
__global__ void __launch_bounds__(128) k_ape_step_fx(Geom g, const double2 *__restrict__ Uin, const int4 *__restrict__ Ufx,
                                                     int vb, double2 *Uout, double alpha) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y;
  if (s >= g.V) return;
  const double2 *ui = Uin + ((size_t)s * 4 + i) * 9;
  double2 *uo = Uout + ((size_t)s * 4 + i) * 9;
  if (i == 3) {
#pragma unroll
    for (int k = 0; k < 9; ++k) uo[k] = ui[k];
    return;
  }
  int c[4];
  coords_full(g, s, c);
  auto hop = [&](const int cc[4], int mu, int dir) {  // neighbour of cc in +-mu (mu: run time)
    int r = 0, stride = 1;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int L = g.L[k];
      int v = cc[k];
      if (k == mu) v = dir > 0 ? (v + 1 == L ? 0 : v + 1) : (v == 0 ? L - 1 : v - 1);
      r += v * stride;
      stride *= L;
    }
    return r;
  };
  auto link = [&](int site, int mu) { return Ufx + ((size_t)mu * vb + (site >> 5)) * 288 + (site & 31); };
  auto load = [&](const int4 *p, int4 u[9]) {
#pragma unroll
    for (int k = 0; k < 9; ++k) u[k] = p[32 * k];
  };
  const int s_i = hop(c, i, 1);
  M3 V;
#pragma unroll 1
  for (int col = 0; col < 3; ++col) {
    long long S[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll 1
    for (int t = 0; t < 4; ++t) {  // two transverse directions, forward and backward staple
      const int j = (t >> 1) == 0 ? (i == 0 ? 1 : 0) : (i == 2 ? 1 : 2);
      const bool up = !(t & 1);
      int cmj[4] = {c[0], c[1], c[2], c[3]};
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (k == j && !up) cmj[k] = c[k] == 0 ? g.L[k] - 1 : c[k] - 1;
      const int sj = up ? hop(c, j, 1) : hop(c, j, -1);
      // forward: U_j(x) U_i(x+j) U_j(x+i)^+, backward: U_j(x-j)^+ U_i(x-j) U_j(x-j+i)
      const int4 *third = link(up ? s_i : hop(cmj, i, 1), j);
      int rh[3], rl[3], ih[3], il[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {  // its column col: of the adjoint for the forward staple
        const int4 e = third[32 * (up ? col * 3 + a : a * 3 + col)];
        rh[a] = e.x;
        rl[a] = e.y;
        ih[a] = up ? -e.z : e.z;
        il[a] = up ? -e.w : e.w;
      }
      int4 u[9];
      long long X[6];
      load(link(sj, i), u);
      fx_su3<true>(u, rh, rl, ih, il, X);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        fx_split(X[2 * a], rh[a], rl[a]);
        fx_split(X[2 * a + 1], ih[a], il[a]);
      }
      load(link(up ? s : sj, j), u);
      if (up) fx_su3<true>(u, rh, rl, ih, il, X);
      else fx_su3<false>(u, rh, rl, ih, il, X);
#pragma unroll
      for (int k = 0; k < 6; ++k) S[k] += X[k];
    }
    // V = U + alpha S, S in units of 2^-58
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double2 u = ui[a * 3 + col];
      const double2 v = make_double2(fma(alpha, __ll2double_rn(S[2 * a]) * 0x1p-58, u.x),
                                     fma(alpha, __ll2double_rn(S[2 * a + 1]) * 0x1p-58, u.y));
      if (col == 0) V.m[a][0] = v;
      else if (col == 1) V.m[a][1] = v;
      else V.m[a][2] = v;
    }
  }
  V = project_su3(V);
#pragma unroll
  for (int k = 0; k < 9; ++k) uo[k] = V.m[k / 3][k % 3];
}

// Component a of one Gaussian step in FP64 at site s: q + alpha (H q)
__device__ __forceinline__ double2 gauss_row64(const Geom &g, const double2 *__restrict__ U,
                                               const double2 *__restrict__ q, int s, int a, double alpha) {
  int c[4];
  coords_full(g, s, c);
  double2 acc = make_double2(0.0, 0.0);
  int stride = 1;
#pragma unroll 1
  for (int i = 0; i < 3; ++i) {
    const int L = g.L[i], ci = i == 0 ? c[0] : (i == 1 ? c[1] : c[2]);
    const int sf = s + (ci + 1 == L ? stride * (1 - L) : stride), sb = s + (ci == 0 ? stride * (L - 1) : -stride);
    stride *= L;
#pragma unroll 1
    for (int b = 0; b < 3; ++b) {
      acc = cmac(acc, U[((size_t)s * 4 + i) * 9 + a * 3 + b], q[(size_t)sf * 12 + b]);    // U_i(x)[a][b] q(x+i)
      acc = cmacc(acc, U[((size_t)sb * 4 + i) * 9 + b * 3 + a], q[(size_t)sb * 12 + b]);  // conj(U_i(x-i)[b][a]) q(x-i)
    }
  }
  return make_double2(fma(alpha, acc.x, q[(size_t)s * 12 + a].x), fma(alpha, acc.y, q[(size_t)s * 12 + a].y));
}

// The n Gaussian steps on integer limbs (fx64.cuh), for SU(3) links: the source is
// converted once, the steps q <- scale (q + alpha H q) run on limbs, and the result is
// converted back once.  In FP64 a step took 864 fused multiply-adds per site at 64
// cycles a warp.
//
// Field: [rhs][4 spins][block of 32 sites][3 colours][32] int4 (re.h, re.l, im.h, im.l)
// and [rhs][4][blocks][32] int, the exponent E of the colour vector: a component is
// (h 2^29 + l) 2^(E - 1075 - GAUSS_SH), below 2^(53 + GAUSS_SH) in size.  The exponent
// is an int, so no step over- or underflows; GAUSS_ZERO marks a zero vector and
// GAUSS_NAN one that is not finite.
// Links: [3 directions][block of 32 sites][9][32] int4.
constexpr int GAUSS_SH = 5;  // six directions of |X| < 2.45 * 2^58 stay below 2^62 (gauss_mul)
constexpr int GAUSS_ZERO = -(1 << 28), GAUSS_NAN = 1 << 28, GAUSS_FP64 = 1 << 29;
struct GaussF {
  int4 *d;
  int *e;
  int vb;  // blocks of 32 sites
  __device__ int4 *at(int rhs, int spin, int s) const {  // + 32 colour
    return d + ((size_t)(rhs * 4 + spin) * vb + (s >> 5)) * 96 + (s & 31);
  }
  __device__ int *exp(int rhs, int spin, int s) const { return e + (size_t)(rhs * 4 + spin) * vb * 32 + s; }
};

// Where links have no limbs (*bad, k_spatial_links) every exponent is GAUSS_FP64, and the
// three kernels below work on FP64 fields in the same memory, [rhs][V][12] double2.
__device__ __forceinline__ double2 *gauss_fp64(const GaussF &f, int V, int rhs) {
  return (double2 *)f.d + (size_t)rhs * V * 12;
}

// FP64 -> limbs; a block takes 32 sites, a warp one spin
__global__ void __launch_bounds__(128) k_gauss_in(int V, const double2 *__restrict__ in, GaussF f, const int *bad) {
  const int rhs = blockIdx.x / f.vb, s = (blockIdx.x % f.vb) * 32 + (threadIdx.x & 31), spin = threadIdx.x >> 5;
  if (s >= V) return;
  const double2 *q = in + ((size_t)rhs * V + s) * 12 + spin * 3;
  const double2 v[3] = {q[0], q[1], q[2]};
  if (*bad) {
    *f.exp(rhs, spin, s) = GAUSS_FP64;
#pragma unroll
    for (int k = 0; k < 3; ++k) gauss_fp64(f, V, rhs)[(size_t)s * 12 + spin * 3 + k] = v[k];
    return;
  }
  const int m = fx_max(fx_max(fx_max(0, v[0]), v[1]), v[2]);
  unsigned low = 0u;
#pragma unroll
  for (int k = 0; k < 3; ++k) low |= __double2loint(v[k].x) | __double2loint(v[k].y);
  const int ex = m >> 20;
  const int E = m == 0 && low == 0u ? GAUSS_ZERO : (ex == 0x7ff ? GAUSS_NAN : max(ex, 1));
  *f.exp(rhs, spin, s) = E;
  if (E == GAUSS_ZERO || E == GAUSS_NAN) return;
  int4 *o = f.at(rhs, spin, s);
  auto conv = [&](double x) {  // as fx_int, with subnormal values too
    const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
    const unsigned long long mant = ((unsigned long long)((hi & 0xfffff) | (e ? 0x100000 : 0)) << 32) | (unsigned)__double2loint(x);
    return fx_negif((long long)((mant << GAUSS_SH) >> min(E - max(e, 1), 63)), hi >> 31);
  };
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    int4 t;
    fx_split(conv(v[k].x), t.x, t.y);
    fx_split(conv(v[k].y), t.z, t.w);
    o[32 * k] = t;
  }
}

// limbs -> FP64
__global__ void __launch_bounds__(128) k_gauss_out(int V, GaussF f, double2 *__restrict__ out) {
  const int rhs = blockIdx.x / f.vb, s = (blockIdx.x % f.vb) * 32 + (threadIdx.x & 31), spin = threadIdx.x >> 5;
  if (s >= V) return;
  const int E = *f.exp(rhs, spin, s);
  const int4 *q = f.at(rhs, spin, s);
  double2 *o = out + ((size_t)rhs * V + s) * 12 + spin * 3;
  if (E == GAUSS_FP64) {
#pragma unroll
    for (int k = 0; k < 3; ++k) o[k] = gauss_fp64(f, V, rhs)[(size_t)s * 12 + spin * 3 + k];
    return;
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (E == GAUSS_ZERO) {
      o[k] = make_double2(0.0, 0.0);
    } else if (E == GAUSS_NAN) {
      const double nan = __longlong_as_double(0x7ff8000000000000ll);
      o[k] = make_double2(nan, nan);
    } else {
      const int4 t = q[32 * k];
      const double re = __ll2double_rn((long long)t.x * (1 << 29) + t.y), im = __ll2double_rn((long long)t.z * (1 << 29) + t.w);
      o[k] = make_double2(scalbn(re, E - 1075 - GAUSS_SH), scalbn(im, E - 1075 - GAUSS_SH));
    }
  }
}

// A real coefficient (kh 2^29 + kl) 2^(ek - 1080), 58 bits
struct GaussCoef {
  int kh, kl, ek;
};
// (v c) 2^-60 with the coefficient's integer, |v| < 2^62 - 2^30
__device__ __forceinline__ long long gauss_mul(long long v, const GaussCoef &c) {
  const int l = (int)((unsigned)v << 1) >> 1, h = (int)((v - l) >> 31);  // v = h 2^31 + l
  return fx_mad(h, c.kh, 0) + ((fx_mad(h, c.kl, 0) * 4 + fx_mad(l, c.kh, 0) + (1ll << 30)) >> 31);
}

// acc += M q of one neighbour (exponent En) at exponent Em; nothing is loaded for a
// neighbour of zeros
template <bool FWD>
__device__ __forceinline__ void gauss_dir(const int4 *__restrict__ link, const int4 *__restrict__ q, int En, int Em,
                                          long long acc[6]) {
  if (En == GAUSS_ZERO) return;
  int4 u[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) u[k] = link[32 * k];
  int rh[3], rl[3], ih[3], il[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int4 t = q[32 * k];
    rh[k] = t.x;
    rl[k] = t.y;
    ih[k] = t.z;
    il[k] = t.w;
  }
  long long X[6];
  fx_su3<FWD>(u, rh, rl, ih, il, X);
  const int d = min(Em - En, 62);
  const long long half = (1ll << d) >> 1;  // rounded: a bias would add up over the steps
#pragma unroll
  for (int k = 0; k < 6; ++k) acc[k] += (X[k] + half) >> d;
}

// One step.  A block takes 32 sites, a warp one spin of them (the four warps read the
// same links).  Bound by the integer pipes: 648 multiply-adds per (site, spin,
// right-hand side), of 4 cycles each where their operands differ, on one of them.  Two
// right-hand sides per thread for each link in registers were slower (12^3 x 24, 12
// sources: 7.8 ms for 25 steps against 6.5).  25 steps on 12 Gaussian sources of
// 16^3 x 32: 58.9 ms in FP64 arithmetic, 22.2 ms here; on 12 point sources, whose
// neighbours are mostly zero, 9.8 ms with each neighbour converted where it is used and
// 3.6 ms here (6.4 while the links of zero neighbours were loaded).
__global__ void __launch_bounds__(128, 4) k_gauss_step(Geom g, const int4 *__restrict__ U, GaussF in, GaussF out,
                                                       GaussCoef alpha, GaussCoef scale, bool scaled,
                                                       const double2 *__restrict__ U64, double alpha64, double scale64) {
  const int vb = in.vb, lane = threadIdx.x & 31, spin = threadIdx.x >> 5;
  const int blk = blockIdx.x % vb, rhs = blockIdx.x / vb;
  const int site = blk * 32 + lane, s = min(site, g.V - 1);
  int c[4];
  coords_full(g, s, c);
  const int stride[3] = {1, g.L[0], g.L[0] * g.L[1]};
  int n[6];  // 2 mu + (0 forward, 1 backward)
#pragma unroll
  for (int mu = 0; mu < 3; ++mu) {
    n[2 * mu] = s + (c[mu] + 1 == g.L[mu] ? stride[mu] * (1 - g.L[mu]) : stride[mu]);
    n[2 * mu + 1] = s + (c[mu] == 0 ? stride[mu] * (g.L[mu] - 1) : -stride[mu]);
  }
  long long acc[6] = {0, 0, 0, 0, 0, 0};
  const int E0 = *in.exp(rhs, spin, s);
  int Em = GAUSS_ZERO;
#pragma unroll
  for (int q = 0; q < 6; ++q) Em = max(Em, *in.exp(rhs, spin, n[q]));
  if (E0 == GAUSS_FP64) {  // rolled: this rare branch shall not take registers from the other
    if (site >= g.V) return;
    *out.exp(rhs, spin, s) = GAUSS_FP64;
    const double2 *q = gauss_fp64(in, g.V, rhs) + spin * 3;
#pragma unroll 1
    for (int k = 0; k < 3; ++k)
      gauss_fp64(out, g.V, rhs)[(size_t)s * 12 + spin * 3 + k] = cscale(gauss_row64(g, U64, q, s, k, alpha64), scale64);
    return;
  }
  if (E0 == GAUSS_ZERO && Em == GAUSS_ZERO) {  // (the values of a zero vector are not read)
    if (site < g.V) *out.exp(rhs, spin, s) = GAUSS_ZERO;
    return;
  }
#pragma unroll 1
  for (int mu = 0; mu < 3; ++mu) {  // one body: the code stays in the instruction cache
    const int nf = mu == 0 ? n[0] : (mu == 1 ? n[2] : n[4]), nb = mu == 0 ? n[1] : (mu == 1 ? n[3] : n[5]);
    gauss_dir<true>(U + ((size_t)mu * vb + blk) * 288 + (s & 31),  // U_mu(x)
                    in.at(rhs, spin, nf), *in.exp(rhs, spin, nf), Em, acc);
    gauss_dir<false>(U + ((size_t)mu * vb + (nb >> 5)) * 288 + (nb & 31),  // U_mu(x - mu)
                     in.at(rhs, spin, nb), *in.exp(rhs, spin, nb), Em, acc);
  }
  if (site >= g.V) return;
  // scale (q + alpha acc); before each product the six values are shifted up to 61 bits
  // together, so that the product's upper 60 bits lose nothing
  const int4 *q = in.at(rhs, spin, s);
  const bool hq = E0 != GAUSS_ZERO, ha = Em != GAUSS_ZERO && alpha.ek > 0;
  auto shift_up = [](long long v[6]) {
    unsigned long long any = 0;
#pragma unroll
    for (int k = 0; k < 6; ++k) any |= (unsigned long long)(v[k] ^ (v[k] >> 63));
    const int n = any ? max(__clzll((long long)any) - 3, 0) : 0;
#pragma unroll
    for (int k = 0; k < 6; ++k) v[k] <<= n;
    return n;
  };
  const int Ea = ha ? Em - shift_up(acc) + alpha.ek - 1020 : GAUSS_ZERO, Eq = hq ? E0 - 2 : GAUSS_ZERO;
  const int Et = max(Eq, Ea), dq = min(Et - Eq, 62), da = min(Et - Ea, 62);
  const long long rq = (1ll << dq) >> 1, ra = (1ll << da) >> 1;
  long long v[6];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int4 t = q[32 * k];
    const long long qv[2] = {((long long)t.x * (1 << 29) + t.y) << 2, ((long long)t.z * (1 << 29) + t.w) << 2};
#pragma unroll
    for (int h = 0; h < 2; ++h)
      v[2 * k + h] = (hq ? (qv[h] + rq) >> dq : 0) + (ha ? (gauss_mul(acc[2 * k + h], alpha) + ra) >> da : 0);
  }
  int Er = Et;
  if (scaled) {
    Er += scale.ek - 1020 - shift_up(v);
#pragma unroll
    for (int k = 0; k < 6; ++k) v[k] = gauss_mul(v[k], scale);
  }
  unsigned long long any = 0;
#pragma unroll
  for (int k = 0; k < 6; ++k) any |= (unsigned long long)(v[k] ^ (v[k] >> 63));
  const bool nan = E0 == GAUSS_NAN || Em == GAUSS_NAN;
  const int sh = 64 - __clzll((long long)any) - (53 + GAUSS_SH);  // > 0: too large by sh bits
  const int E = nan ? GAUSS_NAN : (any == 0 ? GAUSS_ZERO : Er + sh);
  *out.exp(rhs, spin, s) = E;
  if (nan || any == 0) return;
  int4 *o = out.at(rhs, spin, s);
  const long long ro = sh > 0 ? (1ll << sh) >> 1 : 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const long long a = sh > 0 ? (v[2 * k] + ro) >> sh : v[2 * k] << -sh;
    const long long b = sh > 0 ? (v[2 * k + 1] + ro) >> sh : v[2 * k + 1] << -sh;
    int4 t;
    fx_split(a, t.x, t.y);
    fx_split(b, t.z, t.w);
    o[32 * k] = t;
  }
}

// One step in FP64 for links that are not SU(3): thread per (rhs, site, spin)
__global__ void k_gauss_step64(Geom g, const double2 *__restrict__ U, const double2 *__restrict__ in, double2 *out,
                               int nrhs, double alpha, double scale) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (size_t)nrhs * g.V * 4) return;
  const int s = (int)((idx >> 2) % g.V), spin = (int)(idx & 3);
  const size_t rhs = (idx >> 2) / g.V;
#pragma unroll 1
  for (int k = 0; k < 3; ++k)
    out[(rhs * g.V + s) * 12 + spin * 3 + k] =
        cscale(gauss_row64(g, U, in + rhs * g.V * 12 + spin * 3, s, k, alpha), scale);
}

// c + lo as 58 bits below c's exponent, |lo| at most half a unit in the last place of c
static GaussCoef gauss_coef(double c, double lo = 0.0) {
  unsigned long long w;
  memcpy(&w, &c, sizeof(w));
  GaussCoef r;
  r.ek = (int)((w >> 52) & 0x7ff);
  long long k = r.ek ? (long long)((w & 0xfffffffffffffull) | 0x10000000000000ull) << 5 : 0;
  fx_split(((w >> 63) ? -k : k) + (r.ek ? llrint(std::ldexp(lo, 1080 - r.ek)) : 0), r.kh, r.kl);
  return r;
}

// Bytes of limbs kept for a batch of right-hand sides: all steps of as many as stay in
// L2 run before the next ones start, so that the steps read and write L2.
constexpr size_t GAUSS_WS_BYTES = 64u << 20;

// workspace for the limbs of the spatial links and the flag of k_spatial_links.  APE and
// Gaussian smearing have one each (slot): the replays of a captured graph of one are not
// ordered with calls of the other.
static int4 *spatial_limbs(lqcd_ctx *ctx, int slot, int vb, int **bad, int *rc) {
  Carver sizing(nullptr);
  sizing.take<int4>((size_t)3 * vb * 288);
  sizing.take<int>(1);
  void *w = workspace(ctx, slot, sizing.size(), rc);
  if (!w) return nullptr;
  Carver cv(w);
  int4 *links = cv.take<int4>((size_t)3 * vb * 288);
  *bad = cv.take<int>(1);
  return links;
}

// *done: false if the workspace was refused, and nothing was launched
static int gauss_fx(lqcd_ctx *ctx, const double2 *U, const double2 *in, double2 *out, int nrhs, double alpha,
                    double scale, int n_iter, cudaStream_t st, bool *done) {
  const Geom &g = ctx->geom;
  const int vb = (g.V + 31) / 32;
  int rc = LQCD_OK;
  int *bad = nullptr;
  int4 *links = spatial_limbs(ctx, WS_SMEAR_FX, vb, &bad, &rc);
  *done = false;
  if (!links) return rc;
  const size_t nd = (size_t)4 * vb * 96, ne = (size_t)4 * vb * 32;  // per right-hand side
  const size_t per = 2 * (nd * sizeof(int4) + ne * sizeof(int));
  const int chunk = (int)std::max<size_t>(1, std::min<size_t>(nrhs, GAUSS_WS_BYTES / per));
  char *w = (char *)workspace(ctx, WS_SMEAR, per * chunk, &rc);
  const FxUse use(ctx, st);
  if (!w || !use.ok) return rc;
  *done = true;
  LQCD_CUDA_TRY(ctx, cudaMemsetAsync(bad, 0, sizeof(int), st));
  KL k_spatial_links<<<(g.V * 4 + 255) / 256, 256, 0, st>>>(g, U, links, vb, bad);
  LQCD_LAUNCH_CHECK(ctx, "k_spatial_links");
  GaussF f[2];
  for (int k = 0; k < 2; ++k) {
    f[k].d = (int4 *)w + k * nd * chunk;
    f[k].e = (int *)((int4 *)w + 2 * nd * chunk) + k * ne * chunk;
    f[k].vb = vb;
  }
  // The rounding of 1 / (1 + 6 alpha) would add up over the steps, so its remainder is kept.
  // Error of 25 steps on 8^3 x 16 against quadruple precision: 1.3e-16 at alpha = 4 and 0.6
  // (1.7e-16 on APE links); 5.4e-16 and 1.8e-15 in FP64 arithmetic.
  double lo = 0.0;
  if (scale != 1.0) {
    const double a6 = 6.0 * alpha, a6l = std::fma(6.0, alpha, -a6), n = 1.0 + a6, b = n - a6;
    const double nl = ((1.0 - b) + (a6 - (n - b))) + a6l;
    const double rest = std::fma(-scale, nl, std::fma(-scale, n, 1.0)) * scale;
    if (std::fabs(rest) < 0x1p-50 * std::fabs(scale)) lo = rest;
  }
  const GaussCoef ca = gauss_coef(alpha), cs = gauss_coef(scale, lo);
  const bool scaled = scale != 1.0;
  for (int r = 0; r < nrhs; r += chunk) {
    const int n = std::min(chunk, nrhs - r);
    const size_t o = (size_t)r * g.V * 12;
    KL k_gauss_in<<<(unsigned)vb * n, 128, 0, st>>>(g.V, in + o, f[0], bad);
    LQCD_LAUNCH_CHECK(ctx, "k_gauss_in");
    for (int it = 0; it < n_iter; ++it) {
      KL k_gauss_step<<<(unsigned)vb * n, 128, 0, st>>>(g, links, f[it % 2], f[1 - it % 2], ca, cs, scaled, U,
                                                          alpha, scale);
      LQCD_LAUNCH_CHECK(ctx, "k_gauss_step");
    }
    KL k_gauss_out<<<(unsigned)vb * n, 128, 0, st>>>(g.V, f[n_iter % 2], out + o);
    LQCD_LAUNCH_CHECK(ctx, "k_gauss_out");
  }
  return LQCD_OK;
}

}  // namespace lqcd

using namespace lqcd;

extern "C" int lqcd_smear_ape(lqcd_ctx *ctx, double alpha, int n_iter, double *out, lqcd_stream_t stream) {
  LQCD_TRACE("lqcd_smear_ape");
  if (!ctx || n_iter < 0 || !std::isfinite(alpha)) return set_error(ctx, LQCD_ERR_INVALID, "lqcd_smear_ape: bad argument");
  if (!ctx->have_gauge) return set_error(ctx, LQCD_ERR_NO_GAUGE, "lqcd_smear_ape: no gauge field");
  if (out && !is_device_ptr(out)) return set_error(ctx, LQCD_ERR_INVALID, "lqcd_smear_ape: out must be device memory");
  cudaSetDevice(ctx->device);
  cudaStream_t st = (cudaStream_t)stream;
  const Geom &g = ctx->geom;
  const size_t n = (size_t)g.V * 36;
  if (!ctx->Uape) LQCD_CUDA_TRY(ctx, cudaMalloc(&ctx->Uape, n * sizeof(double2)));
  int rc = LQCD_OK;
  double2 *tmp = (double2 *)workspace(ctx, WS_SMEAR_LINKS, n * sizeof(double2), &rc);
  if (!tmp) return rc;
  // ping-pong so that the last step lands in Uape
  double2 *bufs[2] = {n_iter % 2 ? ctx->Uape : tmp, n_iter % 2 ? tmp : ctx->Uape};
  const double2 *src = ctx->U64;
  const int threads = 128, blocks = (g.V * 4 + threads - 1) / threads;
  int4 *links = nullptr;
  int *bad = nullptr;
  const int vb = (g.V + 31) / 32;
  const FxUse use(ctx, st);
  if (use.ok && n_iter > 0)  // (without the workspace: FP64)
    links = spatial_limbs(ctx, WS_APE_FX, vb, &bad, &rc);
  if (links) LQCD_CUDA_TRY(ctx, cudaMemsetAsync(bad, 0, sizeof(int), st));
  for (int it = 0; it < n_iter; ++it) {
    double2 *dst = bufs[it % 2];
    if (links) {
      KL k_spatial_links<<<(g.V * 4 + 255) / 256, 256, 0, st>>>(g, src, links, vb, bad);
      KL k_ape_step_fx<<<dim3((g.V + 127) / 128, 4), 128, 0, st>>>(g, src, links, vb, dst, alpha);
      // in place of what links without limbs gave (in the kernel above, the branch and its
      // registers made a step on 16^3 x 32 10% slower)
      KL k_ape_step<<<std::min(blocks, 512), threads, 0, st>>>(g, src, dst, alpha, bad);
    } else {
      KL k_ape_step<<<blocks, threads, 0, st>>>(g, src, dst, alpha, nullptr);
    }
    LQCD_LAUNCH_CHECK(ctx, "k_ape_step");
    src = dst;
  }
  if (n_iter == 0)
    LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(ctx->Uape, ctx->U64, n * sizeof(double2), cudaMemcpyDeviceToDevice, st));
  if (out) LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(out, ctx->Uape, n * sizeof(double2), cudaMemcpyDeviceToDevice, st));
  ctx->have_ape = true;
  return LQCD_OK;
}

extern "C" int lqcd_smear_gaussian(lqcd_ctx *ctx, const double *in, double *out, int nrhs, double alpha, int n_iter,
                                   int ape_links, int normalise, lqcd_stream_t stream) {
  LQCD_TRACE("lqcd_smear_gaussian");
  if (!ctx || nrhs < 0 || n_iter < 0 || !std::isfinite(alpha) || (nrhs > 0 && (!in || !out)) || (in && in == out))
    return set_error(ctx, LQCD_ERR_INVALID, "lqcd_smear_gaussian: bad argument (in and out must differ)");
  if (!ctx->have_gauge) return set_error(ctx, LQCD_ERR_NO_GAUGE, "lqcd_smear_gaussian: no gauge field");
  if (ape_links && !ctx->have_ape)
    return set_error(ctx, LQCD_ERR_INVALID, "lqcd_smear_gaussian: no APE-smeared links (call lqcd_smear_ape)");
  if (nrhs == 0) return LQCD_OK;
  if (!is_device_ptr(in) || !is_device_ptr(out))
    return set_error(ctx, LQCD_ERR_INVALID, "lqcd_smear_gaussian: in and out must be device memory");
  cudaSetDevice(ctx->device);
  cudaStream_t st = (cudaStream_t)stream;
  const Geom &g = ctx->geom;
  const size_t n = (size_t)nrhs * g.V * 12;
  if (n_iter == 0) {
    LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(out, in, n * sizeof(double2), cudaMemcpyDeviceToDevice, st));
    return LQCD_OK;
  }
  const double2 *U = ape_links ? ctx->Uape : ctx->U64;
  const double scale = normalise ? 1.0 / (1.0 + 6.0 * alpha) : 1.0;
  // FP64 for links that are not SU(3), for a scale or alpha without 58-bit form, and
  // where the limbs' workspace could not be had
  int rc = LQCD_OK;
  if (ctx->fx_links && std::isnormal(scale) && (alpha == 0.0 || std::isnormal(alpha))) {
    bool done = false;
    rc = gauss_fx(ctx, U, (const double2 *)in, (double2 *)out, nrhs, alpha, scale, n_iter, st, &done);
    if (done) return rc;
  }
  double2 *tmp = (double2 *)workspace(ctx, WS_SMEAR, n * sizeof(double2), &rc);
  if (!tmp) return rc;
  double2 *bufs[2] = {n_iter % 2 ? (double2 *)out : tmp, n_iter % 2 ? tmp : (double2 *)out};
  const double2 *src = (const double2 *)in;
  const int threads = 128;
  for (int it = 0; it < n_iter; ++it) {
    double2 *dst = bufs[it % 2];
    const unsigned blocks = (unsigned)((nrhs * (size_t)g.V * 4 + threads - 1) / threads);
    KL k_gauss_step64<<<blocks, threads, 0, st>>>(g, U, src, dst, nrhs, alpha, scale);
    LQCD_LAUNCH_CHECK(ctx, "k_gauss_step64");
    src = dst;
  }
  return LQCD_OK;
}
