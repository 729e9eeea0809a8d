// The iterate of the mixed solver and its true residual b - D x.
//
// The iterate is held as integer limbs with one exponent per site (fxfield.cuh: 57
// bits relative to the site's largest component, which every update restores), so that the residual that
// certifies |M x - b| / |b| (Sec. III) runs on the integer units, exactly but for
// the last of those bits, and reads the iterate in coalesced parity order.  The FP64
// source b is brought to the same form where it is read; the residual goes out in
// FP32 (it only seeds the next inner solve) with an FP64 sum of |r|^2.  The rounding
// error of one evaluation is a few 1e-16 of |x|, far below the 1e-10 residual it
// certifies.  (In double-float arithmetic, pairs of FP32 numbers, it took about
// 10,500 FP32 operations per site and kept 48 bits: 12.1 ms per parity for 384
// right-hand sides of 16^3 x 32, now 10.2; the update of the iterate 4.5 ms, now 2.6
// and 3.7 ms for the first and the later ones, without clearing it before.)
#include <algorithm>
#include <cmath>
#include <vector>

#include "fxfield.cuh"
#include "fxaccum.cuh"
#include "fpconv.cuh"
#include "sloppy.cuh"

namespace lqcd {

// 2^k as two FP32 factors, 0 below and infinity above their range
__device__ __forceinline__ float2 pow2_pair(int k) {
  const int a = max(-126, min(127, k)), b = max(-127, min(128, k - a));
  return make_float2(__int_as_float((a + 127) << 23), __int_as_float((b + 127) << 23));
}

// ------------------------------------------------------------------ update
// x = scale e (FIRST) or x += scale e for the listed right-hand sides, both parities
// (fxaccum.cuh).  Bound by memory, 288 B (FIRST) or 480 B per site and right-hand side,
// and by the registers of a site's 24 sums, which are normalised together: 96 right-hand
// sides of 16^3 x 32 take 0.66 and 0.91 ms (5 and 4 blocks per SM; 0.75 and 1.00 ms with
// the registers that the compiler wants, 0.55 and 0.87 without normalisation).
template <bool FIRST>
__global__ void __launch_bounds__(ST, FIRST ? 5 : 4) k_fx_accum(F32F e0, F32F e1, FxF x0, FxF x1, const double *scale,
                                                 const int *list, const int *count, int nbx, int vh) {
  const int n_items = *count * nbx;
  for (int w = blockIdx.x; w < n_items; w += gridDim.x) {
    const int rhs = list[w / nbx];
    const int i = (w % nbx) * ST + threadIdx.x;
    if (i >= vh) continue;
    const FxScale s = fx_scale(scale[rhs]);  // > 0
#pragma unroll 1
    for (int p = 0; p < 2; ++p) {
      const FxF x = (p ? x1 : x0).at(rhs);
      int4 *xs = x.site(i);
      const float4 *q = (p ? e1 : e0).d + (size_t)rhs * 6 * vh + i;
      float e[24];
      long long v[24];
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const float4 t = q[(size_t)k * vh];
        e[4 * k] = t.x;
        e[4 * k + 1] = t.y;
        e[4 * k + 2] = t.z;
        e[4 * k + 3] = t.w;
      }
      const int old = FIRST ? 0 : x.e[i];
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        int4 t = make_int4(0, 0, 0, 0);
        if (!FIRST && old > 0) t = xs[32 * k];
        v[2 * k] = fx_value(t.x, t.y);
        v[2 * k + 1] = fx_value(t.z, t.w);
      }
      const int E = fx_accum_site(e, s, old, v);
      x.e[i] = E;
      if (E <= 0) continue;  // the limbs of such a site are not read
#pragma unroll
      for (int k = 0; k < 12; ++k) xs[32 * k] = fx_split_c(v[2 * k], v[2 * k + 1]);
    }
  }
}

// ---------------------------------------------------------------- residual
// r = b - x + kappa H x at the sites of parity p_out, FP32, with one |r|^2 partial
// per block.  A block takes 64 sites of one listed right-hand side (lane layout of
// fxf_hop); blocks are ordered (chunk of FXR_CHUNK right-hand sides, site block,
// right-hand side in the chunk), so that blocks issued together share their links.
// kappa = (kh 2^29 + kl) 2^(ek - 1080).  r is stored, and summed, times 2^shift[slot]
// (about one over the last residual): FP32 would hold neither the residual of sources of
// any size nor its square.
constexpr int FXR_SITES = 64;
constexpr int FXR_CHUNK = 8;
__global__ void __launch_bounds__(2 * FXR_SITES, 4) k_fx_resid(Geom g, int p_out, const int4 *__restrict__ U, FxF xin,
                                                            FxF xown, const double2 *__restrict__ b, F32F r, int kh,
                                                            int kl, int ek, const int *list, const int *shift, int n,
                                                            double *part, int nblk) {
  const int in_chunk = blockIdx.x % FXR_CHUNK, rest = blockIdx.x / FXR_CHUNK;
  const int blk = rest % nblk, slot = (rest / nblk) * FXR_CHUNK + in_chunk;
  if (slot >= n) return;  // ragged last chunk: the whole block leaves together
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, hs = warp & 1, vh = g.Vh;
  const int site = blk * FXR_SITES + (warp >> 1) * 32 + lane;
  const int i = min(site, vh - 1);
  const int rhs = list[slot];
  const FxF xo = xown.at(rhs);
  long long up[6], low[6];
  int Em;
  bool bad;
  fxf_hop<false, false>(g, p_out, i, hs, xin.at(rhs), U, up, low, Em, bad);
  int c[4];
  coords_of(g, p_out, i, c);
  const double2 *bp = b + ((size_t)rhs * g.V + site_of(g, c)) * 12;
  double2 bv[6];
  int mb = 0;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    bv[k] = bp[(k < 3 ? hs * 3 : 3 + hs * 3) + k];  // rows hs and 2 + hs
    mb = fx_max(mb, bv[k]);
  }
  const int Eb = mb >> 20, Ex = xo.e[i];
  const int Ey = Em > 0 ? Em + ek - 1017 : 0;  // kappa H x
  bad = bad || Ex < 0 || Eb > FX_EMAX;
  const int Er = max(max(Ey, Ex), max(Eb, FX_EMIN));
  const int dx = min(Er - Ex, 63), dy = min(Er - Ey, 63);
  // r = I 2^(Er - 1079); FP32 as two power-of-two factors
  const float2 f = pow2_pair(Er - 1079 + shift[slot]);
  const int4 *xs = xo.site(i);
  float2 v[6];
  float rn = 0.f;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const int4 t = xs[32 * ((k < 3 ? hs * 3 : 3 + hs * 3) + k)];
    long long y[2], xi[2] = {fx_value(t.x, t.y), fx_value(t.z, t.w)};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const long long acc = (k < 3 ? up[2 * k + h] : low[2 * (k - 3) + h]) >> 5;
      int ah, al;
      fx_split(acc, ah, al);
      y[h] = fx_mad(ah, kh, 0) + ((fx_mad(al, kh, fx_mad(ah, kl, 0)) + (1ll << 28)) >> 29);
    }
    const long long re = fx_int<FXF_SH>(bv[k].x, Er) - (Ex > 0 ? xi[0] >> dx : 0) + (Em > 0 ? y[0] >> dy : 0);
    const long long im = fx_int<FXF_SH>(bv[k].y, Er) - (Ex > 0 ? xi[1] >> dx : 0) + (Em > 0 ? y[1] >> dy : 0);
    v[k] = make_float2(__ll2float_rn(re) * f.x * f.y, __ll2float_rn(im) * f.x * f.y);
    if (bad) v[k] = make_float2(__int_as_float(0x7fffffff), __int_as_float(0x7fffffff));
    rn = fmaf(v[k].x, v[k].x, fmaf(v[k].y, v[k].y, rn));
  }
  if (site < vh) {
    // quads of [6][Vh] float4: row 0 fills quad 0 and half of 1, row 1 the rest of 1 and 2
    float4 *o = r.d + (size_t)rhs * 6 * vh + i;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 *w = v + 3 * h;
      float4 *q = o + (size_t)(3 * h) * vh;
      const float2 p0 = hs ? w[1] : w[0], p1 = hs ? w[2] : w[1], sgl = hs ? w[0] : w[2];
      q[hs ? 2 * (size_t)vh : 0] = make_float4(p0.x, p0.y, p1.x, p1.y);
      reinterpret_cast<float2 *>(q + vh)[hs] = sgl;
    }
  } else {
    rn = 0.f;
  }
  __shared__ float sh[2 * FXR_SITES];
  sh[threadIdx.x] = rn;
  __syncthreads();
  if (threadIdx.x < 32) {
    double t = ((double)sh[lane] + (double)sh[lane + 32]) + ((double)sh[lane + 64] + (double)sh[lane + 96]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) part[((size_t)slot * 2 + p_out) * nblk + blk] = t;
  }
}

__global__ void k_fx_resid_fin(const double *part, int nb, double *rr) {
  double a = 0.0;
  for (int k = threadIdx.x; k < nb; k += 32) a += part[(size_t)blockIdx.x * nb + k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
  if (threadIdx.x == 0) rr[blockIdx.x] = a;
}

// ---------------------------------------------------------- back to FP64
// Canonical FP64 x from the limbs; right-hand sides without a started iterate
// (have == 0) get zeros.  JOIN_SITES parity-local indices own 2 JOIN_SITES
// consecutive canonical sites, staged through shared memory so that reads and
// writes are coalesced (records of 24 + 1 elements against bank conflicts).
constexpr int JOIN_SITES = 64;
__global__ void __launch_bounds__(2 * JOIN_SITES) k_fx_join(Geom g, FxF x0, FxF x1, const double *have, double2 *out,
                                                            int nbj) {
  __shared__ double2 tile[JOIN_SITES * 25];
  const int rhs = blockIdx.x / nbj, i0 = (blockIdx.x % nbj) * JOIN_SITES;
  const int nloc = min(JOIN_SITES, g.Vh - i0);
  double2 *dst = out + ((size_t)rhs * g.V + 2 * (size_t)i0) * 12;
  const int li = threadIdx.x & (JOIN_SITES - 1), p = threadIdx.x / JOIN_SITES;
  if (have[rhs] != 0.0) {
    if (li < nloc) {
      const int i = i0 + li;
      const FxF x = (p ? x1 : x0).at(rhs);
      const int4 *xs = x.site(i);
      const int E = x.e[i];
      int rr = i / g.Lxh;
      const int y = rr % g.L[1];
      rr /= g.L[1];
      const int odd_first = (y + rr % g.L[2] + rr / g.L[2]) & 1;  // is site 2 i the odd one?
      double2 *t = tile + li * 25 + (p == odd_first ? 0 : 12);
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        const int4 q = E > 0 ? xs[32 * k] : make_int4(0, 0, 0, 0);
        t[k] = E < 0 ? make_double2(__longlong_as_double(0x7ff8000000000000ll), __longlong_as_double(0x7ff8000000000000ll))
                     : make_double2(fx_double<FXF_SH>(fx_value(q.x, q.y), E), fx_double<FXF_SH>(fx_value(q.z, q.w), E));
      }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < nloc * 24; k += 2 * JOIN_SITES) dst[k] = tile[k / 24 * 25 + k % 24];
  } else {
    for (int k = threadIdx.x; k < nloc * 24; k += 2 * JOIN_SITES) dst[k] = make_double2(0.0, 0.0);
  }
}

// ------------------------------------------------------------- host side
static FxF fx_parity(const FxIterate &x, int p, int vh) {
  const int vb = fx_blocks(vh);
  return FxF{x.d + (size_t)p * x.cap * vb * 384, x.e + (size_t)p * x.cap * vb * 32, vb};
}

int fx_accum(lqcd_ctx *ctx, const FxIterate &x, const F32F &e, const F32F &o, const double *scale, bool first,
             const int *list, const int *count, int G, cudaStream_t st) {
  const int vh = ctx->geom.Vh;
  const FxF x0 = fx_parity(x, 0, vh), x1 = fx_parity(x, 1, vh);
  const int nbx = (vh + ST - 1) / ST;
  if (first) KL k_fx_accum<true><<<G, ST, 0, st>>>(e, o, x0, x1, scale, list, count, nbx, vh);
  else KL k_fx_accum<false><<<G, ST, 0, st>>>(e, o, x0, x1, scale, list, count, nbx, vh);
  LQCD_LAUNCH_CHECK(ctx, "k_fx_accum");
  return LQCD_OK;
}

int fx_join(lqcd_ctx *ctx, const FxIterate &x, const double *have, double2 *out, int nrhs, cudaStream_t st) {
  const Geom &g = ctx->geom;
  const int nbj = (g.Vh + JOIN_SITES - 1) / JOIN_SITES;
  KL k_fx_join<<<(unsigned)((size_t)nrhs * nbj), 2 * JOIN_SITES, 0, st>>>(g, fx_parity(x, 0, g.Vh),
                                                                         fx_parity(x, 1, g.Vh), have, out, nbj);
  LQCD_LAUNCH_CHECK(ctx, "k_fx_join");
  return LQCD_OK;
}

int fx_residual(lqcd_ctx *ctx, const FxIterate &x, const double2 *b, const F32F r[2], const int *list,
                const int *shift, int n, double *rr, cudaStream_t st) {
  if (n <= 0) return LQCD_OK;
  const Geom &g = ctx->geom;
  const int nblk = (g.Vh + FXR_SITES - 1) / FXR_SITES;
  int rc = LQCD_OK;
  Carver sizing(nullptr);
  sizing.take<double>((size_t)n * 2 * nblk);
  sizing.take<double>((size_t)n);
  sizing.take<int>(2 * (size_t)n);
  void *w = workspace(ctx, WS_F64_PART, sizing.size(), &rc);
  if (!w) return rc;
  Carver cv(w);
  double *part = cv.take<double>((size_t)n * 2 * nblk);
  double *d_rr = cv.take<double>((size_t)n);
  int *d_list = cv.take<int>(2 * (size_t)n);
  std::vector<int> up(list, list + n);
  up.insert(up.end(), shift, shift + n);
  LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(d_list, up.data(), 2 * n * sizeof(int), cudaMemcpyHostToDevice, st));
  // kappa as 58 bits below its exponent
  unsigned long long kb;
  const double kappa = ctx->kappa;
  memcpy(&kb, &kappa, sizeof(kb));
  const int ek = (int)((kb >> 52) & 0x7ff);
  long long K = ek ? (long long)((kb & 0xfffffffffffffull) | 0x10000000000000ull) << 5 : 0;
  if (kb >> 63) K = -K;
  int kh, kl;
  fx_split(K, kh, kl);
  const long long blocks = (long long)((n + FXR_CHUNK - 1) / FXR_CHUNK) * nblk * FXR_CHUNK;
  for (int p = 0; p < 2; ++p) {
    KL k_fx_resid<<<(unsigned)blocks, 2 * FXR_SITES, 0, st>>>(g, p, ctx->Ufx, fx_parity(x, 1 - p, g.Vh),
                                                              fx_parity(x, p, g.Vh), b, r[p], kh, kl, ek, d_list, d_list + n,
                                                              n, part, nblk);
    LQCD_LAUNCH_CHECK(ctx, "k_fx_resid");
  }
  KL k_fx_resid_fin<<<n, 32, 0, st>>>(part, 2 * nblk, d_rr);
  LQCD_LAUNCH_CHECK(ctx, "k_fx_resid_fin");
  std::vector<double> h(n);
  LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(h.data(), d_rr, n * sizeof(double), cudaMemcpyDeviceToHost, st));
  LQCD_CUDA_TRY(ctx, cudaStreamSynchronize(st));
  for (int j = 0; j < n; ++j) rr[list[j]] = std::ldexp(h[j], -2 * shift[j]);
  return LQCD_OK;
}

}  // namespace lqcd
