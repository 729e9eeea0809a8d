// FP64 path: Wilson hopping term, full-operator application, and the plain
// even-odd preconditioned BiCGstab solver (Sec. II: BiCGstab inversions;
// Sec. III: stop on |M x - b| / |b|).
//
// Layouts: canonical fields are [rhs][V][12] double2 (site-lexicographic);
// solver vectors are parity-compact [rhs][Vh][12] double2 with parity-local
// index i = site >> 1.  The gauge field is the canonical [V][4][9] copy.
#include <algorithm>
#include <cmath>
#include <vector>

#include "internal.cuh"
#include "fxfield.cuh"

namespace lqcd {

// ------------------------------------------------------------------ hopping
template <int MU, bool DAG, bool IN_CANON>
__device__ __forceinline__ void hop_dir64(const Geom &g, const int c[4], int s, const double2 *__restrict__ in,
                                          const double2 *__restrict__ U, double2 acc[4][3]) {
  constexpr int SF = DAG ? +1 : -1;  // projector sign of the forward hop
  constexpr int SB = -SF;
  double2 ps[4][3], h[2][3], x[2][3], u[3][3];
  // forward: (1 + SF gamma_mu) U_mu(x) psi(x + mu)
  {
    int cn[4] = {c[0], c[1], c[2], c[3]};
    cn[MU] = (c[MU] + 1 == g.L[MU]) ? 0 : c[MU] + 1;
    int sn = site_of(g, cn);
    const double2 *p = in + (size_t)(IN_CANON ? sn : (sn >> 1)) * 12;
#pragma unroll
    for (int k = 0; k < 12; ++k) ps[k / 3][k % 3] = p[k];
    const double2 *up = U + ((size_t)s * 4 + MU) * 9;
#pragma unroll
    for (int k = 0; k < 9; ++k) u[k / 3][k % 3] = up[k];
    spin_project<MU, SF>(ps, h);
    su3_mul<false>(u, h, x);
    if (MU == 3 && c[3] == g.L[3] - 1) {
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) x[a][b] = cscale(x[a][b], -1.0);
    }
    spin_accum<MU, SF>(acc, x);
  }
  // backward: (1 + SB gamma_mu) U_mu(x - mu)^+ psi(x - mu)
  {
    int cn[4] = {c[0], c[1], c[2], c[3]};
    cn[MU] = (c[MU] == 0) ? g.L[MU] - 1 : c[MU] - 1;
    int sn = site_of(g, cn);
    const double2 *p = in + (size_t)(IN_CANON ? sn : (sn >> 1)) * 12;
#pragma unroll
    for (int k = 0; k < 12; ++k) ps[k / 3][k % 3] = p[k];
    const double2 *up = U + ((size_t)sn * 4 + MU) * 9;
#pragma unroll
    for (int k = 0; k < 9; ++k) u[k / 3][k % 3] = up[k];
    spin_project<MU, SB>(ps, h);
    su3_mul<true>(u, h, x);
    if (MU == 3 && c[3] == 0) {
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) x[a][b] = cscale(x[a][b], -1.0);
    }
    spin_accum<MU, SB>(acc, x);
  }
}

// out = cA*A + cB*B + cH*(H in) at the sites of parity p_out, per RHS (grid.y).
// Bound by the FP64 pipe (about 1.7 operations per cycle and SM): the SU(3) products
// as chains of fused multiply-adds take 864 operations per site instead of 1056;
// D on 12 right-hand sides of 16^3 x 32 3.29 -> 2.63 ms.
// A, B share out's layout; either may be null.  Inactive RHS are skipped.
template <bool DAG, bool IN_CANON, bool OUT_CANON>
__global__ void __launch_bounds__(128) k_hop64(Geom g, int p_out, const double2 *__restrict__ U,
                                               const double2 *__restrict__ in, size_t in_stride, double2 *out,
                                               size_t out_stride, const double2 *A, double cA, const double2 *B,
                                               double cB, double cH, const int *active) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int rhs = blockIdx.y;
  if (i >= g.Vh) return;
  if (active && !active[rhs]) return;
  int c[4];
  coords_of(g, p_out, i, c);
  int s = site_of(g, c);
  double2 acc[4][3];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) acc[a][b] = make_double2(0.0, 0.0);
  const double2 *inr = in + (size_t)rhs * in_stride;
  hop_dir64<0, DAG, IN_CANON>(g, c, s, inr, U, acc);
  hop_dir64<1, DAG, IN_CANON>(g, c, s, inr, U, acc);
  hop_dir64<2, DAG, IN_CANON>(g, c, s, inr, U, acc);
  hop_dir64<3, DAG, IN_CANON>(g, c, s, inr, U, acc);
  size_t o = (size_t)rhs * out_stride + (size_t)(OUT_CANON ? s : i) * 12;
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    double2 v = cscale(acc[k / 3][k % 3], cH);
    if (A) v = cadd(v, cscale(A[o + k], cA));
    if (B) v = cadd(v, cscale(B[o + k], cB));
    out[o + k] = v;
  }
}

// H in at one site in FP64: rows hs and 2 + hs
template <bool DAG, bool IN_CANON>
__device__ __noinline__ void hop_site64(const Geom &g, int p_out, int i, int hs, const double2 *in, const double2 *U,
                                        double2 out[6]) {
  int c[4];
  coords_of(g, p_out, i, c);
  const int s = site_of(g, c);
  double2 acc[4][3];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) acc[a][b] = make_double2(0.0, 0.0);
  hop_dir64<0, DAG, IN_CANON>(g, c, s, in, U, acc);
  hop_dir64<1, DAG, IN_CANON>(g, c, s, in, U, acc);
  hop_dir64<2, DAG, IN_CANON>(g, c, s, in, U, acc);
  hop_dir64<3, DAG, IN_CANON>(g, c, s, in, U, acc);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    out[k] = hs ? acc[1][k] : acc[0][k];
    out[3 + k] = hs ? acc[3][k] : acc[2][k];
  }
}

// The same by a whole warp (all lanes call, with one site; every lane receives the rows):
// lane 4 q + a forms colour a of neighbour q = 2 mu + (0 forward, 1 backward), 48 FP64
// operations in sequence and so about 3,000 cycles, where one lane alone takes 55,000.
constexpr int HOP_WARP_SITES = 16;  // as many of a warp's sites take less time like this
template <bool DAG, bool IN_CANON>
__device__ __noinline__ void hop_site64_warp(const Geom &g, int p_out, int i, int hs, const double2 *in, const double2 *U,
                                             double2 out[6]) {
  const int lane = threadIdx.x & 31, q = lane >> 2, a = min(lane & 3, 2), mu = q >> 1;
  const bool fwd = !(q & 1);
  int c[4];
  coords_of(g, p_out, i, c);
  const int s = site_of(g, c);
  int sn = s, stride = 1;
  bool edge = false;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int L = g.L[m];
    if (m == mu) {
      edge = fwd ? c[m] + 1 == L : c[m] == 0;
      sn = s + (fwd ? (edge ? stride * (1 - L) : stride) : (edge ? stride * (L - 1) : -stride));
    }
    stride *= L;
  }
  const double2 *p = in + (size_t)(IN_CANON ? sn : (sn >> 1)) * 12;
  const double2 *u = U + ((size_t)(fwd ? s : sn) * 4 + mu) * 9;
  const bool minus = fwd != DAG, imag = !(mu & 1);  // projector 1 -+ gamma_mu; its phases
  const bool wrap = mu == 3 && edge;
  // U h_r for row r = 0, 1 of the projection: h_r = psi_r + phase psi_low
  auto eps = [&](int r) { return minus != ((mu == 1 && r == 0) || (mu == 2 && r == 1)); };  // phase < 0
  auto half = [&](int r) {
    const int low = mu < 2 ? 3 - r : 2 + r;
    const bool neg = eps(r);
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const double2 x = p[r * 3 + b], y = p[low * 3 + b], t = imag ? cmuli(y) : y;
      double2 w = u[fwd ? a * 3 + b : b * 3 + a];
      if (!fwd) w.y = -w.y;
      acc = cmac(acc, w, neg ? csub(x, t) : cadd(x, t));
    }
    if (wrap) acc = make_double2(-acc.x, -acc.y);
    return acc;
  };
  const int rl = mu < 2 ? 1 - hs : hs;  // row 2 + hs is the conjugate phase of h_rl
  double2 up = half(hs), lo = half(rl);
  if (imag) lo = make_double2(lo.y, -lo.x);
  if (eps(rl)) lo = make_double2(-lo.x, -lo.y);
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    up.x += __shfl_xor_sync(0xffffffffu, up.x, o);
    up.y += __shfl_xor_sync(0xffffffffu, up.y, o);
    lo.x += __shfl_xor_sync(0xffffffffu, lo.x, o);
    lo.y += __shfl_xor_sync(0xffffffffu, lo.y, o);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    out[k] = make_double2(__shfl_sync(0xffffffffu, up.x, k), __shfl_sync(0xffffffffu, up.y, k));
    out[3 + k] = make_double2(__shfl_sync(0xffffffffu, lo.x, k), __shfl_sync(0xffffffffu, lo.y, k));
  }
}

// out = cA A + cB B + cH v at rows hs and 2 + hs (v) of one site, o: its row hs
__device__ __forceinline__ void hop64_store(const double2 v[6], size_t o, double2 *out, const double2 *A, double cA,
                                            const double2 *B, double cB, double cH) {
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const size_t e = o + (k < 3 ? k : 3 + k);
    double2 w = v[k];
    if (A) {  // one fused multiply-add per component where cA = 1, the usual call
      const double2 a = A[e], t = cA == 1.0 ? a : cscale(a, cA);
      w = make_double2(fma(cH, w.x, t.x), fma(cH, w.y, t.y));
    } else if (cH != 1.0) {
      w = cscale(w, cH);
    }
    if (B) {
      const double2 b = B[e];
      w = make_double2(fma(cB, b.x, w.x), fma(cB, b.y, w.y));
    }
    out[e] = w;
  }
}

// FP64 field -> integer limbs: canonical (both parities) or the compact field of one
// parity (f0).  Thread per site and right-hand side (grid.y).
template <bool CANON>
__global__ void __launch_bounds__(128) k_fx_from64(Geom g, const double2 *__restrict__ in, size_t in_stride, FxF f0,
                                                   FxF f1, const int *active) {
  const int rhs = blockIdx.y, idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (active && !active[rhs]) return;
  if (idx >= (CANON ? g.V : g.Vh)) return;
  int p = 0, i = idx;
  if (CANON) {
    int r = idx / g.L[0];
    const int y = r % g.L[1];
    r /= g.L[1];
    p = (idx % g.L[0] + y + r % g.L[2] + r / g.L[2]) & 1;
    i = idx >> 1;
  }
  const double2 *q = in + (size_t)rhs * in_stride + (size_t)idx * 12;
  const FxF f = (p ? f1 : f0).at(rhs);
  double2 v[12];
  int m[4] = {0, 0, 0, 0};
  unsigned low[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int k = 0; k < 12; ++k) v[k] = q[k];
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    m[k / 3] = fx_max(m[k / 3], v[k]);
    low[k / 3] |= __double2loint(v[k].x) | __double2loint(v[k].y);
  }
  const int E = fx_site_exp(max(max(m[0], m[1]), max(m[2], m[3])), low[0] | low[1] | low[2] | low[3]);
  f.e[i] = E > 0 ? fx_with_rows(E, m, low) : E;
  if (E <= 0) return;  // the limbs of such a site are not read
  int4 *o = f.site(i);
#pragma unroll
  for (int k = 0; k < 12; ++k)
    o[32 * k] = fx_split_c(fx_int<FXF_SH>(v[k].x, E), fx_int<FXF_SH>(v[k].y, E));
}

// The hopping term with its SU(3) products on the integer units (fx64.cuh), on a field
// of integer limbs (fxfield.cuh); the FP64 field `in` it was made from serves the sites
// that have no integer form or whose rows are of very different size.  D on 12
// right-hand sides of 16^3 x 32, conversion included: 2.63 ms in FP64 arithmetic
// (k_hop64), 1.31 ms when each neighbour is converted where it is used, 1.00 ms here;
// one right-hand side of 4^4: 32 us.  Near a point source some sites always have such
// rows: with each of them left to its lane 768 point sources of 4^4 took 5.44 ms to
// solve, by whole warps 5.07 (4.74 without a look at the rows).
template <bool DAG, bool IN_CANON, bool OUT_CANON>
__global__ void __launch_bounds__(128, 4) k_hop64_fxf(Geom g, int p_out, const double2 *__restrict__ U,
                                                      const int4 *__restrict__ Ufx, FxF f,
                                                      const double2 *__restrict__ in, size_t in_stride, double2 *out,
                                                      size_t out_stride, const double2 *A, double cA, const double2 *B,
                                                      double cB, double cH, const int *active) {
  const int rhs = blockIdx.y, warp = threadIdx.x >> 5, hs = warp & 1;
  if (active && !active[rhs]) return;
  const int site = blockIdx.x * 64 + (warp >> 1) * 32 + (threadIdx.x & 31), i = min(site, g.Vh - 1);
  long long up[6], low[6];
  int Em;
  bool bad;
  fxf_hop<DAG, true>(g, p_out, i, hs, f.at(rhs), Ufx, up, low, Em, bad);
  double2 v[6];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    v[k] = make_double2(fx_double<FXF_SH>(up[2 * k], Em), fx_double<FXF_SH>(up[2 * k + 1], Em));
    v[3 + k] = make_double2(fx_double<FXF_SH>(low[2 * k], Em), fx_double<FXF_SH>(low[2 * k + 1], Em));
  }
  bad = bad && site < g.Vh;
  unsigned todo = __ballot_sync(0xffffffffu, bad);
  if (__popc(todo) > HOP_WARP_SITES) {
    if (bad) hop_site64<DAG, IN_CANON>(g, p_out, i, hs, in + (size_t)rhs * in_stride, U, v);
    todo = 0u;
  }
  while (todo) {
    const int src = __ffs(todo) - 1;
    todo &= todo - 1;
    double2 w[6];
    hop_site64_warp<DAG, IN_CANON>(g, p_out, __shfl_sync(0xffffffffu, i, src), hs, in + (size_t)rhs * in_stride, U, w);
    if ((threadIdx.x & 31) == src) {
#pragma unroll
      for (int k = 0; k < 6; ++k) v[k] = w[k];
    }
  }
  if (site >= g.Vh) return;
  size_t s = i;
  if (OUT_CANON) {
    int c[4];
    coords_of(g, p_out, i, c);
    s = site_of(g, c);
  }
  hop64_store(v, (size_t)rhs * out_stride + s * 12 + hs * 3, out, A, cA, B, cB, cH);
}

static bool capturing(cudaStream_t st) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  const bool err = cudaStreamIsCapturing(st, &cap) != cudaSuccess;
  if (err) cudaGetLastError();
  return err || cap != cudaStreamCaptureStatusNone;
}
FxUse::FxUse(lqcd_ctx *c, cudaStream_t s) : ok(c->fx_links), ctx(c), st(s) {
  if (ctx->fx_depth++ > 0) {  // within another use, which is on the same stream
    ok = ctx->fx_ok;
    return;
  }
  if (ok && !capturing(st)) {
    ok = record = cudaStreamWaitEvent(st, ctx->fx_ev, 0) == cudaSuccess;
    if (!ok) cudaGetLastError();
  }
  ctx->fx_ok = ok;
}
FxUse::~FxUse() {
  --ctx->fx_depth;
  if (record && cudaEventRecord(ctx->fx_ev, st) != cudaSuccess) {  // nothing to wait for: be done first
    cudaGetLastError();
    cudaStreamSynchronize(st);
  }
}

// Workspace of integer limbs for both parities of some right-hand sides: as many as keep it
// in L2 (FX_WS_BYTES), at least one and at most FX_WS_RHS.  It is reserved with the gauge
// field: D enqueues its work and allocates nothing.  The first lqcd_set_gauge of a context
// takes 0.19 ms instead of 0.10 on 4^4 for it, as much with room for 128 (a larger
// allocation as such; on 8^3 x 16 0.41 instead of 0.38).
constexpr size_t FX_WS_BYTES = 96u << 20;
constexpr size_t FX_WS_RHS = 1024;
static size_t fx_rhs_bytes(const lqcd_ctx *ctx) {
  return (size_t)2 * fx_blocks(ctx->geom.Vh) * 32 * (12 * sizeof(int4) + sizeof(int));
}
static int fx_max_chunk(const lqcd_ctx *ctx) {
  return (int)std::max<size_t>(1, std::min(FX_WS_RHS, FX_WS_BYTES / fx_rhs_bytes(ctx)));
}
void fx_reserve(lqcd_ctx *ctx) {
  int rc = LQCD_OK;
  workspace(ctx, WS_FX, fx_rhs_bytes(ctx) * fx_max_chunk(ctx), &rc);  // (if refused: FP64 arithmetic)
}
// The workspace and how many right-hand sides it takes at a time, or null: where it was
// refused, and while the stream is being captured, when the caller takes FP64 arithmetic
// (a graph's replays are not ordered with other uses).
static char *fx_workspace(lqcd_ctx *ctx, int nrhs, int *chunk, cudaStream_t st) {
  if (capturing(st)) return nullptr;
  *chunk = std::min(nrhs, fx_max_chunk(ctx));
  return (char *)ctx->ws[WS_FX].p;
}
// one launch; fx: the input as integer limbs, or null
static int launch_hop64_one(lqcd_ctx *ctx, cudaStream_t st, bool dag, bool in_canon, bool out_canon, int p_out,
                            const double2 *in, size_t in_stride, double2 *out, size_t out_stride, const double2 *A,
                            double cA, const double2 *B, double cB, double cH, const int *active, int nrhs,
                            const FxF *fx) {
  const Geom &g = ctx->geom;
  const dim3 grid((g.Vh + 127) / 128, nrhs);
#define HOP64_CASE(D, IC, OC)                                                                                   \
  if (dag == D && in_canon == IC && out_canon == OC) {                                                          \
    if (!fx)                                                                                                    \
      KL k_hop64<D, IC, OC><<<grid, 128, 0, st>>>(g, p_out, ctx->U64, in, in_stride, out, out_stride, A, cA, B, \
                                                  cB, cH, active);                                              \
    else                                                                                                        \
      KL k_hop64_fxf<D, IC, OC><<<dim3((g.Vh + 63) / 64, nrhs), 128, 0, st>>>(                                  \
          g, p_out, ctx->U64, ctx->Ufx, *fx, in, in_stride, out, out_stride, A, cA, B, cB, cH, active);         \
    LQCD_LAUNCH_CHECK(ctx, "k_hop64");                                                                          \
    return LQCD_OK;                                                                                             \
  }
  HOP64_CASE(false, false, false)
  HOP64_CASE(false, true, true)
  HOP64_CASE(true, true, true)
  HOP64_CASE(true, false, false)
#undef HOP64_CASE
  return set_error(ctx, LQCD_ERR_INVALID, "launch_hop64: unsupported layout combination");
}

static FxF fx_carve(char *w, int p, int vh, int chunk) {
  const int vb = fx_blocks(vh);
  const size_t nd = (size_t)chunk * vb * 384;
  return FxF{(int4 *)w + p * nd, (int *)((int4 *)w + 2 * nd) + (size_t)p * chunk * vb * 32, vb};
}

int launch_hop64(lqcd_ctx *ctx, cudaStream_t st, bool dag, bool in_canon, bool out_canon, int p_out,
                 const double2 *in, size_t in_stride, double2 *out, size_t out_stride, const double2 *A, double cA,
                 const double2 *B, double cB, double cH, const int *active, int nrhs) {
  const Geom &g = ctx->geom;
  int chunk = 0;
  char *w = nullptr;
  const FxUse use(ctx, st);
  if (use.ok) w = fx_workspace(ctx, nrhs, &chunk, st);
  if (!w)
    return launch_hop64_one(ctx, st, dag, in_canon, out_canon, p_out, in, in_stride, out, out_stride, A, cA, B, cB, cH,
                            active, nrhs, nullptr);
  const FxF f0 = fx_carve(w, 0, g.Vh, chunk), f1 = fx_carve(w, 1, g.Vh, chunk);
  for (int r = 0; r < nrhs; r += chunk) {
    const int n = std::min(chunk, nrhs - r);
    const int *act = active ? active + r : nullptr;
    const double2 *inr = in + (size_t)r * in_stride;
    const size_t o = (size_t)r * out_stride;
    if (in_canon)
      KL k_fx_from64<true><<<dim3((g.V + 127) / 128, n), 128, 0, st>>>(g, inr, in_stride, f0, f1, act);
    else
      KL k_fx_from64<false><<<dim3((g.Vh + 127) / 128, n), 128, 0, st>>>(g, inr, in_stride, f0, f0, act);
    LQCD_LAUNCH_CHECK(ctx, "k_fx_from64");
    const FxF &f = in_canon && p_out == 0 ? f1 : f0;  // the neighbours' parity
    int rc = launch_hop64_one(ctx, st, dag, in_canon, out_canon, p_out, inr, in_stride, out + o, out_stride,
                              A ? A + o : nullptr, cA, B ? B + o : nullptr, cB, cH, act, n, &f);
    if (rc) return rc;
  }
  return LQCD_OK;
}

int fp64_apply_dirac(lqcd_ctx *ctx, const double2 *in, double2 *out, int nrhs, bool dagger, cudaStream_t st) {
  const Geom &g = ctx->geom;
  const size_t stride = (size_t)g.V * 12;
  int chunk = nrhs;
  char *w = nullptr;
  const FxUse use(ctx, st);
  if (use.ok) w = fx_workspace(ctx, nrhs, &chunk, st);
  if (!w) chunk = nrhs;
  for (int r = 0; r < nrhs; r += chunk) {
    const int n = std::min(chunk, nrhs - r);
    const double2 *inr = in + (size_t)r * stride;
    double2 *outr = out + (size_t)r * stride;
    FxF f[2];
    if (w) {
      f[0] = fx_carve(w, 0, g.Vh, chunk);
      f[1] = fx_carve(w, 1, g.Vh, chunk);
      KL k_fx_from64<true><<<dim3((g.V + 127) / 128, n), 128, 0, st>>>(g, inr, stride, f[0], f[1], nullptr);
      LQCD_LAUNCH_CHECK(ctx, "k_fx_from64");
    }
    for (int p = 0; p < 2; ++p) {
      int rc = launch_hop64_one(ctx, st, dagger, true, true, p, inr, stride, outr, stride, inr, 1.0, nullptr, 0.0,
                                -ctx->kappa, nullptr, n, w ? &f[1 - p] : nullptr);
      if (rc) return rc;
    }
  }
  return LQCD_OK;
}

// --------------------------------------------------------- layout changes
// canonical [rhs][V][12] -> compact parity p [rhs][Vh][12] (and back)
__global__ void k_split64(Geom g, int p, const double2 *__restrict__ full, double2 *half) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int rhs = blockIdx.y;
  if (i >= g.Vh) return;
  int c[4];
  coords_of(g, p, i, c);
  int s = site_of(g, c);
  const double2 *src = full + ((size_t)rhs * g.V + s) * 12;
  double2 *dst = half + ((size_t)rhs * g.Vh + i) * 12;
#pragma unroll
  for (int k = 0; k < 12; ++k) dst[k] = src[k];
}

__global__ void k_merge64(Geom g, int p, const double2 *__restrict__ half, double2 *full, const int *active) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int rhs = blockIdx.y;
  if (i >= g.Vh) return;
  if (active && !active[rhs]) return;
  int c[4];
  coords_of(g, p, i, c);
  int s = site_of(g, c);
  const double2 *src = half + ((size_t)rhs * g.Vh + i) * 12;
  double2 *dst = full + ((size_t)rhs * g.V + s) * 12;
#pragma unroll
  for (int k = 0; k < 12; ++k) dst[k] = src[k];
}

// ------------------------------------------------------------ reductions
struct D4 {
  double a, b, c, d;
};

// Sums over a warp of the four fields, in a fixed order: a on lane 0, b on lane 8, c on
// lane 16, d on lane 24.  A lane hands the fields that its partner keeps over to it, so
// that the warp does 6 FP64 additions, of 64 cycles or more each, instead of 20.
__device__ __forceinline__ double warp_sum4(const D4 &v) {
  const int lane = threadIdx.x & 31;
  const bool up16 = lane & 16, up8 = lane & 8;
  const double t = __shfl_xor_sync(0xffffffffu, up16 ? v.a : v.c, 16);
  const double u = __shfl_xor_sync(0xffffffffu, up16 ? v.b : v.d, 16);
  const double x = (up16 ? v.c : v.a) + t, y = (up16 ? v.d : v.b) + u;
  double z = (up8 ? y : x) + __shfl_xor_sync(0xffffffffu, up8 ? x : y, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
  return z;
}
__device__ __forceinline__ D4 gather4(double z) {  // the four sums of warp_sum4 on every lane
  return D4{__shfl_sync(0xffffffffu, z, 0), __shfl_sync(0xffffffffu, z, 8), __shfl_sync(0xffffffffu, z, 16),
            __shfl_sync(0xffffffffu, z, 24)};
}

// block-wide sum of 4 doubles in a fixed order, for blocks of up to eight warps; valid in
// the first warp.  With 20 + 20 additions, the FP64 solve of 768
// right-hand sides of 4^4 took 4.87 ms, and 4.70 with these.
__device__ __forceinline__ D4 block_sum4(const D4 &v) {
  __shared__ double sh[8][4];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const double z = warp_sum4(v);
  if ((lane & 7) == 0) sh[w][lane >> 3] = z;
  __syncthreads();
  D4 r = {0, 0, 0, 0};
  if (w == 0) {
    double t = (lane & 7) < (int)(blockDim.x >> 5) ? sh[lane & 7][lane >> 3] : 0.0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    r = gather4(t);
  }
  __syncthreads();
  return r;
}

// per-RHS solver scalars
struct S64 {
  double2 rho, alpha, omega, beta;
  double rr, target2, bb, rel;
  int iters, status, restart, pad;
};

#define RED_THREADS 256

// p = r + beta (p - omega v); on restart: rhat = r, p = r.
__global__ void __launch_bounds__(RED_THREADS) k_bicg_p(size_t n, S64 *sc, const int *active, const double2 *r,
                                                        double2 *rhat, double2 *p, const double2 *v) {
  int rhs = blockIdx.y;
  if (!active[rhs]) return;
  const S64 s = sc[rhs];
  size_t off = (size_t)rhs * n;
  for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x) {
    double2 rk = r[off + k];
    if (s.restart) {
      rhat[off + k] = rk;
      p[off + k] = rk;
    } else {
      double2 t = cmac(p[off + k], cscale(s.omega, -1.0), v[off + k]);
      p[off + k] = cmac(rk, s.beta, t);
    }
  }
}

// partial <a, b> (complex), or |a|^2 in .c (NORM; b unused).  These sums are bound by
// the FP64 pipe, so each kernel forms only what its finaliser reads, in chains of
// fused multiply-adds (4 or 2 operations per element).
template <bool NORM>
__global__ void __launch_bounds__(RED_THREADS) k_dot64(size_t n, const int *active, const double2 *a, const double2 *b,
                                                       D4 *part) {
  int rhs = blockIdx.y;
  if (!active[rhs]) return;
  size_t off = (size_t)rhs * n;
  D4 acc = {0, 0, 0, 0};
  for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x) {
    const double2 x = a[off + k];
    if (NORM) {
      acc.c = fma(x.x, x.x, fma(x.y, x.y, acc.c));
    } else {
      const double2 d = cmacc(make_double2(acc.a, acc.b), x, b[off + k]);
      acc.a = d.x;
      acc.b = d.y;
    }
  }
  D4 r = block_sum4(acc);
  if (threadIdx.x == 0) part[(size_t)rhs * gridDim.x + blockIdx.x] = r;
}

// s = r - alpha v
__global__ void __launch_bounds__(RED_THREADS) k_bicg_s(size_t n, const S64 *sc, const int *active, const double2 *r,
                                                        const double2 *v, double2 *s) {
  int rhs = blockIdx.y;
  if (!active[rhs]) return;
  double2 al = sc[rhs].alpha;
  size_t off = (size_t)rhs * n;
  for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x)
    s[off + k] = cmac(r[off + k], cscale(al, -1.0), v[off + k]);
}

// x += alpha p + omega s; r = s - omega t; partials <rhat, r>, |r|^2
__global__ void __launch_bounds__(RED_THREADS) k_bicg_xr(size_t n, const S64 *sc, const int *active, double2 *x,
                                                         const double2 *p, const double2 *s, const double2 *t,
                                                         double2 *r, const double2 *rhat, D4 *part) {
  int rhs = blockIdx.y;
  if (!active[rhs]) return;
  double2 al = sc[rhs].alpha, om = sc[rhs].omega;
  size_t off = (size_t)rhs * n;
  D4 acc = {0, 0, 0, 0};
  for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x) {
    double2 sk = s[off + k];
    x[off + k] = cadd(x[off + k], cmac(cmul(al, p[off + k]), om, sk));
    double2 rk = cmac(sk, cscale(om, -1.0), t[off + k]);
    r[off + k] = rk;
    const double2 d = cmacc(make_double2(acc.a, acc.b), rhat[off + k], rk);
    acc.a = d.x;
    acc.b = d.y;
    acc.c = fma(rk.x, rk.x, fma(rk.y, rk.y, acc.c));
  }
  D4 rr = block_sum4(acc);
  if (threadIdx.x == 0) part[(size_t)rhs * gridDim.x + blockIdx.x] = rr;
}

// fixed-order sum of the nb partials of one RHS by one warp
__device__ __forceinline__ D4 warp_total(const D4 *part, int nb) {
  int lane = threadIdx.x;
  D4 acc = {0, 0, 0, 0};
  for (int k = lane; k < nb; k += 32) {
    D4 v = part[k];
    acc.a += v.a;
    acc.b += v.b;
    acc.c += v.c;
    acc.d += v.d;
  }
  return gather4(warp_sum4(acc));
}

__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
  double d = b.x * b.x + b.y * b.y;
  return make_double2((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}

// init: r = b_hat - A x was computed; partials hold <r, r> in .c
__global__ void k_fin_init(S64 *sc, int *active, const D4 *part, int nb, int max_iter) {
  int rhs = blockIdx.x;
  if (!active[rhs]) return;
  D4 t = warp_total(part + (size_t)rhs * nb, nb);
  if (threadIdx.x != 0) return;
  S64 &s = sc[rhs];
  s.rr = t.c;
  s.rho = make_double2(t.c, 0.0);
  s.alpha = s.omega = make_double2(1.0, 0.0);
  s.beta = make_double2(0.0, 0.0);
  s.restart = 1;
  if (!isfinite(t.c)) {
    s.status = LQCD_ERR_NONFINITE;
    active[rhs] = 0;
  } else if (t.c <= s.target2) {
    active[rhs] = 0;
  } else if (s.iters >= max_iter) {
    s.status = LQCD_ERR_NOT_CONVERGED;
    active[rhs] = 0;
  }
}

__global__ void k_fin_alpha(S64 *sc, const int *active, const D4 *part, int nb) {
  int rhs = blockIdx.x;
  if (!active[rhs]) return;
  D4 t = warp_total(part + (size_t)rhs * nb, nb);
  if (threadIdx.x != 0) return;
  S64 &s = sc[rhs];
  double2 rv = make_double2(t.a, t.b);
  s.alpha = (rv.x == 0.0 && rv.y == 0.0) ? make_double2(0.0, 0.0) : cdiv(s.rho, rv);
  s.restart = 0;
}

__global__ void k_fin_omega(S64 *sc, const int *active, const D4 *part, int nb) {
  int rhs = blockIdx.x;
  if (!active[rhs]) return;
  D4 t = warp_total(part + (size_t)rhs * nb, nb);
  if (threadIdx.x != 0) return;
  S64 &s = sc[rhs];
  // part: a,b = <t, s>, c = |s|^2 (from k_dot64(t, s)); need |t|^2: stored in d by k_dot_ts
  double2 ts = make_double2(t.a, t.b);
  s.omega = (t.d == 0.0) ? make_double2(0.0, 0.0) : make_double2(ts.x / t.d, ts.y / t.d);
}

// partials <t, s> and |t|^2
__global__ void __launch_bounds__(RED_THREADS) k_dot_ts(size_t n, const int *active, const double2 *t, const double2 *s,
                                                        D4 *part) {
  int rhs = blockIdx.y;
  if (!active[rhs]) return;
  size_t off = (size_t)rhs * n;
  D4 acc = {0, 0, 0, 0};
  for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x) {
    const double2 x = t[off + k], d = cmacc(make_double2(acc.a, acc.b), x, s[off + k]);
    acc.a = d.x;
    acc.b = d.y;
    acc.d = fma(x.x, x.x, fma(x.y, x.y, acc.d));
  }
  D4 r = block_sum4(acc);
  if (threadIdx.x == 0) part[(size_t)rhs * gridDim.x + blockIdx.x] = r;
}

__global__ void k_fin_conv(S64 *sc, int *active, const D4 *part, int nb, int max_iter) {
  int rhs = blockIdx.x;
  if (!active[rhs]) return;
  D4 t = warp_total(part + (size_t)rhs * nb, nb);
  if (threadIdx.x != 0) return;
  S64 &s = sc[rhs];
  double2 rho_new = make_double2(t.a, t.b);
  s.rr = t.c;
  s.iters += 1;
  if (!isfinite(t.c) || !isfinite(t.a) || !isfinite(t.b)) {
    s.status = LQCD_ERR_NONFINITE;
    active[rhs] = 0;
    return;
  }
  if (t.c <= s.target2) {
    active[rhs] = 0;
    return;
  }
  if (s.iters >= max_iter) {
    s.status = LQCD_ERR_NOT_CONVERGED;
    active[rhs] = 0;
    return;
  }
  double om2 = s.omega.x * s.omega.x + s.omega.y * s.omega.y;
  double rho2 = rho_new.x * rho_new.x + rho_new.y * rho_new.y;
  if (om2 == 0.0 || rho2 == 0.0 || rho2 < 1e-60 * t.c * t.c) {
    // breakdown: restart the shadow residual at the current residual
    s.restart = 1;
    s.rho = make_double2(t.c, 0.0);
    s.alpha = s.omega = make_double2(1.0, 0.0);
    s.beta = make_double2(0.0, 0.0);
    return;
  }
  s.beta = cmul(cdiv(rho_new, s.rho), cdiv(s.alpha, s.omega));
  s.rho = rho_new;
}

// partial |r|^2 -> .c and |b|^2 -> .d (canonical full fields), for the true
// residual; SAME (r == b) sums once and copies
template <bool SAME>
__global__ void __launch_bounds__(RED_THREADS) k_norms64(size_t n, const double2 *r, const double2 *b, D4 *part) {
  int rhs = blockIdx.y;
  size_t off = (size_t)rhs * n;
  D4 acc = {0, 0, 0, 0};
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  // Four elements loaded before they are summed (in the same order as one at a time).
  // The sums are bound by the FP64 pipe; where a warp's elements are all zero, most of
  // a diluted source, they are left out by an integer test and the pass runs at the
  // rate of the loads (|b|^2 of 384 diluted sources of 16^3 x 32: 3.7 -> 2.4 ms).
  auto add = [&](const double2 &x, const double2 &y) {
    const unsigned bits = ((unsigned)__double2hiint(x.x) << 1) | (unsigned)__double2loint(x.x) |
                          ((unsigned)__double2hiint(x.y) << 1) | (unsigned)__double2loint(x.y);
    if (bits != 0u) acc.c = fma(x.x, x.x, fma(x.y, x.y, acc.c));
    if (!SAME) {
      const unsigned by = ((unsigned)__double2hiint(y.x) << 1) | (unsigned)__double2loint(y.x) |
                          ((unsigned)__double2hiint(y.y) << 1) | (unsigned)__double2loint(y.y);
      if (by != 0u) acc.d = fma(y.x, y.x, fma(y.y, y.y, acc.d));
    }
  };
  for (; k + 3 * stride < n; k += 4 * stride) {
    double2 x[4], y[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      x[u] = r[off + k + u * stride];
      y[u] = SAME ? x[u] : b[off + k + u * stride];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) add(x[u], y[u]);
  }
  for (; k < n; k += stride) add(r[off + k], SAME ? r[off + k] : b[off + k]);
  if (SAME) acc.d = acc.c;
  D4 rr = block_sum4(acc);
  if (threadIdx.x == 0) part[(size_t)rhs * gridDim.x + blockIdx.x] = rr;
}

__global__ void k_fin_norms(const D4 *part, int nb, double *out_rr, double *out_bb) {
  int rhs = blockIdx.x;
  D4 t = warp_total(part + (size_t)rhs * nb, nb);
  if (threadIdx.x == 0) {
    out_rr[rhs] = t.c;
    out_bb[rhs] = t.d;
  }
}

static int red_blocks(size_t n) {
  size_t nb = (n + 2047) / 2048;
  if (nb < 1) nb = 1;
  if (nb > 304) nb = 304;
  return (int)nb;
}

// true residual |b - D x|^2 and |b|^2 per RHS (host arrays), FP64 full lattice
int fp64_true_residual(lqcd_ctx *ctx, const double2 *b, const double2 *x, int nrhs, double *rr, double *bb,
                       cudaStream_t st) {
  const Geom &g = ctx->geom;
  size_t stride = (size_t)g.V * 12;
  int rc = LQCD_OK;
  double2 *res = (double2 *)workspace(ctx, WS_F64_FULL, (size_t)nrhs * stride * sizeof(double2), &rc);
  if (!res) return rc;
  int nb = red_blocks(stride);
  Carver sizing(nullptr);
  sizing.take<D4>((size_t)nrhs * nb);
  sizing.take<double>(2 * (size_t)nrhs);
  void *pw = workspace(ctx, WS_F64_PART, sizing.size(), &rc);
  if (!pw) return rc;
  Carver cv(pw);
  D4 *part = cv.take<D4>((size_t)nrhs * nb);
  double *d_rr = cv.take<double>(2 * (size_t)nrhs);
  double *d_bb = d_rr + nrhs;
  for (int p = 0; p < 2; ++p) {
    // res = b - x + kappa H x
    rc = launch_hop64(ctx, st, false, true, true, p, x, stride, res, stride, b, 1.0, x, -1.0, ctx->kappa, nullptr,
                      nrhs);
    if (rc) return rc;
  }
  KL k_norms64<false><<<dim3(nb, nrhs), RED_THREADS, 0, st>>>(stride, res, b, part);
  LQCD_LAUNCH_CHECK(ctx, "k_norms64");
  KL k_fin_norms<<<nrhs, 32, 0, st>>>(part, nb, d_rr, d_bb);
  LQCD_LAUNCH_CHECK(ctx, "k_fin_norms");
  LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(rr, d_rr, nrhs * sizeof(double), cudaMemcpyDeviceToHost, st));
  LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(bb, d_bb, nrhs * sizeof(double), cudaMemcpyDeviceToHost, st));
  LQCD_CUDA_TRY(ctx, cudaStreamSynchronize(st));
  return LQCD_OK;
}

// |b|^2 per right-hand side (host array), FP64
int fp64_norms(lqcd_ctx *ctx, const double2 *b, int nrhs, double *bb, cudaStream_t st) {
  const size_t stride = (size_t)ctx->geom.V * 12;
  const int nb = red_blocks(stride);
  int rc = LQCD_OK;
  Carver sizing(nullptr);
  sizing.take<D4>((size_t)nrhs * nb);
  sizing.take<double>(2 * (size_t)nrhs);
  void *pw = workspace(ctx, WS_F64_PART, sizing.size(), &rc);
  if (!pw) return rc;
  Carver cv(pw);
  D4 *part = cv.take<D4>((size_t)nrhs * nb);
  double *d_rr = cv.take<double>(2 * (size_t)nrhs);
  double *d_bb = d_rr + nrhs;
  KL k_norms64<true><<<dim3(nb, nrhs), RED_THREADS, 0, st>>>(stride, b, b, part);
  LQCD_LAUNCH_CHECK(ctx, "k_norms64");
  KL k_fin_norms<<<nrhs, 32, 0, st>>>(part, nb, d_rr, d_bb);
  LQCD_LAUNCH_CHECK(ctx, "k_fin_norms");
  LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(bb, d_bb, nrhs * sizeof(double), cudaMemcpyDeviceToHost, st));
  LQCD_CUDA_TRY(ctx, cudaStreamSynchronize(st));
  return LQCD_OK;
}

// ------------------------------------------------------------- the solver
// One block of nrhs right-hand sides, even-odd BiCGstab in FP64.
static int fp64_solve_block(lqcd_ctx *ctx, const double2 *b, double2 *x, int nrhs, const lqcd_solver_params &p,
                            lqcd_solve_stats *stats, cudaStream_t st, double t_start) {
  const Geom &g = ctx->geom;
  const double kappa = ctx->kappa;
  size_t n = (size_t)g.Vh * 12;  // double2 per parity vector
  size_t full = (size_t)g.V * 12;
  const int NV = 10;
  int rc = LQCD_OK;
  double2 *vec = (double2 *)workspace(ctx, WS_F64_VECS, (size_t)NV * nrhs * n * sizeof(double2), &rc);
  if (!vec) return rc;
  double2 *xe = vec, *r = vec + (size_t)nrhs * n, *rhat = r + (size_t)nrhs * n, *pp = rhat + (size_t)nrhs * n;
  double2 *v = pp + (size_t)nrhs * n, *s = v + (size_t)nrhs * n, *t = s + (size_t)nrhs * n;
  double2 *tmp = t + (size_t)nrhs * n, *bo = tmp + (size_t)nrhs * n, *bhat = bo + (size_t)nrhs * n;
  int nb = red_blocks(n);
  Carver sizing(nullptr);
  sizing.take<S64>(nrhs);
  sizing.take<int>(nrhs);
  sizing.take<D4>((size_t)nrhs * nb);
  char *sw = (char *)workspace(ctx, WS_F64_SCAL, sizing.size(), &rc);
  if (!sw) return rc;
  Carver cv(sw);
  S64 *sc = cv.take<S64>(nrhs);
  int *active = cv.take<int>(nrhs);
  D4 *part = cv.take<D4>((size_t)nrhs * nb);

  std::vector<double> rr(nrhs), bb(nrhs), target2(nrhs);
  std::vector<S64> hs(nrhs);
  std::vector<int> hact(nrhs);
  dim3 gv((g.Vh + 127) / 128, nrhs), gr(nb, nrhs);

  // |b|^2 of the full source (FP64)
  {
    LQCD_CUDA_TRY(ctx, cudaMemsetAsync(x, 0, (size_t)nrhs * full * sizeof(double2), st));
    rc = fp64_true_residual(ctx, b, x, nrhs, rr.data(), bb.data(), st);
    if (rc) return rc;
  }
  // b_e, b_o and b_hat = b_e + kappa H_eo b_o
  KL k_split64<<<gv, 128, 0, st>>>(g, 1, b, bo);
  KL k_split64<<<gv, 128, 0, st>>>(g, 0, b, tmp);
  LQCD_LAUNCH_CHECK(ctx, "k_split64");
  rc = launch_hop64(ctx, st, false, false, false, 0, bo, n, bhat, n, tmp, 1.0, nullptr, 0.0, kappa, nullptr, nrhs);
  if (rc) return rc;
  LQCD_CUDA_TRY(ctx, cudaMemsetAsync(xe, 0, (size_t)nrhs * n * sizeof(double2), st));
  for (int k = 0; k < nrhs; ++k) {
    hs[k] = S64{};
    target2[k] = 0.25 * p.tol * p.tol * bb[k];
    hs[k].target2 = target2[k];
    hs[k].bb = bb[k];
    hact[k] = 1;
  }
  LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(sc, hs.data(), nrhs * sizeof(S64), cudaMemcpyHostToDevice, st));
  const int max_restarts = 6;
  for (int restart = 0; restart <= max_restarts; ++restart) {
    LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(active, hact.data(), nrhs * sizeof(int), cudaMemcpyHostToDevice, st));
    // r = b_hat - D_hat x_e = b_hat - x_e + kappa^2 H_eo H_oe x_e
    rc = launch_hop64(ctx, st, false, false, false, 1, xe, n, tmp, n, nullptr, 0.0, nullptr, 0.0, 1.0, active, nrhs);
    if (rc) return rc;
    rc = launch_hop64(ctx, st, false, false, false, 0, tmp, n, r, n, bhat, 1.0, xe, -1.0, kappa * kappa, active, nrhs);
    if (rc) return rc;
    KL k_dot64<true><<<gr, RED_THREADS, 0, st>>>(n, active, r, r, part);
    KL k_fin_init<<<nrhs, 32, 0, st>>>(sc, active, part, nb, p.max_iter);
    LQCD_LAUNCH_CHECK(ctx, "init");
    bool any = true, timed_out = false;
    while (any) {
      for (int it = 0; it < 4; ++it) {
        KL k_bicg_p<<<gr, RED_THREADS, 0, st>>>(n, sc, active, r, rhat, pp, v);
        launch_hop64(ctx, st, false, false, false, 1, pp, n, tmp, n, nullptr, 0.0, nullptr, 0.0, 1.0, active, nrhs);
        launch_hop64(ctx, st, false, false, false, 0, tmp, n, v, n, pp, 1.0, nullptr, 0.0, -kappa * kappa, active,
                     nrhs);
        KL k_dot64<false><<<gr, RED_THREADS, 0, st>>>(n, active, rhat, v, part);
        KL k_fin_alpha<<<nrhs, 32, 0, st>>>(sc, active, part, nb);
        KL k_bicg_s<<<gr, RED_THREADS, 0, st>>>(n, sc, active, r, v, s);
        launch_hop64(ctx, st, false, false, false, 1, s, n, tmp, n, nullptr, 0.0, nullptr, 0.0, 1.0, active, nrhs);
        launch_hop64(ctx, st, false, false, false, 0, tmp, n, t, n, s, 1.0, nullptr, 0.0, -kappa * kappa, active,
                     nrhs);
        KL k_dot_ts<<<gr, RED_THREADS, 0, st>>>(n, active, t, s, part);
        KL k_fin_omega<<<nrhs, 32, 0, st>>>(sc, active, part, nb);
        KL k_bicg_xr<<<gr, RED_THREADS, 0, st>>>(n, sc, active, xe, pp, s, t, r, rhat, part);
        KL k_fin_conv<<<nrhs, 32, 0, st>>>(sc, active, part, nb, p.max_iter);
      }
      LQCD_LAUNCH_CHECK(ctx, "bicgstab iteration");
      LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(hact.data(), active, nrhs * sizeof(int), cudaMemcpyDeviceToHost, st));
      LQCD_CUDA_TRY(ctx, cudaStreamSynchronize(st));
      any = false;
      for (int k = 0; k < nrhs; ++k) any = any || hact[k];
      if (any && p.timeout_ms > 0 && wall_ms() - t_start > p.timeout_ms) {
        timed_out = true;
        break;
      }
    }
    LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(hs.data(), sc, nrhs * sizeof(S64), cudaMemcpyDeviceToHost, st));
    LQCD_CUDA_TRY(ctx, cudaStreamSynchronize(st));
    // x_o = b_o + kappa H_oe x_e ; merge into canonical x
    rc = launch_hop64(ctx, st, false, false, false, 1, xe, n, tmp, n, bo, 1.0, nullptr, 0.0, kappa, nullptr, nrhs);
    if (rc) return rc;
    KL k_merge64<<<gv, 128, 0, st>>>(g, 0, xe, x, nullptr);
    KL k_merge64<<<gv, 128, 0, st>>>(g, 1, tmp, x, nullptr);
    LQCD_LAUNCH_CHECK(ctx, "k_merge64");
    rc = fp64_true_residual(ctx, b, x, nrhs, rr.data(), bb.data(), st);
    if (rc) return rc;
    bool again = false;
    for (int k = 0; k < nrhs; ++k) {
      double rel = bb[k] > 0 ? std::sqrt(rr[k] / bb[k]) : 0.0;
      stats[k].iterations = hs[k].iters;
      stats[k].true_rel_residual = rel;
      stats[k].reliable_updates = 0;
      stats[k].restarts = restart;
      int status = hs[k].status;
      if (timed_out && status == LQCD_OK && !(rel <= p.tol)) status = LQCD_ERR_TIMEOUT;
      if (status == LQCD_OK && !std::isfinite(rel)) status = LQCD_ERR_NONFINITE;
      stats[k].status = status;
      hact[k] = 0;
      if (status == LQCD_OK && rel > p.tol) {
        if (restart == max_restarts) {
          stats[k].status = LQCD_ERR_NOT_CONVERGED;
        } else {
          hact[k] = 1;
          again = true;
          target2[k] *= 0.01;
          hs[k].target2 = target2[k];
        }
      }
    }
    if (!again || timed_out) break;
    LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(sc, hs.data(), nrhs * sizeof(S64), cudaMemcpyHostToDevice, st));
  }
  return LQCD_OK;
}

// ------------------------------------------------------------ CG (CGNR)
// CG on the normal equations of the Schur operator A = D_hat:
// A^+ A x = A^+ b_hat, with A^+ = gamma5 A gamma5 (the dagger hopping term),
// stopping on the Schur residual s = b_hat - A x (tracked by the recursion and
// checked against the true full-lattice FP64 residual afterwards).
struct SCG {
  double alpha, beta, rr, ss, target2;
  int iters, status, pad;
};

__global__ void k_cg_fin_init(SCG *sc, int *active, const D4 *part_r, const D4 *part_s, int nb, int max_iter) {
  int rhs = blockIdx.x;
  if (!active[rhs]) return;
  D4 tr = warp_total(part_r + (size_t)rhs * nb, nb);
  D4 ts = warp_total(part_s + (size_t)rhs * nb, nb);
  if (threadIdx.x) return;
  SCG &c = sc[rhs];
  c.rr = tr.c;
  c.ss = ts.c;
  if (!isfinite(tr.c) || !isfinite(ts.c)) {
    c.status = LQCD_ERR_NONFINITE;
    active[rhs] = 0;
  } else if (ts.c <= c.target2 || tr.c == 0.0) {
    active[rhs] = 0;
  } else if (c.iters >= max_iter) {
    c.status = LQCD_ERR_NOT_CONVERGED;
    active[rhs] = 0;
  }
}

__global__ void k_cg_fin_alpha(SCG *sc, const int *active, const D4 *part, int nb) {
  int rhs = blockIdx.x;
  if (!active[rhs]) return;
  D4 t = warp_total(part + (size_t)rhs * nb, nb);  // |A p|^2 in .c
  if (threadIdx.x) return;
  sc[rhs].alpha = t.c > 0.0 ? sc[rhs].rr / t.c : 0.0;
}

// x += alpha p; s -= alpha q; partial |s|^2
__global__ void __launch_bounds__(RED_THREADS) k_cg_xs(size_t n, const SCG *sc, const int *active, double2 *x,
                                                       const double2 *p, double2 *s, const double2 *q, D4 *part) {
  int rhs = blockIdx.y;
  if (!active[rhs]) return;
  double a = sc[rhs].alpha;
  size_t off = (size_t)rhs * n;
  D4 acc = {0, 0, 0, 0};
  for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x) {
    x[off + k] = cadd(x[off + k], cscale(p[off + k], a));
    const double2 qk = q[off + k], sk = s[off + k], v = make_double2(fma(-a, qk.x, sk.x), fma(-a, qk.y, sk.y));
    s[off + k] = v;
    acc.c = fma(v.x, v.x, fma(v.y, v.y, acc.c));
  }
  D4 r = block_sum4(acc);
  if (threadIdx.x == 0) part[(size_t)rhs * gridDim.x + blockIdx.x] = r;
}

__global__ void k_cg_fin_ss(SCG *sc, int *active, const D4 *part, int nb, int max_iter) {
  int rhs = blockIdx.x;
  if (!active[rhs]) return;
  D4 t = warp_total(part + (size_t)rhs * nb, nb);
  if (threadIdx.x) return;
  SCG &c = sc[rhs];
  c.ss = t.c;
  c.iters += 1;
  if (!isfinite(t.c)) {
    c.status = LQCD_ERR_NONFINITE;
    active[rhs] = 0;
  } else if (t.c <= c.target2) {
    active[rhs] = 0;
  } else if (c.iters >= max_iter) {
    c.status = LQCD_ERR_NOT_CONVERGED;
    active[rhs] = 0;
  }
}

__global__ void k_cg_fin_beta(SCG *sc, const int *active, const D4 *part, int nb) {
  int rhs = blockIdx.x;
  if (!active[rhs]) return;
  D4 t = warp_total(part + (size_t)rhs * nb, nb);
  if (threadIdx.x) return;
  SCG &c = sc[rhs];
  c.beta = c.rr > 0.0 ? t.c / c.rr : 0.0;
  c.rr = t.c;
}

// p = r + beta p (beta = 0 on the first use)
__global__ void __launch_bounds__(RED_THREADS) k_cg_p(size_t n, const SCG *sc, const int *active, const double2 *r,
                                                      double2 *p) {
  int rhs = blockIdx.y;
  if (!active[rhs]) return;
  double b = sc[rhs].beta;
  size_t off = (size_t)rhs * n;
  for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x)
    p[off + k] = cadd(r[off + k], cscale(p[off + k], b));
}

static int fp64_cg_block(lqcd_ctx *ctx, const double2 *b, double2 *x, int nrhs, const lqcd_solver_params &p,
                         lqcd_solve_stats *stats, cudaStream_t st, double t_start) {
  const Geom &g = ctx->geom;
  const double kappa = ctx->kappa, k2 = kappa * kappa;
  size_t n = (size_t)g.Vh * 12;
  int rc = LQCD_OK;
  double2 *vec = (double2 *)workspace(ctx, WS_F64_VECS, (size_t)9 * nrhs * n * sizeof(double2), &rc);
  if (!vec) return rc;
  double2 *xe = vec, *s = vec + (size_t)nrhs * n, *r = s + (size_t)nrhs * n, *pp = r + (size_t)nrhs * n;
  double2 *q = pp + (size_t)nrhs * n, *tmp = q + (size_t)nrhs * n, *bo = tmp + (size_t)nrhs * n;
  double2 *bhat = bo + (size_t)nrhs * n, *be = bhat + (size_t)nrhs * n;
  int nb = red_blocks(n);
  Carver sizing(nullptr);
  sizing.take<SCG>(nrhs);
  sizing.take<int>(nrhs);
  sizing.take<D4>((size_t)nrhs * nb);
  sizing.take<D4>((size_t)nrhs * nb);
  char *sw = (char *)workspace(ctx, WS_F64_SCAL, sizing.size(), &rc);
  if (!sw) return rc;
  Carver cv(sw);
  SCG *sc = cv.take<SCG>(nrhs);
  int *active = cv.take<int>(nrhs);
  D4 *part = cv.take<D4>((size_t)nrhs * nb);
  D4 *part2 = cv.take<D4>((size_t)nrhs * nb);
  std::vector<double> rr(nrhs), bb(nrhs);
  std::vector<SCG> hs(nrhs);
  std::vector<int> hact(nrhs, 1);
  dim3 gv((g.Vh + 127) / 128, nrhs), gr(nb, nrhs);
  LQCD_CUDA_TRY(ctx, cudaMemsetAsync(x, 0, (size_t)nrhs * g.V * 12 * sizeof(double2), st));
  rc = fp64_true_residual(ctx, b, x, nrhs, rr.data(), bb.data(), st);  // |b|^2
  if (rc) return rc;
  KL k_split64<<<gv, 128, 0, st>>>(g, 1, b, bo);
  KL k_split64<<<gv, 128, 0, st>>>(g, 0, b, be);
  rc = launch_hop64(ctx, st, false, false, false, 0, bo, n, bhat, n, be, 1.0, nullptr, 0.0, kappa, nullptr, nrhs);
  if (rc) return rc;
  LQCD_CUDA_TRY(ctx, cudaMemsetAsync(xe, 0, (size_t)nrhs * n * sizeof(double2), st));
  for (int k = 0; k < nrhs; ++k) {
    hs[k] = SCG{};
    hs[k].target2 = 0.25 * p.tol * p.tol * bb[k];
  }
  LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(sc, hs.data(), nrhs * sizeof(SCG), cudaMemcpyHostToDevice, st));
  const int max_restarts = 6;
  for (int restart = 0; restart <= max_restarts; ++restart) {
    LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(active, hact.data(), nrhs * sizeof(int), cudaMemcpyHostToDevice, st));
    // s = b_hat - A x_e ; r = A^+ s ; p = r
    launch_hop64(ctx, st, false, false, false, 1, xe, n, tmp, n, nullptr, 0.0, nullptr, 0.0, 1.0, active, nrhs);
    launch_hop64(ctx, st, false, false, false, 0, tmp, n, s, n, bhat, 1.0, xe, -1.0, k2, active, nrhs);
    launch_hop64(ctx, st, true, false, false, 1, s, n, tmp, n, nullptr, 0.0, nullptr, 0.0, 1.0, active, nrhs);
    launch_hop64(ctx, st, true, false, false, 0, tmp, n, r, n, s, 1.0, nullptr, 0.0, -k2, active, nrhs);
    KL k_dot64<true><<<gr, RED_THREADS, 0, st>>>(n, active, r, r, part);
    KL k_dot64<true><<<gr, RED_THREADS, 0, st>>>(n, active, s, s, part2);
    KL k_cg_fin_init<<<nrhs, 32, 0, st>>>(sc, active, part, part2, nb, p.max_iter);
    LQCD_CUDA_TRY(ctx, cudaMemsetAsync(pp, 0, (size_t)nrhs * n * sizeof(double2), st));
    {  // beta = 0 for the first direction
      std::vector<SCG> tmp_h(nrhs);
      LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(tmp_h.data(), sc, nrhs * sizeof(SCG), cudaMemcpyDeviceToHost, st));
      LQCD_CUDA_TRY(ctx, cudaStreamSynchronize(st));
      for (auto &c : tmp_h) c.beta = 0.0;
      LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(sc, tmp_h.data(), nrhs * sizeof(SCG), cudaMemcpyHostToDevice, st));
    }
    KL k_cg_p<<<gr, RED_THREADS, 0, st>>>(n, sc, active, r, pp);
    bool any = true, timed_out = false;
    while (any) {
      for (int it = 0; it < 4; ++it) {
        // q = A p
        launch_hop64(ctx, st, false, false, false, 1, pp, n, tmp, n, nullptr, 0.0, nullptr, 0.0, 1.0, active, nrhs);
        launch_hop64(ctx, st, false, false, false, 0, tmp, n, q, n, pp, 1.0, nullptr, 0.0, -k2, active, nrhs);
        KL k_dot64<true><<<gr, RED_THREADS, 0, st>>>(n, active, q, q, part);
        KL k_cg_fin_alpha<<<nrhs, 32, 0, st>>>(sc, active, part, nb);
        KL k_cg_xs<<<gr, RED_THREADS, 0, st>>>(n, sc, active, xe, pp, s, q, part);
        KL k_cg_fin_ss<<<nrhs, 32, 0, st>>>(sc, active, part, nb, p.max_iter);
        // r = A^+ s
        launch_hop64(ctx, st, true, false, false, 1, s, n, tmp, n, nullptr, 0.0, nullptr, 0.0, 1.0, active, nrhs);
        launch_hop64(ctx, st, true, false, false, 0, tmp, n, r, n, s, 1.0, nullptr, 0.0, -k2, active, nrhs);
        KL k_dot64<true><<<gr, RED_THREADS, 0, st>>>(n, active, r, r, part);
        KL k_cg_fin_beta<<<nrhs, 32, 0, st>>>(sc, active, part, nb);
        KL k_cg_p<<<gr, RED_THREADS, 0, st>>>(n, sc, active, r, pp);
      }
      LQCD_LAUNCH_CHECK(ctx, "cg iteration");
      LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(hact.data(), active, nrhs * sizeof(int), cudaMemcpyDeviceToHost, st));
      LQCD_CUDA_TRY(ctx, cudaStreamSynchronize(st));
      any = false;
      for (int k = 0; k < nrhs; ++k) any = any || hact[k];
      if (any && p.timeout_ms > 0 && wall_ms() - t_start > p.timeout_ms) {
        timed_out = true;
        break;
      }
    }
    LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(hs.data(), sc, nrhs * sizeof(SCG), cudaMemcpyDeviceToHost, st));
    rc = launch_hop64(ctx, st, false, false, false, 1, xe, n, tmp, n, bo, 1.0, nullptr, 0.0, kappa, nullptr, nrhs);
    if (rc) return rc;
    KL k_merge64<<<gv, 128, 0, st>>>(g, 0, xe, x, nullptr);
    KL k_merge64<<<gv, 128, 0, st>>>(g, 1, tmp, x, nullptr);
    LQCD_LAUNCH_CHECK(ctx, "k_merge64");
    rc = fp64_true_residual(ctx, b, x, nrhs, rr.data(), bb.data(), st);
    if (rc) return rc;
    bool again = false;
    for (int k = 0; k < nrhs; ++k) {
      double rel = bb[k] > 0 ? std::sqrt(rr[k] / bb[k]) : 0.0;
      stats[k].iterations = hs[k].iters;
      stats[k].true_rel_residual = rel;
      stats[k].reliable_updates = 0;
      stats[k].restarts = restart;
      int status = hs[k].status;
      if (timed_out && status == LQCD_OK && !(rel <= p.tol)) status = LQCD_ERR_TIMEOUT;
      if (status == LQCD_OK && !std::isfinite(rel)) status = LQCD_ERR_NONFINITE;
      stats[k].status = status;
      hact[k] = 0;
      if (status == LQCD_OK && rel > p.tol) {
        if (restart == max_restarts) {
          stats[k].status = LQCD_ERR_NOT_CONVERGED;
        } else {
          hact[k] = 1;
          again = true;
          hs[k].target2 *= 0.01;
        }
      }
    }
    if (!again || timed_out) break;
    LQCD_CUDA_TRY(ctx, cudaMemcpyAsync(sc, hs.data(), nrhs * sizeof(SCG), cudaMemcpyHostToDevice, st));
  }
  return LQCD_OK;
}

int fp64_solve(lqcd_ctx *ctx, const double2 *b, double2 *x, int nrhs, const lqcd_solver_params &p,
               lqcd_solve_stats *stats, cudaStream_t st) {
  int blk = p.rhs_block > 0 ? p.rhs_block : 1;  // the plain solver: one RHS at a time
  if (blk > 65535) blk = 65535;
  double t0 = wall_ms();
  size_t full = (size_t)ctx->geom.V * 12;
  int worst = LQCD_OK;
  const FxUse use(ctx, st);  // one for all hops of the solve
  for (int k0 = 0; k0 < nrhs; k0 += blk) {
    int nk = nrhs - k0 < blk ? nrhs - k0 : blk;
    int rc = p.solver == LQCD_SOLVER_CG ? fp64_cg_block(ctx, b + k0 * full, x + k0 * full, nk, p, stats + k0, st, t0)
                                        : fp64_solve_block(ctx, b + k0 * full, x + k0 * full, nk, p, stats + k0, st, t0);
    if (rc) return rc;
    for (int k = 0; k < nk; ++k)
      if (worst == LQCD_OK && stats[k0 + k].status != LQCD_OK) worst = stats[k0 + k].status;
  }
  if (worst != LQCD_OK) set_error(ctx, worst, "lqcd_solve_batch: some right-hand sides did not converge");
  return worst;
}

}  // namespace lqcd
