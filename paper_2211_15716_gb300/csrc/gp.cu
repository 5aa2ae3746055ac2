// Gross-Pitaevskii half steps on the implicit global grid: a complex field
// psi = u + i v kept as two real fields of the grid's layout, u at whole and
// v at half time steps:
//   which 0:  u += dt * H(v),   which 1:  v -= dt * H(u),
//   H w = -1/2 lap(w) + (V + g (u^2 + v^2)) w,
// on inner points (psi fixed on each array's boundary), lap the 7-point
// operator with the grid's spacings. With w the field read and o the field
// written, scaled by dt and the sign s (+1, -1):
//   o += s (kc w + kx (w[-x] + w[+x]) + ky (..) + kz (..) + q w),
//   kd = -dt/(2 dd^2), kc = -2 (kx + ky + kz), q = dt (V + g (u^2 + v^2)).
//
// Per-point arithmetic (shared by both kernels, so they give the same bits):
// FP32 fields in FP32 with FMAs. FP64 fields: q and the seven-term sum in
// float pairs (pair.cuh: error-free products and two-sums, a compensated
// dot product starting from o) and one FP64 add, within about 2^-45 of
// |o| + sum |terms| (the FP64 sum: 13 FP64 instructions per point, which
// bound the step by the FP64 pipe); points whose values leave the pair
// ranges take the FP64 sum.
//
// Kernels: k_gp_tma (3-D grids, rows of a multiple of 16 bytes): the
// persistent TMA column kernel of the adjoint's design (W x 16 tiles, one
// warp per row, equal shares of (z chunk, column, plane) over all
// subdomains, loads issued by thread 0 after each barrier); per plane the w
// box with a one-vector / one-row halo and the o and V boxes; FP64 fields
// form the pairs of w once per point into triple-buffered shared planes.
// k_gp_half: one thread per (x, y) column marching in z (any grid,
// including 2-D and 1-D ones: absent dimensions have zero neighbour strides
// and zero weights).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <mutex>

#include "cell.cuh"
#include "igg_internal.h"
#include "pair.cuh"
#include "tma_util.cuh"

namespace igg {
namespace {

// pair ranges: |w|, |o| in [2^-40, 2^41), |q| in [2^-36, 2^37) (or zero),
// weights zero or in [2^-18, 2^18]: no partial product or error term leaves
// the normal FP32 range
constexpr unsigned kGpWE = 40, kGpQE = 36;
static_assert(kGpWE <= kPairMaxRadius && kGpQE <= kPairMaxRadius,
              "pair_ok radii must stay inside pair_split's range");

// A half step's weights as pairs, its sign applied (x, y, z, centre), dt and g
// as pairs, and the FP32 kernels' weights (kf: kx, ky, kz, kc without the
// sign), all formed on the host (see Coef).
struct GpPairW {
  double k[4];  // s kx, s ky, s kz, s kc (FP64)
  float kh[4], kl[4], kf[4];
  double dt, g;
  float dth, dtl, gh, gl;
  float s;
  int pair;
};

GpPairW make_gp_w(const GpCoef &c, int which) {
  GpPairW w;
  const double sg = which == 0 ? 1.0 : -1.0;
  const double d[4] = {c.kx, c.ky, c.kz, c.kc};
  bool ok = true;
  for (int i = 0; i < 4; ++i) {
    w.k[i] = sg * d[i];
    w.kh[i] = (float)w.k[i];
    w.kl[i] = (float)(w.k[i] - (double)w.kh[i]);
    w.kf[i] = (float)d[i];
    // (a zero weight: an absent dimension)
    if (i < 3) ok = ok && (d[i] == 0.0 || (fabs(d[i]) >= 0x1p-18 && fabs(d[i]) <= 0x1p18));
  }
  w.dt = c.dt;
  w.g = c.g;
  w.dth = (float)c.dt;
  w.dtl = (float)(c.dt - (double)w.dth);
  w.gh = (float)c.g;
  w.gl = (float)(c.g - (double)w.gh);
  w.s = (float)sg;
  // dt and g enter the pair products: dt in [2^-40, 2^20], g zero or in
  // [2^-40, 2^40]
  ok = ok && c.dt >= 0x1p-40 && c.dt <= 0x1p20 &&
       (c.g == 0.0 || (fabs(c.g) >= 0x1p-40 && fabs(c.g) <= 0x1p40));
  w.pair = ok;
  return w;
}

// w as a pair, NaN in h outside the pair range
__device__ __forceinline__ FF gp_pair(double x) {
  FF q = pair_split(x);
  q.h = pair_ok(x, kGpWE) ? q.h : __int_as_float(0x7FC00000);
  return q;
}

// the pairs of two points
__device__ __forceinline__ FF2 gp_pair2(double a, double b) {
  const FF p = gp_pair(a), q = gp_pair(b);
  return {make_float2(p.h, q.h), make_float2(p.l, q.l)};
}

// q = dt (V + g (u^2 + v^2)) in FP64 (uc, vc: u and v at the point)
__device__ __forceinline__ double gp_q(double uc, double vc, double pot, const GpPairW &w) {
  return __dmul_rn(w.dt, __fma_rn(w.g, __fma_rn(uc, uc, __dmul_rn(vc, vc)), pot));
}

// q as a normalised pair from the pairs of u, v and the potential (NaN in h
// when one of theirs is): error-free squares and sum for rho, then g rho + V
// and dt (..) with FMA product splits, about 2^-45 of dt (|V| + |g| rho). One
// point, or two as float2 (the same roundings).
template <class F>
__device__ __forceinline__ FFv<F> gp_q_pair(const FFv<F> &u, const FFv<F> &v, const FFv<F> &vp,
                                            const GpPairW &w) {
  const F zero = vset(0.f, F());
  const F p1 = vfma(u.h, u.h, zero);
  F e1 = vfma(u.h, u.h, vneg(p1));
  e1 = vfma(vadd(u.h, u.h), u.l, e1);
  const F p2 = vfma(v.h, v.h, zero);
  F e2 = vfma(v.h, v.h, vneg(p2));
  e2 = vfma(vadd(v.h, v.h), v.l, e2);
  F t;
  const F rs = vtwo_sum(p1, p2, t);
  t = vadd(t, vadd(e1, e2));
  const F gh = vset(w.gh, F()), dth = vset(w.dth, F());
  const F a = vfma(gh, rs, zero);
  F ae = vfma(gh, rs, vneg(a));
  ae = vfma(gh, t, ae);
  ae = vfma(vset(w.gl, F()), rs, ae);
  F be;
  const F b = vtwo_sum(a, vp.h, be);
  be = vadd(be, vadd(ae, vp.l));
  const F cq = vfma(dth, b, zero);
  F ce = vfma(dth, b, vneg(cq));
  ce = vfma(dth, be, ce);
  ce = vfma(vset(w.dtl, F()), b, ce);
  FFv<F> q;
  q.h = vfast_two_sum(cq, ce, q.l);
  return q;
}

// the pair range of q: zero or |q| in [2^-36, 2^37) (from the leading part)
__device__ __forceinline__ bool gp_q_ok(float qh) {
  const unsigned b = __float_as_uint(qh);
  const unsigned e = (b >> 23) & 0xFFu;
  return e - (127u - kGpQE) <= 2u * kGpQE || (b << 1) == 0u;
}

// o + s h on the pair path as acc + err, from the pairs of o, q and w (one
// point, or two as float2)
template <int WHICH, class F>
__device__ __forceinline__ void gp_sum_pair(const FFv<F> &op, const FFv<F> &qp, const FFv<F> &wc,
                                            const FFv<F> &wxm, const FFv<F> &wxp,
                                            const FFv<F> &wym, const FFv<F> &wyp,
                                            const FFv<F> &wzm, const FFv<F> &wzp,
                                            const GpPairW &w, F &acc, F &err) {
  acc = op.h;
  err = op.l;
  dot2_term(acc, err, vset(w.kh[3], F()), vset(w.kl[3], F()), wc.h, wc.l);
  dot2_term(acc, err, WHICH == 0 ? qp.h : vneg(qp.h), WHICH == 0 ? qp.l : vneg(qp.l), wc.h, wc.l);
  dot2_pair(acc, err, w.kh[0], w.kl[0], wxm, wxp);
  dot2_pair(acc, err, w.kh[1], w.kl[1], wym, wyp);
  dot2_pair(acc, err, w.kh[2], w.kl[2], wzm, wzp);
}

// the sum rounded to FP64; false: take gp_out_f64 (o_ok: o in range)
__device__ __forceinline__ bool gp_out_pair(float acc, float err, bool o_ok, float qh,
                                            const GpPairW &w, double &res) {
  res = __dadd_rn(f2d_finite(acc), f2d_finite(err));
  return w.pair && o_ok && gp_q_ok(qh) && acc == acc;
}

// o + s h in FP64
__device__ __forceinline__ double gp_out_f64(double o, double q, double wc, double wxm,
                                             double wxp, double wym, double wyp, double wzm,
                                             double wzp, const GpPairW &w) {
  // s is applied through the signed weights: s h = sum of the signed terms
  double h = __dmul_rn(w.k[3], wc);
  h = __fma_rn(w.k[0], __dadd_rn(wxm, wxp), h);
  h = __fma_rn(w.k[1], __dadd_rn(wym, wyp), h);
  h = __fma_rn(w.k[2], __dadd_rn(wzm, wzp), h);
  h = __fma_rn(__dmul_rn((double)w.s, q), wc, h);
  return __dadd_rn(o, h);
}

// o + s h for FP32 fields
__device__ __forceinline__ float gp_out_f32(float o, float uc, float vc, float pot, float wc,
                                            float wxm, float wxp, float wym, float wyp, float wzm,
                                            float wzp, const GpPairW &w, int which) {
  float h = __fmul_rn(w.kf[3], wc);
  h = __fmaf_rn(w.kf[0], __fadd_rn(wxm, wxp), h);
  h = __fmaf_rn(w.kf[1], __fadd_rn(wym, wyp), h);
  h = __fmaf_rn(w.kf[2], __fadd_rn(wzm, wzp), h);
  const float q = __fmul_rn(w.dth, __fmaf_rn(w.gh, __fmaf_rn(uc, uc, __fmul_rn(vc, vc)), pot));
  h = __fmaf_rn(q, wc, h);
  return which == 0 ? __fadd_rn(o, h) : __fadd_rn(o, -h);
}

// ---------------------------------------------------------------------------
// tiled kernel (any grid)

constexpr int kGpX = 32, kGpY = 8, kGpZ = 32;

// blockIdx.z = subdomain * zchunks + z chunk; inner ranges [lo, hi) per
// dimension (absent dimensions: [0, 1) with zero stride)
template <class S, int WHICH>
__global__ void __launch_bounds__(kGpX *kGpY)
    k_gp_half(int nx, int ny, int nz, int zchunks, S *__restrict__ u, S *__restrict__ v,
              const S *__restrict__ V, const GpPairW pw) {
  const int ylo = ny > 1 ? 1 : 0, yhi = ny > 1 ? ny - 1 : 1;
  const int zlo = nz > 1 ? 1 : 0, zhi = nz > 1 ? nz - 1 : 1;
  const int i = 1 + blockIdx.x * kGpX + threadIdx.x, j = ylo + blockIdx.y * kGpY + threadIdx.y;
  // lanes past the last column run along (the FP64 path votes across the
  // warp) and store nothing
  const bool act = i < nx - 1 && j < yhi;
  const long long sub = blockIdx.z / zchunks;
  const int k0 = zlo + (int)(blockIdx.z % zchunks) * kGpZ, k1 = min(k0 + kGpZ, zhi);
  if (k0 >= k1) return;  // uniform over the block
  const int ii = act ? i : 1, jj = act ? j : ylo;
  const long long nloc = (long long)nx * ny * nz;
  const long long sy = ny > 1 ? nx : 0, sz = nz > 1 ? (long long)nx * ny : 0;
  S *out = (WHICH == 0 ? u : v) + sub * nloc;
  const S *w = (WHICH == 0 ? v : u) + sub * nloc;
  const S *Vs = V + sub * nloc;
  long long p = ii + (long long)nx * jj + (long long)nx * ny * k0;
  if constexpr (sizeof(S) == 8) {
    double wm = w[p - sz], wc = w[p];
    for (int k = k0; k < k1; ++k, p += (long long)nx * ny) {
      const double wp = w[p + sz];
      const double o = out[p], pot = Vs[p];
      const double xm = w[p - 1], xp = w[p + 1], ym = w[p - sy], yp = w[p + sy];
      const FF op = gp_pair(o), cp = gp_pair(wc);
      const FF vp = gp_pair(pot);
      const FF qp = WHICH == 0 ? gp_q_pair(op, cp, vp, pw) : gp_q_pair(cp, op, vp, pw);
      float acc, err;
      gp_sum_pair<WHICH>(op, qp, cp, gp_pair(xm), gp_pair(xp), gp_pair(ym), gp_pair(yp),
                         gp_pair(wm), gp_pair(wp), pw, acc, err);
      double r;
      const bool ok = gp_out_pair(acc, err, pair_ok(o, kGpWE), qp.h, pw, r);
      if (__any_sync(0xffffffffu, !ok)) {
        if (!ok) {
          const double q = WHICH == 0 ? gp_q(o, wc, pot, pw) : gp_q(wc, o, pot, pw);
          r = gp_out_f64(o, q, wc, xm, xp, ym, yp, wm, wp, pw);
        }
      }
      if (act) out[p] = r;
      wm = wc;
      wc = wp;
    }
  } else {
    S wm = w[p - sz], wc = w[p];
    for (int k = k0; k < k1; ++k, p += (long long)nx * ny) {
      const S wp = w[p + sz];
      const S o = out[p];
      const S uc = WHICH == 0 ? o : wc, vc = WHICH == 0 ? wc : o;
      const S r = gp_out_f32(o, uc, vc, Vs[p], wc, w[p - 1], w[p + 1], w[p - sy], w[p + sy], wm,
                             wp, pw, WHICH);
      if (act) out[p] = r;
      wm = wc;
      wc = wp;
    }
  }
}

// ---------------------------------------------------------------------------
// TMA-pipelined kernel (3-D grids)

template <class S>
struct GpShape {
  static constexpr bool PAIRS = sizeof(S) == 8;          // FP64: w as pairs in shared planes
  static constexpr int V = 16 / (int)sizeof(S);          // points per lane
  static constexpr int W = 32 * V;                       // points per row
  static constexpr int BW = W + 2 * V;                   // w box width
  // rows per tile and stages: FP64 8 and 4, three CTAs per SM (24 warps); FP32 16
  // and 6, one. The FP64 launch is bound by instruction issue (263 instructions
  // per point, issue 66 %), then by the barrier of each plane; the shape matters
  // little: 2x2x2 x 256^3, four steps, three CTAs of 8 rows 10.76, one of 16 rows
  // 10.79, two of 8 (six stages) 11.29 ms
  static constexpr int H = sizeof(S) == 8 ? 8 : 16;
  static constexpr int BH = H + 2;
  static constexpr int WARPS = H;
  static constexpr int MINB = H == 8 ? 3 : 1;            // resident CTAs per SM
  static constexpr int NS = H == 8 ? 4 : 6;                           // loads issued NS - 2 ahead
  static constexpr int FB = BW * BH * (int)sizeof(S);    // w box bytes
  static constexpr int FBA = (FB + 127) / 128 * 128;
  static constexpr int OB = W * H * (int)sizeof(S);      // o and V box bytes
  static constexpr int STAGE = FBA + 2 * OB;
  static constexpr int VPL = BW * BH;                    // pair plane points
  static constexpr int VBA = PAIRS ? (3 * VPL * 8 + 127) / 128 * 128 : 0;
  static constexpr int SMEM = NS * STAGE + VBA + NS * 8 + 16;
  static constexpr int RING = 2 * (W + 2) + 2 * H;
  static constexpr int RPT = (RING + 32 * WARPS - 1) / (32 * WARPS);
  static_assert(OB % 128 == 0, "stage alignment");
  static_assert(BW <= 256 && W <= 256 && BH <= 256, "TMA box dims");
};

template <class S>
__device__ __forceinline__ void gp_lds16(const void *p, Vec<S> &o) {
  unpack(*reinterpret_cast<const uint4 *>(p), o);
}

// mW, mO, mV: tensor maps of the field read (w), the field written (o) and
// the potential over [nsub * nz][ny][nx]; ncxy columns per subdomain
template <class S, int WHICH>
__global__ void __launch_bounds__(32 * GpShape<S>::WARPS, GpShape<S>::MINB)
    k_gp_tma(const __grid_constant__ CUtensorMap mW, const __grid_constant__ CUtensorMap mO,
             const __grid_constant__ CUtensorMap mV, int nx, int ny, int nz, int ncx, int ncxy,
             int ncol, S *out, const S *rd, const GpPairW pw, const int *__restrict__ nbr, int ox,
             int xsend, unsigned *__restrict__ dev_err) {
  using Sh = GpShape<S>;
  constexpr int V = Sh::V, W = Sh::W, BW = Sh::BW, H = Sh::H, NS = Sh::NS;
  constexpr unsigned NT = 32 * Sh::WARPS;
  extern __shared__ __align__(128) unsigned char smem[];
  const unsigned sbase = smem_u32(smem);
  // FP64: pair planes, two neighbouring points of a row as h0 h1 l0 l1
  float *planes = reinterpret_cast<float *>(smem + NS * Sh::STAGE);
  const unsigned full0 = sbase + NS * Sh::STAGE + Sh::VBA;
  volatile int *flags = reinterpret_cast<volatile int *>(smem + NS * Sh::STAGE + Sh::VBA + NS * 8);

  const int nzi = nz - 2;  // inner planes per column (z = m + 1)
  const long long U = (long long)ncol * nzi;
  const long long u0 = U * blockIdx.x / gridDim.x, u1 = U * (blockIdx.x + 1) / gridDim.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto origin = [&](int col, int &x0, int &r0, int &zoff) {
    const int sub = col / ncxy, cc = col - sub * ncxy;
    x0 = (cc % ncx) * W;
    r0 = (cc / ncx) * H;
    zoff = sub * nz;
  };

  // load cursor (thread 0): a segment's loads are its planes z0 - 1 .. z1
  Share cur{u0, u1, nzi, ncol};
  Seg cs{0, 0, 0};
  int cj = 0, cK = 0, issued = 0;
  auto issue_upto = [&](int last) {
    while (issued <= last) {
      if (cj >= cK) {
        if (!cur.next(cs)) return;
        cj = 0;
        cK = cs.m1 - cs.m0 + 2;
      }
      int x0, r0, zoff;
      origin(cs.col, x0, r0, zoff);
      const int s = issued % NS;
      const bool ov = cj >= 1 && cj <= cK - 2;  // o and V of the computed planes
      const unsigned bar = full0 + 8 * s, dst = sbase + s * Sh::STAGE;
      mbar_expect_tx(bar, Sh::FB + (ov ? 2 * Sh::OB : 0));
      const int p = zoff + cs.m0 + cj;  // plane z = m0 + 1 - 1 + cj
      tma_load_3d(dst, &mW, x0 - V, r0 - 1, p, bar);
      if (ov) {
        tma_load_3d(dst + Sh::FBA, &mO, x0, r0, p, bar);
        tma_load_3d(dst + Sh::FBA + Sh::OB, &mV, x0, r0, p, bar);
      }
      ++cj;
      ++issued;
    }
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < NS; ++s) mbar_init(full0 + 8 * s, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    pdl_trigger();
    pdl_wait();  // (and the CTA's other accesses follow its first load)
    issue_upto(NS - 2);
  }
  __syncthreads();

  const int r = warp;
  const int ob = (r + 1) * BW + V + lane * V;  // own points in the w box / pair plane
  const int oo = r * W + lane * V;             // own points in the o and V boxes
  const long long sz = (long long)nx * ny;
  auto stage = [&](int kk) { return smem + (kk % NS) * Sh::STAGE; };
  auto wbox = [&](int kk) { return reinterpret_cast<const S *>(stage(kk)); };
  auto wait_full = [&](int kk) {
    return __all_sync(0xffffffffu, mbar_wait(full0 + 8 * (kk % NS), (kk / NS) & 1));
  };

  Share sh{u0, u1, nzi, ncol};
  Seg sg;
  int k = 0, q = 0;
  bool stop = false;
  // own w of planes z-1, z, z+1 (FP64: also as pairs)
  S tm[V], tc[V], tp[V];  // (FP64: unused)
  FF2 pm, pc, pp;
  while (!stop && sh.next(sg)) {
    int x0, r0, zoff;
    origin(sg.col, x0, r0, zoff);
    const int xs = x0 + lane * V, y = r0 + r;
    const bool yin = y >= 1 && y <= ny - 2;
    bool xyin[V];
#pragma unroll
    for (int i = 0; i < V; ++i) xyin[i] = yin && xs + i >= 1 && xs + i <= nx - 2;
    // the halo update's x exchange (GpCoef::xsend): this lane's points of the
    // sent planes nx - o (bits 0..V-1: to the right neighbour's column 0) and
    // o - 1 (bits 8..8+V-1: to the left neighbour's column nx - 1), and the
    // element offsets of their copies
    unsigned sendm = 0u;
    long long dr = 0, dl = 0;
    if (xsend) {
      const int sub = zoff / nz, xl = nbr[6 * sub], xr = nbr[6 * sub + 1];
      const long long nloc = sz * nz, h = nx - ox;
      dr = (long long)(xr - sub) * nloc - h;
      dl = (long long)(xl - sub) * nloc + h;
#pragma unroll
      for (int i = 0; i < V; ++i) {
        if (!xyin[i]) continue;
        if (xr >= 0 && xs + i == nx - ox) sendm |= 1u << i;
        if (xl >= 0 && xs + i == ox - 1) sendm |= 1u << (8 + i);
      }
    }
    int rb[Sh::RPT];
#pragma unroll
    for (int j = 0; j < Sh::RPT; ++j) {
      const int i = threadIdx.x + j * NT;
      int xo = 0, yo = -1;
      if (i < 2 * (W + 2)) {
        xo = i % (W + 2) - 1;
        yo = i < W + 2 ? -1 : H;
      } else {
        const int t = i - 2 * (W + 2);
        xo = t < H ? -1 : W;
        yo = t % H;
      }
      rb[j] = i < Sh::RING ? (yo + 1) * BW + xo + V : -1;
    }
    // own w of load kk (and, FP64, its pairs)
    auto own = [&](int kk, S *t, FF2 &pr) {
      Vec<S> a;
      gp_lds16<S>(wbox(kk) + ob, a);
      if constexpr (Sh::PAIRS) {
        pr = gp_pair2(a.v[0], a.v[1]);
      } else {
#pragma unroll
        for (int i = 0; i < V; ++i) t[i] = a.v[i];
      }
    };
    // FP64: the pair plane of load kk (own pairs, then the ring)
    auto form = [&](int kk, float *pl, const FF2 &pr) {
      if constexpr (Sh::PAIRS) {
        *reinterpret_cast<float4 *>(pl + 2 * ob) = make_float4(pr.h.x, pr.h.y, pr.l.x, pr.l.y);
        const S *Wb = wbox(kk);
#pragma unroll
        for (int j = 0; j < Sh::RPT; ++j)
          if (rb[j] >= 0) {
            const FF q = gp_pair(Wb[rb[j]]);
            float *d = pl + 4 * (rb[j] >> 1) + (rb[j] & 1);
            d[0] = q.h;
            d[2] = q.l;
          }
      }
    };
    bool good = wait_full(k);
    if (good) {
      own(k, tm, pm);
      ++k;
      good = wait_full(k);
    }
    float *pl = planes + (q % 3) * 2 * Sh::VPL;
    if (good) {
      own(k, tc, pc);
      form(k, pl, pc);
    }
    if (all_any(!good, NT)) {
      stop = true;
      break;
    }
    if (threadIdx.x == 0) issue_upto(k + NS - 2);
    int kc = k;
    ++k;
    const float *plm = pl;
    ++q;
    for (int m = sg.m0; m < sg.m1; ++m) {
      const int z = m + 1;
      good = wait_full(k);
      float *pln = planes + (q % 3) * 2 * Sh::VPL;
      if (good) {
        own(k, tp, pp);
        form(k, pln, pp);
      }
      if (all_any(!good, NT)) {
        stop = true;
        break;
      }
      if (threadIdx.x == 0) issue_upto(k + NS - 2);
      // plane z
      const S *Wb = wbox(kc);
      const S *Ob = reinterpret_cast<const S *>(stage(kc) + Sh::FBA) + oo;
      const S *Pb = reinterpret_cast<const S *>(stage(kc) + Sh::FBA + Sh::OB) + oo;
      Vec<S> ov, pv;
      gp_lds16<S>(Ob, ov);
      gp_lds16<S>(Pb, pv);
      const long long p0 = zoff * sz + xs + (long long)nx * y + sz * z;
      S res[V];
      if constexpr (Sh::PAIRS) {
        // (the plane's row pitch and ob are even: ob and ob +- BW start pairs)
        auto two = [&](int o) {
          const float4 a = *reinterpret_cast<const float4 *>(plm + 2 * o);
          return FF2{make_float2(a.x, a.y), make_float2(a.z, a.w)};
        };
        const float *xl = plm + 2 * ob - 4, *xr = plm + 2 * ob + 4;
        const FF2 xm = {make_float2(xl[1], pc.h.x), make_float2(xl[3], pc.l.x)};
        const FF2 xp = {make_float2(pc.h.y, xr[0]), make_float2(pc.l.y, xr[2])};
        const FF2 op = gp_pair2(ov.v[0], ov.v[1]), vp = gp_pair2(pv.v[0], pv.v[1]);
        const FF2 qp = WHICH == 0 ? gp_q_pair(op, pc, vp, pw) : gp_q_pair(pc, op, vp, pw);
        float2 acc, err;
        gp_sum_pair<WHICH>(op, qp, pc, xm, xp, two(ob - BW), two(ob + BW), pm, pp, pw, acc, err);
        const bool ok0 =
            gp_out_pair(acc.x, err.x, pair_ok(ov.v[0], kGpWE), qp.h.x, pw, res[0]);
        const bool ok1 =
            gp_out_pair(acc.y, err.y, pair_ok(ov.v[1], kGpWE), qp.h.y, pw, res[1]);
        const bool bad = (!ok0 && xyin[0]) || (!ok1 && xyin[1]);
        // (a NaN marks the point)
        if (!ok0) res[0] = __longlong_as_double(0x7FF8000000000000ll);
        if (!ok1) res[1] = __longlong_as_double(0x7FF8000000000000ll);
        if (__any_sync(0xffffffffu, bad)) {
#pragma unroll
          for (int i = 0; i < V; ++i) {
            if (res[i] != res[i]) {
              // (the field read is not written by this launch; planes z and
              // z + 1 are in shared memory, z - 1 may have been overwritten)
              const double *wc = reinterpret_cast<const double *>(Wb) + ob + i;
              const double wzm = xyin[i] ? rd[p0 + i - sz] : 0.0;
              const double wzp = reinterpret_cast<const double *>(wbox(k))[ob + i];
              const double q = WHICH == 0 ? gp_q(ov.v[i], wc[0], pv.v[i], pw)
                                          : gp_q(wc[0], ov.v[i], pv.v[i], pw);
              res[i] = gp_out_f64(ov.v[i], q, wc[0], wc[-1], wc[1], wc[-BW], wc[BW], wzm, wzp, pw);
            }
          }
        }
      } else {
        Vec<S> wym, wyp;
        gp_lds16<S>(Wb + ob - BW, wym);
        gp_lds16<S>(Wb + ob + BW, wyp);
        const S wl = Wb[ob - 1], wr = Wb[ob + V];
#pragma unroll
        for (int i = 0; i < V; ++i) {
          const S xm = i == 0 ? wl : tc[i - 1];
          const S xp = i == V - 1 ? wr : tc[i + 1];
          const S uc = WHICH == 0 ? ov.v[i] : tc[i], vc = WHICH == 0 ? tc[i] : ov.v[i];
          res[i] = gp_out_f32(ov.v[i], uc, vc, pv.v[i], tc[i], xm, xp, wym.v[i], wyp.v[i], tm[i],
                              tp[i], pw, WHICH);
        }
      }
      bool all_in = true;
#pragma unroll
      for (int i = 0; i < V; ++i) all_in = all_in && xyin[i];
      if (all_in) {
        Vec<S> o;
#pragma unroll
        for (int i = 0; i < V; ++i) o.v[i] = res[i];
        *reinterpret_cast<uint4 *>(out + p0) = pack(o);
      } else {
#pragma unroll
        for (int i = 0; i < V; ++i)
          if (xyin[i]) out[p0 + i] = res[i];
      }
      if (sendm) {
        // the sent points stored again into the neighbours' halo columns
        // (the halo launch then copies the face rows only)
#pragma unroll
        for (int i = 0; i < V; ++i) {
          if (sendm >> i & 1u) out[p0 + i + dr] = res[i];
          if (sendm >> (8 + i) & 1u) out[p0 + i + dl] = res[i];
        }
      }
      kc = k;
      ++k;
      plm = pln;
      ++q;
      if constexpr (!Sh::PAIRS) {
#pragma unroll
        for (int i = 0; i < V; ++i) {
          tm[i] = tc[i];
          tc[i] = tp[i];
        }
      }
      pm = pc;
      pc = pp;
    }
  }
  if (threadIdx.x == 0) flags[0] = issued;
  __syncthreads();
  if (threadIdx.x == 0 && stop) {
    atomicOr(dev_err, IGG_DEV_ERR_TIMEOUT);
    for (int kk = k; kk < flags[0]; ++kk) {
      if (!mbar_wait(full0 + 8 * (kk % NS), (kk / NS) & 1)) {
        atomicOr(dev_err, IGG_DEV_ERR_DRAIN);
        break;
      }
    }
  }
}

template <class S, int WHICH>
cudaError_t launch_tma(int nsub, int nx, int ny, int nz, void *u, void *v, const void *V,
                       const GpCoef &c, unsigned *dev_err, cudaStream_t s) {
  using Sh = GpShape<S>;
  static cudaError_t attr = cudaErrorNotReady;
  static std::mutex mu;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (attr == cudaErrorNotReady)
      attr = cudaFuncSetAttribute(k_gp_tma<S, WHICH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  Sh::SMEM);
  }
  if (attr != cudaSuccess) return attr;
  void *o = WHICH == 0 ? u : v;
  const void *w = WHICH == 0 ? v : u;
  const long long nzt = (long long)nsub * nz;
  CUtensorMap mW, mO, mV;
  if (!encode<S>(&mW, w, nx, ny, nzt, Sh::BW, Sh::BH, 1) ||
      !encode<S>(&mO, o, nx, ny, nzt, Sh::W, Sh::H, 1) ||
      !encode<S>(&mV, V, nx, ny, nzt, Sh::W, Sh::H, 1))
    return cudaErrorInvalidValue;
  int per_sm = 0, dev = 0, sms = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gp_tma<S, WHICH>,
                                                                32 * Sh::WARPS, Sh::SMEM);
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const int ncx = (nx + Sh::W - 1) / Sh::W, ncy = (ny + Sh::H - 1) / Sh::H;
  const long long ncol = (long long)nsub * ncx * ncy;
  if (ncol > (1ll << 30)) return cudaErrorInvalidValue;
  const long long U = ncol * (nz - 2);
  const long long G = std::min<long long>((long long)per_sm * sms, std::max<long long>(1, U / 4));
  return launch_pdl(pdl_on((long long)nsub * nx * ny * nz), k_gp_tma<S, WHICH>, (unsigned)G, 32 * Sh::WARPS, Sh::SMEM, s, mW, mO, mV, nx,
                    ny, nz, ncx, ncx * ncy, (int)ncol, (S *)o, (const S *)w, make_gp_w(c, WHICH), c.nbr, c.ox,
                    c.xsend, dev_err);
}

template <class S, int WHICH>
cudaError_t launch_w(int nsub, int nx, int ny, int nz, void *u, void *v, const void *V,
                     const GpCoef &c, cudaStream_t s) {
  const int ny_in = ny > 1 ? ny - 2 : 1, nz_in = nz > 1 ? nz - 2 : 1;
  const int zchunks = (nz_in + kGpZ - 1) / kGpZ;
  const long long gz = (long long)nsub * zchunks;
  if (gz > 65535 || nx < 3) return cudaErrorInvalidValue;
  const dim3 grid((nx - 2 + kGpX - 1) / kGpX, (ny_in + kGpY - 1) / kGpY, (unsigned)gz);
  k_gp_half<S, WHICH><<<grid, dim3(kGpX, kGpY), 0, s>>>(nx, ny, nz, zchunks, (S *)u, (S *)v,
                                                       (const S *)V, make_gp_w(c, WHICH));
  return cudaGetLastError();
}

template <class S>
bool tma_fits(int nx, int ny, int nz, const void *u, const void *v, const void *V) {
  if (!tma_available() || ny < 3 || nz < 3 || nx < 3) return false;
  if (((size_t)nx * sizeof(S)) % 16 != 0) return false;
  for (const void *p : {u, v, V})
    if (reinterpret_cast<uintptr_t>(p) % 16 != 0) return false;
  return true;
}

}  // namespace

cudaError_t launch_gp_half(igg_dtype dt, int which, int nsub, int nx, int ny, int nz, void *u,
                           void *v, const void *V, const GpCoef &c, bool tma, unsigned *dev_err,
                           cudaStream_t s, bool *xsent) {
  *xsent = false;
  GpCoef cw = c;  // the tiled kernel does no x sends
  cw.xsend = 0;
  switch (dt) {
    case IGG_F64:
      if (tma && tma_fits<double>(nx, ny, nz, u, v, V)) {
        *xsent = c.xsend != 0;
        return which == 0 ? launch_tma<double, 0>(nsub, nx, ny, nz, u, v, V, c, dev_err, s)
                          : launch_tma<double, 1>(nsub, nx, ny, nz, u, v, V, c, dev_err, s);
      }
      return which == 0 ? launch_w<double, 0>(nsub, nx, ny, nz, u, v, V, cw, s)
                        : launch_w<double, 1>(nsub, nx, ny, nz, u, v, V, cw, s);
    case IGG_F32:
      if (tma && tma_fits<float>(nx, ny, nz, u, v, V)) {
        *xsent = c.xsend != 0;
        return which == 0 ? launch_tma<float, 0>(nsub, nx, ny, nz, u, v, V, c, dev_err, s)
                          : launch_tma<float, 1>(nsub, nx, ny, nz, u, v, V, c, dev_err, s);
      }
      return which == 0 ? launch_w<float, 0>(nsub, nx, ny, nz, u, v, V, cw, s)
                        : launch_w<float, 1>(nsub, nx, ny, nz, u, v, V, cw, s);
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace igg
