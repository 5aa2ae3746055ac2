// Staggered-grid acoustics (a multi-field stencil on the implicit global grid
// whose fields have different sizes): P at cells [nz][ny][nx], Vx at x faces
// [nz][ny][nx+1], Vy at y faces [nz][ny+1][nx], Vz at z faces [nz+1][ny][nx],
// every field of every subdomain in one buffer [nsub][...]. One leapfrog step:
//   Vx[i] -= dt/(rho dx) (P[i] - P[i-1]) on faces 1..nx-1 (all y, z), likewise
//   Vy, Vz;  then  P -= dt K / dx (Vx[i+1] - Vx[i]) + ... on every cell.
// The outermost faces are never written (walls, or halo faces of a
// subdomain that the halo update fills). One thread per (x, y) column marches
// along z, keeping the z neighbour in a register.
#include "igg_internal.h"

namespace igg {
namespace {

constexpr int kAcX = 32, kAcY = 8, kAcZ = 32;

// Coefficients in the storage type (formed on the host), and the number 1:
// FP64 differences a - b are computed as fma(a, 1, -b), the same rounding by the
// FMA instruction. The FP64 launches are bound by the FP64 pipe, which takes
// FMAs faster than additions (598 against 504 G/s in independent chains): 2x2x2
// x 256^3 cells, four steps, 11.89 to 11.25 ms.
template <class S>
struct AcW {
  S ax, ay, az, bx, by, bz, one;
};

template <class S>
struct AcNum;
template <>
struct AcNum<double> {
  static __device__ __forceinline__ double sub(double a, double b, double one) {
    return __fma_rn(a, one, -b);
  }
  static __device__ __forceinline__ double fma(double a, double b, double c) {
    return __fma_rn(a, b, c);
  }
};
template <>
struct AcNum<float> {
  static __device__ __forceinline__ float sub(float a, float b, float) { return __fsub_rn(a, b); }
  static __device__ __forceinline__ float fma(float a, float b, float c) {
    return __fmaf_rn(a, b, c);
  }
};

// blockIdx.z = subdomain * zchunks + z chunk. The z march is software
// pipelined: the loads of plane k + 1 are issued before the stores of plane
// k, so that each thread keeps two planes of loads in flight (the launches
// are bound by memory latency otherwise).
//
// x sends (AcCoef::xsend): update_halo!'s x exchange done by the launches
// themselves. A field of x size nf and x overlap of sends its plane nf - of
// to the right neighbour's plane 0 and its plane of - 1 to the left
// neighbour's plane nf - 1 (P, Vy, Vz: of = o; Vx: nf = nx + 1, of = o + 1);
// the thread of a sent column stores every value of it as the launch leaves
// it (computed, or a wall face it does not compute) a second time into the
// neighbour, and the threads of receiving columns do not store there. The y
// and z exchanges run after both launches.
// The x sends of one thread: sm bit 0 / 1 its column is sent right / left;
// dr, dl the neighbours' subdomain offsets (xr - sub, xl - sub). The copy of
// the value at own index q of a field of np points per subdomain and x send
// distance h = nf - of goes to q + dr np - h (right) and q + dl np + h (left).
struct AcSend {
  unsigned sm;
  int dr, dl;
};

__device__ __forceinline__ AcSend ac_send(int i, int nf, int of, long long sub, int xl, int xr) {
  AcSend a;
  a.sm = (xr >= 0 && i == nf - of ? 1u : 0u) | (xl >= 0 && i == of - 1 ? 2u : 0u);
  a.dr = xr - (int)sub;
  a.dl = xl - (int)sub;
  return a;
}

template <class S>
__device__ __forceinline__ void ac_put(S *p, S v, const AcSend &a, long long np, int h) {
  if (a.sm & 1u) p[(long long)a.dr * np - h] = v;
  if (a.sm & 2u) p[(long long)a.dl * np + h] = v;
}

// FP32: the planes kAcAhead ahead go into L2. Two planes of loads per thread are
// 20 KB in flight per SM, short of what the latency of device memory asks for
// (FP64 launches, bound by the FP64 pipe, only lose issue slots to it): 2x1x2 x
// 255x193x130, ten steps, 2.71 to 2.59 ms; 2x2x2 x 256^3 FP64, four, 11.28 with-
// out, 11.62 ms with it. Not where the fields fit in L2: 16 steps of 2x1x2 x 96^3
// (57 MB) 0.70 ms without, 0.84 with it; of 2x2x1 x 128^3 (134 MB) 1.77 and 1.66.
constexpr int kAcAhead = 3;
template <class S>
__device__ __forceinline__ void ac_ahead(const S *p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

template <class S>
__global__ void __launch_bounds__(kAcX *kAcY)
    k_acoustic_v(int nx, int ny, int nz, int zchunks, const S *P, S *Vx, S *Vy, S *Vz,
                 const AcW<S> w, const int *__restrict__ nbr, int ox, int xsend, int ahead) {
  using N = AcNum<S>;
  const int i = blockIdx.x * kAcX + threadIdx.x, j = blockIdx.y * kAcY + threadIdx.y;
  if (i >= nx || j >= ny) return;
  const long long sub = blockIdx.z / zchunks;
  const int k0 = (int)(blockIdx.z % zchunks) * kAcZ, k1 = min(k0 + kAcZ, nz);
  const long long np = (long long)nx * ny * nz;
  const long long sp = (long long)nx * ny, sx = (long long)(nx + 1) * ny,
                  sy = (long long)nx * (ny + 1);
  const long long npx = sx * nz, npy = sy * nz, npz = sp * (nz + 1);
  const S *Ps = P + sub * np + i + (long long)nx * j;
  S *Vxs = Vx + sub * npx + i + (long long)(nx + 1) * j;
  S *Vys = Vy + sub * npy + i + (long long)nx * j;
  S *Vzs = Vz + sub * npz + i + (long long)nx * j;
  // x sends (Vx: nf = nx + 1, of = o + 1; Vy, Vz: nf = nx, of = o; the
  // send distance nf - of is nx - o for all three) and the receiving columns
  // (halo cells: Vy and Vz not stored)
  AcSend ex{0u, 0, 0}, ev = ex;
  bool keep = true;
  const int h = nx - ox;
  if (xsend) {
    const int xl = nbr[6 * sub], xr = nbr[6 * sub + 1];
    ex = ac_send(i, nx + 1, ox + 1, sub, xl, xr);
    ev = ac_send(i, nx, ox, sub, xl, xr);
    keep = !((i == 0 && xl >= 0) || (i == nx - 1 && xr >= 0));
  }
  const bool sv = ev.sm != 0u;  // sends Vy and Vz (wall faces too)
  pdl_trigger();
  pdl_wait();
  S pzm = k0 > 0 ? Ps[sp * (k0 - 1)] : S(0);
  // plane k0
  S pc = Ps[sp * k0];
  S pxm = i > 0 ? Ps[sp * k0 - 1] : S(0);
  S pym = j > 0 ? Ps[sp * k0 - nx] : S(0);
  S vx = i > 0 ? Vxs[sx * k0] : S(0);
  S vy = (j > 0 || sv) ? Vys[sy * k0] : S(0);
  S vz = (k0 > 0 || sv) ? Vzs[sp * k0] : S(0);
  for (int k = k0; k < k1; ++k) {
    // plane k + 1
    const bool nxt = k + 1 < k1;
    S pc1 = S(0), pxm1 = S(0), pym1 = S(0), vx1 = S(0), vy1 = S(0), vz1 = S(0);
    if (sizeof(S) == 4 && k + ahead < k1) {
      ac_ahead(Ps + sp * (k + ahead));
      ac_ahead(Vxs + sx * (k + ahead));
      ac_ahead(Vys + sy * (k + ahead));
      ac_ahead(Vzs + sp * (k + ahead));
    }
    if (nxt) {
      pc1 = Ps[sp * (k + 1)];
      if (i > 0) {
        pxm1 = Ps[sp * (k + 1) - 1];
        vx1 = Vxs[sx * (k + 1)];
      }
      if (j > 0) pym1 = Ps[sp * (k + 1) - nx];
      if (j > 0 || sv) vy1 = Vys[sy * (k + 1)];
      vz1 = Vzs[sp * (k + 1)];
    }
    if (i > 0) {
      vx = N::fma(-w.ax, N::sub(pc, pxm, w.one), vx);
      Vxs[sx * k] = vx;
    }
    if (j > 0) {
      vy = N::fma(-w.ay, N::sub(pc, pym, w.one), vy);
      if (keep) Vys[sy * k] = vy;
    }
    if (k > 0) {
      vz = N::fma(-w.az, N::sub(pc, pzm, w.one), vz);
      if (keep) Vzs[sp * k] = vz;
    }
    if (ex.sm) ac_put(Vxs + sx * k, vx, ex, npx, h);
    if (sv) {
      ac_put(Vys + sy * k, vy, ev, npy, h);
      ac_put(Vzs + sp * k, vz, ev, npz, h);
      // the last face row of Vy (y = ny, a wall or halo face no thread
      // computes)
      if (j == ny - 1) ac_put(Vys + sy * k + nx, Vys[sy * k + nx], ev, npy, h);
    }
    pzm = pc;
    pc = pc1;
    pxm = pxm1;
    pym = pym1;
    vx = vx1;
    vy = vy1;
    vz = vz1;
  }
  // the last plane of Vz (z = nz, a wall or halo face no thread computes)
  if (sv && k1 == nz) ac_put(Vzs + sp * nz, Vzs[sp * nz], ev, npz, h);
}

template <class S>
__global__ void __launch_bounds__(kAcX *kAcY)
    k_acoustic_p(int nx, int ny, int nz, int zchunks, S *P,
                 const S *Vx, const S *Vy, const S *Vz, const AcW<S> w,
                 const int *__restrict__ nbr, int ox, int xsend, int ahead) {
  using N = AcNum<S>;
  const int i = blockIdx.x * kAcX + threadIdx.x, j = blockIdx.y * kAcY + threadIdx.y;
  if (i >= nx || j >= ny) return;
  const long long sub = blockIdx.z / zchunks;
  const int k0 = (int)(blockIdx.z % zchunks) * kAcZ, k1 = min(k0 + kAcZ, nz);
  const long long np = (long long)nx * ny * nz;
  const long long sp = (long long)nx * ny, sx = (long long)(nx + 1) * ny,
                  sy = (long long)nx * (ny + 1);
  S *Ps = P + sub * np + i + (long long)nx * j;
  const S *Vxs = Vx + sub * (long long)(nx + 1) * ny * nz + i + (long long)(nx + 1) * j;
  const S *Vys = Vy + sub * (long long)nx * (ny + 1) * nz + i + (long long)nx * j;
  const S *Vzs = Vz + sub * (long long)nx * ny * (nz + 1) + i + (long long)nx * j;
  AcSend ep{0u, 0, 0};
  bool keep = true;
  const int h = nx - ox;
  if (xsend) {
    const int xl = nbr[6 * sub], xr = nbr[6 * sub + 1];
    ep = ac_send(i, nx, ox, sub, xl, xr);
    keep = !((i == 0 && xl >= 0) || (i == nx - 1 && xr >= 0));
  }
  pdl_trigger();
  pdl_wait();
  S vzc = Vzs[sp * k0];
  // plane k0
  S pc = Ps[sp * k0], x0 = Vxs[sx * k0], x1 = Vxs[sx * k0 + 1], y0 = Vys[sy * k0],
    y1 = Vys[sy * k0 + nx], vzp = Vzs[sp * (k0 + 1)];
  for (int k = k0; k < k1; ++k) {
    // plane k + 1
    const bool nxt = k + 1 < k1;
    S pc1 = S(0), x01 = S(0), x11 = S(0), y01 = S(0), y11 = S(0), vzp1 = S(0);
    if (sizeof(S) == 4 && k + ahead < k1) {
      ac_ahead(Ps + sp * (k + ahead));
      ac_ahead(Vxs + sx * (k + ahead));
      ac_ahead(Vys + sy * (k + ahead));
      ac_ahead(Vzs + sp * (k + ahead));
    }
    if (nxt) {
      pc1 = Ps[sp * (k + 1)];
      x01 = Vxs[sx * (k + 1)];
      x11 = Vxs[sx * (k + 1) + 1];
      y01 = Vys[sy * (k + 1)];
      y11 = Vys[sy * (k + 1) + nx];
      vzp1 = Vzs[sp * (k + 2)];
    }
    // P - bx dVx - by dVy - bz dVz, one FMA per term (6 FP64 instructions
    // per cell for FP64 fields, whose launches the FP64 pipe bounds)
    S pn = N::fma(-w.bx, N::sub(x1, x0, w.one), pc);
    pn = N::fma(-w.by, N::sub(y1, y0, w.one), pn);
    pn = N::fma(-w.bz, N::sub(vzp, vzc, w.one), pn);
    if (keep) Ps[sp * k] = pn;
    if (ep.sm) ac_put(Ps + sp * k, pn, ep, np, h);
    vzc = vzp;
    pc = pc1;
    x0 = x01;
    x1 = x11;
    y0 = y01;
    y1 = y11;
    vzp = vzp1;
  }
}

template <class S>
cudaError_t launch_t(int nsub, int nx, int ny, int nz, void *P, void *Vx, void *Vy, void *Vz,
                     const AcCoef &c, cudaStream_t s) {
  const int zchunks = (nz + kAcZ - 1) / kAcZ;
  const long long gz = (long long)nsub * zchunks;
  if (gz > 65535) return cudaErrorInvalidValue;
  const dim3 grid((nx + kAcX - 1) / kAcX, (ny + kAcY - 1) / kAcY, (unsigned)gz);
  const dim3 block(kAcX, kAcY);
  const AcW<S> w = {(S)c.ax, (S)c.ay, (S)c.az, (S)c.bx, (S)c.by, (S)c.bz, S(1)};
  // FP64: the CTAs of a dependent launch fill the SMs that the one before leaves
  // room on, and where those are neither idle nor soon drained the FP64 pipes end
  // up with unequal shares (16 steps, early start against none: 64^3, 32 CTAs,
  // 547 and 610 us; 2x1x2 x 70x60x64, 192, 1762 and 1022; 2x1x1 x 128^3, 512,
  // 2137 and 2023; 2x1x2 x 200x160x128, 2240, 6492 and 6590). So up to one CTA per
  // SM (152 SMs), and again above eight; where between 512 and 2240 CTAs the
  // upper line lies was not measured. FP32 launches gain at every size.
  const long long ctas = (long long)grid.x * grid.y * grid.z;
  const bool pdl = sizeof(S) == 4 || ctas <= 152 || ctas > 2 * 4 * 152;
  // (kAcAhead: fields that stay in L2 only lose issue slots to the prefetches)
  const long long bytes = 4ll * nsub * nx * ny * nz * (long long)sizeof(S);
  const int ahead = bytes > (96ll << 20) ? kAcAhead : nz;
  cudaError_t e = launch_pdl(pdl, k_acoustic_v<S>, grid, block, 0, s, nx, ny, nz, zchunks, (const S *)P,
                             (S *)Vx, (S *)Vy, (S *)Vz, w, c.nbr, c.ox, c.xsend, ahead);
  if (e != cudaSuccess) return e;
  return launch_pdl(pdl, k_acoustic_p<S>, grid, block, 0, s, nx, ny, nz, zchunks, (S *)P, (const S *)Vx,
                    (const S *)Vy, (const S *)Vz, w, c.nbr, c.ox, c.xsend, ahead);
}

}  // namespace

cudaError_t launch_acoustic(igg_dtype dt, int nsub, int nx, int ny, int nz, void *P, void *Vx,
                            void *Vy, void *Vz, const AcCoef &c, cudaStream_t s) {
  switch (dt) {
    case IGG_F64: return launch_t<double>(nsub, nx, ny, nz, P, Vx, Vy, Vz, c, s);
    case IGG_F32: return launch_t<float>(nsub, nx, ny, nz, P, Vx, Vy, Vz, c, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace igg
