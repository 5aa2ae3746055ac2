// Row-copy stencil kernel: the full FP64 step on 3-D grids of odd row length
// (255 or 127 points, say), whose rows are not a multiple of 16 bytes: no tensor
// map takes them (a pitch is a multiple of 16 bytes), and they start at either
// alignment. T and Ci themselves start on 16 bytes (use_rows, runtime.cu): a
// copy's 16-byte boundary is found from the element index.
//
// What bounds it: with plain loads, one point per thread and step in flight, it
// was the latency of the loads (2x2x2 x 255x127x129 FP64, ten steps: 2.57 ms,
// 0.46 of the copy bandwidth; now 1.81, 0.66). As in the TMA kernel (tma.cu) a producer warp
// keeps several planes of a tile in flight with bulk copies, here one untiled
// cp.async.bulk per row, issued by a lane each: the row from the 16-byte
// boundary at or before its first point, so that it lies in its shared-memory
// row with a shift of 0 or 1 points (V = 2 points are 16 bytes), the same for
// producer and consumers, who both get it from the row's index. A lane of a
// consumer warp takes the points lane, lane + 32, .. of its row: shared-memory
// loads and global stores of one point each stay contiguous over the warp at
// any shift. The producer's copies of a row each bound it then (the consumers
// wait for them): FP64 tiles of 64 points by 16 rows (512 bytes a copy) took 2.21 ms,
// of 128 by 8 2.08 with two CTAs per SM and 1.81 with three. The same on FP32 and
// BF16 fields, whose copies of a row are a half and a quarter as long, took
// 1.11 and 1.14 ms where the scalar kernel takes 0.93 and 0.79: theirs stay
// with the scalar kernel.
//
// Ring protocol as in the TMA kernel: load k brings T plane m0 - 1 + k and Ci
// plane m0 - 2 + k into stage k % NS (full[s]: count 1 + transaction bytes;
// empty[s]: one arrival per consumer warp), step j reads loads j and j + 1.
// Every wait is bounded; on a timeout the kernel records IGG_DEV_ERR_TIMEOUT,
// waits (bounded) for its copies in flight and returns.
//
// No copy leaves the field: a row's copy starts at a multiple of V elements
// that is at least 0 and ends at one that is at most the field's length. What
// is cut off at the end (less than V points of the very last row, y = ny - 1 and
// z = nz - 1 of the last subdomain) is read by no stencil: rows have at least
// kRowsMinNx > V points.
#include "cell.cuh"
#include "fixlist.cuh"
#include "igg_internal.h"
#include "tma_util.cuh"

namespace igg {
namespace {

// fix-up entries a consumer warp stages (FP64: three CTAs per SM leave room for
// eight)
constexpr unsigned kRowsPend = 8;

struct Sh {
  static constexpr int V = 2;                           // points per 16 bytes
  static constexpr int P = 4;                           // points per lane and row
  static constexpr int W = 32 * P;                      // points per row of a tile
  static constexpr int BW = (W + 2 + V - 1 + V - 1) / V * V;  // T row in shared memory
  static constexpr int CW = (W + V - 1 + V - 1) / V * V;      // Ci row
  static constexpr int H = 8;                            // rows of a tile
  static constexpr int BH = H + 2;
  static constexpr int NS = 4;
  static constexpr int CONSUMERS = 8;
  static constexpr int RPT = H / CONSUMERS;             // rows per consumer warp
  static constexpr int TB = BW * BH * 8;                  // (multiples of 16 bytes)
  static constexpr int CB = CW * H * 8;
  static constexpr int STAGE = TB + CB;
  static constexpr int BARS = NS * STAGE;
  static constexpr int PEND = BARS + 2 * NS * 8 + 64;
  static constexpr int SMEM = PEND + CONSUMERS * (int)kRowsPend * 16;
  static_assert(H % CONSUMERS == 0 && V < kRowsMinNx, "tile");
  static_assert(3 * (SMEM + 1024) <= 228 * 1024, "three CTAs per SM");
  static_assert(BH <= 32 && H <= 32, "one copy per lane");
};

__device__ __forceinline__ void bulk_row(unsigned dst, const void *src, unsigned bytes,
                                         unsigned bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}

// MODE 1: the FP64 cell; 2 + (3 - NG): the emulated cell's fast path with NG
// weight groups
template <int MODE>
__global__ void __launch_bounds__(32 * 9, 3)
    k_stencil_rows(const TmaTile *__restrict__ tiles, double *T2, const double *T,
                   const double *Ci, int nx, int ny,
                   Coef c0, unsigned *dev_err, void *fix, size_t fix_cap) {
  constexpr int V = Sh::V, NS = Sh::NS, P = Sh::P;
  constexpr bool EMU = MODE >= 2;
  extern __shared__ __align__(128) unsigned char smem[];
  const unsigned sbase = smem_u32(smem);
  const unsigned full0 = sbase + Sh::BARS, empty0 = full0 + NS * 8;
  volatile int *flags = reinterpret_cast<volatile int *>(smem + Sh::BARS + 2 * NS * 8);
  // flags[0]: abort; flags[1]: loads issued; flags[2]: loads consumed
  const TmaTile t = tiles[blockIdx.x];
  const int K = (t.m1 - t.m0) + 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long sz = (long long)nx * ny;
  if (threadIdx.x == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, Sh::CONSUMERS);
    }
    flags[0] = 0;
    flags[1] = 0;
    flags[2] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();

  if (warp == Sh::CONSUMERS) {
    // ---------------- producer (all lanes; lane l copies row l) ----------------
    pdl_trigger();
    pdl_wait();
    const long long lim = c0.npts / V * V;  // no copy beyond it
    // T rows r0 - 1 .. re (r0 >= 1, re <= ny - 1), points xb - 1 .. xe; Ci rows
    // r0 .. re - 1, points xb .. xe - 1
    const bool hasT = lane < t.re - t.r0 + 2, hasC = lane < t.re - t.r0;
    int k = 0;
    for (; k < K; ++k) {
      const int s = k % NS;
      bool ok = true;
      if (k >= NS) ok = __all_sync(0xffffffffu, mbar_wait(empty0 + 8 * s, ((k / NS) - 1) & 1));
      if (!ok) {
        if (lane == 0) {
          atomicOr(dev_err, IGG_DEV_ERR_TIMEOUT);
          flags[0] = 1;
        }
        break;
      }
      if (__any_sync(0xffffffffu, flags[0] != 0)) break;
      const long long pT = t.base + sz * (t.m0 - 1 + k);
      // (a tile has m0, r0, xb >= 1: eT >= 0)
      const long long eT = pT + (long long)nx * (t.r0 - 1 + lane) + t.xb - 1;
      const long long eC = pT - sz + (long long)nx * (t.r0 + lane) + t.xb;
      const long long aT = eT - (eT & (V - 1)), aC = eC - (eC & (V - 1));
      long long bT = (eT + (t.xe - t.xb) + 2 + V - 1) / V * V;
      long long bC = (eC + (t.xe - t.xb) + V - 1) / V * V;
      bT = min(bT, lim);
      bC = min(bC, lim);
      const unsigned nT = hasT && bT > aT ? (unsigned)(bT - aT) * 8u : 0u;
      const unsigned nC = k >= 2 && hasC && bC > aC ? (unsigned)(bC - aC) * 8u : 0u;
      const unsigned total = __reduce_add_sync(0xffffffffu, nT + nC);
      const unsigned bar = full0 + 8 * s, dst = sbase + s * Sh::STAGE;
      if (lane == 0) mbar_expect_tx(bar, total);
      __syncwarp();
      if (nT) bulk_row(dst + (unsigned)(lane * Sh::BW * 8), T + aT, nT, bar);
      if (nC)
        bulk_row(dst + Sh::TB + (unsigned)(lane * Sh::CW * 8), Ci + aC, nC, bar);
    }
    if (lane == 0) flags[1] = k;
  } else {
    // ---------------- consumers ----------------
    const W<double> w = make_w(c0, 0.0);
    // this lane's points of a row: x = xb + lane + 32 i
    unsigned inm = 0u;
#pragma unroll
    for (int i = 0; i < P; ++i)
      if (t.xb + lane + 32 * i < t.xe) inm |= 1u << i;
    // shared-memory index of the lane's first point in a T or Ci row whose first
    // copied point has element index e (the row's shift is e mod V)
    auto shT = [&](int e) { return (e & (V - 1)) + 1 + lane; };
    auto shC = [&](int e) { return (e & (V - 1)) + lane; };
    // element indices mod 2^32 (only their low bits matter): the T row r0 + r of
    // plane m starts at e0 + sz (m - m0) + nx r
    const unsigned usz = (unsigned)sz;
    const unsigned e0 = (unsigned)(t.base + sz * t.m0 + (long long)nx * t.r0 + t.xb - 1);
    int rowi[Sh::RPT];
    bool comp[Sh::RPT];
#pragma unroll
    for (int j = 0; j < Sh::RPT; ++j) {
      rowi[j] = warp + j * Sh::CONSUMERS;
      comp[j] = t.r0 + rowi[j] < t.re;
    }
    double zm[Sh::RPT][P];
    bool ok = __all_sync(0xffffffffu, mbar_wait(full0, 0) && mbar_wait(full0 + 8, 0));
    if (!ok) {
      atomicOr(dev_err, IGG_DEV_ERR_TIMEOUT);
      flags[0] = 1;
    } else {
      const double *Tb = reinterpret_cast<const double *>(smem);
#pragma unroll
      for (int j = 0; j < Sh::RPT; ++j) {
        const double *row = Tb + (rowi[j] + 1) * Sh::BW + shT((int)(e0 - usz + (unsigned)(nx * rowi[j])));
#pragma unroll
        for (int i = 0; i < P; ++i) zm[j][i] = row[32 * i];
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty0);
    }
    int consumed = 2;
    // the warp's staged fix-up entries (emulated FP64 cell)
    FixEntry *pend = reinterpret_cast<FixEntry *>(smem + Sh::PEND) + warp * kRowsPend;
    unsigned npend = 0u;  // warp-uniform
    auto flush = [&]() {
      __syncwarp();
      if (npend) {
        const FixList fl = fix_list(fix, fix_cap);
        unsigned base = 0u;
        if (lane == 0) base = atomicAdd(fl.count, npend);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (lane < npend && base + lane < fix_cap) fl.e[base + lane] = pend[lane];
        npend = 0u;
      }
      __syncwarp();
    };
    unsigned e = e0;
#pragma unroll 1
    for (int m = t.m0; ok && m < t.m1; ++m, e += usz) {
      const int k = m - t.m0 + 1;
      const int s = k % NS, s1 = (k + 1) % NS;
      if (!__all_sync(0xffffffffu, mbar_wait(full0 + 8 * s1, ((k + 1) / NS) & 1))) {
        atomicOr(dev_err, IGG_DEV_ERR_TIMEOUT);
        flags[0] = 1;
        ok = false;
        break;
      }
      consumed = k + 2;
      const double *Tc = reinterpret_cast<const double *>(smem + s * Sh::STAGE);
      const double *Tn = reinterpret_cast<const double *>(smem + s1 * Sh::STAGE);
      const double *Cn = reinterpret_cast<const double *>(smem + s1 * Sh::STAGE + Sh::TB);
#pragma unroll
      for (int j = 0; j < Sh::RPT; ++j) {
        const int r = rowi[j];
        const int er = (int)(e + (unsigned)(nx * r));
        const double *row = Tc + (r + 1) * Sh::BW + shT(er);
        const double *up = Tc + r * Sh::BW + shT(er - nx);
        const double *dn = Tc + (r + 2) * Sh::BW + shT(er + nx);
        const double *zpr = Tn + (r + 1) * Sh::BW + shT((int)((unsigned)er + usz));
        const double *cir = Cn + r * Sh::CW + shC(er + 1);
        double c[P], out[P];
#pragma unroll
        for (int i = 0; i < P; ++i) c[i] = row[32 * i];
        unsigned okm = (1u << P) - 1u;
        if constexpr (EMU) {
          constexpr int NG = 5 - MODE;
          // two points' FP32 sums at a time as float2, the tests per point
          okm = 0u;
#pragma unroll
          for (int i2 = 0; i2 < P; i2 += 2) {
            int gh[2][NG];
            unsigned gm[2][NG], o[2] = {0u, 0u}, rr[2] = {0u, 0u};
            double ci[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int i = i2 + h;
              const unsigned long long nb[6] = {
                  dbits(row[32 * i - 1]), dbits(row[32 * i + 1]), dbits(up[32 * i]),
                  dbits(dn[32 * i]),      dbits(zm[j][i]),        dbits(zpr[32 * i])};
              emu2_int<NG>(dbits(c[i]), nb, dhi(c[i]), gh[h], gm[h], o[h], rr[h]);
              ci[h] = cir[32 * i];
            }
            float2 fh[NG], fl[NG];
#pragma unroll
            for (int g = 0; g < NG; ++g) {
              fh[g] = make_float2(__int2float_rn(gh[0][g]), __int2float_rn(gh[1][g]));
              fl[g] = make_float2(__uint_as_float(gm[0][g]), __uint_as_float(gm[1][g]));
            }
            float2 Sv, Cv;
            emu2_sum<NG>(fh, fl, w, Sv, Cv);
            const float2 Kr = vfma(make_float2(emu2_cif(ci[0]), emu2_cif(ci[1])), Cv,
                                   vset(kMagic, float2()));
            const float2 Kd = vadd(Kr, vset(-kMagic, float2()));
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int i = i2 + h;
              const unsigned hc = dhi(c[i]);
              out[i] = emu2_apply(dbits(c[i]), hc, ci[h], h ? Sv.y : Sv.x, h ? Kr.y : Kr.x);
              if (emu2_centre_ok(hc) &&
                  emu2_ok(o[h] | (dhi(out[i]) ^ hc), rr[h], ci[h], h ? Kd.y : Kd.x))
                okm |= 1u << i;
            }
          }
        } else {
#pragma unroll
          for (int i = 0; i < P; ++i) {
            const double xm = row[32 * i - 1], xp = row[32 * i + 1];
            const double ym = up[32 * i], yp = dn[32 * i];
            const double zp = zpr[32 * i], ci = cir[32 * i];
            out[i] = cell_f64(c[i], xm, xp, ym, yp, zm[j][i], zp, ci, w);
          }
        }
        const long long di = t.base + t.xb + lane + (long long)nx * (t.r0 + r) + sz * m;
        if (comp[j]) {
#pragma unroll
          for (int i = 0; i < P; ++i)
            if ((inm >> i & 1u) && in_bounds(di + 32 * i, c0.npts)) T2[di + 32 * i] = out[i];
        }
        if constexpr (EMU) {
          // list each 32-point segment of the row with refused points
          const unsigned defm = comp[j] ? (~okm & inm) : 0u;
          if (__any_sync(0xffffffffu, defm != 0u)) {
#pragma unroll
            for (int i = 0; i < P; ++i) {
              const unsigned bits = __ballot_sync(0xffffffffu, defm >> i & 1u);
              if (bits) {
                if (lane == 0) {
                  FixEntry en;
                  en.p = di + 32 * i;
                  en.bits = bits;
                  en.pad = 0u;
                  pend[npend] = en;
                }
                ++npend;
              }
            }
            if (npend > kRowsPend - P) flush();
          }
        }
#pragma unroll
        for (int i = 0; i < P; ++i) zm[j][i] = c[i];
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty0 + 8 * s);
    }
    if constexpr (EMU) flush();
    if (warp == 0 && lane == 0) flags[2] = consumed;
  }
  __syncthreads();
  // After an abort, wait (bounded) for copies issued but never consumed, so
  // that no bulk copy writes into this CTA's shared memory after it exits.
  if (threadIdx.x == 0 && flags[0]) {
    for (int k = flags[2]; k < flags[1]; ++k) {
      if (!mbar_wait(full0 + 8 * (k % NS), (k / NS) & 1)) {
        atomicOr(dev_err, IGG_DEV_ERR_DRAIN);
        break;
      }
    }
  }
}

template <int MODE>
cudaError_t prepare_t(int *ctas) {
  cudaError_t e = cudaFuncSetAttribute(k_stencil_rows<MODE>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, Sh::SMEM);
  if (e == cudaSuccess && ctas)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas, k_stencil_rows<MODE>,
                                                      32 * (Sh::CONSUMERS + 1), Sh::SMEM);
  return e;
}

template <int MODE>
cudaError_t launch_t(const TmaTile *tiles, int ntiles, void *T2, const void *T, const void *Ci,
                     int nx, int ny, const Coef &c, unsigned *dev_err, FixBuf fix, cudaStream_t s) {
  return launch_pdl(pdl_on(c.npts), k_stencil_rows<MODE>, ntiles, 32 * (Sh::CONSUMERS + 1), Sh::SMEM, s, tiles,
                    (double *)T2, (const double *)T, (const double *)Ci, nx, ny, c, dev_err, fix.p, fix.cap);
}

}  // namespace

int rows_tile_width() { return Sh::W; }
int rows_tile_rows() { return Sh::H; }

cudaError_t rows_prepare(int *ctas) {
  cudaError_t e = prepare_t<1>(nullptr);
  if (e == cudaSuccess) e = prepare_t<2>(nullptr);
  if (e == cudaSuccess) e = prepare_t<4>(nullptr);
  return e == cudaSuccess ? prepare_t<3>(ctas) : e;
}

cudaError_t launch_stencil_rows(const TmaTile *tiles, int ntiles, void *T2, const void *T,
                                const void *Ci, int nx, int ny, long long nzt, const Coef &c,
                                unsigned *dev_err, FixBuf fix, cudaStream_t s) {
  if (ntiles <= 0) return cudaSuccess;
  Coef cc = c;
  cc.npts = (long long)nx * ny * nzt;
  if (!c.f64_emu) return launch_t<1>(tiles, ntiles, T2, T, Ci, nx, ny, cc, dev_err, fix, s);
  if (!fix.p) return cudaErrorInvalidValue;
  cudaError_t e;
  switch (weight_groups(c.wx, c.wy, c.wz)) {
    case 1: e = launch_t<4>(tiles, ntiles, T2, T, Ci, nx, ny, cc, dev_err, fix, s); break;
    case 2: e = launch_t<3>(tiles, ntiles, T2, T, Ci, nx, ny, cc, dev_err, fix, s); break;
    default: e = launch_t<2>(tiles, ntiles, T2, T, Ci, nx, ny, cc, dev_err, fix, s);
  }
  return e == cudaSuccess ? launch_fixup(fix, T2, T, Ci, nx, ny, cc, s) : e;
}

cudaError_t rows_bounds_flag(unsigned *out, bool clear) { return read_bounds_flag(out, clear); }

}  // namespace igg
