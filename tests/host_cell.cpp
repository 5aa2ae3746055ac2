// The cells of csrc/cell.cuh on the CPU: its device functions compiled as C++,
// with the CUDA intrinsics that they use written out (built by
// test_emu_cell_host.py with -ffp-contract=off, so every operation rounds as
// written).
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

template <class A, class B>
static A as(B b) {
  static_assert(sizeof(A) == sizeof(B), "size");
  A a;
  std::memcpy(&a, &b, sizeof a);
  return a;
}
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
static inline double __dadd_rn(double a, double b) { return a + b; }
static inline double __dsub_rn(double a, double b) { return a - b; }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
static inline float2 __fadd2_rn(float2 a, float2 b) { return {a.x + b.x, a.y + b.y}; }
static inline float2 __ffma2_rn(float2 a, float2 b, float2 c) {
  return {std::fmaf(a.x, b.x, c.x), std::fmaf(a.y, b.y, c.y)};
}
static inline float __int2float_rn(int a) { return (float)a; }
static inline float __uint2float_rn(unsigned a) { return (float)a; }
static inline float __double2float_rn(double a) { return (float)a; }
static inline float __int_as_float(int a) { return as<float>(a); }
static inline float __uint_as_float(unsigned a) { return as<float>(a); }
static inline unsigned __float_as_uint(float a) { return as<unsigned>(a); }
static inline long long __double_as_longlong(double a) { return as<long long>(a); }
static inline double __longlong_as_double(long long a) { return as<double>(a); }
static inline int __double2hiint(double a) { return (int)(as<unsigned long long>(a) >> 32); }
static inline int __double2loint(double a) { return (int)as<unsigned long long>(a); }
static inline double __hiloint2double(int h, int l) {
  return as<double>(((unsigned long long)(unsigned)h << 32) | (unsigned)l);
}
static inline unsigned __funnelshift_r(unsigned lo, unsigned hi, unsigned s) {
  return (unsigned)((((unsigned long long)hi << 32) | lo) >> (s & 31u));
}
static inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) {
  return (unsigned)((((unsigned long long)hi << 32 | lo) << (s & 31u)) >> 32);
}
template <class T>
static T __ldg(const T *p) { return *p; }
template <class T>
static T min(T a, T b) { return b < a ? b : a; }
template <class T>
static T max(T a, T b) { return a < b ? b : a; }

#include "cell.cuh"

using namespace igg;

// n stencils t[7] = centre, x-, x+, y-, y+, z-, z+ with Ci: out the result of
// the path that the cell takes, path 0 = fast, 1 = aligned, 2 = FP64.
template <int NG>
static void run(int n, const double *t, const double *ci, const W<double> &w, double *out, int *path) {
  for (int i = 0; i < n; ++i) {
    const double *s = t + 7 * i;
    unsigned long long nb[6];
    for (int k = 0; k < 6; ++k) nb[k] = dbits(s[1 + k]);
    bool ok;
    path[i] = 0;
    out[i] = cell_emu_fast<NG>(s[0], nb, ci[i], w, ok);
    if (ok) continue;
    path[i] = 1;
    out[i] = cell_emu_aligned<NG>(s[0], nb, ci[i], w, ok);
    if (ok) continue;
    path[i] = 2;
    out[i] = cell_f64(s[0], s[1], s[2], s[3], s[4], s[5], s[6], ci[i], w);
  }
}

extern "C" int host_cells(int n, const double *t, const double *ci, const double *wts, double *out,
                          int *path) {
  W<double> w = {};
  const double d[3] = {wts[0], wts[1], wts[2]};
  w.wx = d[0];
  w.wy = d[1];
  w.wz = d[2];
  w.wc = -2.0 * (d[0] + d[1] + d[2]);
  for (int i = 0; i < 3; ++i) {
    w.wh[i] = (float)d[i];
    w.wl[i] = (float)(d[i] - (double)w.wh[i]);
    w.ah[i] = 8388608.0f * w.wh[i];
    w.al[i] = 8388608.0f * w.wl[i];
  }
  w.emu = true;
  w.ng = weight_groups(d[0], d[1], d[2]);
  if (w.ng == 1) run<1>(n, t, ci, w, out, path);
  else if (w.ng == 2) run<2>(n, t, ci, w, out, path);
  else run<3>(n, t, ci, w, out, path);
  return w.ng;
}
