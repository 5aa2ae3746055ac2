// Float-pair ("double-float") arithmetic on the FP32 pipe for FP64 data:
// bit-move conversions between FP64 values and pairs h + l of FP32 values
// (~48-bit significands), and the steps of a compensated dot product (Dot2
// of Ogita, Rump and Oishi) on pairs. GB300 issues about two FP64
// instructions per SM and clock against 128 FP32 lanes, so sums of many
// FP64 terms whose signs vary (where exact integer differences do not
// apply) run faster this way, ending in one FP64 add.
#pragma once

#include <cuda_runtime.h>

namespace igg {
namespace {

// FP32 arithmetic on one number or, as float2, on two points at once (packed
// instructions: half the issue slots). The sums below are
// written so that no product feeds an addition (products are FMAs with a
// zero addend, or folded into the FMA that uses them): the compiler may fuse
// a packed multiply into a following packed addition, which would change the
// rounding against the scalar form.
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ float2 vneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float vset(float w, float) { return w; }
__device__ __forceinline__ float2 vset(float w, float2) { return make_float2(w, w); }

// error-free sum a + b = s + e (Knuth's two-sum), per lane
template <class V>
__device__ __forceinline__ V vtwo_sum(V a, V b, V &e) {
  const V s = vadd(a, b);
  const V bb = vadd(s, vneg(a));
  e = vadd(vadd(a, vneg(vadd(s, vneg(bb)))), vadd(b, vneg(bb)));
  return s;
}

// float pair h + l (F = float2: of two points)
template <class F>
struct FFv {
  F h, l;
};
using FF = FFv<float>;
using FF2 = FFv<float2>;

// True when x is zero or its exponent field lies in [1023 - r, 1023 + r].
// Radii of at most 127 keep that inside pair_split's range [949, 1150].
constexpr unsigned kPairMaxRadius = 127;
__device__ __forceinline__ bool pair_ok(double x, unsigned r) {
  const unsigned hw = (unsigned)__double2hiint(x), lw = (unsigned)__double2loint(x);
  const unsigned E = (hw >> 20) & 0x7FFu;
  return E - (1023u - r) <= 2u * r || ((hw << 1) | lw) == 0u;
}

// x = h + l by bit moves; meaningful for zero and exponent fields in
// [949, 1150] (at 1151 the head's FP32 exponent field would be 255; callers
// check pair_ok with radii of at most 127), any input runs without faults.
__device__ __forceinline__ FF pair_split(double x) {
  const unsigned hw = (unsigned)__double2hiint(x), lw = (unsigned)__double2loint(x);
  const unsigned s = hw & 0x80000000u;
  // (E - 896) << 20 | top fraction bits, then shifted in with the next 3 bits
  const unsigned t = (hw & 0x7FFFFFFFu) - (896u << 20);
  const unsigned hb = __funnelshift_l(lw, t, 3) | s;
  // +-2^(E-1075): the weight of the last fraction bit
  const unsigned sc = (((hw & 0x7FF00000u) - (948u << 20)) << 3) | s;
  FF r;
  r.h = __uint_as_float(hb);
  r.l = __fmul_rn(__uint2float_rn(lw & 0x1FFFFFFFu), __uint_as_float(sc));
  const bool zero = ((hw << 1) | lw) == 0u;
  r.h = zero ? 0.f : r.h;
  r.l = zero ? 0.f : r.l;
  return r;
}

// float -> double by bit moves: exact for normal numbers, infinities and
// NaNs; zero and subnormal inputs give a zero of the same sign.
__device__ __forceinline__ double f2d_bits(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned s = b & 0x80000000u, e8 = b & 0x7F800000u;
  unsigned hi = s | (((b & 0x7FFFFFFFu) >> 3) + (896u << 20));
  hi = e8 == 0x7F800000u ? (s | 0x7FF00000u | ((b & 0x007FFFFFu) >> 3)) : hi;
  hi = e8 == 0u ? s : hi;
  const unsigned lo = e8 == 0u ? 0u : b << 29;
  return __hiloint2double((int)hi, (int)lo);
}

// float -> double by bit moves for finite inputs: exact for normal numbers,
// zero and subnormal inputs give a zero of the same sign.
__device__ __forceinline__ double f2d_finite(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned s = b & 0x80000000u;
  const bool z = (b & 0x7F800000u) == 0u;
  const unsigned hi = z ? s : s | (((b & 0x7FFFFFFFu) >> 3) + (896u << 20));
  return __hiloint2double((int)hi, z ? 0 : (int)(b << 29));
}

// error-free sum when |a| >= |b| or a == 0 (Dekker): a + b = s + e exactly
template <class F>
__device__ __forceinline__ F vfast_two_sum(F a, F b, F &e) {
  const F s = vadd(a, b);
  e = vadd(b, vneg(vadd(s, vneg(a))));
  return s;
}

// acc + err += w * v (w, v pairs): error-free leading product and sum, the
// small parts into err
template <class F>
__device__ __forceinline__ void dot2_term(F &acc, F &err, F wh, F wl, F vh, F vl) {
  const F p = vfma(wh, vh, vset(0.f, F()));
  F q = vfma(wh, vh, vneg(p));
  q = vfma(wh, vl, q);
  q = vfma(wl, vh, q);
  F e;
  acc = vtwo_sum(acc, p, e);
  err = vadd(err, vadd(e, q));
}

// acc + err += w * (a + b) for the neighbour pair (a, b)
template <class F>
__device__ __forceinline__ void dot2_pair(F &acc, F &err, float wh, float wl, const FFv<F> &a,
                                          const FFv<F> &b) {
  F t;
  const F s = vtwo_sum(a.h, b.h, t);
  t = vadd(t, vadd(a.l, b.l));
  const F h = vset(wh, F());
  const F p = vfma(h, s, vset(0.f, F()));
  F q = vfma(h, s, vneg(p));
  q = vfma(h, t, q);
  q = vfma(vset(wl, F()), s, q);
  F e;
  acc = vtwo_sum(acc, p, e);
  err = vadd(err, vadd(e, q));
}

}  // namespace
}  // namespace igg
