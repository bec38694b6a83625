// Box-Muller transform of two Philox words, evaluated in float-float arithmetic so
// that the FP32 Gaussian is the correctly rounded value of
//   g_even = sqrt(-2 ln u0) cos(2 pi u1),   g_odd = sqrt(-2 ln u0) sin(2 pi u1),
// u_j = ((x_j >> 8) + 1) 2^-24, except where the float-float value (relative error
// below about 2^-44) falls within that distance of a rounding midpoint.
//
// A float-float number is an unevaluated sum h + l of two floats.  Sums and products
// use the error-free transforms of Dekker (1971) and Knuth (TAOCP vol. 2): two_sum,
// fast_two_sum and two_prod (the rounding error of a product from one FMA).  Every
// operation is written with intrinsics of fixed rounding, which the compiler never contracts
// into FMAs, so each transform is exact as written.
//
//  ln u0  Table-driven logarithm after Tang (1990, ACM TOMS 16, "Table-driven
//         implementation of the logarithm function in IEEE floating-point arithmetic"):
//         u0 = 2^e f with f in [sqrt(1/2), sqrt(2)], c = a float near 1/F for the table
//         point F = 1 + j/128 nearest to f, t = f c - 1 (exact as a float-float,
//         |t| < 2^-7.5), ln u0 = e ln 2 - ln c + ln(1 + t), the last term by its Taylor
//         series (t and t^2/2 in float-float, t^3 (1/3 - t/4 + ...) in float).
//  sqrt   One Newton correction of the float square root with the exact residual.
//  sincos Quadrant and octant symmetry reduce 2 pi u1 exactly to phi in [0, pi/4];
//         phi = a_j + delta with a table point a_j = 2 pi j / 4096 and 0 <= delta <
//         2 pi / 4096; angle addition with the table's cos a_j, sin a_j (float-float)
//         and the Taylor series of cos delta, sin delta.
//
// The table (kBmTableLen float4, built in FP64 on the host by lpt2::bm_table):
//   [0, 513)          (cos a_j hi, lo, sin a_j hi, lo), a_j = 2 pi j / 4096, j = 0..512
//   [513, 604)        (c_j, -ln c_j hi, lo, 0), c_j = float(1 / (1 + j/128)), j = -37..53
//   604               (2 pi hi, lo, ln 2 hi, lo)
#pragma once
#include <stdint.h>

#include "packed.cuh"

namespace lpt2 {

constexpr int kBmSinCos = 513;
constexpr int kBmLogLo = -37, kBmLogHi = 53;
constexpr int kBmLog0 = kBmSinCos;                           // entry of j = kBmLogLo
constexpr int kBmConst = kBmSinCos + (kBmLogHi - kBmLogLo + 1);
constexpr int kBmTableLen = kBmConst + 1;

// Fills the table on the host (FP64 values split into float pairs).
void bm_table(float4* t);

// Two draws at a time: every float operation is the packed form of both draws' (packed.cuh),
// which halves the issue slots of the float-float arithmetic that bounds the noise pass
// (z_r2c_noise at 512^3 750 -> 684 us: then
// the FMA pipe, which a packed instruction holds for two cycles, and Philox bound it).
struct ffl {   // float-float values h + l of two draws
  float2 h, l;
};

__device__ __forceinline__ ffl ff_two_sum(float2 a, float2 b) {
  const float2 s = padd(a, b);
  const float2 bb = psub(s, a);
  return {s, padd(psub(a, psub(s, bb)), psub(b, bb))};
}
__device__ __forceinline__ ffl ff_two_diff(float2 a, float2 b) {   // a - b
  const float2 s = psub(a, b);
  const float2 bb = psub(s, a);
  return {s, psub(psub(a, psub(s, bb)), padd(b, bb))};
}
__device__ __forceinline__ ffl ff_fast_two_sum(float2 a, float2 b) {   // |a| >= |b| or a = 0
  const float2 s = padd(a, b);
  return {s, psub(b, psub(s, a))};
}
__device__ __forceinline__ ffl ff_two_prod(float2 a, float2 b) {
  const float2 p = pmul(a, b);
  return {p, pfma(a, b, pneg(p))};
}
__device__ __forceinline__ ffl ff_mul(ffl a, ffl b) {
  const ffl p = ff_two_prod(a.h, b.h);
  const float2 t = pfma(a.h, b.l, pmul(a.l, b.h));
  return ff_fast_two_sum(p.h, padd(p.l, t));
}
__device__ __forceinline__ ffl ff_add(ffl a, ffl b) {
  const ffl s = ff_two_sum(a.h, b.h);
  return ff_fast_two_sum(s.h, padd(s.l, padd(a.l, b.l)));
}
__device__ __forceinline__ ffl ff_sub(ffl a, ffl b) {
  const ffl s = ff_two_diff(a.h, b.h);
  return ff_fast_two_sum(s.h, padd(s.l, psub(a.l, b.l)));
}

// m = 2^e f 2^24 with f in [sqrt(1/2), sqrt(2)]; the table entry of f.
__device__ __forceinline__ float4 bm_log_entry(uint32_t m, const float4* tab, float& f, float& e) {
  const float fm = __uint2float_rn(m);                            // exact: m <= 2^24
  const int b = (int)((__float_as_uint(fm) >> 23) & 0xff) - 126;   // bit length of m, 1..25
  f = __uint_as_float((__float_as_uint(fm) & 0x807fffffu) | 0x3f800000u);   // m / 2^(b-1)
  int ei = b - 25;
  if (f > 1.41421353816986083984375f) {   // the float just below sqrt 2
    f = __fmul_rn(f, 0.5f);
    ei += 1;
  }
  e = (float)ei;
  const int j = __float2int_rn(__fmul_rn(__fsub_rn(f, 1.0f), 128.0f));   // f - 1 is exact
  return tab[kBmLog0 + (j - kBmLogLo)];                           // c, -ln c (hi, lo)
}

// ln(m 2^-24) for m in [1, 2^24], as float-floats.
__device__ __forceinline__ ffl bm_log_u(uint32_t m0, uint32_t m1, const float4* tab) {
  float2 f, e;
  const float4 L0 = bm_log_entry(m0, tab, f.x, e.x), L1 = bm_log_entry(m1, tab, f.y, e.y);
  const ffl pc = ff_two_prod(f, make_float2(L0.x, L1.x));
  const ffl t = ff_two_sum(psub(pc.h, pair(1.0f)), pc.l);               // pc.h - 1 is exact
  // ln(1 + t) = t - t^2/2 + t^3 (1/3 - t/4 + t^2/5 - t^3/6 + t^4/7)
  ffl t2 = ff_two_prod(t.h, t.h);
  t2.l = pfma(pmul(pair(2.0f), t.h), t.l, t2.l);
  float2 poly = pfma(t.h, pair(1.0f / 7.0f), pair(-1.0f / 6.0f));
  poly = pfma(t.h, poly, pair(0.2f));
  poly = pfma(t.h, poly, pair(-0.25f));
  poly = pfma(t.h, poly, pair(1.0f / 3.0f));
  const float2 cube = pmul(pmul(t.h, t2.h), poly);
  ffl l1 = ff_two_sum(t.h, pmul(pair(-0.5f), t2.h));
  l1 = ff_fast_two_sum(l1.h, padd(l1.l, padd(pfma(pair(-0.5f), t2.l, t.l), cube)));
  const float4 C = tab[kBmConst];                                  // 2 pi, ln 2
  ffl el = ff_two_prod(e, pair(C.z));
  el.l = pfma(e, pair(C.w), el.l);
  return ff_add(ff_add(el, ffl{make_float2(L0.y, L1.y), make_float2(L0.z, L1.z)}), l1);
}

// Quadrant q and octant swap of 2 pi m 2^-24; table entry of the angle in [0, pi/4] and the
// remainder 2^-24 rem.
__device__ __forceinline__ float4 bm_angle_entry(uint32_t m, const float4* tab, uint32_t& q, bool& swap, float& x) {
  m &= 0xffffffu;                          // 2^24 -> 0 (angle 2 pi)
  q = m >> 22;
  uint32_t r = m & 0x3fffffu;
  swap = r > (1u << 21);                   // second octant of the quadrant: pi/2 - phi
  if (swap) r = (1u << 22) - r;
  x = __fmul_rn(__uint2float_rn(r & 0xfffu), 5.9604644775390625e-8f);   // exact
  return tab[r >> 12];                     // cos a_j, sin a_j
}
// (cos, sin) of the first octant -> of quadrant q, one half (h or l) of one draw
__device__ __forceinline__ void bm_octant(uint32_t q, bool swap, float c, float s, float& cs, float& sn) {
  const float c1 = swap ? s : c, s1 = swap ? c : s;   // angle of the quadrant
  cs = q & 1 ? s1 : c1;
  sn = q & 1 ? c1 : s1;
  if (q == 1 || q == 2) cs = -cs;
  if (q >= 2) sn = -sn;
}

// (cos, sin)(2 pi m 2^-24) for m in [1, 2^24], as float-floats.
__device__ __forceinline__ void bm_sincos_u(uint32_t m0, uint32_t m1, const float4* tab, ffl& cs, ffl& sn) {
  uint32_t q0, q1;
  bool w0, w1;
  float2 x;
  const float4 T0 = bm_angle_entry(m0, tab, q0, w0, x.x), T1 = bm_angle_entry(m1, tab, q1, w1, x.y);
  const float4 C = tab[kBmConst];
  ffl d = ff_two_prod(pair(C.x), x);                                         // delta = 2 pi x
  d.l = pfma(pair(C.y), x, d.l);
  const float2 d2h = pmul(d.h, d.h);
  // sin delta = delta - delta^3/6 + delta^5/120
  const float2 s3 = pmul(pmul(d.h, d2h), pfma(d2h, pair(1.0f / 120.0f), pair(-1.0f / 6.0f)));
  const ffl sd = ff_fast_two_sum(d.h, padd(d.l, s3));
  // cos delta = 1 - delta^2/2 + delta^4/24
  ffl dd = ff_two_prod(d.h, d.h);
  dd.l = pfma(pmul(pair(2.0f), d.h), d.l, dd.l);
  ffl cd = ff_fast_two_sum(pair(1.0f), pmul(pair(-0.5f), dd.h));
  cd.l = padd(cd.l, pfma(pmul(dd.h, dd.h), pair(1.0f / 24.0f), pmul(pair(-0.5f), dd.l)));
  const ffl ca{make_float2(T0.x, T1.x), make_float2(T0.y, T1.y)}, sa{make_float2(T0.z, T1.z), make_float2(T0.w, T1.w)};
  const ffl sphi = ff_add(ff_mul(sa, cd), ff_mul(ca, sd));
  const ffl cphi = ff_sub(ff_mul(ca, cd), ff_mul(sa, sd));
  bm_octant(q0, w0, cphi.h.x, sphi.h.x, cs.h.x, sn.h.x);
  bm_octant(q0, w0, cphi.l.x, sphi.l.x, cs.l.x, sn.l.x);
  bm_octant(q1, w1, cphi.h.y, sphi.h.y, cs.h.y, sn.h.y);
  bm_octant(q1, w1, cphi.l.y, sphi.l.y, cs.l.y, sn.l.y);
}

// Copies the table from global to shared memory (all threads of the CTA take part; the
// caller synchronises before the first use).  The lookups of a warp hit random entries,
// which shared memory serves with far fewer transactions than the L1 cache.
__device__ __forceinline__ void bm_load_table(float4* s_tab, const float4* __restrict__ g_tab) {
  for (int i = threadIdx.x; i < kBmTableLen; i += blockDim.x) s_tab[i] = __ldg(g_tab + i);
}

// (g_even, g_odd) of the Box-Muller transforms of the Philox word pairs a and b, rounded once to
// FP32: .x, .y those of a, .z, .w those of b; tab is the table in shared (or global) memory.
__device__ __forceinline__ float4 bm_pair2(uint2 a, uint2 b, const float4* tab) {
  const ffl lu = bm_log_u((a.x >> 8) + 1u, (b.x >> 8) + 1u, tab);
  const float2 lh = pmul(pair(-2.0f), lu.h), ll = pmul(pair(-2.0f), lu.l);   // -2 ln u0 >= 0
  ffl r;
  r.h = make_float2(__fsqrt_rn(lh.x), __fsqrt_rn(lh.y));
  // 1 / (2 r), 0 where ln u0 = 0 (the radius is 0)
  const float2 q = make_float2(lh.x > 0.0f ? 0.5f * __frcp_rn(r.h.x) : 0.0f, lh.y > 0.0f ? 0.5f * __frcp_rn(r.h.y) : 0.0f);
  const ffl sq = ff_two_prod(r.h, r.h);
  r.l = pmul(padd(psub(psub(lh, sq.h), sq.l), ll), q);
  ffl cs, sn;
  bm_sincos_u((a.y >> 8) + 1u, (b.y >> 8) + 1u, tab, cs, sn);
  const ffl ge = ff_mul(r, cs), go = ff_mul(r, sn);   // ff_mul normalises: h is the rounded sum
  return make_float4(ge.h.x, go.h.x, ge.h.y, go.h.y);
}

}  // namespace lpt2
