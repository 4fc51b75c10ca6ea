// Float-pair (hi + lo) arithmetic and float-pair phasors shared by the k-space sums of the
// potential and the forces.
#pragma once

#include "cpm_internal.cuh"

namespace cpm {

// a * b for float pairs, to ~2^-44 relative (the lo * lo term dropped).
__device__ __forceinline__ void ff_mul(float ah, float al, float bh, float bl, float& ph,
                                       float& pl) {
  ph = __fmul_rn(ah, bh);  // not fused with the sums it enters
  pl = fmaf(ah, bh, -ph) + fmaf(ah, bl, al * bh);
}

// a + b for float pairs (two-sum of the high parts).
__device__ __forceinline__ void ff_add(float ah, float al, float bh, float bl, float& sh,
                                       float& sl) {
  const float s = ah + bh;
  const float bb = s - ah;
  sl = ((ah - (s - bb)) + (bh - bb)) + (al + bl);
  sh = s;
}

// exp(2 pi i ph 2^-32) as float pairs, to ~1e-13: the top 12 bits of the phase index the
// exact table, the low 20 bits give an angle t < 2 pi 2^-12 whose sine and cosine follow
// from their Taylor series (t - t^3/6, 1 - t^2/2 + t^4/24; the next terms are below
// 1e-16), and the two rotations are multiplied in float pairs.
__device__ __forceinline__ void phasor_ff(uint32_t ph, const float4* __restrict__ T, float& ch,
                                          float& cl, float& sh, float& sl) {
  const float4 t4 = __ldg(T + (ph >> 20));
  const float low = (float)(ph & 0xFFFFFu);
  constexpr float kCh = 1.462918119976564e-09f;   // 2 pi 2^-32, high part
  constexpr float kCl = -4.070940267922164e-17f;  // and the rest
  const float th = low * kCh;
  const float tl = fmaf(low, kCh, -th) + low * kCl;
  const float p = th * th;
  const float pe = fmaf(th, th, -p) + 2.0f * th * tl;
  // cos t = 1 - t^2/2 + t^4/24
  const float half = 0.5f * p;
  const float c0 = 1.0f - half;
  const float c0l = ((1.0f - c0) - half) - 0.5f * pe + p * p * (1.0f / 24.0f);
  // sin t = t - t^3/6
  const float t3 = th * p * (1.0f / 6.0f);
  const float s0 = th - t3;
  const float s0l = ((th - s0) - t3) + tl;
  // (Tc + i Ts)(c0 + i s0)
  float ah, al, bh, bl;
  ff_mul(t4.x, t4.y, c0, c0l, ah, al);
  ff_mul(t4.z, t4.w, s0, s0l, bh, bl);
  ff_add(ah, al, -bh, -bl, ch, cl);
  ff_mul(t4.z, t4.w, c0, c0l, ah, al);
  ff_mul(t4.x, t4.y, s0, s0l, bh, bl);
  ff_add(ah, al, bh, bl, sh, sl);
}

// (h, l) += x by an error-free two-sum of the high part.
__device__ __forceinline__ void pair_add1(float& h, float& l, float x) {
  const float s = h + x;
  const float bb = s - h;
  l += (h - (s - bb)) + (x - bb);
  h = s;
}

// (h, l) += x, two float pairs at once in paired IEEE instructions (a - b as fma(b, -1, a)):
// the values of pair_add1 on each component.
__device__ __forceinline__ void pair_add2(float2& h, float2& l, float2 x) {
  const float2 m1 = make_float2(-1.f, -1.f);
  const float2 s = __fadd2_rn(h, x);
  const float2 bb = __ffma2_rn(h, m1, s);                       // s - h
  const float2 a = __ffma2_rn(__ffma2_rn(bb, m1, s), m1, h);    // h - (s - bb)
  l = __fadd2_rn(l, __fadd2_rn(a, __ffma2_rn(bb, m1, x)));      // + (x - bb)
  h = s;
}

// (h, l) += a b, two float pairs at once in paired IEEE instructions: the two-sum's form with
// the product unrounded (s - h as -fma(s, -1, h)).  Good to ~2^-24 of h where h and a b cancel
// (s then holds bits below both addends' ulps), so for sums whose terms are float anyway.
__device__ __forceinline__ void pair_fma2(float2& h, float2& l, float2 a, float2 b) {
  const float2 m1 = make_float2(-1.f, -1.f);
  const float2 s = __ffma2_rn(a, b, h);
  const float2 nb = __ffma2_rn(s, m1, h);                                // h - s
  const float2 e = __ffma2_rn(__fadd2_rn(s, nb), m1, h);                 // h - (s - (s - h))
  l = __fadd2_rn(l, __fadd2_rn(e, __ffma2_rn(a, b, nb)));                // + (a b - (s - h))
  h = s;
}

// (h, l) += (ah + al) (bh + bl), two at once: the product of the high parts split exactly
// (two-product), its rounded part added by a two-sum, to ~2^-47.  na = -ah.
__device__ __forceinline__ void pair_dot2(float2& h, float2& l, float2 ah, float2 na, float2 al,
                                          float2 bh, float2 bl) {
  const float2 m1 = make_float2(-1.f, -1.f);
  const float2 n = __fmul2_rn(na, bh);                         // -p, p = ah bh rounded
  const float2 pe = __ffma2_rn(ah, bh, n);                     // ah bh - p
  const float2 s = __ffma2_rn(n, m1, h);                       // h + p
  const float2 nb = __ffma2_rn(s, m1, h);                      // h - s
  const float2 e = __ffma2_rn(__fadd2_rn(s, nb), m1, h);       // h - (s - (s - h))
  const float2 q = __fadd2_rn(e, __ffma2_rn(n, m1, nb));       // + (p - (s - h))
  l = __fadd2_rn(__ffma2_rn(ah, bl, __ffma2_rn(al, bh, l)), __fadd2_rn(q, pe));
  h = s;
}

// (h, l) += (bh, bl): two-sum of the high parts, the low parts added once.
__device__ __forceinline__ void pair_add_pair(float& h, float& l, float bh, float bl) {
  const float s = h + bh;
  const float bb = s - h;
  l = (l + bl) + ((h - (s - bb)) + (bh - bb));
  h = s;
}

// Per-axis FP64 phasors of a point: entries off[d] + j hold exp(2 pi i j s_d), s_d the
// fractional coordinate, j = 0 .. the table's largest index of axis d.  A k-vector's phasor
// is the product of three of them (conjugated for negative indices): eight FP64 operations
// to ~4e-16 instead of a sincospi.
struct AxisPhasors {
  int off[3];
  int len;  // entries a point

  __device__ __forceinline__ double2 phasor(const double2* __restrict__ row, int h, int k,
                                            int l) const {
    double2 a = __ldca(row + off[0] + abs(h)), b = __ldca(row + off[1] + abs(k)),
            c = __ldca(row + off[2] + abs(l));
    if (h < 0) a.y = -a.y;
    if (k < 0) b.y = -b.y;
    if (l < 0) c.y = -c.y;
    const double2 ab = make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
    return make_double2(ab.x * c.x - ab.y * c.y, ab.x * c.y + ab.y * c.x);
  }
};

}  // namespace cpm
