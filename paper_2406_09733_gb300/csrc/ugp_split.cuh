// Sums of three floats (a + b + c, each at most half an ulp of the one before) for the BVH build:
// about 70 bits from FP32 arithmetic, for values that are then stored as two floats (48 bits). The
// error-free transformations are those of Dekker (1971) and Knuth (TAOCP 2, 4.2.2); products take
// their error from an fma. On this GPU an FP64 instruction takes 32 to 64 times the issue of an
// FP32 one, so the 200 of a primitive's record bounded the build.
#pragma once

#include <math.h>

namespace ugp {
namespace split {

struct t3 {
  float a, b, c;
};

// not contracted into fmas
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = add(a, b);
  const float bb = sub(s, a);
  e = add(sub(a, sub(s, bb)), sub(b, bb));
}
__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e) {
  p = mul(a, b);
  e = fmaf(a, b, -p);
}
__device__ __forceinline__ t3 renorm(float a, float b, float c) {
  float s, t, u, v, w;
  two_sum(b, c, s, t);
  two_sum(a, s, u, v);
  two_sum(v, t, w, c);
  return {u, w, c};
}
__device__ __forceinline__ t3 neg(t3 x) { return {-x.a, -x.b, -x.c}; }

// p q + r s of floats.
__device__ __forceinline__ t3 dot2(float p, float q, float r, float s) {
  float ph, pl, rh, rl, h, e, l, f, m, g;
  two_prod(p, q, ph, pl);
  two_prod(r, s, rh, rl);
  two_sum(ph, rh, h, e);
  two_sum(pl, rl, l, f);
  two_sum(e, l, m, g);
  return renorm(h, m, add(g, f));
}
__device__ __forceinline__ t3 add3(t3 x, t3 y) {
  float s, e, t, f, m, g;
  two_sum(x.a, y.a, s, e);
  two_sum(x.b, y.b, t, f);
  two_sum(e, t, m, g);
  return renorm(s, m, add(add(g, f), add(x.c, y.c)));
}
__device__ __forceinline__ t3 mulf(t3 x, float m) {
  float p, e, q, g, s, t;
  two_prod(x.a, m, p, e);
  two_prod(x.b, m, q, g);
  two_sum(e, q, s, t);
  return renorm(p, s, add(add(t, g), mul(x.c, m)));
}
__device__ __forceinline__ t3 mul3(t3 x, t3 y) {
  float p, e, q, g, h, k, s, t, u, v;
  two_prod(x.a, y.a, p, e);
  two_prod(x.a, y.b, q, g);
  two_prod(x.b, y.a, h, k);
  two_sum(q, h, s, t);
  two_sum(e, s, u, v);
  const float c = fmaf(x.a, y.c, fmaf(x.b, y.b, mul(x.c, y.a)));
  return renorm(p, u, add(add(add(t, v), add(g, k)), c));
}
// 1 / x by the series of r0 / (1 - e), e = 1 - x r0 with r0 = 1 / x.a rounded (|e| <= 2^-23).
__device__ __forceinline__ t3 recip3(t3 x) {
  const float r0 = 1.f / x.a;
  const float e0 = fmaf(-x.a, r0, 1.f);  // exact
  float q, g, E, f, p, pe;
  two_prod(-x.b, r0, q, g);
  two_sum(e0, q, E, f);
  f = add(f, fmaf(-x.c, r0, g));
  two_prod(r0, E, p, pe);
  pe = add(pe, fmaf(r0, f, mul(r0, mul(E, E))));
  return renorm(r0, p, pe);
}

// Whitening matrix W = S^-1 R^T (row r, column c: R_cr / s_r) of the quaternion (w, x, y, z), which
// need not have unit length, as hi + lo, and g0 = mag / ((2 pi)^(3/2) s_x s_y s_z). The quaternion and
// the scales enter by their mantissas (powers of two are exact), so nothing over- or underflows
// on the way.
__device__ __forceinline__ void whitening(float w, float x, float y, float z, const float s[3], float mag, float hi[9],
                                          float lo[9], float& g0) {
  int eq, em;
  frexpf(fmaxf(fmaxf(fabsf(w), fabsf(x)), fmaxf(fabsf(y), fabsf(z))), &eq);
  const float sc = ldexpf(1.f, -eq);
  w = mul(w, sc);
  x = mul(x, sc);
  y = mul(y, sc);
  z = mul(z, sc);
  const t3 wx = dot2(w, w, x, x), yz = dot2(y, y, z, z);
  const t3 n = add3(wx, yz);  // squared length
  // n R, column by column (the columns are the principal axes)
  const t3 R[9] = {add3(wx, neg(yz)), dot2(x, y, -w, z), dot2(x, z, w, y),
                   dot2(x, y, w, z), add3(dot2(w, w, -x, x), dot2(y, y, -z, z)), dot2(y, z, -w, x),
                   dot2(x, z, -w, y), dot2(y, z, w, x), add3(dot2(w, w, -x, x), dot2(z, z, -y, y))};
  float m[3];
  int es[3];
  for (int r = 0; r < 3; ++r) {
    m[r] = frexpf(s[r], &es[r]);
    const t3 f = recip3(mulf(n, m[r]));
    for (int c = 0; c < 3; ++c) {
      const t3 v = mul3(R[3 * c + r], f);
      const int e = (c == r ? 0 : 1) - es[r];  // off the diagonal n R holds twice the products
      hi[3 * r + c] = ldexpf(v.a, e);
      lo[3 * r + c] = ldexpf(add(v.b, v.c), e);
    }
  }
  // (2 pi)^(3/2) = 15.749609945722419 as three floats
  const float mm = frexpf(mag, &em);
  float p, e;
  two_prod(m[0], m[1], p, e);
  const t3 vol = mul3(mulf({p, e, 0.f}, m[2]), {0x1.f7fccep+3f, -0x1.976a8p-30f, 0.f});
  g0 = ldexpf(mulf(recip3(vol), mm).a, em - es[0] - es[1] - es[2]);
}

}  // namespace split
}  // namespace ugp
