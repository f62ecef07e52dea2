// rbc_stencil.cuh -- the leapfrog update of Eq. 1 for four consecutive nodes,
// in packed fp32x2 arithmetic (sm_100 family FADD2/FMUL2/FFMA2: two lanes of
// fp32 per instruction, each correctly rounded, so the results equal those of
// the scalar sequence).
//
//   out = (2 p - p_old) + a * sum_k c_k s_k,
//   s_k = sum over the axes of [(p_{-k} - p) + (p_{+k} - p)]   (k = 1..4)
//
// The weights c1..c4 are those of rbc_internal.cuh; summing differences from
// the centre makes the fp32 rounding relative to the second differences
// instead of |p|, because c0 = -2 (c1 + c2 + c3 + c4) cancels exactly.
#pragma once

#include "rbc_internal.cuh"

namespace rbc {

__device__ __forceinline__ float2 lo2(const float4 &v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(const float4 &v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float2 half2of(const float4 &v, int j) { return j ? hi2(v) : lo2(v); }
__device__ __forceinline__ float2 neg2(const float2 v) { return make_float2(-v.x, -v.y); }
__device__ __forceinline__ float2 sum_diff2(const float2 m, const float2 p, const float2 np) {
  return __fadd2_rn(__fadd2_rn(m, np), __fadd2_rn(p, np));
}

// w[0..11]: x window x0-4 .. x0+7 (centre at w[4..7]); zq[0..8]: z window
// (zq[4] = centre).
__device__ __forceinline__ float4 leap4p(const float *w, const float4 *zq, const float4 po, const float4 av) {
  float2 out[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const float2 p = make_float2(w[4 + 2 * j], w[5 + 2 * j]);
    const float2 np = neg2(p);
    float2 s[5];
#pragma unroll
    for (int k = 1; k <= 4; ++k) {
      const float2 xm = make_float2(w[4 + 2 * j - k], w[5 + 2 * j - k]);
      const float2 xp = make_float2(w[4 + 2 * j + k], w[5 + 2 * j + k]);
      float2 t = sum_diff2(xm, xp, np);
      t = __fadd2_rn(t, sum_diff2(half2of(zq[4 - k], j), half2of(zq[4 + k], j), np));
      s[k] = t;
    }
    float2 lap = __fmul2_rn(make_float2(kC4, kC4), s[4]);
    lap = __ffma2_rn(make_float2(kC3, kC3), s[3], lap);
    lap = __ffma2_rn(make_float2(kC2, kC2), s[2], lap);
    lap = __ffma2_rn(make_float2(kC1, kC1), s[1], lap);
    const float2 base = __fadd2_rn(__fadd2_rn(p, p), neg2(half2of(po, j)));
    out[j] = __ffma2_rn(half2of(av, j), lap, base);
  }
  return make_float4(out[0].x, out[0].y, out[1].x, out[1].y);
}

// Same update split as out = base + inc, inc = a * lap (the discrete second
// time difference p^{n+1} - 2 p^n + p^{n-1} without the point terms), for
// callers that need the increment itself (the FWI gradient).
__device__ __forceinline__ float4 leap4p_inc(const float *w, const float4 *zq, const float4 po, const float4 av,
                                             float4 *inc) {
  float2 out[2], dd[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const float2 p = make_float2(w[4 + 2 * j], w[5 + 2 * j]);
    const float2 np = neg2(p);
    float2 s[5];
#pragma unroll
    for (int k = 1; k <= 4; ++k) {
      const float2 xm = make_float2(w[4 + 2 * j - k], w[5 + 2 * j - k]);
      const float2 xp = make_float2(w[4 + 2 * j + k], w[5 + 2 * j + k]);
      float2 t = sum_diff2(xm, xp, np);
      t = __fadd2_rn(t, sum_diff2(half2of(zq[4 - k], j), half2of(zq[4 + k], j), np));
      s[k] = t;
    }
    float2 lap = __fmul2_rn(make_float2(kC4, kC4), s[4]);
    lap = __ffma2_rn(make_float2(kC3, kC3), s[3], lap);
    lap = __ffma2_rn(make_float2(kC2, kC2), s[2], lap);
    lap = __ffma2_rn(make_float2(kC1, kC1), s[1], lap);
    const float2 base = __fadd2_rn(__fadd2_rn(p, p), neg2(half2of(po, j)));
    dd[j] = __fmul2_rn(half2of(av, j), lap);
    out[j] = __fadd2_rn(base, dd[j]);
  }
  *inc = make_float4(dd[0].x, dd[0].y, dd[1].x, dd[1].y);
  return make_float4(out[0].x, out[0].y, out[1].x, out[1].y);
}

// ---- the update with shared differences (resident 2-D loops, 3-D steps) ----
// The same roundings as leap4p, bit for bit, with fewer operations: with
// D_k[i] = p_{i+k} - p_i, the term (p_{-k} - p) + (p_{+k} - p) is D_k[i] -
// D_k[i-k] (rounding is symmetric in the sign), and every D_k serves two
// nodes: along x within the float4, along z by a march down the rows.  59
// packed operations per float4 against 70.
// a - b as one packed operation (b * -1 is exact: one rounding)
__device__ __forceinline__ float2 sub2(const float2 a, const float2 b) {
  return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
}
__device__ __forceinline__ float4 sub4(const float4 a, const float4 b) {
  const float2 l = sub2(lo2(a), lo2(b)), h = sub2(hi2(a), hi2(b));
  return make_float4(l.x, l.y, h.x, h.y);
}

// h^2 Laplacian at four consecutive nodes: x window (lf, c, rt); z[k-1] =
// D_k[row] - D_k[row - k] (3-D: y[k-1] along the third axis).
template <bool kThreeD = false>
__device__ __forceinline__ float4 lap_shared(const float4 lf, const float4 c, const float4 rt, const float4 *z,
                                             const float4 *y = nullptr) {
  const float w[12] = {lf.x, lf.y, lf.z, lf.w, c.x, c.y, c.z, c.w, rt.x, rt.y, rt.z, rt.w};
  float d1[5], d3[7];
  float2 d2[3], d4[4];
#pragma unroll
  for (int i = 0; i < 5; ++i) d1[i] = w[i + 4] - w[i + 3];
#pragma unroll
  for (int i = 0; i < 7; ++i) d3[i] = w[i + 4] - w[i + 1];
#pragma unroll
  for (int i = 0; i < 3; ++i)
    d2[i] = sub2(make_float2(w[2 * i + 4], w[2 * i + 5]), make_float2(w[2 * i + 2], w[2 * i + 3]));
#pragma unroll
  for (int i = 0; i < 4; ++i) d4[i] = sub2(make_float2(w[2 * i + 4], w[2 * i + 5]), make_float2(w[2 * i], w[2 * i + 1]));
  float2 out[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    float2 s[4];
    s[0] = make_float2(d1[2 * j + 1] - d1[2 * j], d1[2 * j + 2] - d1[2 * j + 1]);
    s[1] = sub2(d2[j + 1], d2[j]);
    s[2] = make_float2(d3[2 * j + 3] - d3[2 * j], d3[2 * j + 4] - d3[2 * j + 1]);
    s[3] = sub2(d4[j + 2], d4[j]);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      s[k] = __fadd2_rn(s[k], half2of(z[k], j));
      if (kThreeD) s[k] = __fadd2_rn(s[k], half2of(y[k], j));
    }
    float2 lap = __fmul2_rn(make_float2(kC4, kC4), s[3]);
    lap = __ffma2_rn(make_float2(kC3, kC3), s[2], lap);
    lap = __ffma2_rn(make_float2(kC2, kC2), s[1], lap);
    out[j] = __ffma2_rn(make_float2(kC1, kC1), s[0], lap);
  }
  return make_float4(out[0].x, out[0].y, out[1].x, out[1].y);
}

// (m - p) + (q - p) for the neighbours m, q of p on either side
__device__ __forceinline__ float4 pair_diff(const float4 m, const float4 p, const float4 q) {
  return sub4(sub4(q, p), sub4(p, m));
}

// (2 p - p_old) + a lap; *inc (kInc) = a lap, rounded by itself as in leap4p_inc.
template <bool kInc>
__device__ __forceinline__ float4 leap_fin(const float4 c, const float4 po, const float4 av, const float4 lap,
                                           float4 *inc) {
  const float2 bl = sub2(__fadd2_rn(lo2(c), lo2(c)), lo2(po)), bh = sub2(__fadd2_rn(hi2(c), hi2(c)), hi2(po));
  float2 l, h;
  if (kInc) {
    l = __fmul2_rn(lo2(av), lo2(lap));
    h = __fmul2_rn(hi2(av), hi2(lap));
    *inc = make_float4(l.x, l.y, h.x, h.y);
    l = __fadd2_rn(bl, l);
    h = __fadd2_rn(bh, h);
  } else {
    l = __ffma2_rn(lo2(av), lo2(lap), bl);
    h = __ffma2_rn(hi2(av), hi2(lap), bh);
  }
  return make_float4(l.x, l.y, h.x, h.y);
}

} // namespace rbc
