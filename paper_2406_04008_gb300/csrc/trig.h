// The rotation-scale matrix of an element: s res (+-sin z or cos z) as float pairs (hi + lo).
//
// FP64 runs at 1/64 of the FP32 rate on this part.  The library's sine and cosine of one element were a
// dependent chain of about a hundred such instructions (2 us of the transform's 12 at 1000 elements, most of
// its 100 at 26 k), and even a table with eight of them cost 0.5 us of an iteration.  So an entry is formed in
// error-free float arithmetic with three floats where FP64 has 53 bits, and rounded once to the pair: its
// error is half a unit of lo, as that of an FP64 value split into a pair.
#pragma once
#include <cmath>

#include "arith.h"
#include "internal.h"

namespace collage {

// |z| <= kTrigMax: z = k step + x with the step 2 pi / 4096 in three floats (Cody & Waite 1980), then
// sin(k + x) = S cos x + C sin x with the tabled S, C of k (three floats each, one quadrant of them),
// sin x = x - x^3/6 + x^5/120 and cos x - 1 = -x^2/2 + x^4/24, |x| <= 0.001.
constexpr float kTrigMax = 8192.0f;
constexpr int kTrigQuarter = kTrigSteps / 4;
constexpr double kTrigStep = 6.283185307179586 / kTrigSteps;
constexpr double kTrigStepLow = 2.4492935982947064e-16 / kTrigSteps;  // ... beyond a double
constexpr float kTrigC1 = (float)kTrigStep;
constexpr float kTrigC2 = (float)(kTrigStep - (double)kTrigC1);
constexpr float kTrigC3 = (float)(kTrigStep - (double)kTrigC1 - (double)kTrigC2 + kTrigStepLow);

// Sine of i steps.
__device__ __forceinline__ float4 trig_sine(int i, const float4* table) {
  const int r = i & (kTrigQuarter - 1);
  float4 t = table[i & kTrigQuarter ? kTrigQuarter - r : r];
  if (i & (2 * kTrigQuarter)) t = make_float4(-t.x, -t.y, -t.z, 0.0f);
  return t;
}

// a b (sin z, or cos z) as m[0] + m[1].
__device__ __forceinline__ void trig_entry(float z, bool cosine, float a, float b, const float4* table, float (&m)[2]) {
  const float k = rintf(__fmul_rn(z, 1.0f / kTrigC1));
  const int i = (int)k + (cosine ? kTrigQuarter : 0);
  const float4 S = trig_sine(i, table), C = trig_sine(i + kTrigQuarter, table);
  // x = xh + xl, to 2^-58
  float e, q, u0, u1;
  const float p = two_prod(k, kTrigC1, e), u = two_prod(k, kTrigC2, q);
  const float a1 = two_sum(__fsub_rn(z, p), -e, u0);  // z - p is exact: p is within a factor 2 of z
  const float a2 = two_sum(a1, -u, u1);
  float xl;
  const float xh = fast_two_sum(a2, __fsub_rn(__fadd_rn(u0, u1), __fmaf_rn(k, kTrigC3, q)), xl);
  // sin x = xh + sl, cos x - 1 = ch + cl
  float yl;
  const float y = two_prod(xh, xh, yl);
  yl = __fmaf_rn(2.0f * xh, xl, yl);
  const float sl = __fmaf_rn(__fmul_rn(xh, y), __fmaf_rn(y, 1.0f / 120.0f, -1.0f / 6.0f), xl);
  const float ch = -0.5f * y, cl = __fmaf_rn(__fmul_rn(y, y), 1.0f / 24.0f, -0.5f * yl);
  // S + C sin x + S (cos x - 1) = t0 + t1 + t2, to 2^-55
  float e1, e2, f1, f2, g1, g2, t2;
  const float p1 = two_prod(C.x, xh, e1), p2 = two_prod(S.x, ch, e2);
  const float low = __fadd_rn(__fadd_rn(e1, e2), __fmaf_rn(C.x, sl, __fmaf_rn(C.y, xh, __fmaf_rn(S.x, cl, __fmul_rn(S.y, ch)))));
  const float t0 = two_sum(two_sum(S.x, p1, f1), p2, f2);
  const float r = two_sum(two_sum(f1, f2, g1), S.y, g2);
  const float t1 = two_sum(r, __fadd_rn(__fadd_rn(g1, g2), __fadd_rn(S.z, low)), t2);
  // times a b
  float hl, pl, q1l, q2l, h1, h2, lo;
  const float h = two_prod(a, b, hl), pp = two_prod(h, t0, pl);
  const float q1 = two_prod(h, t1, q1l), q2 = two_prod(hl, t0, q2l);
  const float tail = two_sum(two_sum(pl, q1, h1), q2, h2);
  m[0] = fast_two_sum(pp, tail, lo);
  m[1] = __fadd_rn(lo, __fadd_rn(__fadd_rn(h1, h2), __fadd_rn(__fadd_rn(q1l, q2l), __fmaf_rn(h, t2, __fmul_rn(hl, t1)))));
}

static __device__ __noinline__ void trig_wide(float z, bool cosine, float a, float b, float (&m)[2]) {  // any other angle
  const double v = (double)a * (double)b * (cosine ? cos((double)z) : sin((double)z));
  m[0] = (float)v;
  m[1] = (float)(v - (double)m[0]);
}

// The table: sines of 0 to a quarter turn, each as the sum of three floats.
inline void trig_table(float4* t) {
  for (int k = 0; k <= kTrigQuarter; ++k) {
    const double s = 2 * k <= kTrigQuarter ? sin(k * kTrigStep) : cos((kTrigQuarter - k) * kTrigStep);
    const float h = (float)s, m = (float)(s - (double)h);
    t[k] = make_float4(h, m, (float)(s - (double)h - (double)m), 0.0f);
  }
}

}  // namespace collage
