// trig.cuh -- the elementary functions of the rollout step, branch-free, in
// Vec<N>: sin / cos of the state angles, and the logarithm and the angle of
// Box-Muller from small tables.  A branch in the step (such as the
// large-argument path of sincosf) splits it into separate scheduling regions;
// these have none.  All but the MUFU forms build for the host too: the scalar
// forms at the end are the same code, over which the accuracy tests run.
#pragma once

#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

#include "vec.cuh"

namespace brmppi {

// ------------------------------------------------------------ state angles
// sin and cos of |e| <= pi/4: Taylor series of sin to e^9 and of cos to e^10,
// truncation below 2e-9.
template <int N>
BRMPPI_HD void turn_sincos(Vec<N> e, Vec<N>* s, Vec<N>* c) {
  using T = Vec<N>;
  const T e2 = e * e, e4 = e2 * e2;
  // sin e = e + e^3 (-1/3! + e^2/5! + e^4 (-1/7! + e^2/9!))
  *s = fma(e * e2,
           fma(e4, fma(e2, T(2.7557318844628753e-06f), T(-1.9841270113829523e-04f)),
               fma(e2, T(8.333333767950535e-03f), T(-0.1666666716337204f))),
           e);
  // cos e = 1 + e^2 (-1/2! + e^2/4! + e^4 (-1/6! + e^2/8!) - e^8/10!)
  *c = fma(e2,
           fma(e4 * e4, T(-2.755731998149713e-07f),
               fma(e4, fma(e2, T(2.4801587642286904e-05f), T(-1.3888889225199820e-03f)),
                   fma(e2, T(0.0416666679084301f), T(-0.5f)))),
           T(1.0f));
}

// sin and cos of a state angle.  Cody-Waite reduction by pi/2 (Cody and Waite,
// 1980): pi/2 split into the float nearest it and the float nearest the
// remainder; x - k hi is exact for |x| < 2^24 pi/2, so r carries one rounding;
// then turn_sincos on |r| <= pi/4 and the quadrant.  k = round(x 2/pi) by the
// shifter 1.5 * 2^23: adding it rounds the product to an integer (one rounding,
// ties to even) for |x 2/pi| < 2^22, and the sum's low mantissa bits are k mod
// 4 -- no rounding or conversion instruction on the steer angle's dependency
// chain.  Within 1.5 ulp of the exact values for |x| <= 2^16 (host test against
// FP64); up to |x| = 2^24 the outputs stay within 4e-6 of [-1, 1] (beyond 2^22
// pi/2 the shifted sum loses integer resolution and |r| reaches pi/2, where the
// Taylor pair is still within 3.6e-6); NaN for NaN or infinite x.  Beyond 2^24
// rad the outputs grow: only a rollout whose steering came within ~1e-7 rad of
// +-pi/2 gets there, and the huge or non-finite cost it then accrues carries
// zero weight in the softmin.
template <int N>
BRMPPI_HD void state_sincos(Vec<N> x, Vec<N>* s, Vec<N>* c) {
  using T = Vec<N>;
  const T t = fma(x, T(0.636619746685028f), T(12582912.0f));  // 2 / pi; 1.5 * 2^23
  const T kf = t + T(-12582912.0f);
  T r = fma(kf, T(-1.5707963705062866f), x);
  r = fma(kf, T(4.371138828673793e-08f), r);
  T sr, cr;
  turn_sincos(r, &sr, &cr);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const uint32_t q = float_bits(t.get(i));  // k mod 4 in the low bits (the shifter is 0 mod 4)
    const bool odd = q & 1u;                  // x = r + k pi/2
    const float ss = odd ? cr.get(i) : sr.get(i), cc = odd ? sr.get(i) : cr.get(i);
    s->set(i, (q & 2u) ? -ss : ss);
    c->set(i, ((q + 1u) & 2u) ? -cc : cc);
  }
}

// -------------------------------------------------- Box-Muller from tables
// Angle: the top 9 bits of the word pick the nearest of 512 directions, the
// other 14 leave |d| <= pi/512: cos and sin are the table's direction turned
// by d (sin d = d - d^3/6, cos d = 1 - d^2/2: truncation below 1e-10).  Over
// all 2^23 uniforms they are within 0.51 ulp of 1.0f (a quadrant reduction with
// turn_sincos: 0.74).  One table of cosines serves both, 128 entries (a
// quarter turn) apart.  It needs no quadrant selection.
// Logarithm: u = 2^e m with m in [0.705, 1.410), the next 7 bits pick
// 1/c and 2 ln c of a centre c of m's cell (c = 1 in the cell around 1, so
// that u near 1 keeps its relative accuracy), t = m/c - 1 in one fused
// multiply-add, |t| <= 2^-8, and 2 ln(1 + t) = t (2 + t (-1 + 2/3 t)):
// within 1.42 ulp, 3.0e-8 relative in the root mean square, over all 2^23
// uniforms (both figures: host test).
// (aligned for the 16-byte copies that stage them)
struct alignas(16) NoiseTables {
  float cosine[640];  // cos(2 pi (i + 1/2) / 512 - pi/2), so sin at i and cos at i + 128
  float rcp[128], log[128];  // 1 / c, 2 ln c
};
constexpr int kNoiseTableFloats = 896;
constexpr uint32_t kLogBase = 0x3f348000u;  // the float 0.705078125: where m's cells begin
static_assert(sizeof(NoiseTables) == 4 * kNoiseTableFloats, "tables are staged as one array");
static_assert(alignof(NoiseTables) >= 16, "tables are staged in 16-byte copies");

namespace table_math {  // compile-time series in double
constexpr double kPi = 3.14159265358979323846;
constexpr double sin_small(double x) {  // |x| <= pi/4
  double term = x, sum = x;
  for (int n = 1; n < 12; ++n) {
    term *= -x * x / ((2 * n) * (2 * n + 1));
    sum += term;
  }
  return sum;
}
constexpr double cos_small(double x) {
  double term = 1, sum = 1;
  for (int n = 1; n < 12; ++n) {
    term *= -x * x / ((2 * n - 1) * (2 * n));
    sum += term;
  }
  return sum;
}
// sin of 2 pi j / 1024 for an integer j
constexpr double sin_1024(int j) {
  j &= 1023;
  const double sign = j >= 512 ? -1.0 : 1.0;
  j &= 511;
  if (j > 256) j = 512 - j;
  const double x = kPi * j / 512.0;
  return sign * (j <= 128 ? sin_small(x) : cos_small(kPi / 2 - x));
}
constexpr double log_near_one(double c) {  // 2 atanh((c - 1) / (c + 1))
  const double s = (c - 1) / (c + 1), z = s * s;
  double p = s, sum = 0;
  for (int n = 0; n < 24; ++n) {
    sum += p / (2 * n + 1);
    p *= z;
  }
  return 2 * sum;
}
}  // namespace table_math

// The tables in device memory (one copy a translation unit, read through L2).
constexpr NoiseTables make_noise_tables() {
  NoiseTables t{};
  for (int i = 0; i < 640; ++i) t.cosine[i] = static_cast<float>(table_math::sin_1024(2 * i + 1));
  for (int i = 0; i < 128; ++i) {
    // the floats with bits kLogBase + 65536 i ..: mantissa steps of 2^-24
    // below 1 and 2^-23 above, 65536 of them a cell; the cell of 1 is i = 75
    const int bits = 0x348000 + 65536 * i + 32768;  // the cell's middle, bits above 0x3f000000
    const double c = bits < 0x800000 ? 0.5 + bits / 16777216.0 : 1.0 + (bits - 0x800000) / 8388608.0;
    const float r = i == 75 ? 1.0f : static_cast<float>(1.0 / c);
    t.rcp[i] = r;
    t.log[i] = static_cast<float>(-2.0 * table_math::log_near_one(static_cast<double>(r)));  // 2 ln(1 / r)
  }
  return t;
}

static __device__ constexpr NoiseTables kNoiseTables = make_noise_tables();

// Words wa, wb of N samples -> their two normals: u = ((w >> 9) + 1/2) 2^-23 of
// each word, r = sqrt(-2 ln u_a), (r cos, r sin)(2 pi u_b).  `tab` points to a
// NoiseTables (shared or global memory).  PARTS: 2 ln u_a and -cos, -sin of
// 2 pi u_b too, for the scalar forms below.  (In one piece: with the lookups in
// functions of their own the producer warps' schedule is 0.4% longer.)
template <int N, bool PARTS = false>
BRMPPI_HD void box_muller(const uint32_t* wa, const uint32_t* wb, const float* tab, Vec<N>& n0, Vec<N>& n1,
                          Vec<N>* parts = nullptr) {
  using T = Vec<N>;
  // the uniform from bits: 1 + (w >> 9) 2^-23 less 1 - 2^-24, exact (Sterbenz)
  T ua;
#pragma unroll
  for (int i = 0; i < N; ++i) ua.set(i, bits_float(0x3f800000u | (wa[i] >> 9)));
  ua = ua + T(-0.999999940395355224609375f);
  T m, ef, rc, lg, o, cs, sn;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const uint32_t b = float_bits(ua.get(i)), d = b - kLogBase, de = d & 0xff800000u;
    m.set(i, bits_float(b - de));
    ef.set(i, static_cast<float>(static_cast<int32_t>(de)));  // e 2^23
    const float* cell = tab + 640 + ((d >> 16) & 127u);
    rc.set(i, cell[0]);
    lg.set(i, cell[128]);
    o.set(i, bits_float(0x3f800000u | (wb[i] & 0x007ffe00u)));  // 1 + (14 bits) 2^-14
    const float* dir = tab + ((wb[i] >> 23) ^ 256u);  // the opposite direction: minus signs
    sn.set(i, dir[0]);
    cs.set(i, dir[128]);
  }
  const T t = fma(m, rc, T(-1.0f));
  const T lm = fma(t, fma(t, fma(t, T(0.666666666666666667f), T(-1.0f)), T(2.0f)), lg);  // 2 ln m
  const T q2 = fma(ef, T(1.6525916589735634e-07f), lm);                                  // 2 ln u; 2 ln 2 2^-23
  // -sqrt(-q2), -q2 in [1.2e-7, 33.3]: MUFU reciprocal square root and one
  // Newton step (0.6 ulp against 2.5)
  const T y = vrsqrt(-q2);
  T nrad = q2 * y;
  nrad = fma(T(0.5f) * y, fma(nrad, nrad, q2), nrad);
  // d = (o + 2^-15 - 3/2) 2 pi / 512
  const T dd = fma(o, T(0.01227184630308513f), T(-0.018407394947599402f));
  const T w = (T(-0.5f) * dd) * dd;  // cos d - 1
  const T sd = dd * fma(w, T(0.333333333333333333f), T(1.0f));
  // the turn's small part by itself: one rounding at the size of the result
  const T c = cs + fma(-sn, sd, cs * w);
  n0 = nrad * c;
  const T s = sn + fma(cs, sd, sn * w);
  n1 = nrad * s;
  if constexpr (PARTS) {
    parts[0] = q2;
    parts[1] = c;
    parts[2] = s;
  }
}

// ------------------------------------------------------------ scalar forms
BRMPPI_HD void turn_sincos(float e, float* s, float* c) {
  Vec<1> sv, cv;
  turn_sincos<1>(Vec<1>(e), &sv, &cv);
  *s = sv.x;
  *c = cv.x;
}
BRMPPI_HD void state_sincos(float x, float* s, float* c) {
  Vec<1> sv, cv;
  state_sincos<1>(Vec<1>(x), &sv, &cv);
  *s = sv.x;
  *c = cv.x;
}
inline const float* host_noise_tables() {
  static const NoiseTables t = make_noise_tables();
  return reinterpret_cast<const float*>(&t);
}
// -2 ln u of u = (k + 1/2) 2^-23, and sin and cos of 2 pi u; k < 2^23
inline float neg2_log_unit(float u) {
  const uint32_t w = static_cast<uint32_t>(u * 8388608.0f) << 9;
  Vec<1> n0, n1, parts[3];
  box_muller<1, true>(&w, &w, host_noise_tables(), n0, n1, parts);
  return -parts[0].x;
}
inline void unit_turn_sincos(uint32_t k, float* s, float* c) {
  const uint32_t w = k << 9;
  Vec<1> n0, n1, parts[3];
  box_muller<1, true>(&w, &w, host_noise_tables(), n0, n1, parts);
  *c = -parts[1].x;
  *s = -parts[2].x;
}

}  // namespace brmppi
