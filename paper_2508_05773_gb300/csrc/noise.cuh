// noise.cuh -- the noise of the rollouts: Philox4x32-10 blocks with their
// first rounds shared, and Box-Muller from small tables.
//
// What bounds it.  A Philox block is 20 multiplies of 32 x 32 to 64 bits, and
// IMAD.WIDE holds the FMA pipe for 4.25 clocks of a scheduler (measured on
// GB300; an FFMA 1.07), so a block costs as much FMA time as 80 FFMAs.  Its
// four normals took 64 more FP32 operations with polynomial logarithms and
// angles.  Both are cut here without changing a Philox word: 16 multiplies a
// block, and 48 FP32 operations and 2 MUFU for the four normals.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "vec.cuh"

namespace brmppi {

// ------------------------------------------------------------------ Philox
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): counter (b, tau, s, ctr),
// key (k0, k1); a round maps (x, y, z, w) to
//   (hi(M1 z) ^ y ^ k0, lo(M1 z), hi(M0 x) ^ w ^ k1, lo(M0 x))
// and the keys advance by the Weyl increments between rounds.  Over a solve
// most of the first three rounds repeat:
//   round 1: M0 b belongs to the block, M1 s to the sample;
//   round 2: M0 x with x = hi(M1 s) ^ tau ^ k0 to (sample, step), shared by
//            the step's blocks; M1 z with z = hi(M0 b) ^ ctr ^ k1 to the block;
//   round 3: M1 z needs all of (block, sample, step), M0 x the block and
//            the sample.
// So a block costs two multiplies of round 3 and 14 of rounds 4 to 10, and a
// (sample, step) one more.
constexpr uint32_t kPhiloxM0 = 0xD2511F53u, kPhiloxM1 = 0xCD9E8D57u;
constexpr uint32_t kPhiloxW0 = 0x9E3779B9u, kPhiloxW1 = 0xBB67AE85u;

// Both halves of a product in one IMAD.WIDE (apart, the compiler may take an
// IMAD and an IMAD.HI, two instructions for the same pipe).
__device__ __forceinline__ uint2 mul_wide(uint32_t a, uint32_t b) {
  uint2 r;
  asm("{.reg .u64 p; mul.wide.u32 p, %2, %3; mov.b64 {%0, %1}, p;}" : "=r"(r.x), "=r"(r.y) : "r"(a), "r"(b));
  return r;  // lo, hi
}

// Of block b (for one key and counter): hi(M1 z) ^ k0 of round 2, lo(M1 z) ^
// k0 of round 3, lo(M0 b) ^ k1 of round 2.
struct PhiloxBlock {
  uint32_t a, b, c, unused;
};
__device__ __forceinline__ PhiloxBlock philox_block(uint32_t b, uint32_t ctr, uint32_t k0, uint32_t k1) {
  const uint2 p = mul_wide(kPhiloxM0, b), q = mul_wide(kPhiloxM1, p.y ^ ctr ^ k1);
  return {q.y ^ (k0 + kPhiloxW0), q.x ^ (k0 + 2u * kPhiloxW0), p.x ^ (k1 + kPhiloxW1), 0u};
}
// Of sample s: M1 s.
struct PhiloxSample {
  uint32_t lo, hi;
};
__device__ __forceinline__ PhiloxSample philox_sample(uint32_t s) {
  const uint2 p = mul_wide(kPhiloxM1, s);
  return {p.x, p.y};
}
// Of sample s at step tau: hi and lo (^ k1 of round 3) of M0 x of round 2.
struct PhiloxStep {
  uint32_t hi, lo;
};
__device__ __forceinline__ PhiloxStep philox_step(PhiloxSample s, uint32_t tau, uint32_t k0, uint32_t k1) {
  const uint2 p = mul_wide(kPhiloxM0, s.hi ^ tau ^ k0);
  return {p.y, p.x ^ (k1 + 2u * kPhiloxW1)};
}
// The four words of block `b` of a sample at a step.
__device__ __forceinline__ uint4 philox_words(PhiloxBlock b, PhiloxSample s, PhiloxStep st, uint32_t k0, uint32_t k1) {
  const uint2 p2 = mul_wide(kPhiloxM0, b.a ^ s.lo), q2 = mul_wide(kPhiloxM1, st.hi ^ b.c);
  uint4 c = make_uint4(q2.y ^ b.b, q2.x, p2.y ^ st.lo, p2.x);
  k0 += 3u * kPhiloxW0;
  k1 += 3u * kPhiloxW1;
#pragma unroll
  for (int r = 3; r < 10; ++r) {
    const uint2 p = mul_wide(kPhiloxM0, c.x), q = mul_wide(kPhiloxM1, c.z);
    c = make_uint4(q.y ^ c.y ^ k0, q.x, p.y ^ c.w ^ k1, p.x);
    k0 += kPhiloxW0;
    k1 += kPhiloxW1;
  }
  return c;
}

// -------------------------------------------------------------- Box-Muller
// Two words -> two standard normals: u = ((w >> 9) + 1/2) 2^-23 of each word,
// r = sqrt(-2 ln u_a), (r cos, r sin)(2 pi u_b).
//
// Angle: the top 9 bits of the word pick the nearest of 512 directions, the
// other 14 leave |d| <= pi/512: cos and sin are the table's direction turned
// by d (sin d = d - d^3/6, cos d = 1 - d^2/2: truncation below 1e-10).  Over
// all 2^23 uniforms they are within 0.51 ulp of 1.0f (the polynomial pair of
// unit_turn_sincos: 0.74).  One
// table of cosines serves both, 128 entries (a quarter turn) apart.  It needs
// no quadrant selection.
// Logarithm: u = 2^e m with m in [0.705, 1.410), the next 7 bits pick
// 1/c and 2 ln c of a centre c of m's cell (c = 1 in the cell around 1, so
// that u near 1 keeps its relative accuracy), t = m/c - 1 in one fused
// multiply-add, |t| <= 2^-8, and 2 ln(1 + t) = t (2 + t (-1 + 2/3 t)):
// within 1.42 ulp, 3.0e-8 relative in the root mean square, over all 2^23
// uniforms (neg2_log_unit with an exact division: 2.5 ulp, 4.1e-8).
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

// Words wa, wb of N samples -> their two normals; `tab` points to a
// NoiseTables (shared or global memory).
template <int N>
__device__ __forceinline__ void box_muller(const uint32_t* wa, const uint32_t* wb, const float* tab, Vec<N>& n0,
                                           Vec<N>& n1) {
  using T = Vec<N>;
  // the uniform from bits: 1 + (w >> 9) 2^-23 less 1 - 2^-24, exact (Sterbenz)
  T ua;
#pragma unroll
  for (int i = 0; i < N; ++i) ua.set(i, __uint_as_float(0x3f800000u | (wa[i] >> 9)));
  ua = ua + T(-0.999999940395355224609375f);
  T m, ef, rc, lg, o, cs, sn;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const uint32_t b = __float_as_uint(ua.get(i)), d = b - kLogBase, de = d & 0xff800000u;
    m.set(i, __uint_as_float(b - de));
    ef.set(i, static_cast<float>(static_cast<int32_t>(de)));  // e 2^23
    const float* cell = tab + 640 + ((d >> 16) & 127u);
    rc.set(i, cell[0]);
    lg.set(i, cell[128]);
    o.set(i, __uint_as_float(0x3f800000u | (wb[i] & 0x007ffe00u)));  // 1 + (14 bits) 2^-14
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
  n0 = nrad * (cs + fma(-sn, sd, cs * w));
  n1 = nrad * (sn + fma(cs, sd, sn * w));
}

}  // namespace brmppi
