// noise.cuh -- the noise of the rollouts: Philox4x32-10 blocks with their
// first rounds shared; their words become normals by box_muller (trig.cuh).
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

#include "trig.cuh"
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

}  // namespace brmppi
