// vec.cuh -- binary32 values of one or two samples in one lane.
//
// Vec<1> is a float, Vec<2> the values of two samples in a register pair:
// its products, sums and fused multiply-adds are the packed instructions
// (mul / add / fma .rn.f32x2), which take one issue slot for two lanes of
// arithmetic.  They run at the scalar instructions' FMA-pipe rate (measured
// on GB300: 2.15 clocks a packed fma on one scheduler against 1.07 for a
// scalar one), so a loop whose issue slots are the limit gains, one whose
// FMA pipe is full does not.
//
// Every operation rounds by itself: a product is never fused into a sum
// unless fma() says so.  A step written in Vec<N> gives a sample the same
// bits in every instantiation (lanes a sample, samples a lane).  The
// arithmetic also builds for the host, in the same roundings (without
// contraction), so that the accuracy tests run what the kernels run.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>

namespace brmppi {

#define BRMPPI_HD __host__ __device__ __forceinline__

BRMPPI_HD uint32_t float_bits(float v) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(v);
#else
  uint32_t b;
  std::memcpy(&b, &v, sizeof(b));
  return b;
#endif
}
BRMPPI_HD float bits_float(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float v;
  std::memcpy(&v, &b, sizeof(v));
  return v;
#endif
}
BRMPPI_HD float mul_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}
BRMPPI_HD float add_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  return a + b;
#endif
}
BRMPPI_HD float sub_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fsub_rn(a, b);
#else
  return a - b;
#endif
}
BRMPPI_HD float fma_rn(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return std::fmaf(a, b, c);
#endif
}

template <int N>
struct Vec;

template <>
struct Vec<1> {
  float x;
  Vec() = default;
  BRMPPI_HD Vec(float v) : x(v) {}
  BRMPPI_HD float get(int) const { return x; }
  BRMPPI_HD void set(int, float v) { x = v; }
};

template <>
struct Vec<2> {
  float2 x;
  Vec() = default;
  BRMPPI_HD Vec(float v) : x(make_float2(v, v)) {}
  BRMPPI_HD explicit Vec(float2 v) : x(v) {}
  BRMPPI_HD float get(int i) const { return i ? x.y : x.x; }
  BRMPPI_HD void set(int i, float v) {
    if (i) x.y = v;
    else x.x = v;
  }
};

BRMPPI_HD Vec<1> operator*(Vec<1> a, Vec<1> b) { return mul_rn(a.x, b.x); }
BRMPPI_HD Vec<1> operator+(Vec<1> a, Vec<1> b) { return add_rn(a.x, b.x); }
BRMPPI_HD Vec<1> operator-(Vec<1> a, Vec<1> b) { return sub_rn(a.x, b.x); }
BRMPPI_HD Vec<1> operator-(Vec<1> a) { return -a.x; }
BRMPPI_HD Vec<1> fma(Vec<1> a, Vec<1> b, Vec<1> c) { return fma_rn(a.x, b.x, c.x); }

// (the packed forms exist from sm_100 on)
BRMPPI_HD Vec<2> operator*(Vec<2> a, Vec<2> b) {
#if defined(__CUDA_ARCH__) && __CUDA_ARCH__ >= 1000
  return Vec<2>(__fmul2_rn(a.x, b.x));
#else
  return Vec<2>(make_float2(mul_rn(a.x.x, b.x.x), mul_rn(a.x.y, b.x.y)));
#endif
}
BRMPPI_HD Vec<2> operator+(Vec<2> a, Vec<2> b) {
#if defined(__CUDA_ARCH__) && __CUDA_ARCH__ >= 1000
  return Vec<2>(__fadd2_rn(a.x, b.x));
#else
  return Vec<2>(make_float2(add_rn(a.x.x, b.x.x), add_rn(a.x.y, b.x.y)));
#endif
}
BRMPPI_HD Vec<2> operator-(Vec<2> a) { return Vec<2>(make_float2(-a.x.x, -a.x.y)); }
BRMPPI_HD Vec<2> fma(Vec<2> a, Vec<2> b, Vec<2> c) {
#if defined(__CUDA_ARCH__) && __CUDA_ARCH__ >= 1000
  return Vec<2>(__ffma2_rn(a.x, b.x, c.x));
#else
  return Vec<2>(make_float2(fma_rn(a.x.x, b.x.x, c.x.x), fma_rn(a.x.y, b.x.y, c.x.y)));
#endif
}
// a - b in one packed instruction: -1 b + a rounds once, as the difference does
BRMPPI_HD Vec<2> operator-(Vec<2> a, Vec<2> b) { return fma(b, Vec<2>(-1.f), a); }

// component by component: no packed form exists
template <int N, typename F>
__device__ __forceinline__ Vec<N> vmap(Vec<N> a, F f) {
  Vec<N> r;
#pragma unroll
  for (int i = 0; i < N; ++i) r.set(i, f(a.get(i)));
  return r;
}
template <int N, typename F>
__device__ __forceinline__ Vec<N> vmap(Vec<N> a, Vec<N> b, F f) {
  Vec<N> r;
#pragma unroll
  for (int i = 0; i < N; ++i) r.set(i, f(a.get(i), b.get(i)));
  return r;
}
template <int N>
__device__ __forceinline__ Vec<N> vclamp(Vec<N> a, float lo, float hi) {
  return vmap(a, [=](float v) { return fminf(fmaxf(v, lo), hi); });
}
// MUFU reciprocal (about 1 ulp) and reciprocal square root (about 2 ulp) of
// normal arguments: the bare instruction, without the scaling of subnormal
// ones that __fdividef and rsqrtf carry (three more instructions each)
template <int N>
__device__ __forceinline__ Vec<N> vrcp(Vec<N> a) {
  return vmap(a, [](float v) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
  });
}
template <int N>
BRMPPI_HD Vec<N> vrsqrt(Vec<N> a) {
  Vec<N> r;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float v = a.get(i);
    float q;
#ifdef __CUDA_ARCH__
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(q) : "f"(v));
#else
    q = 1.0f / std::sqrt(v);
#endif
    r.set(i, q);
  }
  return r;
}
template <int N>
__device__ __forceinline__ Vec<N> vshfl_xor(Vec<N> a, int m) {
  return vmap(a, [=](float v) { return __shfl_xor_sync(0xffffffffu, v, m); });
}

// Compensated accumulation (TwoSum): (h, l) += inc with the rounding error
// of the float sum carried in l.
template <int N>
__device__ __forceinline__ void acc2(Vec<N>& h, Vec<N>& l, Vec<N> inc) {
  const Vec<N> sum = h + inc;
  const Vec<N> bp = sum - h;
  l = l + ((h - (sum - bp)) + (inc - bp));
  h = sum;
}

// into [-pi, pi]; only the square of the result is used.  The turn count is
// rounded by the 1.5 * 2^23 shifter (as rintf for |a| < 2^22 2 pi)
template <int N>
__device__ __forceinline__ Vec<N> wrap_pi(Vec<N> a) {
  using T = Vec<N>;
  const T n = fma(a, T(0.15915494309189533577f), T(12582912.0f)) + T(-12582912.0f);
  return fma(n, T(-6.28318530717958647692f), a);
}

}  // namespace brmppi
