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
// bits in every instantiation (lanes a sample, samples a lane).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace brmppi {

template <int N>
struct Vec;

template <>
struct Vec<1> {
  float x;
  Vec() = default;
  __device__ __forceinline__ Vec(float v) : x(v) {}
  __device__ __forceinline__ float get(int) const { return x; }
  __device__ __forceinline__ void set(int, float v) { x = v; }
};

template <>
struct Vec<2> {
  float2 x;
  Vec() = default;
  __device__ __forceinline__ Vec(float v) : x(make_float2(v, v)) {}
  __device__ __forceinline__ explicit Vec(float2 v) : x(v) {}
  __device__ __forceinline__ float get(int i) const { return i ? x.y : x.x; }
  __device__ __forceinline__ void set(int i, float v) {
    if (i) x.y = v;
    else x.x = v;
  }
};

__device__ __forceinline__ Vec<1> operator*(Vec<1> a, Vec<1> b) { return __fmul_rn(a.x, b.x); }
__device__ __forceinline__ Vec<1> operator+(Vec<1> a, Vec<1> b) { return __fadd_rn(a.x, b.x); }
__device__ __forceinline__ Vec<1> operator-(Vec<1> a, Vec<1> b) { return __fsub_rn(a.x, b.x); }
__device__ __forceinline__ Vec<1> operator-(Vec<1> a) { return -a.x; }
__device__ __forceinline__ Vec<1> fma(Vec<1> a, Vec<1> b, Vec<1> c) { return __fmaf_rn(a.x, b.x, c.x); }

__device__ __forceinline__ Vec<2> operator*(Vec<2> a, Vec<2> b) { return Vec<2>(__fmul2_rn(a.x, b.x)); }
__device__ __forceinline__ Vec<2> operator+(Vec<2> a, Vec<2> b) { return Vec<2>(__fadd2_rn(a.x, b.x)); }
__device__ __forceinline__ Vec<2> operator-(Vec<2> a) { return Vec<2>(make_float2(-a.x.x, -a.x.y)); }
__device__ __forceinline__ Vec<2> fma(Vec<2> a, Vec<2> b, Vec<2> c) { return Vec<2>(__ffma2_rn(a.x, b.x, c.x)); }
// a - b in one packed instruction: -1 b + a rounds once, as the difference does
__device__ __forceinline__ Vec<2> operator-(Vec<2> a, Vec<2> b) { return fma(b, Vec<2>(-1.f), a); }

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
__device__ __forceinline__ Vec<N> vrsqrt(Vec<N> a) {
  return vmap(a, [](float v) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
  });
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

// turn_sincos and state_sincos of trig.cuh (their derivation and accuracy
// are stated there), the same operations in the same order.
template <int N>
__device__ __forceinline__ void turn_sincos(Vec<N> e, Vec<N>* s, Vec<N>* c) {
  using T = Vec<N>;
  const T e2 = e * e, e4 = e2 * e2;
  *s = fma(e * e2,
           fma(e4, fma(e2, T(2.7557318844628753e-06f), T(-1.9841270113829523e-04f)),
               fma(e2, T(8.333333767950535e-03f), T(-0.1666666716337204f))),
           e);
  *c = fma(e2,
           fma(e4 * e4, T(-2.755731998149713e-07f),
               fma(e4, fma(e2, T(2.4801587642286904e-05f), T(-1.3888889225199820e-03f)),
                   fma(e2, T(0.0416666679084301f), T(-0.5f)))),
           T(1.0f));
}

template <int N>
__device__ __forceinline__ void state_sincos(Vec<N> x, Vec<N>* s, Vec<N>* c) {
  using T = Vec<N>;
  const T t = fma(x, T(0.636619746685028f), T(12582912.0f));
  const T kf = t + T(-12582912.0f);
  T r = fma(kf, T(-1.5707963705062866f), x);
  r = fma(kf, T(4.371138828673793e-08f), r);
  T sr, cr;
  turn_sincos(r, &sr, &cr);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const uint32_t q = __float_as_uint(t.get(i));
    const bool odd = q & 1u;
    const float ss = odd ? cr.get(i) : sr.get(i), cc = odd ? sr.get(i) : cr.get(i);
    s->set(i, (q & 2u) ? -ss : ss);
    c->set(i, ((q + 1u) & 2u) ? -cc : cc);
  }
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
