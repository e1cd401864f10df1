// variants.h -- the solve-kernel instantiations of a family, one table a group;
// each (group, family) is a translation unit of its own (compiled in
// parallel).  Every family holds the same (tps, bpt) pairs of one sample a
// team.
#pragma once

#include "launch.h"

namespace brmppi {

template <int N>
const Variant* table(const Variant (&v)[N], int* n) {
  *n = N;
  return v;
}

// Noise drawn in registers: 1, 2, 4 or 8 lanes per sample, any number of
// rows, their state in shared memory or, where it does not fit there, in
// local memory; and two samples a team in packed registers (the throughput
// shapes of batches, serving and large single solves; with a steer-rate
// column one lane a sample only: wider teams spill about 1 KB a thread).
template <int F>
const Variant* narrow_variants(int* n) {
  if constexpr (F == kPlain || F == kMoving) {
    static const Variant v[] = {
        {1, 1, F, &solve_kernel<1, 1, F>},
        {2, 3, F, &solve_kernel<2, 3, F>},
        {4, 3, F, &solve_kernel<4, 3, F>},
        {8, 3, F, &solve_kernel<8, 3, F>},
        {1, 1, F, &solve_kernel<1, 1, F, 0, 1, true>, 0, 1, true},
        {2, 3, F, &solve_kernel<2, 3, F, 0, 1, true>, 0, 1, true},
        {4, 3, F, &solve_kernel<4, 3, F, 0, 1, true>, 0, 1, true},
        {8, 3, F, &solve_kernel<8, 3, F, 0, 1, true>, 0, 1, true},
        {1, 1, F, &solve_kernel<1, 1, F, 0, 2>, 0, 2},
        {2, 3, F, &solve_kernel<2, 3, F, 0, 2>, 0, 2},
        {4, 3, F, &solve_kernel<4, 3, F, 0, 2>, 0, 2},
        {8, 3, F, &solve_kernel<8, 3, F, 0, 2>, 0, 2},
    };
    return table(v, n);
  } else {
    static const Variant v[] = {
        {1, 1, F, &solve_kernel<1, 1, F>},
        {2, 3, F, &solve_kernel<2, 3, F>},
        {4, 3, F, &solve_kernel<4, 3, F>},
        {8, 3, F, &solve_kernel<8, 3, F>},
        {1, 1, F, &solve_kernel<1, 1, F, 0, 1, true>, 0, 1, true},
        {2, 3, F, &solve_kernel<2, 3, F, 0, 1, true>, 0, 1, true},
        {4, 3, F, &solve_kernel<4, 3, F, 0, 1, true>, 0, 1, true},
        {8, 3, F, &solve_kernel<8, 3, F, 0, 1, true>, 0, 1, true},
        {1, 1, F, &solve_kernel<1, 1, F, 0, 2>, 0, 2},
    };
    return table(v, n);
  }
}

// Noise from producer warps, up to two Philox blocks of rows a lane: the
// latency shapes.
template <int F>
const Variant* wide_variants(int* n) {
  static const Variant v[] = {
      {2, 1, F, &solve_kernel<2, 1, F>},   {2, 2, F, &solve_kernel<2, 2, F>},   {4, 1, F, &solve_kernel<4, 1, F>},
      {4, 2, F, &solve_kernel<4, 2, F>},   {8, 1, F, &solve_kernel<8, 1, F>},   {8, 2, F, &solve_kernel<8, 2, F>},
      {16, 1, F, &solve_kernel<16, 1, F>}, {16, 2, F, &solve_kernel<16, 2, F>}, {32, 1, F, &solve_kernel<32, 1, F>},
  };
  return table(v, n);
}

// Single solves on the latency shapes with an exact number of rows a lane (1
// to 4): the step runs without a branch on the row count.
template <int F>
const Variant* latency_variants(int* n) {
  if constexpr (F == kPlain || F == kMoving) {
    static const Variant v[] = {
        {2, 1, F, &solve_kernel<2, 1, F, 1>, 1}, {2, 1, F, &solve_kernel<2, 1, F, 2>, 2},
        {2, 1, F, &solve_kernel<2, 1, F, 3>, 3}, {2, 1, F, &solve_kernel<2, 1, F, 4>, 4},
        {4, 1, F, &solve_kernel<4, 1, F, 1>, 1}, {4, 1, F, &solve_kernel<4, 1, F, 2>, 2},
        {4, 1, F, &solve_kernel<4, 1, F, 3>, 3}, {4, 1, F, &solve_kernel<4, 1, F, 4>, 4},
        {8, 1, F, &solve_kernel<8, 1, F, 1>, 1}, {8, 1, F, &solve_kernel<8, 1, F, 2>, 2},
        {8, 1, F, &solve_kernel<8, 1, F, 3>, 3}, {8, 1, F, &solve_kernel<8, 1, F, 4>, 4},
    };
    return table(v, n);
  } else {
    static const Variant v[] = {
        {4, 1, F, &solve_kernel<4, 1, F, 1>, 1},
        {4, 1, F, &solve_kernel<4, 1, F, 2>, 2},
        {4, 1, F, &solve_kernel<4, 1, F, 3>, 3},
        {4, 1, F, &solve_kernel<4, 1, F, 4>, 4},
    };
    return table(v, n);
  }
}

}  // namespace brmppi
