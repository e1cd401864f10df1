// variants_pair.cu -- solve-kernel instantiations that roll out two samples a
// team in packed registers (Vec<2>): the throughput shapes of batches,
// serving and large single solves.
#include "launch.h"

namespace brmppi {

const Variant* variants_pair(int* n) {
  static const Variant v[] = {
      {1, 1, false, &solve_kernel<1, 1, false, 0, 2>, 0, 2},
      {2, 3, false, &solve_kernel<2, 3, false, 0, 2>, 0, 2},
      {4, 3, false, &solve_kernel<4, 3, false, 0, 2>, 0, 2},
      {8, 3, false, &solve_kernel<8, 3, false, 0, 2>, 0, 2},
  };
  *n = static_cast<int>(sizeof(v) / sizeof(v[0]));
  return v;
}

}  // namespace brmppi
