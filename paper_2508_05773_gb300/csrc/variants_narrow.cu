// variants_narrow.cu -- solve-kernel instantiations that draw their noise in
// registers and keep the rows' state in shared memory (or, where it does not
// fit there, in local memory): 1, 2, 4 or 8 lanes per sample, any number of
// rows, one sample a team.
#include "launch.h"

namespace brmppi {

const Variant* variants_narrow(int* n) {
  static const Variant v[] = {
      {1, 1, false, &solve_kernel<1, 1, false>},
      {2, 3, false, &solve_kernel<2, 3, false>},
      {4, 3, false, &solve_kernel<4, 3, false>},
      {8, 3, false, &solve_kernel<8, 3, false>},
      {1, 1, false, &solve_kernel<1, 1, false, 0, 1, true>, 0, 1, true},
      {2, 3, false, &solve_kernel<2, 3, false, 0, 1, true>, 0, 1, true},
      {4, 3, false, &solve_kernel<4, 3, false, 0, 1, true>, 0, 1, true},
      {8, 3, false, &solve_kernel<8, 3, false, 0, 1, true>, 0, 1, true},
  };
  *n = static_cast<int>(sizeof(v) / sizeof(v[0]));
  return v;
}

}  // namespace brmppi
