// variants_pair_ext.cu -- solve-kernel instantiations that roll out two samples
// a team in packed registers (Vec<2>), with the optional terms.  One lane a
// sample only: wider teams spill about 1 KB a thread in this family.
#include "launch.h"

namespace brmppi {

const Variant* variants_pair_ext(int* n) {
  static const Variant v[] = {
      {1, 1, true, &solve_kernel<1, 1, true, 0, 2>, 0, 2},
  };
  *n = static_cast<int>(sizeof(v) / sizeof(v[0]));
  return v;
}

}  // namespace brmppi
