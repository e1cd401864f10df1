// variants_wide_moving.cu -- the wide group (variants.h) of family kMoving.
#include "variants.h"

namespace brmppi {

const Variant* variants_wide_moving(int* n) { return wide_variants<kMoving>(n); }

}  // namespace brmppi
