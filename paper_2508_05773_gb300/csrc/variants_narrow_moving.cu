// variants_narrow_moving.cu -- the narrow group (variants.h) of family kMoving.
#include "variants.h"

namespace brmppi {

const Variant* variants_narrow_moving(int* n) { return narrow_variants<kMoving>(n); }

}  // namespace brmppi
