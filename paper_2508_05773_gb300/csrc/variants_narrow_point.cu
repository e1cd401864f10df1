// variants_narrow_point.cu -- the narrow group (variants.h) of family kPoint.
#include "variants.h"

namespace brmppi {

const Variant* variants_narrow_point(int* n) { return narrow_variants<kPoint>(n); }

}  // namespace brmppi
