// variants_wide_point.cu -- the wide group (variants.h) of family kPoint.
#include "variants.h"

namespace brmppi {

const Variant* variants_wide_point(int* n) { return wide_variants<kPoint>(n); }

}  // namespace brmppi
