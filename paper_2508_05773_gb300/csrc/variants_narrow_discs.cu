// variants_narrow_discs.cu -- the narrow group (variants.h) of family kDiscs.
#include "variants.h"

namespace brmppi {

const Variant* variants_narrow_discs(int* n) { return narrow_variants<kDiscs>(n); }

}  // namespace brmppi
