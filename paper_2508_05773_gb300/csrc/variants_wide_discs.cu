// variants_wide_discs.cu -- the wide group (variants.h) of family kDiscs.
#include "variants.h"

namespace brmppi {

const Variant* variants_wide_discs(int* n) { return wide_variants<kDiscs>(n); }

}  // namespace brmppi
