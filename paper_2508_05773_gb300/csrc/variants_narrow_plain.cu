// variants_narrow_plain.cu -- the narrow group (variants.h) of family kPlain.
#include "variants.h"

namespace brmppi {

const Variant* variants_narrow_plain(int* n) { return narrow_variants<kPlain>(n); }

}  // namespace brmppi
