// variants_wide_plain.cu -- the wide group (variants.h) of family kPlain.
#include "variants.h"

namespace brmppi {

const Variant* variants_wide_plain(int* n) { return wide_variants<kPlain>(n); }

}  // namespace brmppi
