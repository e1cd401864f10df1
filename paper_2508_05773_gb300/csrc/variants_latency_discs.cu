// variants_latency_discs.cu -- the latency group (variants.h) of family kDiscs.
#include "variants.h"

namespace brmppi {

const Variant* variants_latency_discs(int* n) { return latency_variants<kDiscs>(n); }

}  // namespace brmppi
