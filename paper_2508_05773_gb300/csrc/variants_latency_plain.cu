// variants_latency_plain.cu -- the latency group (variants.h) of family kPlain.
#include "variants.h"

namespace brmppi {

const Variant* variants_latency_plain(int* n) { return latency_variants<kPlain>(n); }

}  // namespace brmppi
