// variants_latency_point.cu -- the latency group (variants.h) of family kPoint.
#include "variants.h"

namespace brmppi {

const Variant* variants_latency_point(int* n) { return latency_variants<kPoint>(n); }

}  // namespace brmppi
