// variants_latency_moving.cu -- the latency group (variants.h) of family kMoving.
#include "variants.h"

namespace brmppi {

const Variant* variants_latency_moving(int* n) { return latency_variants<kMoving>(n); }

}  // namespace brmppi
