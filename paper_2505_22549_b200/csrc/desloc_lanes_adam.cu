// desloc_lanes_kernel for ADAM.
#include "desloc_lanes.cuh"

namespace desloc {

const void *lookup_lanes_adam(bool post, bool bf16, int mt, int mask) {
    return bf16 ? lookup_lanes<OPT_ADAM, bf16_t>(post, mt, mask) : lookup_lanes<OPT_ADAM, float>(post, mt, mask);
}

}  // namespace desloc
