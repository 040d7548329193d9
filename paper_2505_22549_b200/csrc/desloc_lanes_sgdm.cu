// desloc_lanes_kernel for SGDM.
#include "desloc_lanes.cuh"

namespace desloc {

const void *lookup_lanes_sgdm(bool post, bool bf16, int mt, int mask) {
    return bf16 ? lookup_lanes<OPT_SGDM, bf16_t>(post, mt, mask) : lookup_lanes<OPT_SGDM, float>(post, mt, mask);
}

}  // namespace desloc
