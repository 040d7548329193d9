// desloc_lanes_kernel for ADOPT.
#include "desloc_lanes.cuh"

namespace desloc {

const void *lookup_lanes_adopt(bool post, bool bf16, int mt, int mask) {
    return bf16 ? lookup_lanes<OPT_ADOPT, bf16_t>(post, mt, mask) : lookup_lanes<OPT_ADOPT, float>(post, mt, mask);
}

}  // namespace desloc
