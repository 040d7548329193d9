// desloc_crowd_kernel for ADOPT.
#include "desloc_crowd.cuh"

namespace desloc {

const void *lookup_crowd_adopt(bool post, bool bf16, int kind, int mask) {
    return bf16 ? lookup_crowd<OPT_ADOPT, bf16_t>(post, kind, mask) : lookup_crowd<OPT_ADOPT, float>(post, kind, mask);
}

}  // namespace desloc
