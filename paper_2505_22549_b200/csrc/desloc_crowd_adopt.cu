// desloc_crowd_kernel for ADOPT.
#include "desloc_crowd.cuh"

namespace desloc {

const void *lookup_crowd_adopt(bool post, bool bf16, int kind, int mask, bool diag) {
    return bf16 ? lookup_crowd<OPT_ADOPT, bf16_t>(post, kind, mask, diag) : lookup_crowd<OPT_ADOPT, float>(post, kind, mask, diag);
}

}  // namespace desloc
