// desloc_crowd_kernel for SGDM.
#include "desloc_crowd.cuh"

namespace desloc {

const void *lookup_crowd_sgdm(bool post, bool bf16, int kind, int mask, bool diag) {
    return bf16 ? lookup_crowd<OPT_SGDM, bf16_t>(post, kind, mask, diag) : lookup_crowd<OPT_SGDM, float>(post, kind, mask, diag);
}

}  // namespace desloc
