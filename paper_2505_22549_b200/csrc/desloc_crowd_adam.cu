// desloc_crowd_kernel for ADAM.
#include "desloc_crowd.cuh"

namespace desloc {

const void *lookup_crowd_adam(bool post, bool bf16, int kind, int mask, bool diag) {
    return bf16 ? lookup_crowd<OPT_ADAM, bf16_t>(post, kind, mask, diag) : lookup_crowd<OPT_ADAM, float>(post, kind, mask, diag);
}

}  // namespace desloc
