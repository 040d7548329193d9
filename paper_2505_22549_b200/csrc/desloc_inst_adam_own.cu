// Adam kernels for gradients that the copy engine cannot take, see desloc_inst.cuh.
#include "desloc_inst.cuh"

namespace desloc {
const void *lookup_adam_own(bool post, bool bf16, int mt, int mask) {
    return bf16 ? lookup_own<OPT_ADAM, bf16_t>(post, mt, mask) : lookup_own<OPT_ADAM, float>(post, mt, mask);
}
}  // namespace desloc
