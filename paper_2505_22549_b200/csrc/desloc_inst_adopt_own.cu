// ADOPT kernels for gradients that the copy engine cannot take, see desloc_inst.cuh.
#include "desloc_inst.cuh"

namespace desloc {
const void *lookup_adopt_own(bool post, bool bf16, int mt, int mask) {
    return bf16 ? lookup_own<OPT_ADOPT, bf16_t>(post, mt, mask) : lookup_own<OPT_ADOPT, float>(post, mt, mask);
}
}  // namespace desloc
