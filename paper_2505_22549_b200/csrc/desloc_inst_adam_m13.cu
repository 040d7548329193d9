// desloc_step_kernel instantiations: ADAM, pre-average ordering, 13 to 16 workers.
#include "desloc_inst.cuh"

namespace desloc {
const void *lookup_adam_m13(bool bf16, int mt, int mask) {
    return lookup_sync<OPT_ADAM, false, false, 13, 16>(bf16, mt, mask);
}
}  // namespace desloc
