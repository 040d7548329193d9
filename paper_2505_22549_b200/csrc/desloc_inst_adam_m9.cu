// desloc_step_kernel instantiations: ADAM, pre-average ordering, 9 to 12 workers.
#include "desloc_inst.cuh"

namespace desloc {
const void *lookup_adam_m9(bool bf16, int mt, int mask) {
    return lookup_sync<OPT_ADAM, false, false, 9, 12>(bf16, mt, mask);
}
}  // namespace desloc
