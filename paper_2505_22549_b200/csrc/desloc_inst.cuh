// Instantiation tables for desloc_step_kernel.  Each optimizer x averaging order x (with or
// without norm diagnostics) is its own translation unit (they compile in parallel); this header
// builds the (MT, mask) -> kernel table for one of them.
#pragma once
#include <utility>

#include "desloc_kernels.cuh"

namespace desloc {

template <int OPT, bool POST, bool DIAG, typename GT, int MT, int MASK>
const void *kernel_ptr() {
    return reinterpret_cast<const void *>(&desloc_step_kernel<OPT, MASK, MT, GT, POST, DIAG>);
}

// Masks 1..NMASK for every MT in MT0..MT1.  NMASK = 7 for Adam / ADOPT, 3 for SGDM (no second
// state).  Mask 0, the local step, is the one-replica kernel whatever the worker count.
template <int OPT, bool POST, bool DIAG, typename GT, int NMASK, int MT0, int MT1, int... I>
const void *pick_sync(int mt, int mask, std::integer_sequence<int, I...>) {
    static const void *const tbl[] = {
        kernel_ptr<OPT, POST, DIAG, GT, MT0 + I / NMASK, 1 + I % NMASK>()...};
    if (mt < MT0 || mt > MT1 || mask < 1 || mask > NMASK) return nullptr;
    return tbl[(mt - MT0) * NMASK + (mask - 1)];
}

template <int OPT, bool POST, bool DIAG, int MT0 = 2, int MT1 = MAX_MT>
const void *lookup_sync(bool bf16, int mt, int mask) {
    constexpr int NMASK = (OPT == OPT_SGDM) ? 3 : 7;
    using Seq = std::make_integer_sequence<int, (MT1 - MT0 + 1) * NMASK>;
    return bf16 ? pick_sync<OPT, POST, DIAG, bf16_t, NMASK, MT0, MT1>(mt, mask, Seq{})
                : pick_sync<OPT, POST, DIAG, float, NMASK, MT0, MT1>(mt, mask, Seq{});
}

// One unit per (optimizer, ordering, diagnostics).  mt = 1 is the one-replica-per-tile kernel (a
// single worker, or a local step: the same code for either ordering); it lives in the pre units.
template <int OPT, bool POST, bool DIAG>
const void *lookup_unit(bool bf16, int mt, int mask) {
    if (mt == 1) {
        if constexpr (!POST) {
            if (mask != 0) return nullptr;
            return bf16 ? kernel_ptr<OPT, false, DIAG, bf16_t, 1, 0>() : kernel_ptr<OPT, false, DIAG, float, 1, 0>();
        }
        return nullptr;
    }
    return lookup_sync<OPT, POST, DIAG>(bf16, mt, mask);
}

#define DESLOC_DECLARE_UNIT(name) const void *lookup_##name(bool bf16, int mt, int mask)
DESLOC_DECLARE_UNIT(adam_pre);
DESLOC_DECLARE_UNIT(adam_m9);    // MT = 9..12, pre-average
DESLOC_DECLARE_UNIT(adam_m13);   // MT = 13..16
DESLOC_DECLARE_UNIT(adopt_m9);
DESLOC_DECLARE_UNIT(adopt_m13);
DESLOC_DECLARE_UNIT(sgdm_m9);
DESLOC_DECLARE_UNIT(sgdm_m13);
DESLOC_DECLARE_UNIT(adam_post);
DESLOC_DECLARE_UNIT(adopt_pre);
DESLOC_DECLARE_UNIT(adopt_post);
DESLOC_DECLARE_UNIT(sgdm_pre);
DESLOC_DECLARE_UNIT(sgdm_post);
DESLOC_DECLARE_UNIT(adam_pre_diag);
DESLOC_DECLARE_UNIT(adam_post_diag);
DESLOC_DECLARE_UNIT(adopt_pre_diag);
DESLOC_DECLARE_UNIT(adopt_post_diag);
DESLOC_DECLARE_UNIT(sgdm_pre_diag);
DESLOC_DECLARE_UNIT(sgdm_post_diag);
#undef DESLOC_DECLARE_UNIT

}  // namespace desloc
