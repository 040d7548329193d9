/*
 * desloc_testing.h -- hooks for the library's own tests.  NOT part of the API: nothing here is
 * needed to use the library, and it may change without notice.
 */
#ifndef DESLOC_TESTING_H_
#define DESLOC_TESTING_H_

#include "desloc.h"

#ifdef __cplusplus
extern "C" {
#endif

/*
 * Cap the grid of the step kernels of this context at max_blocks thread blocks, per worker on local
 * steps (0 = no cap, the default: one block per chunk or part of one).  With a cap every size runs in the tile
 * kernels, whose blocks stride over the parts (the runtime-M kernel ignores the cap).  Results do not
 * depend on it; the tests use it to run the striding path, which the default launch never takes
 * below 2^31 chunks.  DESLOC_E_RANGE for a negative value.
 */
DESLOC_API int desloc_testing_set_max_blocks(desloc_ctx *ctx, int64_t max_blocks);

/*
 * Whether the tile kernels stage their tiles through shared memory: -1 = the library decides (the default:
 * small and mid-sized problems do not run in tile kernels at all, and of the launches that do, one of at most two
 * blocks per SM of single tiles -- seven on local steps -- skips the staging, since it has nothing to overlap, and
 * so do blocks that take whole chunks because the gradients cannot be staged), 0 = tile kernels for every size,
 * staged whenever alignment allows (but for those whole chunks), 1 = tile kernels that never stage (every chunk is
 * updated straight from global memory), 2 = tile kernels (or the runtime-M kernel) for every size, staged as the library
 * decides.  Results do not depend on it.  DESLOC_E_RANGE for other values.
 */
DESLOC_API int desloc_testing_set_staging(desloc_ctx *ctx, int32_t mode);

/*
 * How often a thread block polls for its tile's copies before it gives up (default: about four
 * million polls).  polls = 0 makes every block give up at once: the step then stores nothing,
 * the blocks still let their copies land before they leave, and every later step call returns
 * DESLOC_E_DEVICE_WAIT -- the way the tests exercise the bounded-wait path without hanging or
 * faulting anything.  A negative value restores the default and clears the recorded failure.
 */
DESLOC_API int desloc_testing_set_wait_limit(desloc_ctx *ctx, int32_t polls);

/*
 * Which kernel a step with this sync mask runs over nchunks chunks (0: all) of a context created from cfg whose x starts on
 * 2 KB boundaries, with diagnostics if diag is not 0: 0 = tiles, 1 = runtime-M, 2 = replicas in the lanes of a warp, 3 = a block of all
 * replicas.  layout: how the gradients lie towards 16-byte pieces -- 0 = they fit, 1 = they do not, 2 = nor do bf16 ones
 * towards 8-byte pieces.  blocks, if not NULL: how many thread blocks.
 * Host-only.  Negative desloc_status on bad input.
 */
DESLOC_API int32_t desloc_testing_kernel_of(const desloc_config *cfg, uint32_t mask, int64_t nchunks, int32_t layout, int32_t diag, int64_t *blocks);

/* Groups of pieces that desloc_step_host() has had brought by a kernel, not by copies, in this context so far. */
DESLOC_API int64_t desloc_testing_gathers(const desloc_ctx *ctx);

#ifdef __cplusplus
}
#endif
#endif /* DESLOC_TESTING_H_ */
