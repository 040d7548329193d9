"""Averaging steps of more than eight workers: tiles of all replicas up to sixteen (their length follows the worker count, the
optimizer and the gradient type), the runtime-M form beyond, and what cannot be staged -- at the edges of tiles and parts."""
import pytest

import desloc_inputs as di
from test_parity_gpu import check, run_both

pytestmark = pytest.mark.gpu


def _workload(opt, gd, M, numel):
    return di.Workload("many", opt, M, numel, gd, "student_t3" if sum(numel) > 1_000_000 else "normal1", beta2=0.99,
                       eps=1e-2, lr=1e-2, weight_decay=0.01, clip_rho=2.0, adopt_norm_clip=(opt == "adopt"), seed=3 + M)


@pytest.mark.parametrize("M", [9, 10, 11, 12, 13, 14, 15, 16, 17])
@pytest.mark.parametrize("opt,gd", [("adam", "bf16"), ("adam", "f32"), ("adopt", "f32"), ("sgdm", "bf16"), ("sgdm", "f32")])
@pytest.mark.parametrize("staging", [None, 0, 2])     # a block of all replicas; tiles and the runtime-M kernel
def test_every_mask_at_tile_edges(M, opt, gd, staging):
    numel = (1, 31, 225, 256, 289, 447, 449, 513, 2049, 8192 + 8)
    masks = [1, 2, 3] if opt == "sgdm" else [1, 2, 3, 4, 5, 6, 7]
    for align in (4, 1):
        check(run_both(_workload(opt, gd, M, numel), len(masks), align=align, forced_masks=masks, v_init=0.5, staging=staging))


@pytest.mark.parametrize("M,opt,gd", [(9, "adam", "bf16"), (16, "adopt", "f32"), (12, "sgdm", "f32")])
@pytest.mark.parametrize("align,max_blocks,g_shift", [(4, 0, None), (1, 0, None), (4, 40, None), (4, 0, 4)])
def test_chunks_in_several_parts(M, opt, gd, align, max_blocks, g_shift):
    numel = (592 * 1024 * 2 + 700, 2047, 2049, 5)     # chunks of 2048 elements and more; blocks that stride
    masks = [3 if opt == "sgdm" else 7, 2]
    check(run_both(_workload(opt, gd, M, numel), 2, align=align, forced_masks=masks, v_init=0.5, max_blocks=max_blocks,
                   g_shift=g_shift))


@pytest.mark.parametrize("M,opt,gd", [(9, "adam", "bf16"), (16, "adopt", "f32"), (12, "sgdm", "bf16")])
@pytest.mark.parametrize("chunks", [148, 149, 296, 297, 444, 445, 593, 888, 889, 1183])
@pytest.mark.parametrize("staging", [None, 2])       # (smaller ones run in a block of all replicas by themselves)
def test_sizes_where_the_runtime_kernel_takes_over(M, opt, gd, chunks, staging):
    """Single-tile chunks of 1024 elements: between one round of tiles (296 blocks) and one of the runtime-M kernel (444), and
    so on for more rounds, the latter runs."""
    w = _workload(opt, gd, M, (1024 * chunks - 5,))
    masks = [3 if opt == "sgdm" else 7, 2]
    check(run_both(w, 2, forced_masks=masks, v_init=0.5, staging=staging))
