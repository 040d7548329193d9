"""Steps with the replicas of a coordinate in the lanes of a warp (small and mid-sized problems): against the oracle, and bit for bit
against the tile kernels, whose sums have the same order."""
import numpy as np
import pytest

import desloc_inputs as di
from test_parity_gpu import _lib, check, run_both

pytestmark = pytest.mark.gpu


def both_ways(w, T, masks_in_lanes=None, **kw):
    d = _lib()
    cfg = d.make_config(w.M, w.numel, w.opt, w.grad_dtype)
    for mask in kw["forced_masks"] if masks_in_lanes is None else masks_in_lanes:
        assert d.desloc_testing_kernel_of(cfg, mask)[0] == "lanes"
    lanes, tiles = run_both(w, T, **kw), run_both(w, T, staging=0, **kw)
    check(lanes)
    for name in ("gx", "gu") + (("gv",) if lanes["gv"] is not None else ()):
        assert np.array_equal(lanes[name].view(np.uint32), tiles[name].view(np.uint32)), name


@pytest.mark.parametrize("M", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("opt,gd,rho", [("adam", "bf16", 0.0), ("adopt", "f32", 1.5), ("sgdm", "bf16", 0.0), ("adam", "f32", 1.5)])
@pytest.mark.parametrize("post", [False, True])
@pytest.mark.parametrize("align,g_shift", [(4, 0), (1, 0), (8, 1), (8, 4)])
def test_every_mask_at_the_edges_of_a_piece(M, opt, gd, rho, post, align, g_shift):
    # a warp's piece of a worker: 128 coordinates for one, 64, 40, 32 for two to four, 16 for more; four warps a block
    piece = {1: 128, 2: 64, 3: 40, 4: 32}.get(M, 16)
    numel = (1, 2, 3, 4, 5, piece - 1, piece, piece + 1, piece + 4, 4 * piece - 4, 4 * piece, 4 * piece + 1, 511, 516, 1031, 2053)
    masks = list(range(4 if opt == "sgdm" else 8))
    w = di.Workload("lanes", opt, M, numel, gd, "normal1", beta1=0.9, beta2=0.99, eps=1e-2, lr=1e-2, weight_decay=0.05,
                    clip_rho=rho, adopt_norm_clip=(opt == "adopt"), seed=M)
    both_ways(w, len(masks), align=align, g_shift=g_shift, forced_masks=masks, v_init=0.25, post=post)


@pytest.mark.parametrize("M", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("opt,gd,align", [("adam", "bf16", 4), ("sgdm", "f32", 1)])
@pytest.mark.parametrize("numel", [(2, 1, 3), (64, 5, 63, 65, 64), (161, 7, 160, 159, 256, 257)])
def test_lists_of_small_tensors_have_fewer_parts(M, opt, gd, align, numel):
    masks = [3 if opt == "sgdm" else 7, 0, 1]
    w = di.Workload("lanes", opt, M, numel, gd, "normal1", beta2=0.99, eps=1e-2, lr=1e-2, seed=M)
    both_ways(w, len(masks), align=align, forced_masks=masks, v_init=0.25)


# (the second five a chunk off the limit: a buffer off a 2 KB boundary has one chunk more)
@pytest.mark.parametrize("M,opt,gd,n", [(8, "adam", "bf16", 374784), (8, "adam", "bf16", 374785), (3, "sgdm", "f32", 532480),
                                        (2, "adopt", "bf16", 2490368), (4, "adam", "f32", 1249280),
                                        (8, "adam", "bf16", 372736), (8, "adam", "bf16", 375297), (3, "sgdm", "f32", 531968),
                                        (2, "adopt", "bf16", 2437120), (4, "adam", "f32", 1244160)])
def test_sizes_on_either_side_of_the_tile_kernels(M, opt, gd, n):
    top = 3 if opt == "sgdm" else 7
    w = di.Workload("lanes", opt, M, (n,), gd, "student_t3", lr=1e-2, clip_rho=1.5, eps=1e-3,
                    adopt_norm_clip=(opt == "adopt"), seed=M)
    both_ways(w, 2, masks_in_lanes=[0] if n in (374785, 375297, 1249280) else [top, 0], align=4, v_init=0.25, forced_masks=[top, 0])


# 444 blocks load into registers, 445 through shared memory: pieces of 512 coordinates of one worker, of 128 of four, 64 of eight (the last
# ragged; a first chunk off a 2 KB boundary adds a block)
@pytest.mark.parametrize("M,opt,gd,blocks", [(1, "adam", "bf16", 512), (3, "adopt", "f32", 512), (4, "adam", "f32", 128), (8, "sgdm", "bf16", 64)])
@pytest.mark.parametrize("more", [-516, -4, 4, 129])
def test_loads_on_either_side_of_the_registers(M, opt, gd, blocks, more):
    local = blocks == 512
    n = 444 * blocks // (M if local else 1) + more
    masks = [0] if local else [3 if opt == "sgdm" else 7, 1]
    w = di.Workload("lanes", opt, M, (n,), gd, "normal1", eps=1e-2, lr=1e-2, weight_decay=0.05, seed=M)
    both_ways(w, len(masks), align=4, forced_masks=masks, v_init=0.25)
