"""Averaging steps of more than eight workers on small problems: against the oracle, and bit for bit against the tile kernels (up to
sixteen workers) and the runtime-M kernel, whose sums have the same order."""
import numpy as np
import pytest

import desloc_inputs as di
from test_parity_gpu import _lib, check, run_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [9, 11, 12, 16, 17, 32, 33, 64, 65, 128, 129, 256])
@pytest.mark.parametrize("opt,gd,rho,align,g_shift", [("adam", "bf16", 0.0, 4, 0), ("adopt", "f32", 1.5, 1, 0),
                                                      ("sgdm", "bf16", 0.0, 8, 4), ("adam", "f32", 1.5, 8, 1)])
@pytest.mark.parametrize("post", [False, True])
def test_every_mask_at_the_edges_of_a_piece(M, opt, gd, rho, align, g_shift, post):
    piece = 64 if M < 12 else 32 if M <= 32 else 16
    numel = (1, 2, 3, piece - 1, piece, piece + 1, piece + 4, 2 * piece, 516, 1031)
    masks = list(range(1, 4 if opt == "sgdm" else 8))
    cfg = _lib().make_config(M, numel, opt, gd)
    assert all(_lib().desloc_testing_kernel_of(cfg, mask)[0] == "crowd" for mask in masks)
    w = di.Workload("crowd", opt, M, numel, gd, "normal1", beta1=0.9, beta2=0.99, eps=1e-2, lr=1e-2, weight_decay=0.05,
                    clip_rho=rho, adopt_norm_clip=(opt == "adopt"), seed=M)
    kw = dict(align=align, g_shift=g_shift, forced_masks=masks, v_init=0.25, post=post)
    crowd, other = run_both(w, len(masks), **kw), run_both(w, len(masks), staging=0, **kw)
    check(crowd)
    check(other)
    for name in ("gx", "gu") + (("gv",) if crowd["gv"] is not None else ()):
        assert np.array_equal(crowd[name].view(np.uint32), other[name].view(np.uint32)), name


@pytest.mark.parametrize("M", [9, 12, 33, 129])
@pytest.mark.parametrize("opt,gd,post", [("adam", "bf16", False), ("adopt", "f32", True)])
@pytest.mark.parametrize("numel", [(2, 1, 3), (16, 5, 15, 17), (65, 7, 64, 63)])
def test_lists_of_small_tensors_have_fewer_parts(M, opt, gd, post, numel):
    w = di.Workload("crowd", opt, M, numel, gd, "normal1", beta2=0.99, eps=1e-2, lr=1e-2, adopt_norm_clip=(opt == "adopt"), seed=M)
    kw = dict(align=4, forced_masks=[7, 1], v_init=0.25, post=post)
    crowd, other = run_both(w, 2, **kw), run_both(w, 2, staging=0, **kw)
    check(crowd)
    for name in ("gx", "gu", "gv"):
        assert np.array_equal(crowd[name].view(np.uint32), other[name].view(np.uint32)), name


@pytest.mark.parametrize("M,opt,gd,n", [(12, "adam", "bf16", 190_000), (16, "sgdm", "f32", 140_001), (24, "adopt", "bf16", 150_000),
                                        (64, "adam", "f32", 110_003), (128, "adopt", "f32", 60_000), (256, "adam", "bf16", 30_001)])
def test_more_blocks_than_fit_at_once(M, opt, gd, n):
    d = _lib()
    top = 3 if opt == "sgdm" else 7
    kernel, blocks = d.desloc_testing_kernel_of(d.make_config(M, [n], opt, gd, flags=1 if opt == "adopt" else 0), top)
    # (64 warps an SM at most)
    lanes = 16 if M < 12 else 8 if M <= 32 else 4
    assert kernel == "crowd" and blocks > 148 * (64 // -(-M * lanes // 32))
    w = di.Workload("crowd", opt, M, (n,), gd, "student_t3", lr=1e-2, clip_rho=1.5, eps=1e-3,
                    adopt_norm_clip=(opt == "adopt"), seed=M)
    kw = dict(align=4, v_init=0.25, forced_masks=[top, 2])
    crowd, other = run_both(w, 2, **kw), run_both(w, 2, staging=2, **kw)
    check(crowd)
    for name in ("gx", "gu") + (("gv",) if crowd["gv"] is not None else ()):
        assert np.array_equal(crowd[name].view(np.uint32), other[name].view(np.uint32)), name
