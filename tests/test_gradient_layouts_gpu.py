"""Gradients laid out differently from the state, so that the copy engine cannot take them.  Chunks go straight from global memory
then, with 128-bit accesses or element by element; in large problems a block takes a whole chunk of one or two replicas, and the
runtime-M kernel the averaging steps of nine workers and more.  Offsets of the gradient buffers within 16 bytes, at the edges of
tiles and chunks, and problems where only a part of the tensors is off."""
import pytest

import desloc_inputs as di
from test_parity_gpu import check, run_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 2, 3, 4, 9, 16])
@pytest.mark.parametrize("opt,gd", [("adam", "bf16"), ("adopt", "f32"), ("sgdm", "bf16")])
@pytest.mark.parametrize("g_shift", [1, 4])
def test_gradients_off_the_states_layout(M, opt, gd, g_shift):
    numel = (13 * 512 + 8, 511, 520, 2047, 4096, 7)
    top = 3 if opt == "sgdm" else 7
    w = di.Workload("layouts", opt, M, numel, gd, "normal1", lr=1e-2, weight_decay=0.05, clip_rho=1.5, beta2=0.99, eps=1e-2,
                    adopt_norm_clip=(opt == "adopt"), seed=M + g_shift)
    check(run_both(w, 4, align=8, forced_masks=[0, top, 2, 1], v_init=0.25, g_shift=g_shift, staging=0))


@pytest.mark.parametrize("M,opt,gd,g_shift", [(7, "adopt", "f32", 1), (8, "adam", "f32", 2), (6, "adam", "bf16", 1), (3, "sgdm", "f32", 3)])
@pytest.mark.parametrize("numel", [(3448,) * 100 + (372_003,), (2_100_000 // 3, 511, 1025)])
def test_mid_sized_problems_off_the_states_layout(M, opt, gd, g_shift, numel):
    w = di.Workload("layouts", opt, M, numel, gd, "student_t3", lr=1e-2, clip_rho=1.5, beta2=0.99, eps=1e-2,
                    adopt_norm_clip=(opt == "adopt"), seed=M)
    check(run_both(w, 2, align=4, forced_masks=[3 if opt == "sgdm" else 7, 2], v_init=0.25, g_shift=g_shift))


@pytest.mark.parametrize("M,opt,gd,g_shift", [(1, "adam", "bf16", 4), (1, "sgdm", "f32", 1), (2, "adam", "f32", 1),
                                              (2, "sgdm", "bf16", 4), (4, "adopt", "bf16", 4), (4, "adam", "bf16", 3),
                                              (12, "sgdm", "bf16", 4), (16, "adam", "bf16", 1), (16, "adam", "bf16", 4)])
@pytest.mark.parametrize("align,max_blocks,staging", [(8, 0, None), (8, 40, 0), (4, 0, None)])
def test_large_problems_off_the_states_layout(M, opt, gd, g_shift, align, max_blocks, staging):
    # more than four rounds of blocks; chunks that end short, tensors of less than a tile
    numel = (9_000_000 // min(M, 4) + 700, 2049, 512 * 9, 3_000_000 // min(M, 4) + 4, 13)
    w = di.Workload("layouts", opt, M, numel, gd, "student_t3", lr=1e-2, clip_rho=1.5, beta2=0.99, eps=1e-2,
                    adopt_norm_clip=(opt == "adopt"), seed=M)
    check(run_both(w, 2, align=align, forced_masks=[0, 3 if opt == "sgdm" else 7], v_init=0.25, g_shift=g_shift,
                   max_blocks=max_blocks, staging=staging))
