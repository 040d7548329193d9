"""Gradients laid out differently from the state, so that the copy engine cannot take them: in large problems threads read
their own gradients, in one access or element by element, while the state is staged (one, two and four replicas per tile), or the
runtime-M kernel runs (nine to sixteen); else the whole chunk goes straight from global memory.  Offsets of the gradient
buffers within 16 bytes, at the edges of tiles and parts."""
import pytest

import desloc_inputs as di
from test_parity_gpu import check, run_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 2, 3, 4, 9, 16])
@pytest.mark.parametrize("opt,gd", [("adam", "bf16"), ("adopt", "f32"), ("sgdm", "bf16")])
@pytest.mark.parametrize("g_shift", [1, 2, 4, 6])
def test_gradients_off_the_states_layout(M, opt, gd, g_shift):
    numel = (13 * 512 + 8, 511, 520, 2047, 4096, 7)
    top = 3 if opt == "sgdm" else 7
    w = di.Workload("layouts", opt, M, numel, gd, "normal1", lr=1e-2, weight_decay=0.05, clip_rho=1.5, beta2=0.99, eps=1e-2,
                    adopt_norm_clip=(opt == "adopt"), seed=M + g_shift)
    check(run_both(w, 4, align=8, forced_masks=[0, top, 2, 1], v_init=0.25, g_shift=g_shift, staging=0))


@pytest.mark.parametrize("M,opt,gd,g_shift", [(1, "adam", "bf16", 4), (1, "sgdm", "f32", 1), (2, "adam", "f32", 1),
                                              (2, "sgdm", "bf16", 4), (4, "adopt", "bf16", 3), (4, "adam", "bf16", 4),
                                              (4, "sgdm", "f32", 2), (12, "sgdm", "f32", 2), (16, "adam", "bf16", 1)])
@pytest.mark.parametrize("post,max_blocks", [(False, 0), (False, 40), (True, 0)])
def test_large_problems_off_the_states_layout(M, opt, gd, g_shift, post, max_blocks):
    # more than four rounds of blocks; a tensor that ends inside a tile, small ones, blocks that stride
    numel = (13_000_000 // min(M, 4) + 700, 2049, 512 * 9, 13)
    w = di.Workload("layouts", opt, M, numel, gd, "student_t3", lr=1e-2, clip_rho=1.5, beta2=0.99, eps=1e-2,
                    adopt_norm_clip=(opt == "adopt"), seed=M)
    check(run_both(w, 2, align=8, forced_masks=[0, 3 if opt == "sgdm" else 7], v_init=0.25, g_shift=g_shift, post=post,
                   max_blocks=max_blocks))
