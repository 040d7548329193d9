"""Local steps (nothing averaged) run one replica per block, a chunk cut into parts of up to three 512-element tiles, or
single tiles straight from global memory where one wave of blocks covers the problem: sizes around those edges against the
oracle."""
import pytest

import desloc_inputs as di
from test_parity_gpu import check, run_both

pytestmark = pytest.mark.gpu

CHUNK = 8 * 512                       # of a large problem with three to eight workers
LARGE = 592 * CHUNK                   # from here on chunks have their full length


@pytest.mark.parametrize("opt,gd", [("adam", "bf16"), ("adam", "f32"), ("adopt", "f32"), ("sgdm", "f32"), ("sgdm", "bf16")])
@pytest.mark.parametrize("M,numel", [
    (3, (LARGE + 2048 + 1, 1535, 1537, 4095, 4097, 511, 513, 5)),    # full chunks; parts that end short, empty parts
    (4, (3 * LARGE // 8 + 700, 2047, 2049)),                         # chunks of three tiles
    (2, (2 * LARGE + 1024 * 7 + 3, 8191)),                           # chunks of eight 1024-element tiles: four or six parts
    (8, (129 * 512 - 3, 400)), (8, (130 * 512, 512)),                # one tile per block: just within a wave, just beyond
    (9, (592 * 8192 // 4 + 5, 1025)),                                # local steps of more than eight workers
])
@pytest.mark.parametrize("staging", [None, 2])       # 2: the smaller ones in tiles, too
def test_local_steps_at_part_and_wave_edges(opt, gd, M, numel, staging):
    w = di.Workload("parts", opt, M, numel, gd, "normal1" if sum(numel) < 100_000 else "student_t3", lr=1e-2, weight_decay=0.05,
                    clip_rho=1.5, K=(0, 0, 0), adopt_norm_clip=(opt == "adopt"), eps=1e-3, seed=M)
    check(run_both(w, 2, align=4, v_init=0.25, staging=staging))


@pytest.mark.parametrize("opt,gd", [("adam", "bf16"), ("adopt", "f32"), ("sgdm", "f32")])
@pytest.mark.parametrize("M,numel", [
    (2, (2 * LARGE + 1024 * 7 + 3, 8191, 2047, 2049)),               # two replicas: a chunk in four parts
    (2, (296 * 512 - 8, 8)), (2, (298 * 512,)),                      # one tile per block, and just beyond a wave
    (8, (LARGE + 255, 257, 4097, 3)),                                # eight replicas: 256-element tiles with fp32 gradients
])
@pytest.mark.parametrize("staging", [None, 2])
def test_averaging_steps_at_part_and_tile_edges(opt, gd, M, numel, staging):
    w = di.Workload("parts", opt, M, numel, gd, "normal1" if sum(numel) < 400_000 else "student_t3", lr=1e-2, weight_decay=0.05,
                    clip_rho=1.5, adopt_norm_clip=(opt == "adopt"), eps=1e-3, seed=M)
    top = 3 if opt == "sgdm" else 7
    check(run_both(w, 2, align=4, v_init=0.25, forced_masks=[top, 1], staging=staging))


@pytest.mark.parametrize("opt", ["adam", "adopt", "sgdm"])
@pytest.mark.parametrize("M", [2, 4, 12])
@pytest.mark.parametrize("eps", [0.0, 1e-22, 1.2e-19, 1e-8])
@pytest.mark.parametrize("staging", [None, 2])
def test_epsilon_whose_square_is_no_normal_number(opt, M, eps, staging):
    """The square of epsilon is zero, a denormal number, or just a normal one: the last two decide between two forms of
    1/sqrt.  v starts at 0.25, so that epsilon 0 is defined."""
    w = di.Workload("eps", opt, M, (700_000, 513), "bf16", "normal1", lr=1e-2, eps=eps, beta2=0.99, seed=M)
    top = 3 if opt == "sgdm" else 7
    check(run_both(w, 3, align=4, v_init=0.25, forced_masks=[0, top, 0], staging=staging))
