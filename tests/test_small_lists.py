"""Lists of small tensors: no thread block without work beside those of chunks that end short."""
import pytest

import paper_2505_22549_b200.binding as B


def plan(M, numel, opt, mask):
    return B.desloc_testing_kernel_of(B.make_config(M, numel, opt, "bf16"), mask)


@pytest.mark.parametrize("M,count,size,local,averaging", [
    # coordinates of a worker per block: 512 on local steps; 256, 160, 128, 64 for two, three, four, five to eight workers;
    # 64, 32, 16 for nine, twelve, from 33 workers on
    (1, 100, 5, 1, 1), (2, 56, 200, 1, 1), (2, 30, 257, 1, 2), (3, 30, 161, 1, 2), (4, 56, 200, 1, 2), (5, 200, 73, 1, 2),
    (8, 200, 64, 1, 1), (8, 20, 511, 1, 8), (9, 100, 28, 1, 1), (12, 200, 78, 1, 3), (24, 100, 600, 2, 19), (64, 38, 200, 1, 13),
    (128, 70, 2, 1, 1), (256, 38, 17, 1, 2),
])
def test_as_many_blocks_as_have_work(M, count, size, local, averaging):
    assert plan(M, [size] * count, "sgdm", 0) == ("lanes", count * M * local)
    if M > 1:
        assert plan(M, [size] * count, "sgdm", 3) == ("lanes" if M <= 8 else "crowd", count * averaging)


@pytest.mark.parametrize("M,numel,opt,kernel", [
    (128, [600] + [2] * 46, "adam", "tiles"), (128, [600] + [300] * 46, "adam", "lanes"),    # three quarters of the blocks' room empty, or less
    (128, [600] + [470] * 46, "sgdm", "lanes"), (128, [600] + [450] * 46, "sgdm", "tiles"),  # 55 % of it
    (128, [500] + [2] * 46, "sgdm", "lanes"),                                                # a block to each chunk
    (125, [600] + [2] * 46, "adopt", "lanes"), (126, [600] + [2] * 46, "adopt", "tiles"),    # four waves of 1480 chunks, or more
    (62, [600] + [2] * 46, "sgdm", "lanes"), (63, [600] + [2] * 46, "sgdm", "tiles"),        # two
])
def test_sparse_lists_stay_with_the_tiles(M, numel, opt, kernel):
    assert plan(M, numel, opt, 0)[0] == kernel


@pytest.mark.parametrize("M,numel,kernel", [
    # what counts are the coordinates, not the chunks: lists of many tensors as large as a single one
    (16, [2_600] * 100, "crowd"), (16, [262_400], "crowd"), (16, [2_700] * 100, "runtime_m"), (6, [3_300] * 100, "lanes"), (6, [3_400] * 100, "tiles"),
    (8, [4_700] * 100, "lanes"), (8, [4_800] * 100, "tiles"), (24, [1_870] * 100, "crowd"), (24, [1_900] * 100, "runtime_m"),
    # blocks with room for twice the line: as many for each tiny tensor as for a whole chunk
    (4, [300_000] + [2] * 1_200, "lanes"), (4, [300_000] + [2] * 1_300, "tiles"), (12, [100_000] + [2] * 400, "crowd"),
    (12, [100_000] + [2] * 450, "tiles"),
])
def test_lists_are_counted_by_coordinates(M, numel, kernel):
    assert plan(M, numel, "adam", 7)[0] == kernel


@pytest.mark.parametrize("M", [12, 13, 14, 15, 16])
def test_momentum_of_twelve_to_sixteen_workers(M):
    """Up to 2.5 million coordinates, where the tiles and the runtime-M kernel take up to 1.66 times as long."""
    assert plan(M, [2_496_000 // M], "sgdm", 3)[0] == plan(M, [2_330_000 // M], "sgdm", 1)[0] == "crowd"
    assert plan(M, [2_504_000 // M + 1], "sgdm", 3)[0] != "crowd"


@pytest.mark.parametrize("M,n,opt,gd,flags,mask,kernel", [
    (5, 360_000, "adam", "f32", 0, 7, "tiles"), (5, 399_000, "adopt", "f32", 1, 7, "tiles"), (5, 360_000, "adam", "f32", 0, 3, "lanes"),
    (5, 310_000, "adam", "f32", 0, 7, "lanes"),                                                             # 1.55 million
    (5, 360_000, "sgdm", "f32", 0, 3, "lanes"), (5, 360_000, "adam", "f32", 2, 7, "lanes"),                 # (averaging behind the update)
    (5, 360_000, "adam", "bf16", 0, 7, "lanes"), (6, 310_000, "adam", "f32", 0, 7, "lanes"), (4, 500_000, "adam", "f32", 0, 7, "lanes"),
])
def test_a_full_round_of_three_tiles_is_left_to_them(M, n, opt, gd, flags, mask, kernel):
    of = lambda numel, layout: B.desloc_testing_kernel_of(B.make_config(M, numel, opt, gd, flags=flags), mask, 0, layout)[0]
    assert of([n], 0) == kernel
    assert of([n], 1) == "lanes"                   # gradients off the state's layout
    assert of([n // 1000] * 1000, 0) == "lanes"    # as many coordinates in tensors that leave tiles half empty
