"""Chunk lengths of mid-sized problems of three to eight workers: with the short first chunks that tensors off a 2 KB boundary get, the
blocks of an averaging step come in few rounds, none of them for a few blocks, and a round is as many blocks as the
optimizer and the gradient type leave room for."""
import numpy as np
import pytest

import paper_2505_22549_b200.binding as B


def model(width, layers=5):
    w = width
    kv, f = w // 3, w * 8 // 3
    return [w * 3 * w] + [w * w, w * kv, w * kv, w * w, f * w, f * w, w * f, w, w] * layers + [w]


def blocks(M, opt, gd, numel, off):
    cfg = B.make_config(M, numel, opt, gd, 0.9, 0.99, 1e-8, 0.0, 0.0, 1, 1, 1, 0)
    length = B.desloc_chunk_elems(cfg)
    at = np.cumsum([0] + [-(-n // 4) * 4 for n in numel])[:-1] * 4 + (1 << 30) + off
    return length, B.desloc_plan_chunks(numel, length, cap=0, x0=[int(a) for a in at])[0]


@pytest.mark.parametrize("M,opt,gd,per_sm", [(8, "adam", "bf16", 2), (6, "adam", "bf16", 2), (6, "sgdm", "bf16", 3), (8, "adopt", "f32", 3),
                                             (4, "adam", "bf16", 4), (3, "adam", "f32", 4)])
@pytest.mark.parametrize("width", [97, 104, 128, 150])
def test_no_round_is_for_a_few_blocks(M, opt, gd, per_sm, width):
    length, n = blocks(M, opt, gd, model(width), 16)
    most = 2048 if (M, gd) == (8, "f32") else 4096
    assert length % 512 == 0 and 512 <= length <= most
    slots = 148 * per_sm
    # (the rule takes every tensor's last chunk as half full, so that a list can be off by some)
    assert n <= slots or n % slots == 0 or n % slots > 0.4 * slots


@pytest.mark.parametrize("M,opt,gd,per_sm", [(8, "adam", "bf16", 2), (6, "adam", "bf16", 2), (6, "sgdm", "bf16", 3), (8, "adopt", "f32", 3),
                                             (4, "adam", "bf16", 4), (3, "adam", "f32", 4)])
@pytest.mark.parametrize("width", [104, 112, 128, 150, 176])
def test_few_rounds_wherever_the_tensors_lie(M, opt, gd, per_sm, width):
    """Tensors packed from 16 bytes behind a 2 KB boundary, packed from one, and each on one (no short first chunks: the rule,
    which knows no addresses, counts them all the same): the rounds that chunks of the greatest length need, or one more, where
    many tensors end in chunks that the rule takes for half full."""
    numel, slots, most = model(width), 148 * per_sm, 2048 if (M, gd) == (8, "f32") else 4096
    assert sum(-(-n // 512) for n in numel) > 2 * slots            # (what the rule asks for)
    length, packed = blocks(M, opt, gd, numel, 16)
    rounds = lambda n: -(-n // slots)
    at = np.cumsum([0] + [-(-n // 4) * 4 for n in numel])[:-1] * 4 + (1 << 30) + 16
    longest = B.desloc_plan_chunks(numel, most, cap=0, x0=[int(a) for a in at])[0]
    for n in (packed, blocks(M, opt, gd, numel, 0)[1], B.desloc_plan_chunks(numel, length, cap=0)[0]):
        assert rounds(n) <= rounds(longest) + 1


@pytest.mark.parametrize("M,opt,gd,layout,finest", [(7, "adopt", "f32", 1, True), (7, "adopt", "bf16", 2, True), (7, "adopt", "bf16", 1, False),
                                                    (7, "adopt", "f32", 0, False)])
def test_gradients_that_nothing_wide_takes_leave_no_block_idle(M, opt, gd, layout, finest):
    """100 tensors of seven tiles: one round of blocks with a chunk each would leave a third of the chip idle; a tile to a
    block where the gradients are read coordinate by coordinate."""
    numel = [3448] * 100
    cfg = B.make_config(M, numel, opt, gd)
    chunks, length = B.desloc_plan_chunks(numel, B.desloc_chunk_elems(cfg), cap=0)[0], B.desloc_chunk_elems(cfg)
    kernel, blocks = B.desloc_testing_kernel_of(cfg, 7, 0, layout)
    assert kernel == "tiles"
    assert (blocks == chunks * (length // 512)) == finest


def test_what_no_context_accepts_counts_as_adam_and_fp32():
    numel = model(128)
    want = B.desloc_chunk_elems(B.make_config(8, numel, "adam", "f32"))
    assert want != B.desloc_chunk_elems(B.make_config(8, numel, "sgdm", "bf16"))
    assert B.desloc_chunk_elems(B.make_config(8, numel, 7, 9)) == want
