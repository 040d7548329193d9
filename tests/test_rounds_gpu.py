"""How a step is cut into blocks follows the size of the problem: single tiles, runs that fill whole rounds of blocks, full-length
runs; parts of a chunk for two and for more than eight workers.  Sizes on either side of each change, against the oracle."""
import pytest

import desloc_inputs as di
from test_parity_gpu import check, run_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,opt,gd,tiles", [
    (8, "adam", "bf16", 592), (8, "adam", "bf16", 593), (8, "adopt", "f32", 2368), (8, "sgdm", "bf16", 2369),
    (4, "adam", "bf16", 888), (4, "adam", "bf16", 889), (4, "adopt", "bf16", 3553), (3, "sgdm", "f32", 1185),
    (2, "adam", "f32", 1036), (2, "adam", "bf16", 1038), (2, "sgdm", "bf16", 4200),
    (16, "adam", "bf16", 196), (12, "adopt", "f32", 593), (9, "sgdm", "bf16", 1200),
])
@pytest.mark.parametrize("extra", [0, -7])
@pytest.mark.parametrize("staging", [None, 2])       # 2: the smaller ones in tiles, too
def test_sizes_where_the_split_changes(M, opt, gd, tiles, extra, staging):
    w = di.Workload("rounds", opt, M, (512 * tiles + extra,), gd, "student_t3", lr=1e-2, weight_decay=0.05, clip_rho=1.5,
                    adopt_norm_clip=(opt == "adopt"), eps=1e-3, seed=M)
    top = 3 if opt == "sgdm" else 7
    check(run_both(w, 2, align=4, v_init=0.25, forced_masks=[top, 0], staging=staging))


@pytest.mark.parametrize("numel,launches,M", [
    # three quarters of what is left each time, as long as that is more than 1.6 M
    ((300_000 + 3,) * 40, 3, 3),                   # 9 M, 2.25 M of the 3 M left, and the rest
    ((1_000_000,) * 3 + (7_000_001,), 3, 2),       # 7.5 M, 1.9 M and the rest: both cuts inside the last tensor
    ((2_000_003, 2_999_999), 2, 3),                # 3.75 M and the rest
    ((3_200_005,), 2, 2), ((1_500_000,), 1, 2),    # one tensor: 2.4 M and the rest, or too small to cut
    ((2_400_000, 700_000, 70_000), 2, 12),         # ends with the first tensor
])
def test_host_gradients_in_groups_of_falling_size(numel, launches, M):
    """The groups together give the plain step, and there are as many as the sizes ask for."""
    import numpy as np
    import torch
    import paper_2505_22549_b200 as d
    from _util import State, f32r
    from test_parity_gpu import make_engine
    w = di.Workload("groups", "adam", M, numel, "bf16", "student_t3", lr=1e-2, K=(2, 3, 4), seed=1)
    dev = torch.device("cuda:0")
    a, b = State(w, dev), State(w, dev)
    ea, eb = make_engine(d, w, a), make_engine(d, w, b)
    host = [torch.empty(b.nflat, dtype=b.g[0].dtype).pin_memory() for _ in range(w.M)]
    views = [[h[o:o + n] for o, n in zip(b.offs, w.numel)] for h in host]
    for t in range(4):
        a.fill_grads(t)
        for m in range(w.M):
            host[m].copy_(a.g[m])
            b.g[m].zero_()
        torch.cuda.synchronize()
        assert ea.step(t, f32r(w.lr), a.views(a.g)) == eb.step_host(t, f32r(w.lr), views, b.views(b.g))
    torch.cuda.synchronize()
    for pa, pb in ((a.x, b.x), (a.u, b.u), (a.v, b.v)):
        assert np.array_equal(a.to_numpy(pa), b.to_numpy(pb))
    assert eb.launches() == 4 * launches and ea.launches() == 4
    ea.close(); eb.close()
