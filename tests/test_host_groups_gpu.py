"""step_host in groups whose kernels are not the whole list's: nine and more workers, with no other step of the process in front, bit
for bit against step."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import desloc_inputs as di
from _util import State, f32r

pytestmark = pytest.mark.gpu

# workers, optimizer, gradients, tensors, post-average, the kernels of the whole list and of the two groups
R, T, C = "runtime_m", "tiles", "crowd"
CASES = [
    (9, "adam", "bf16", (239_000, 75_500), False, (R, T, C)),
    (9, "adopt", "f32", (239_000, 75_500), False, (R, T, C)),
    (11, "sgdm", "f32", (470_000, 145_000), False, (R, T, T)),
    (12, "adam", "f32", (266_000, 84_000), False, (R, T, C)),
    (16, "adopt", "bf16", (266_000, 84_000), False, (R, T, C)),
    (16, "sgdm", "bf16", (520_000, 160_000), False, (R, T, T)),
    (200, "adam", "f32", (60_000, 20_000), False, (R, R, C)),
    (192, "adopt", "f32", (60_000, 6_000), True, (R, R, C)),
    (256, "adam", "bf16", (60_000, 6_000), False, (R, R, C)),
    (256, "adopt", "bf16", (60_000, 20_000), False, (R, R, C)),
    (256, "sgdm", "f32", (60_000, 20_000), True, (R, R, C)),
]


def run(M, opt, gd, numel, post, kernels):
    import paper_2505_22549_b200 as d
    from test_parity_gpu import _flags, make_engine
    w = di.Workload("hostgroups", opt, M, numel, gd, "normal1", lr=1e-2, eps=1e-3, adopt_norm_clip=(opt == "adopt"), K=(1, 1, 1), seed=M)
    dev = torch.device("cuda:0")
    a, b = (State(w, dev, align=512, v_init=0.25) for _ in range(2))
    cfg = d.make_config(M, numel, opt, gd, eps=1e-3, flags=_flags(d, w, post))
    chunks = [-(-n // d.desloc_chunk_elems(cfg)) for n in numel]
    mask = 3 if opt == "sgdm" else 7
    assert tuple(d.desloc_testing_kernel_of(cfg, mask, n)[0] for n in (sum(chunks), *chunks)) == kernels
    ea, eb = make_engine(d, w, a, post), make_engine(d, w, b, post)
    host = [torch.empty(b.nflat, dtype=b.g[0].dtype).pin_memory() for _ in range(M)]
    views = [[h[o:o + n] for o, n in zip(b.offs, numel)] for h in host]
    for t in range(2):
        a.fill_grads(t)
        for m in range(M):
            host[m].copy_(a.g[m])
        torch.cuda.synchronize()
        assert eb.step_host(t, f32r(w.lr), views, b.views(b.g), clip_bound=1.0) == ea.step(
            t, f32r(w.lr), a.views(a.g), clip_bound=1.0) == mask
    torch.cuda.synchronize()
    for pa, pb in ((a.x, b.x), (a.u, b.u)) + (((a.v, b.v),) if a.v is not None else ()):
        assert np.array_equal(a.to_numpy(pa).view(np.uint32), b.to_numpy(pb).view(np.uint32))
    assert eb.launches() == 4       # two groups a step
    ea.close(), eb.close()


@pytest.mark.parametrize("case", range(len(CASES)))
def test_groups_in_other_kernels_than_the_whole_list(case):
    """In a process of its own: a kernel that an earlier step prepared stays prepared."""
    r = subprocess.run([sys.executable, __file__, str(case)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


if __name__ == "__main__":
    run(*CASES[int(sys.argv[1])])
