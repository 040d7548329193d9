"""Gradients of small problems in pinned host memory, brought by a kernel: the bytes that arrive, whatever the alignments of the two
sides, and the same step as with gradients on the device; pageable memory and many pieces, which the copy engine takes."""
import numpy as np
import pytest
import torch

import desloc_inputs as di
from _util import State, f32r
from test_parity_gpu import make_engine

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gd", ["bf16", "f32"])
@pytest.mark.parametrize("shift_h,shift_d", [(0, 0), (1, 0), (3, 5), (8, 0)])
@pytest.mark.parametrize("M,numel,separate,pinned,by_kernel", [
    (2, (1,), False, True, True), (3, (4095, 17, 8193, 1), False, True, True), (4, (2053, 64, 7), True, True, True),
    (8, (4096 + 31,), False, False, False),                 # pageable
    (8, (33,) * 9, True, True, False), (8, (33,) * 8 + (99,), True, True, False),      # 72 pieces
])
def test_host_gradients_of_small_problems(gd, shift_h, shift_d, M, numel, separate, pinned, by_kernel):
    w = di.Workload("hostcopy", "adam", M, numel, gd, "normal1", lr=1e-2, K=(2, 3, 4), eps=1e-3, seed=1)
    dev = torch.device("cuda:0")
    a, b = State(w, dev, align=1, v_init=0.25), State(w, dev, align=1, v_init=0.25, g_shift=shift_d)
    import paper_2505_22549_b200 as d
    ea, eb = make_engine(d, w, a), make_engine(d, w, b)
    dt = b.g[0].dtype
    pin = lambda n: torch.empty(n + shift_h, dtype=dt, pin_memory=pinned)[shift_h:]
    flat = [pin(b.nflat) for _ in range(M)]
    host = [[pin(n) for n in numel] for _ in range(M)] if separate else [[f[o:o + n] for o, n in zip(b.offs, numel)] for f in flat]
    for t in range(5):
        a.fill_grads(t)
        for m in range(M):
            for h, src in zip(host[m], a.views(a.g)[m]):
                h.copy_(src)
            b.g[m].zero_()
        torch.cuda.synchronize()
        before = eb.launches()
        assert ea.step(t, f32r(w.lr), a.views(a.g)) == eb.step_host(t, f32r(w.lr), host, b.views(b.g))
        torch.cuda.synchronize()
        # by the kernel, the copies and the step; else the step alone, in two groups where a tensor ends at three quarters
        assert eb.launches() == before + (2 if by_kernel or numel == (33,) * 9 else 1)
        for m in range(M):
            for x, y in zip(a.views(a.g)[m], b.views(b.g)[m]):
                assert torch.equal(x, y)
    for pa, pb in ((a.x, b.x), (a.u, b.u), (a.v, b.v)):
        assert np.array_equal(a.to_numpy(pa), b.to_numpy(pb))
    ea.close(); eb.close()


@pytest.mark.parametrize("gd", ["bf16", "f32"])
@pytest.mark.parametrize("shift_h,shift_d", [(0, 0), (1, 0), (3, 5)])
@pytest.mark.parametrize("M,numel,separate,pinned", [
    (3, (33, 4095, 4096, 4097, 8193) * 4 + (2_500_007,), True, True),        # a cut inside the last tensor
    (2, (1_900_001,) + (7, 1, 4100) * 12 + (900_003,), True, True),          # inside the first, and the last
    (12, (40_003,) * 9, False, True), (2, (33, 5000) * 16 + (2_100_000,), True, False),      # pageable: copies
])
def test_many_pieces_arrive_group_by_group(gd, shift_h, shift_d, M, numel, separate, pinned):
    """Every byte of the pieces, nothing around them, and other addresses at every step."""
    import paper_2505_22549_b200 as d
    w = di.Workload("pieces", "sgdm", M, numel, gd, "normal1", lr=1e-2, K=(2, 3, 4), seed=2)
    dev = torch.device("cuda:0")
    st = State(w, dev, align=3, g_shift=shift_d)          # (elements in between that belong to nobody)
    eng = make_engine(d, w, st)
    dt, gen = st.g[0].dtype, torch.Generator().manual_seed(3)
    inside = torch.from_numpy(st.valid_mask()).to(dev)
    for t in range(4):
        def pin(n):
            h = torch.empty(n + shift_h + t, dtype=dt, pin_memory=pinned)[shift_h + t:]
            return h.copy_(torch.randn(n, generator=gen))
        flat = [pin(st.nflat + 1) for _ in range(M)]
        host = [[pin(n) for n in numel] for _ in range(M)] if separate else [[f[o + 1:o + 1 + n] for o, n in zip(st.offs, numel)] for f in flat]
        for g in st.g:
            g.fill_(7.0)
        before = d.desloc_testing_gathers(eng.ctx)
        eng.step_host(t, 1e-2, host, st.views(st.g))
        torch.cuda.synchronize()
        assert (d.desloc_testing_gathers(eng.ctx) > before) == pinned
        for m in range(M):
            for x, y in zip(host[m], st.views(st.g)[m]):
                assert torch.equal(x, y.cpu())
            assert bool((st.g[m][~inside] == 7.0).all())
    eng.close()
