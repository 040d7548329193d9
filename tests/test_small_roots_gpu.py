"""1/sqrt of denormal numbers and of the smallest normal ones: second moments and epsilons so small that v + epsilon^2 (Adam) or
max(v, epsilon^2) (ADOPT) is one, with first moments and gradients of the root's size, so that the update is of order one."""
import numpy as np
import pytest
import torch

import desloc_inputs as di
import oracle
from _util import State, compare_per_tensor, f32r, oracle_cfg
from test_parity_gpu import make_engine

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opt", ["adam", "adopt"])
@pytest.mark.parametrize("M", [1, 4, 12])
@pytest.mark.parametrize("eps", [0.0, 2.0 ** -70, 1.2e-19])    # epsilon^2: zero, denormal (exact), just a normal number
@pytest.mark.parametrize("sync", [False, True])
def test_update_from_a_denormal_second_moment(opt, M, eps, sync):
    import paper_2505_22549_b200 as d
    K = (1, 1, 1) if sync else (0, 0, 0)
    w = di.Workload("roots", opt, M, (5000, 513, 7), "f32", "normal1", lr=1e-2, beta2=0.5, eps=eps, K=K, seed=M)
    st = State(w, torch.device("cuda:0"))
    gen = torch.Generator(device="cuda").manual_seed(M)
    # an odd number of units of 2^-149, doubled where beta2 = 1/2 halves it again: exact in fp32 and in the oracle
    units = 2 * torch.randint(0, 1 << 10, (st.nflat,), device="cuda", generator=gen, dtype=torch.int64) + 1
    v = units.to(torch.float64) * 2.0 ** -149 if eps == 0.0 else torch.zeros(st.nflat, device="cuda", dtype=torch.float64)
    root = torch.sqrt(v) if eps == 0.0 else torch.full_like(v, f32r(eps))
    for m in range(M):
        z = torch.randn(st.nflat, device="cuda", generator=gen, dtype=torch.float64)
        st.v[m].copy_((2 * v if opt == "adam" else v).float())
        st.u[m].copy_((root * z if opt == "adam" else z).float())
        st.g[m].copy_((root * z.flip(0) if opt == "adopt" else torch.zeros_like(z)).float())
    ox, ou, ov = st.to_numpy(st.x), st.to_numpy(st.u), st.to_numpy(st.v)
    assert eps or np.count_nonzero(ov) == ov.size          # (the copies kept the denormal numbers)
    before = ox.copy()
    eng = make_engine(d, w, st)
    eng.step(0, f32r(w.lr), st.views(st.g))
    oracle.step(oracle_cfg(w), 0, f32r(w.lr), ox, ou, ov, st.to_numpy(st.g))
    assert np.mean(np.abs(ox - before)[:, st.valid_mask()]) > 1e-4
    for got, want, what in ((st.x, ox, "x"), (st.u, ou, "u")):
        compare_per_tensor(st, st.to_numpy(got), want, what)
    eng.close()
