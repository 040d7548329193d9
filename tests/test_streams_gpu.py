"""Gradient tables across streams: a loop records an event only behind the first kernel of a table; a context that moves between
streams (each step ordered behind the one before, as steps on the same state have to be) and changes its gradients at every
step must not overwrite a table that is still being read."""
import numpy as np
import pytest
import torch

import desloc_inputs as di
from _util import State, f32r
from test_parity_gpu import make_engine

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("repeats", [1, 3])
def test_resident_table_then_another_stream(repeats):
    import paper_2505_22549_b200 as d
    w = di.Workload("hop", "adam", 4, (300_000, 5000, 33), "bf16", "student_t3", lr=1e-2, K=(2, 3, 4), seed=6)
    dev = torch.device("cuda:0")
    ends = []
    for hop in (False, True):
        st = State(w, dev)
        eng = make_engine(d, w, st)
        st.fill_grads(0)
        # every step's gradients in buffers of their own, as many tables as two rounds of slots
        sets = []
        for j in range(18):
            st.fill_grads(j)
            sets.append([b.clone() for b in st.g])
        plan = [j for j in range(len(sets)) for _ in range(repeats)]
        streams = [torch.cuda.Stream(), torch.cuda.Stream()]
        torch.cuda.synchronize()
        for t, j in enumerate(plan):
            s = streams[1 if hop and (t >= len(plan) // 2 or t % 5 == 4) else 0]
            if hop and t:
                s.wait_stream(last)
            with torch.cuda.stream(s):
                eng.step(t, f32r(w.lr), st.views(sets[j]))
            last = s
        torch.cuda.synchronize()
        ends.append([st.to_numpy(a) for a in (st.x, st.u, st.v)])
        eng.close()
    for a, b in zip(*ends):
        assert np.array_equal(a, b)
