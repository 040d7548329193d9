"""Failure detection without a fault: every wait in the kernels is bounded.  A thread block that
does not see its tile arrive within the limit records that, lets the copies it requested land,
stores nothing and leaves; the host reports DESLOC_E_DEVICE_WAIT on the next call.  Here the
limit is set to zero polls through the test hook, so every block takes that path at once --
nothing hangs, nothing faults, and the context (and the GPU) stay usable."""
import numpy as np
import pytest
import torch

import desloc_inputs as di
from _util import State, f32r
from test_parity_gpu import make_engine

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["cfg2_adam_135m", "cfg3_adopt_360m", "cfg5_sgdm_desloc"])
def test_a_wait_that_runs_out_is_reported_and_nothing_is_stored(name):
    import paper_2505_22549_b200 as d
    w = di.mini(di.WORKLOADS[name], T=4).replace(K=(1, 1, 1))
    dev = torch.device("cuda:0")
    st = State(w, dev)
    eng = make_engine(d, w, st)
    st.fill_grads(0)
    eng.step(0, f32r(w.lr), st.views(st.g), clip_bound=1.0)
    torch.cuda.synchronize()
    before = [st.to_numpy(b) for b in (st.x, st.u) + ((st.v,) if st.v is not None else ())]

    d.desloc_testing_set_staging(eng.ctx, 0)                # stage even if the launch is small
    d.desloc_testing_set_wait_limit(eng.ctx, 0)             # every block gives up at once
    st.fill_grads(1)
    eng.step(1, f32r(w.lr), st.views(st.g), clip_bound=1.0)  # enqueues; the failure is on the device
    torch.cuda.synchronize()                                 # completes: no hang, no fault
    with pytest.raises(d.DeslocError) as e:
        eng.step(2, f32r(w.lr), st.views(st.g), clip_bound=1.0)
    assert e.value.status == d.DESLOC_E_DEVICE_WAIT
    with pytest.raises(d.DeslocError) as e:                  # and stays reported
        eng.step_masked(0, f32r(w.lr), st.views(st.g))
    assert e.value.status == d.DESLOC_E_DEVICE_WAIT
    after = [st.to_numpy(b) for b in (st.x, st.u) + ((st.v,) if st.v is not None else ())]
    # aligned full tiles stored nothing; the few ragged tiles (straight from global memory, no
    # wait involved) did their update: most of the state is untouched
    same = np.mean([np.mean(a == b) for a, b in zip(before, after)])
    assert same > 0.9

    d.desloc_testing_set_wait_limit(eng.ctx, -1)            # default limit, failure cleared
    ref = State(w, dev)
    eng2 = make_engine(d, w, ref)
    for b_dst, b_src in zip((ref.x, ref.u) + ((ref.v,) if ref.v is not None else ()),
                            (st.x, st.u) + ((st.v,) if st.v is not None else ())):
        for m in range(w.M):
            b_dst[m].copy_(b_src[m])
    for m in range(w.M):
        ref.g[m].copy_(st.g[m])
    eng.step(2, f32r(w.lr), st.views(st.g), clip_bound=1.0)      # the context works again
    eng2.step(2, f32r(w.lr), ref.views(ref.g), clip_bound=1.0)
    torch.cuda.synchronize()
    assert np.array_equal(st.to_numpy(st.x), ref.to_numpy(ref.x))
    assert not np.array_equal(st.to_numpy(st.x), after[0])
    eng.close(); eng2.close()


@pytest.mark.parametrize("gd", ["bf16", "f32"])
def test_read_outs_after_a_wait_that_ran_out_say_so(gd):
    """Norms whose partial sums were never written are no norms: every read-out reports the failure, and works again once
    it is cleared."""
    import paper_2505_22549_b200 as d
    w = di.Workload("readouts", "adam", 2, (70_000, 4096, 33), gd, "normal1", lr=1e-2, K=(1, 1, 1), seed=2)
    dev = torch.device("cuda:0")
    for step, read in ((lambda e, t, g: e.step_normclip(t, 1e-3, g, 1.0), lambda e: e.grad_norms()),
                       (lambda e, t, g: e.step_diag(t, 1e-3, g), lambda e: e.diag_norms()),
                       (lambda e, t, g: e.step_diag(t, 1e-3, g, max_norm=1.0), lambda e: e.grad_norms())):
        st = State(w, dev)
        eng = make_engine(d, w, st)
        st.fill_grads(0)
        d.desloc_testing_set_staging(eng.ctx, 0)
        step(eng, 0, st.views(st.g))
        assert np.all(np.isfinite(np.concatenate([np.ravel(a) for a in read(eng)])))
        d.desloc_testing_set_wait_limit(eng.ctx, 0)
        step(eng, 1, st.views(st.g))
        with pytest.raises(d.DeslocError) as e:
            read(eng)
        assert e.value.status == d.DESLOC_E_DEVICE_WAIT
        d.desloc_testing_set_wait_limit(eng.ctx, -1)
        step(eng, 2, st.views(st.g))
        read(eng)
        eng.close()


@pytest.mark.parametrize("gd", ["bf16", "f32"])
def test_a_reduction_whose_wait_ran_out_says_so(gd):
    """More parameters than the norms of one launch take, and steps that have no bounded wait of their own: the wait that runs out is the
    reduction's.  Norms and rates of change of incomplete sums are refused, time and again, and the next good ones are right."""
    import paper_2505_22549_b200 as d
    w = di.Workload("reductions", "adam", 2, (150_000, 4096, 33), gd, "normal1", lr=1e-2, K=(1, 1, 1), seed=3)
    dev = torch.device("cuda:0")
    st = State(w, dev)
    eng = make_engine(d, w, st)
    assert d.desloc_testing_kernel_of(d.make_config(2, w.numel, "adam", gd), 7)[0] == "lanes"
    gv = st.views(st.g)
    st.fill_grads(0)
    eng.step_normclip(0, 1e-3, gv, 1.0)
    norms, then = eng.grad_norms(), [[b.clone() for b in row] for row in st.views(st.x)]
    for row in then:
        for b in row:
            b.mul_(0.5)
    for _ in range(8):
        d.desloc_testing_set_wait_limit(eng.ctx, 0)
        with pytest.raises(d.DeslocError) as e:
            eng.rel_change(0, then)
        assert e.value.status == d.DESLOC_E_DEVICE_WAIT
        d.desloc_testing_set_wait_limit(eng.ctx, -1)
        assert np.allclose(eng.rel_change(0, then), 1.0, rtol=1e-5)
    d.desloc_testing_set_wait_limit(eng.ctx, 0)
    eng.step_normclip(1, 1e-3, gv, 1.0)
    with pytest.raises(d.DeslocError) as e:
        eng.grad_norms()
    assert e.value.status == d.DESLOC_E_DEVICE_WAIT
    d.desloc_testing_set_wait_limit(eng.ctx, -1)
    eng.step_normclip(2, 1e-3, gv, 1.0)
    assert np.array_equal(eng.grad_norms()[0], norms[0])
    eng.close()
