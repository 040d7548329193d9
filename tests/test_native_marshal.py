"""The native marshalling of nested tensor lists: addresses in worker-major order, and the refusals of module.py."""
import ctypes

import pytest
import torch


@pytest.fixture(scope="module")
def native():
    import paper_2505_22549_b200.module as m
    return m._native


@pytest.mark.parametrize("kind,dtype", [(0, torch.float32), (1, torch.bfloat16)])
def test_addresses_are_those_of_the_tensors(native, kind, dtype):
    shapes, M = [(4,), (2, 3), (1,)], 3
    lists = [[torch.zeros(s, dtype=dtype) for s in shapes] for _ in range(M)]
    lists[1][1] = torch.nn.Parameter(lists[1][1])
    table = native.Table([4, 6, 1], M)
    for nested in (lists, tuple(tuple(r) for r in lists)):
        at = table.fill(nested, kind, 1, "misfit")
        got = list((ctypes.c_void_p * 9).from_address(at))
        assert got == [t.data_ptr() for row in lists for t in row]


@pytest.mark.parametrize("spoil", ["dtype", "size", "layout", "workers", "short"])
def test_misfits_are_refused(native, spoil):
    good = lambda: [[torch.zeros(4), torch.zeros(6)] for _ in range(2)]
    table, lists = native.Table([4, 6], 2), good()
    if spoil == "dtype":
        lists[1][0] = torch.zeros(4, dtype=torch.bfloat16)
    elif spoil == "size":
        lists[0][1] = torch.zeros(5)
    elif spoil == "layout":
        lists[0][1] = torch.zeros(12)[::2]
    elif spoil == "workers":
        lists = lists[:1]
    else:
        lists[1] = lists[1][:1]
    with pytest.raises(ValueError):
        table.fill(lists, 0, 0, "misfit")
    assert table.fill(good(), 0, 0, "misfit")
    assert table.fill([[1, 2], [3, 4]], 0, 0, "misfit") is None      # not tensors: the caller says so


def test_binding_gradients_leaves_the_table_of_a_running_step_alone():
    """A step reads its pointers with the interpreter's lock released; a thread that binds the next gradients meanwhile must
    not write into the same buffer."""
    import paper_2505_22549_b200 as d
    eng = d.DesLoc.__new__(d.DesLoc)                       # no context: marshalling only
    eng.ctx, eng.M, eng.numel, eng.grad_dtype = None, 2, [4, 6], d.DESLOC_F32
    eng._tables()
    lists = lambda: [[torch.zeros(4), torch.zeros(6)] for _ in range(2)]
    first, second = lists(), lists()
    at = eng._grad_address(first)
    bound = eng.bind_grads(second)
    want = lambda nested: [t.data_ptr() for row in nested for t in row]
    assert list((ctypes.c_void_p * 4).from_address(at)) == want(first)
    assert list(bound.array) == want(second) and eng.bind_grads(bound) is bound


class _Like:
    """Answers what a step asks of a gradient, but is no torch.Tensor."""

    def __init__(self, t):
        self.t, self.dtype, self.is_cuda = t, t.dtype, t.is_cuda
        self.numel, self.is_contiguous, self.data_ptr = t.numel, t.is_contiguous, t.data_ptr


@pytest.mark.parametrize("where", [0, 1])
def test_objects_like_tensors_are_taken(where):
    import paper_2505_22549_b200 as d
    eng = d.DesLoc.__new__(d.DesLoc)
    eng.ctx, eng.M, eng.numel, eng.grad_dtype = None, 2, [4, 6], d.DESLOC_F32
    eng._tables()
    real = [[torch.zeros(4), torch.zeros(6)] for _ in range(2)]
    like = [[real[0][0], _Like(real[0][1])], [_Like(t) for t in real[1]]]
    want = [t.data_ptr() for row in real for t in row]
    for nested in (like, tuple(like), (row for row in like)):
        at = eng._fill(eng._table, nested, d.DESLOC_F32, where, "misfit")
        assert list((ctypes.c_void_p * 4).from_address(at)) == want
    for spoiled in ([like[0], [_Like(torch.zeros(5)), like[1][1]]], [like[0], [_Like(torch.zeros(4).bfloat16()), like[1][1]]],
                    like[:1], [like[0], like[1][:1]]):
        with pytest.raises(ValueError):
            eng._fill(eng._table, spoiled, d.DESLOC_F32, where, "misfit")


def test_a_module_built_for_another_torch_is_refused():
    """It reads torch's objects directly: another build's layout would be misread in silence."""
    import os
    import subprocess
    import sys
    code = "import torch; torch.__version__ = '0.0.1'\nimport paper_2505_22549_b200.module"
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert r.returncode != 0 and "was built for torch" in r.stderr and "paper_2505_22549_b200.build" in r.stderr
