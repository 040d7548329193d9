"""Worker means divide by the count with a corrected reciprocal: every count against the exact quotient.  One worker holds the
value and the others zero, so the sum is the value itself; the step has learning rate zero."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts", [range(2, 17), range(17, 257)])
def test_quotients_of_every_count(counts):
    import paper_2505_22549_b200 as d
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(1)
    n = 4096
    # random mantissas over exponents from -60 to 60, both signs: all quotients are normal numbers
    v = (torch.rand(n, device=dev, generator=gen) + 1) * torch.exp2(torch.randint(-60, 61, (n,), device=dev, generator=gen).float())
    v[::2].neg_()
    g = torch.zeros(n, device=dev)
    for M in counts:
        x, u = torch.zeros(M, n, device=dev), torch.zeros(M, n, device=dev)
        x[M // 2] = v
        eng = d.DesLoc([[r] for r in x], [[r] for r in u], None, opt="sgdm", grad_dtype="f32", K=(1, 1, 1))
        eng.step(0, 0.0, [[g]] * M)
        want = (v.cpu().numpy().astype(np.float64) / M).astype(np.float32)
        got = x.cpu().numpy()
        assert np.array_equal(got, np.broadcast_to(want, got.shape)), M
        eng.close()
