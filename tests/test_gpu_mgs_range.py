"""MGS against rows whose inner products with one another leave the FP64 range while
w is orthogonal to some or all of them: h and w are those of one row at a time."""
import pytest

from paper_2405_01599_gb300 import gen
from tests._gpu import lib_and_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [64, 700_001])  # blocks of 4, blocks of 2
def test_products_out_of_range(n):
    xb, dev = lib_and_device()
    import torch
    V = torch.zeros(6, n, dtype=torch.float64, device=dev)
    for i in range(5):  # the first five share their elements 0 .. i
        V[i, :i + 1] = 1e200
    V[5, n - 1] = 1.0
    plan = xb.Plan.from_host(gen.laplace1d(64), dev)
    for at, h5 in ((None, 0.0), (n - 2, 0.0), (n - 1, 2.0)):
        w = torch.zeros(n, dtype=torch.float64, device=dev)
        if at is not None:
            w[at] = 2.0
        left = w.clone()
        left[n - 1] -= h5
        want = torch.tensor([0.0] * 5 + [h5, float(left.norm())], dtype=torch.float64, device=dev)
        for call in (plan.mgs, lambda V, u: plan.orth(V, u, xb.ORTHO_MGS)):
            u = w.clone()
            assert torch.equal(call(V, u), want) and torch.equal(u, left), (n, at)
