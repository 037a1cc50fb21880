"""The numbers that the exchanges of an orthogonalisation carry, where the count
passes 2^32: the sums are those of any other number, bit for bit (they are
taken in a fixed order), for the first, a middle and the last exchange of a
launch, and also when a slot last held a number that comes up again."""
import pytest

from paper_2405_01599_gb300 import gen
from tests._gpu import lib_and_device

pytestmark = pytest.mark.gpu
LAST = 2 ** 32 - 1


@pytest.mark.parametrize("k,method", [(3, 0), (12, 0), (12, 3), (70, 1), (70, 2)])
def test_numbers_pass_the_largest(k, method):
    xb, dev = lib_and_device()
    import torch
    g = torch.Generator(device=dev)
    g.manual_seed(k)
    plan = xb.Plan.from_host(gen.laplace1d(64), dev)
    cases = []
    for n in (200_003, 300):  # many clusters, then one
        V = torch.randn(k, n, dtype=torch.float64, generator=g, device=dev) / n ** 0.5
        w = torch.randn(n, dtype=torch.float64, generator=g, device=dev)
        cases.append((V, w))

    def go(V, w):
        u = w.clone()
        return plan.orth(V, u, method), u

    plan.orth_config(xb.ORTH_NUMBER, 0)
    want = [go(*c) for c in cases]  # the slots of many clusters hold numbers from 1 on
    for before in range(2 * (k // 4 + 3)):
        plan.orth_config(xb.ORTH_NUMBER, 0)
        go(*cases[0])
        plan.orth_config(xb.ORTH_NUMBER, LAST - before)
        for i in (1, 0, 1, 0):
            h, u = go(*cases[i])
            assert torch.equal(h, want[i][0]) and torch.equal(u, want[i][1]), (before, i)


def test_controls_out_of_range():
    xb, dev = lib_and_device()
    plan = xb.Plan.from_host(gen.laplace1d(64), dev)
    for what, value in ((-1, 0), (99, 0), (xb.ORTH_NUMBER, -1), (xb.ORTH_NUMBER, LAST + 1)):
        with pytest.raises(Exception):
            plan.orth_config(what, value)
