"""The bounded waits of the orthogonalisation: with one poll a wait, a warp that
finds the value it needs not yet there gives up, the others leave at their next
look, the call reports XB_ETIMEOUT (a bounded wait, no fault), and the plan
stays usable: with the default limit the next call, on another stream too,
returns what another plan does, bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2405_01599_gb300 import gen
from tests._gpu import lib_and_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return lib_and_device()


# w in the CTAs' shared memory, and too long for it; few tiles, and more than stages
@pytest.mark.parametrize("n", [5000, 300_000, 3_300_000])
@pytest.mark.parametrize("method", [0, 1, 2, 3])
def test_sweep_gives_up_and_recovers(env, n, method):
    xb, dev = env
    import torch
    g = torch.Generator(device=dev)
    g.manual_seed(n + method)
    k = 17
    V = torch.randn(k, n, dtype=torch.float64, generator=g, device=dev) / n ** 0.5
    w = torch.randn(n, dtype=torch.float64, generator=g, device=dev)
    plan, other = (xb.Plan.from_host(gen.laplace1d(64), dev) for _ in range(2))
    want = w.clone()
    h = other.orth(V, want, method)
    side = torch.cuda.Stream()
    for s in (torch.cuda.current_stream(), side):
        for _ in range(3):
            plan.orth_config(xb.ORTH_POLLS, 1)
            with pytest.raises(xb.XbError) as e:
                plan.orth(V, w.clone(), method)
            assert e.value.code == xb.XB_ETIMEOUT
            plan.orth_config(xb.ORTH_POLLS, 0)
            u = w.clone()
            torch.cuda.synchronize()
            got = plan.orth(V, u, method, stream=s)
            torch.cuda.synchronize()
            assert torch.equal(got, h) and torch.equal(u, want)


@pytest.mark.parametrize("ortho", [0, 3])
def test_solvers_report_it(env, ortho):
    xb, dev = env
    import torch
    A = gen.convdiff3d(N=20, dims=(23, 21, 20))
    b = torch.tensor(oracle.spmv(A, np.ones(A["n"])), device=dev)
    plan = xb.Plan.from_host(A, dev)
    solves = [lambda x: plan.gmres(b, x, m=20, tol=1e-9, ortho=ortho, small_n=0, maxiter=500),
              lambda x: plan.gmres(b, x, m=20, tol=1e-9, ortho=ortho, precision=xb.PREC_MIXED, maxiter=500),
              lambda x: plan.gmres(b, x, m=20, tol=1e-9, ortho=ortho, precond=xb.PRECOND_ILU0, maxiter=500)]
    for solve in solves:
        plan.orth_config(xb.ORTH_POLLS, 1)
        info = solve(torch.zeros_like(b))
        assert info["status"] == xb.XB_ETIMEOUT, info
        plan.orth_config(xb.ORTH_POLLS, 0)
        x = torch.zeros_like(b)
        assert solve(x)["status"] == 0
        r = b.cpu().numpy() - oracle.spmv(A, x.cpu().numpy())
        assert np.linalg.norm(r) <= 1e-9 * np.linalg.norm(b.cpu().numpy())


def test_eigensolver_reports_it(env):
    xb, dev = env
    A = gen.laplace3d(20)
    plan = xb.Plan.from_host(A, dev)
    plan.orth_config(xb.ORTH_POLLS, 1)
    assert plan.lanczos(2, m=20)[2]["status"] == xb.XB_ETIMEOUT
    plan.orth_config(xb.ORTH_POLLS, 0)
    assert plan.lanczos(2, m=20)[2]["status"] == 0
