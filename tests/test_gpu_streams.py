"""Plans of several host threads on streams of their own, and a plan beside a
kernel that keeps an SM busy until the plan's calls are over: launches that hold
their SMs together wait for one another, and every result is the one that the
plan returns alone, bit for bit."""
import threading
import time

import numpy as np
import pytest

import oracle
from paper_2405_01599_gb300 import gen
from tests._gpu import lib_and_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return lib_and_device()


def _work(xb, dev, A, m):
    import torch
    b = torch.tensor(oracle.spmv(A, np.ones(A["n"])), device=dev)
    plan = xb.Plan.from_host(A, dev)
    plan.ilu0_setup()

    def go(stream):
        out = []
        for kw in (dict(small_n=0), dict(precond=xb.PRECOND_ILU0), dict(precision=xb.PREC_MIXED)):
            x = torch.zeros_like(b)
            info = plan.gmres(b, x, m=m, tol=1e-9, ortho=xb.ORTHO_MGS, maxiter=400, stream=stream, **kw)
            assert info["status"] == 0, info
            out.append(x)
        return out
    return go


def test_solves_on_two_streams(env):
    xb, dev = env
    import torch
    jobs = [_work(xb, dev, gen.convdiff3d(N=20, dims=(41, 40, 39)), 20),
            _work(xb, dev, gen.convdiff3d(N=20, dims=(70, 69, 68)), 13)]
    want = [go(torch.cuda.current_stream()) for go in jobs]
    torch.cuda.synchronize()
    got, errors = [[], []], []

    def thread(i):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for _ in range(5):
                    got[i].append(jobs[i](s))
                s.synchronize()
        except BaseException as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=thread, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for i in range(2):
        assert len(got[i]) == 5
        for xs in got[i]:
            for x, w in zip(xs, want[i]):
                assert torch.equal(x, w)


@pytest.mark.parametrize("ctas", [2, 7, 64])
@pytest.mark.parametrize("n", [40, 50_000, 1_000_003])
def test_limited_ctas(env, n, ctas):
    """The same sums in another split: within the rounding of n terms."""
    xb, dev = env
    import torch
    g = torch.Generator(device=dev)
    g.manual_seed(n + ctas)
    k = 9
    V = torch.randn(k, n, dtype=torch.float64, generator=g, device=dev)
    V = torch.linalg.inv(torch.linalg.cholesky(V @ V.T)) @ V
    w = torch.randn(n, dtype=torch.float64, generator=g, device=dev)
    w /= w.norm()
    plan = xb.Plan.from_host(gen.laplace1d(64), dev)
    for method in range(4):
        plan.orth_config(xb.ORTH_CTAS, 0)
        a, b = w.clone(), w.clone()
        ha = plan.orth(V, a, method)
        plan.orth_config(xb.ORTH_CTAS, ctas)
        hb = plan.orth(V, b, method)
        tol = 8 * k * np.sqrt(n) * 2.0 ** -53 + 1e-15
        assert float((ha - hb).abs().max()) <= tol and float((a - b).norm()) <= tol
    for bad in (1, -1):
        with pytest.raises(xb.XbError):
            plan.orth_config(xb.ORTH_CTAS, bad)


def test_beside_a_kernel_that_stays(env):
    """One thread of another stream's kernel holds an SM for ~0.4 s; a plan that
    is left the others' SMs does not wait for it."""
    xb, dev = env
    import torch
    A = gen.convdiff3d(N=20, dims=(41, 40, 39))
    plan = xb.Plan.from_host(A, dev)
    plan.orth_config(xb.ORTH_CTAS, torch.cuda.get_device_properties(dev).multi_processor_count - 24)
    plan.ilu0_config(0)
    b = torch.tensor(oracle.spmv(A, np.ones(A["n"])), device=dev)
    x = torch.zeros_like(b)
    solve = lambda s: plan.gmres(b, x.zero_(), m=20, tol=1e-9, precond=xb.PRECOND_ILU0, stream=s)  # noqa: E731
    s, other = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(s):
        assert solve(s)["status"] == 0
        torch.cuda.synchronize()
        with torch.cuda.stream(other):
            torch.cuda._sleep(800_000_000)
            done = torch.cuda.Event()
            done.record()
        t = time.perf_counter()
        assert solve(s)["status"] == 0
        t = time.perf_counter() - t
        assert not done.query(), t  # the solve ended while the kernel stayed
    torch.cuda.synchronize()
