"""One orthogonalisation of w against k rows (xb_orth, xb_mgs, the Arnoldi step
inside GMRES) at the sizes where its launch shape changes, against the same
Gram-Schmidt in plain FP64 torch.

Sizes: one element, CTAs without elements, the edges of a CTA's 256 elements
and of its tiles, the edges of the cluster-size rule (150,000 and 400,000), of
the MGS block rule (600,000), and a vector too long for the CTAs' shared memory
(3.3M); basis rows around the blocks of 2, 4 and 8 and the 64 values of an
exchange; rows that are not 16-byte aligned.

Tolerance: the rows are orthonormal and ||w|| = 1, so a projection of n terms
carries a rounding error of about sqrt(n) eps and the k of them at most add:
8 k sqrt(n) eps, with eps = 1.1e-16."""
import numpy as np
import pytest

import oracle
from paper_2405_01599_gb300 import gen
from tests._gpu import lib_and_device

pytestmark = pytest.mark.gpu
NAMES = {"mgs": 0, "cgs": 1, "dgks": 2, "bcgs": 3}
EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def env():
    return lib_and_device()


def _case(dev, n, k, ld, shift, seed):
    """k orthonormal rows (stride ld, starting shift elements into a buffer) and w."""
    import torch
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    V = torch.randn(k, n, dtype=torch.float64, generator=g, device=dev)
    if n >= k:
        for _ in range(2):
            V = torch.linalg.qr(V.T, mode="reduced")[0].T.contiguous() if n < 100_000 else \
                torch.linalg.inv(torch.linalg.cholesky(_gram(V))) @ V
    else:
        V = V / V.norm(dim=1, keepdim=True)
    w = torch.randn(n, dtype=torch.float64, generator=g, device=dev)
    w /= w.norm()
    buf = torch.full((shift + k * ld + 2,), float("nan"), dtype=torch.float64, device=dev)
    rows = buf[shift:shift + k * ld].view(k, ld)
    rows[:, :n] = V
    return rows, V, w


def _gram(V):
    import torch
    G = torch.zeros(V.shape[0], V.shape[0], dtype=torch.float64, device=V.device)
    for a in range(0, V.shape[1], 4096):
        G += V[:, a:a + 4096] @ V[:, a:a + 4096].T
    return G


def _reference(V, w, name):
    import torch
    k = V.shape[0]
    block = {"mgs": 1, "bcgs": 4}.get(name, k)
    h = torch.zeros(k + 1, dtype=torch.float64, device=V.device)
    w = w.clone()
    for _ in range(2 if name == "dgks" else 1):
        for i in range(0, k, block):
            c = (V[i:i + block] * w).sum(dim=1)
            w -= c @ V[i:i + block]
            h[i:i + c.numel()] += c
    h[k] = w.norm()
    return w, h


def _check(env, n, k, name, ld=None, shift=0):
    xb, dev = env
    import torch
    ld = ld or n
    rows, V, w = _case(dev, n, k, ld, shift, seed=n + 7 * k)
    plan = xb.Plan.from_host(gen.laplace1d(64), dev)
    wr, hr = _reference(V, w, name)
    tol = 8 * k * np.sqrt(n) * EPS + 1e-15
    for call in (lambda u: plan.orth(rows, u, NAMES[name]),) + \
            ((lambda u: plan.mgs(rows, u),) if name == "mgs" else ()):
        out = w.clone()
        h = call(out)
        assert float((h - hr).abs().max()) <= tol, (n, k, name)
        assert float((out - wr).norm()) <= tol, (n, k, name)
        again = w.clone()
        h2 = call(again)
        assert torch.equal(h, h2) and torch.equal(out, again)


@pytest.mark.parametrize("name", list(NAMES))
@pytest.mark.parametrize("n", [1, 3, 255, 257, 2047, 2049, 30_001, 149_999, 150_000])
def test_sizes(env, n, name):
    _check(env, n, min(n, 9), name)


@pytest.mark.parametrize("name", list(NAMES))
@pytest.mark.parametrize("n", [399_999, 400_000, 599_999, 600_001, 3_300_001])
def test_large_sizes(env, n, name):
    _check(env, n, 6, name)


@pytest.mark.parametrize("name", list(NAMES))
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 7, 8, 16, 17, 63, 64, 65, 130])
def test_row_counts(env, k, name):
    _check(env, 5000, k, name)


@pytest.mark.parametrize("name", list(NAMES))
@pytest.mark.parametrize("n,ld,shift", [(5003, 5003, 0), (5003, 5003, 1), (5000, 5001, 1), (5000, 5008, 0)])
def test_unaligned_rows(env, n, ld, shift, name):
    _check(env, n, 10, name, ld, shift)


@pytest.mark.parametrize("name", ["mgs", "dgks"])
@pytest.mark.parametrize("m", [7, 8, 9, 40])
def test_gmres_step_by_step(env, name, m):
    """The stored inner products of the MGS blocks inside GMRES: the solve takes
    the oracle's number of steps at restart lengths around the block of 8, on a
    system whose rows end inside a tile."""
    xb, dev = env
    import torch
    A = gen.convdiff3d(N=20, dims=(23, 21, 20))
    b = oracle.spmv(A, np.ones(A["n"]))
    _, io = oracle.gmres(A, b, m=m, tol=1e-10, ortho=NAMES[name])
    plan = xb.Plan.from_host(A, dev)
    x = torch.zeros(A["n"], dtype=torch.float64, device=dev)
    info = plan.gmres(torch.tensor(b, device=dev), x, m=m, tol=1e-10, ortho=NAMES[name], small_n=0)
    r = b - oracle.spmv(A, x.cpu().numpy())
    assert info["status"] == 0 and np.linalg.norm(r) <= 1e-10 * np.linalg.norm(b), info
    assert info["persistent"] == 0
    assert abs(info["iters"] - io["iters"]) <= max(3, 0.05 * io["iters"]), (info["iters"], io["iters"])


@pytest.mark.parametrize("name", list(NAMES))
def test_mixed_inner_solve(env, name):
    xb, dev = env
    import torch
    A = gen.convdiff3d(N=24, dims=(27, 25, 24))
    b = oracle.spmv(A, np.ones(A["n"]))
    plan = xb.Plan.from_host(A, dev)
    x = torch.zeros(A["n"], dtype=torch.float64, device=dev)
    info = plan.gmres(torch.tensor(b, device=dev), x, m=30, tol=1e-10, precision=xb.PREC_MIXED,
                      ortho=NAMES[name])
    r = b - oracle.spmv(A, x.cpu().numpy())
    assert info["status"] == 0 and info["fallback"] == 0, info
    assert np.linalg.norm(r) <= 1e-10 * np.linalg.norm(b)


@pytest.mark.parametrize("check_every", [1, 2, 5, 100])
def test_late_look(env, check_every):
    """The host sees a cycle's end one check late and only in the word of the
    step that ended it: the counts are those of the steps taken."""
    xb, dev = env
    import torch
    A = gen.convdiff3d(N=20, dims=(23, 21, 20))
    b = oracle.spmv(A, np.ones(A["n"]))
    plan = xb.Plan.from_host(A, dev)
    infos = []
    for every in (1, check_every):
        for prec in (xb.PREC_FP64, xb.PREC_MIXED):
            x = torch.zeros(A["n"], dtype=torch.float64, device=dev)
            infos.append(plan.gmres(torch.tensor(b, device=dev), x, m=17, tol=1e-9, precision=prec,
                                    check_every=every, small_n=0))
            assert infos[-1]["status"] == 0
    for i, j in ((0, 2), (1, 3)):
        for k in ("iters", "inner_iters", "restarts", "outer"):
            assert infos[i][k] == infos[j][k], k
    # one SpMV per step and per residual, none for the step that did nothing
    assert infos[0]["spmv_calls"] == infos[0]["iters"] + infos[0]["restarts"] + 1
