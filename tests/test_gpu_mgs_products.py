"""Modified Gram-Schmidt in blocks: the dots of a block are taken with one w and
corrected by the rows' own inner products.  With rows that are far from
orthogonal, or a w that is large along the first of them, the corrections decide
the result, and a sweep without them (block CGS) misses it by far.

Sweeps (xb_mgs, xb_orth): unit rows with products of 0.2-0.5, and rows of norm
0.7-1.2 with the same angles, against MGS one row at a time in FP64 torch, at
row counts around the blocks of 2, 4 and 8 and on both sides of the lines by
length.  Every operator I - V_i V_i^T has norm 1 here, so an error is not
amplified from row to row; inside a block a coefficient's error reaches the next
ones by at most a factor 1 + 0.72 each (product times norm squared), 5 over a
block of 4.  A dot of n terms carries sqrt(n) eps: 40 k sqrt(n) eps in all.

GMRES (the products that are kept from step to step): A = B + s u v^T with u = b /
||b||, so every A v_j is s times as large along v_0 as beyond it.  Rounding leaves
(v_0, v_i) ~ eps s; MGS keeps the coefficients on the other vectors exact to eps s,
block CGS to s eps s only.  x after m steps against the oracle's: 32 eps s
(measured on the host: 0.03 eps s); block CGS misses that 100 times over.  In an
FP32 basis 4 eps s, missed 10 times over."""
import numpy as np
import pytest

import oracle
from paper_2405_01599_gb300 import gen
from tests._gpu import lib_and_device

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def env():
    return lib_and_device()


def _gram_schmidt(V, w, block):
    import torch
    w, h = w.clone(), []
    for i in range(0, V.shape[0], block):
        c = (V[i:i + block] * w).sum(dim=1)
        w -= (c[:, None] * V[i:i + block]).sum(dim=0)
        h.append(c)
    return w, torch.cat(h + [w.norm()[None]])


@pytest.mark.parametrize("scaled", [False, True])
@pytest.mark.parametrize("k", [2, 3, 4, 5, 8, 9])
@pytest.mark.parametrize("n", [7, 300, 50_003, 599_999, 700_001, 3_000_001])
def test_rows_far_from_orthogonal(env, n, k, scaled):
    xb, dev = env
    import torch
    g = torch.Generator(device=dev)
    g.manual_seed(n + k)
    V = torch.randn(k, n, dtype=torch.float64, generator=g, device=dev) / n ** 0.5
    V += 0.8 * torch.randn(1, n, dtype=torch.float64, generator=g, device=dev) / n ** 0.5
    V /= V.norm(dim=1, keepdim=True)
    if scaled:
        V *= torch.linspace(0.7, 1.2, k, dtype=torch.float64, device=dev)[:, None]
    w = V.sum(dim=0) + torch.randn(n, dtype=torch.float64, generator=g, device=dev) / n ** 0.5
    w /= w.norm()
    wr, hr = _gram_schmidt(V, w, 1)
    tol = 40 * k * np.sqrt(n) * EPS
    wb, hb = _gram_schmidt(V, w, k)
    assert float((hb - hr).abs().max()) > 1e6 * tol  # without the corrections
    plan = xb.Plan.from_host(gen.laplace1d(64), dev)
    for call in (lambda u: plan.orth(V, u, xb.ORTHO_MGS), lambda u: plan.mgs(V, u)):
        u = w.clone()
        h = call(u)
        assert float((h - hr).abs().max()) <= tol and float((u - wr).norm()) <= tol, (n, k)


def _system(n, s, seed, single):
    """Rows of n entries; exact in FP32 when single."""
    rng = np.random.default_rng(seed)
    b = rng.standard_normal(n)
    if single:
        b = b.astype(np.float32).astype(np.float64)
    M = np.eye(n) + 0.3 * rng.standard_normal((n, n)) / np.sqrt(n)
    v = rng.standard_normal(n)
    M += s * np.outer(b / np.linalg.norm(b), v / np.linalg.norm(v))
    if single:
        M = M.astype(np.float32).astype(np.float64)
    A = dict(n=n, nnz=n * n, rowptr=np.arange(0, n * n + 1, n, dtype=np.int32),
             col=np.tile(np.arange(n, dtype=np.int32), n), val=M.ravel().copy(), sym_upper=False)
    return A, b


def _distance(x, xo):
    return np.linalg.norm(x - xo) / np.linalg.norm(xo)


@pytest.mark.parametrize("path", ["resident", "multi", "batch CTA", "batch cluster"])
@pytest.mark.parametrize("m", [3, 4, 5, 8, 9, 12, 17])
def test_products_kept_in_gmres(env, m, path, monkeypatch):
    xb, dev = env
    import torch
    s = 1e6
    A, b = _system(60, s, 3, False)
    t = {k: torch.as_tensor(A[k], device=dev) for k in ("rowptr", "col", "val")}
    bt = torch.tensor(b, device=dev)
    plan = xb.Plan(t["rowptr"], t["col"], t["val"])
    xo = oracle.gmres(A, b, m=m, tol=1e-300, maxiter=m, ortho=0)[0]
    tol = 32 * EPS * s
    got = {}
    for ortho in (0, 3):
        x = torch.zeros_like(bt)
        if path.startswith("batch"):
            monkeypatch.setenv("XB_BATCH_COOP_MIN_N", "1" if path.endswith("cluster") else "1000000000")
            for mode in (0, 1):
                x = torch.zeros_like(bt)
                bat = xb.Batch([dict(t, b=bt, x=x, m=m, mode=mode)], tol=1e-300, maxiter=m, ortho=ortho)
                bat.run()
                bat.results()
                got.setdefault(ortho, []).append(_distance(x.cpu().numpy(), xo))
        else:
            info = plan.gmres(bt, x, m=m, tol=1e-300, maxiter=m, ortho=ortho,
                              **(dict(small_n=0) if path == "multi" else {}))
            assert info["persistent"] == (0 if path == "multi" else 2) and info["iters"] == m
            got[ortho] = [_distance(x.cpu().numpy(), xo)]
    assert max(got[0]) <= tol, got
    assert min(got[3]) > 100 * tol, got


@pytest.mark.parametrize("m", [3, 5, 8, 9])
def test_products_kept_in_fp32(env, m):
    xb, dev = env
    import torch
    s = 1e4
    A, b = _system(60, s, 3, True)
    plan = xb.Plan.from_host(A, dev)
    bt = torch.tensor(b, device=dev)
    xo = oracle.gmres(A, b, m=m, tol=1e-300, maxiter=m, ortho=0)[0]
    tol = 4 * 2.0 ** -24 * s
    got = {}
    for ortho in (0, 3):
        x = torch.zeros_like(bt)
        info = plan.gmres(bt, x, m=m, tol=1e-300, ortho=ortho, precision=xb.PREC_MIXED, max_outer=1,
                          tol_inner=1e-30, maxiter_inner=m)
        assert info["inner_iters"] == m and info["outer"] == 1, info
        got[ortho] = _distance(x.cpu().numpy(), xo)
    assert got[0] <= tol, got
    assert got[3] > 10 * tol, got
