"""GMRES(m) in the shared-memory-resident and the batched kernel, whose
Gram-Schmidt takes the basis four vectors at a time, against the oracle's
one-at-a-time GMRES: x after a full cycle and three steps of the next.

Sizes: restart lengths around the blocks of 4 and the 32 lanes of the
triangular solve; 1 to 2049 rows, so that CTAs and lanes stand empty; MGS
(corrected blocks) and BCGS; every cluster size; batched in one CTA, in
a cluster and by the default rule, there with rows of up to 1025 entries, which
mode 1's tiles of 256 cut, and rows without entries.  A batched system of one row
at values near the ends of the FP64 range converges as at 1.

Tolerance: A = I + E with ||E|| <= 0.45, so cond(A) <= 2.7.  Each of the m + 3
steps carries a few eps cond^2 into x: 32 (m + 3) 2.7^2 eps, eps = 1.1e-16,
times ||x||, for both sides."""
import numpy as np
import pytest

import oracle
from tests._gpu import lib_and_device

pytestmark = pytest.mark.gpu
LONG = (9, 17, 33, 63, 64, 65, 255, 1023, 1024, 1025)
EPS = 2.0 ** -53
MS = [1, 2, 3, 4, 5, 7, 8, 9, 31, 32, 33, 64]


@pytest.fixture(scope="module")
def env():
    return lib_and_device()


def _matrix(n, seed, long=()):
    """I + four cyclic diagonals of entries in (-0.1, 0.1); long: the numbers of
    entries (of 1e-4 at most) added to the rows 3, 20, 37, ..."""
    rng = np.random.default_rng(seed)
    rows = [dict() for _ in range(n)]
    for i in range(n):
        rows[i][i] = 1.0
        for o in (1, 5, n // 2, n - 3):
            c = (i + o) % n
            rows[i][c] = rows[i].get(c, 0.0) + rng.uniform(-0.1, 0.1)
    for i, k in enumerate(long):
        r = rows[3 + 17 * i]
        for c in rng.permutation(n)[:k]:
            if len(r) < k:
                r.setdefault(int(c), rng.uniform(-1e-4, 1e-4))
    b = rng.standard_normal(n)
    if long:  # rows without entries (and b = 0 there), alone and several at a time
        for i in [0, 1, 2, n - 1] + list(range(300, 340)) + list(range(400, n, 97)):
            rows[i] = {}
            b[i] = 0.0
    rp = np.cumsum([0] + [len(r) for r in rows]).astype(np.int32)
    col = np.concatenate([np.array(sorted(r), np.int32) for r in rows])
    val = np.concatenate([np.array([r[c] for c in sorted(r)]) for r in rows])
    return dict(n=n, rowptr=rp, col=col, val=val), b


def _close(x, xo, m):
    assert np.linalg.norm(x - xo) <= 2 * 32 * (m + 3) * 2.7 ** 2 * EPS * np.linalg.norm(xo)


@pytest.mark.parametrize("ortho", [0, 3])
@pytest.mark.parametrize("cl", [2, 4, 8, 16])
@pytest.mark.parametrize("n", [1, 2, 127, 129, 700])
def test_resident_steps_match_oracle(env, n, cl, ortho, monkeypatch):
    import torch
    xb, dev = env
    monkeypatch.setenv("XB_RESIDENT_CL", str(cl))
    A, b = _matrix(n, n)
    plan = xb.Plan(*(torch.as_tensor(A[k], device=dev) for k in ("rowptr", "col", "val")))
    for m in MS[:9]:
        x = torch.zeros(n, dtype=torch.float64, device=dev)
        info = plan.gmres(torch.as_tensor(b, device=dev), x, m=m, tol=1e-15, maxiter=m + 3, ortho=ortho)
        assert info["persistent"] == 2
        _close(x.cpu().numpy(), oracle.gmres(A, b, m=m, tol=1e-15, maxiter=m + 3, ortho=ortho)[0], m)


def _route(monkeypatch, coop_min):
    if coop_min:
        monkeypatch.setenv("XB_BATCH_COOP_MIN_N", coop_min)
    else:
        monkeypatch.delenv("XB_BATCH_COOP_MIN_N", raising=False)


@pytest.mark.parametrize("ortho", [0, 3])
@pytest.mark.parametrize("coop_min", ["", "1", "1000000000"])
def test_batch_steps_match_oracle(env, coop_min, ortho, monkeypatch):
    import torch
    xb, dev = env
    _route(monkeypatch, coop_min)
    for m in MS:
        mats = [_matrix(n, 10 * m + n, LONG if n > 1024 else ())
                for n in (1, 2, 3, 31, 511, 512, 513, 1024, 1025, 2049)]
        systems = [dict(rowptr=torch.as_tensor(A["rowptr"], device=dev), col=torch.as_tensor(A["col"], device=dev),
                        val=torch.as_tensor(A["val"], device=dev), b=torch.as_tensor(b, device=dev),
                        x=torch.zeros(A["n"], dtype=torch.float64, device=dev), m=m, mode=i % 2)
                   for i, (A, b) in enumerate(mats)]
        xb.Batch(systems, tol=1e-15, maxiter=m + 3, ortho=ortho).run()
        for s, (A, b) in zip(systems, mats):
            _close(s["x"].cpu().numpy(), oracle.gmres(A, b, m=m, tol=1e-15, maxiter=m + 3, ortho=ortho)[0], m)


@pytest.mark.parametrize("coop_min", ["", "1", "1000000000"])
def test_batch_one_row_over_the_range(env, coop_min, monkeypatch):
    import torch
    xb, dev = env
    _route(monkeypatch, coop_min)
    vals = [1.0, 2.0 ** -900, 2.0 ** -500, 2.0 ** 500, 2.0 ** 900]
    systems = [dict(rowptr=torch.tensor([0, 1], dtype=torch.int32, device=dev),
                    col=torch.zeros(1, dtype=torch.int32, device=dev),
                    val=torch.tensor([v], dtype=torch.float64, device=dev),
                    b=torch.ones(1, dtype=torch.float64, device=dev),
                    x=torch.zeros(1, dtype=torch.float64, device=dev), m=4, mode=0) for v in vals]
    bt = xb.Batch(systems, tol=1e-12, maxiter=50)
    bt.run()
    for s, r, v in zip(systems, bt.results(), vals):
        assert r["status"] == 0 and s["x"].item() * v == 1.0
