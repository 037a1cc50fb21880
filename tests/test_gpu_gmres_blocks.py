"""GMRES(m) in the shared-memory-resident kernel, whose Gram-Schmidt takes the
basis four vectors at a time, against the oracle's one-at-a-time GMRES: x after
a full cycle and three steps of the next.

Sizes: restart lengths around the blocks of 4 and the 32 lanes of the
triangular solve; 1 to 700 rows, so that CTAs and lanes stand empty; MGS
(corrected blocks) and BCGS; every cluster size.

Tolerance: A = I + E with ||E|| <= 0.4, so cond(A) <= 2.4.  Each of the m + 3
steps carries a few eps cond^2 into x: 32 (m + 3) 2.4^2 eps, eps = 1.1e-16,
times ||x||, for both sides."""
import numpy as np
import pytest

import oracle
from tests._gpu import lib_and_device

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53
MS = [1, 2, 3, 4, 5, 7, 8, 9, 31, 33]


@pytest.fixture(scope="module")
def env():
    return lib_and_device()


def _matrix(n, seed):
    """I + four cyclic diagonals of entries in (-0.1, 0.1)."""
    rng = np.random.default_rng(seed)
    rows = [dict() for _ in range(n)]
    for i in range(n):
        rows[i][i] = 1.0
        for o in (1, 5, n // 2, n - 3):
            c = (i + o) % n
            rows[i][c] = rows[i].get(c, 0.0) + rng.uniform(-0.1, 0.1)
    rp = np.cumsum([0] + [len(r) for r in rows]).astype(np.int32)
    col = np.concatenate([np.array(sorted(r), np.int32) for r in rows])
    val = np.concatenate([np.array([r[c] for c in sorted(r)]) for r in rows])
    return dict(n=n, rowptr=rp, col=col, val=val), rng.standard_normal(n)


def _close(x, xo, m):
    assert np.linalg.norm(x - xo) <= 2 * 32 * (m + 3) * 2.4 ** 2 * EPS * np.linalg.norm(xo)


@pytest.mark.parametrize("ortho", [0, 3])
@pytest.mark.parametrize("cl", [2, 4, 8, 16])
@pytest.mark.parametrize("n", [1, 2, 127, 129, 700])
def test_resident_steps_match_oracle(env, n, cl, ortho, monkeypatch):
    import torch
    xb, dev = env
    monkeypatch.setenv("XB_RESIDENT_CL", str(cl))
    A, b = _matrix(n, n)
    plan = xb.Plan(*(torch.as_tensor(A[k], device=dev) for k in ("rowptr", "col", "val")))
    for m in MS:
        x = torch.zeros(n, dtype=torch.float64, device=dev)
        info = plan.gmres(torch.as_tensor(b, device=dev), x, m=m, tol=1e-15, maxiter=m + 3, ortho=ortho)
        assert info["persistent"] == 2
        _close(x.cpu().numpy(), oracle.gmres(A, b, m=m, tol=1e-15, maxiter=m + 3, ortho=ortho)[0], m)
