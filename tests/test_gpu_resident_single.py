"""Resident GMRES with MGS on both sides of the cycle lengths up to which it takes a
vector at a time (5, 10, 13 steps for 1, 2, 4 and more rows a thread), against the
oracle's one-at-a-time GMRES: x after a full cycle and three steps of the next.

Tolerance: that of the blocks' tests, 32 (m + 3) 2.7^2 eps ||x|| for both sides."""
import pytest

import oracle
from tests._gpu import lib_and_device
from tests.test_gpu_gmres_blocks import _close, _matrix

pytestmark = pytest.mark.gpu


# rows a thread: 1, 1, 2, 4, 8, 8
@pytest.mark.parametrize("cl,n", [(2, 256), (16, 2048), (16, 2049), (2, 1024), (2, 1025), (2, 2047)])
def test_both_sides_match_oracle(cl, n, monkeypatch):
    xb, dev = lib_and_device()
    import torch
    monkeypatch.setenv("XB_RESIDENT_CL", str(cl))
    A, b = _matrix(n, n + cl)
    plan = xb.Plan(*(torch.as_tensor(A[k], device=dev) for k in ("rowptr", "col", "val")))
    for m in (2, 5, 6, 10, 11, 13, 14):
        x = torch.zeros(n, dtype=torch.float64, device=dev)
        info = plan.gmres(torch.as_tensor(b, device=dev), x, m=m, tol=1e-15, maxiter=m + 3, ortho=0)
        assert info["persistent"] == 2
        _close(x.cpu().numpy(), oracle.gmres(A, b, m=m, tol=1e-15, maxiter=m + 3, ortho=0)[0], m)
