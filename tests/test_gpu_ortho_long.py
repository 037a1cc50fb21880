"""The orthogonalisation of long vectors, which takes blocks of as many rows as
there are (up to 2, 4, 8) and more threads from n = 3,000,000 on, and of FP32
bases, which take blocks of 4 from n = 1,500,000 on, on both sides of those lines.

Tolerances: the sweep tests' 8 k sqrt(n) eps for orthonormal rows and ||w|| = 1.
GMRES against the oracle: x after a cycle and two steps with A = I + E, ||E|| <=
0.3, a few eps cond^2 a step as in the block tests, 64 (m + 2) 2.7^2 eps; in an
FP32 basis the refined solution meets tol."""
import numpy as np
import pytest

import oracle
from paper_2405_01599_gb300 import gen
from tests._gpu import lib_and_device
from tests.test_gpu_ortho_sweep import NAMES, _check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return lib_and_device()


@pytest.mark.parametrize("name", list(NAMES))
@pytest.mark.parametrize("n,k", [(n, k) for n in (2_999_999, 3_000_000) for k in (1, 2, 3, 4, 5)] +
                         [(n, k) for n in (3_000_001, 4_100_003) for k in (1, 2, 3, 4, 5, 8, 9, 17)])
def test_rows_of_long_vectors(env, n, k, name):
    _check(env, n, k, name)


@pytest.mark.parametrize("name", ["mgs", "bcgs", "dgks"])
@pytest.mark.parametrize("side", [144, 145])  # 2,985,984 and 3,048,625 rows
def test_gmres_on_long_vectors(env, side, name):
    xb, dev = env
    import torch
    A = gen.laplace3d(side)
    A["val"] = np.where(A["val"] > 0, 1.0, 0.05)  # I + E, ||E|| <= 0.3
    n, m = A["n"], 5
    b = np.random.default_rng(1).standard_normal(n)
    xo, io = oracle.gmres(A, b, m=m, tol=1e-15, maxiter=m + 2, ortho=NAMES[name])
    plan = xb.Plan.from_host(A, dev)
    x = torch.zeros(n, dtype=torch.float64, device=dev)
    info = plan.gmres(torch.tensor(b, device=dev), x, m=m, tol=1e-15, maxiter=m + 2, ortho=NAMES[name])
    assert info["iters"] == io["iters"] == m + 2
    assert np.linalg.norm(x.cpu().numpy() - xo) <= 64 * (m + 2) * 2.7 ** 2 * 2.0 ** -53 * np.linalg.norm(xo)


@pytest.mark.parametrize("name", list(NAMES))
@pytest.mark.parametrize("side", [62, 114, 115])  # 238,328, 1,481,544 and 1,520,875 rows
def test_fp32_basis(env, side, name):
    xb, dev = env
    import torch
    A = gen.laplace3d(side)
    A["val"] = np.where(A["val"] > 0, 1.0, 0.125)
    n = A["n"]
    b = oracle.spmv(A, np.ones(n))
    plan = xb.Plan.from_host(A, dev)
    x = torch.zeros(n, dtype=torch.float64, device=dev)
    info = plan.gmres(torch.tensor(b, device=dev), x, m=12, tol=1e-12, precision=xb.PREC_MIXED, ortho=NAMES[name])
    assert info["status"] == 0 and info["fallback"] == 0, info
    r = b - oracle.spmv(A, x.cpu().numpy())
    assert np.linalg.norm(r) <= 1e-12 * np.linalg.norm(b)
    other = xb.Plan.from_host(A, dev)
    y = torch.zeros_like(x)
    ref = other.gmres(torch.tensor(b, device=dev), y, m=12, tol=1e-12, ortho=xb.ORTHO_DGKS)
    assert ref["status"] == 0 and info["inner_iters"] <= 2 * ref["iters"] + 12, (info, ref)
