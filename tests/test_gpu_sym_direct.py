"""Symmetric SpMV over tiles (XB_VAR_SYM_TILE) on both sides of its row-length
rule (32 stored entries: rows read straight from memory, longer ones staged) and
at tile edges, against the oracle.  Tolerance per row: 1e-12 of sum |a||x| in
FP64, 2 (k + 2) 6e-8 of it in FP32 (k terms, one rounding each)."""
import numpy as np
import pytest

import oracle
from paper_2405_01599_gb300 import gen
from tests._gpu import lib_and_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return lib_and_device()


def _upper(n, longest, seed):
    """Upper rows of up to `longest` stored entries (the diagonal included),
    near and far columns mixed."""
    rng = np.random.default_rng(seed)
    rp, ci = [0], []
    for i in range(n):
        k = min(longest if i % 7 == 0 else int(rng.integers(1, longest + 1)), n - i)
        near = np.arange(i, min(n, i + (k + 1) // 2))
        rest = np.setdiff1d(np.arange(i, n), near)
        far = rng.choice(rest, size=min(k - near.size, rest.size), replace=False)
        c = np.sort(np.concatenate([near, far]))
        ci.append(c)
        rp.append(rp[-1] + c.size)
    ci = np.concatenate(ci).astype(np.int32)
    return dict(n=n, nnz=ci.size, rowptr=np.array(rp, np.int32), col=ci,
                val=rng.uniform(-1, 1, ci.size), sym_upper=True)


@pytest.mark.parametrize("n", [1, 63, 256, 257, 1025])
@pytest.mark.parametrize("longest", [1, 5, 32, 33])
def test_both_sides_of_the_row_rule(env, n, longest):
    xb, dev = env
    import torch
    A = _upper(n, longest, seed=n + longest)
    F = gen.full_from_upper(A)
    absum = oracle.spmv(dict(F, val=np.abs(F["val"])), np.ones(n))
    k = np.diff(F["rowptr"])
    plan = xb.Plan.from_host(A, dev)
    rng = np.random.default_rng(1)
    x, y0 = rng.uniform(-1, 1, n), rng.uniform(-1, 1, n)
    s = oracle.spmv(F, x)
    for block in (64, 128, 256, 512):
        for alpha, beta in ((1.0, 0.0), (-0.5, 0.0), (1.0, 1.0), (2.0, -0.25)):
            y = torch.tensor(y0 if beta else np.full(n, np.nan), device=dev)
            plan.spmv(torch.tensor(x, device=dev), y, alpha=alpha, beta=beta, variant=xb.VAR_SYM_TILE,
                      block=block, ipt=8)
            ref = alpha * s + (beta * y0 if beta else 0.0)
            assert np.all(np.abs(y.cpu().numpy() - ref) <= 1e-12 * (abs(alpha) * absum + abs(beta) + 1e-300))
    x32 = torch.tensor(x, dtype=torch.float32, device=dev)
    y32 = torch.empty(n, dtype=torch.float32, device=dev)
    plan.spmv_f32(x32, y32)
    ref = oracle.spmv(dict(F, val=F["val"].astype(np.float32).astype(np.float64)), x32.cpu().numpy().astype(np.float64))
    assert np.all(np.abs(y32.cpu().numpy() - ref) <= 2 * (k + 2) * 6e-8 * absum)


def test_two_products_in_a_row(env):
    """The scaling of the second product's y must not overtake the first's sums."""
    xb, dev = env
    import torch
    A = gen.laplace3d(34, upper=True)
    F = gen.full_from_upper(A)
    plan = xb.Plan.from_host(A, dev)
    x = torch.rand(A["n"], dtype=torch.float64, device=dev)
    y, z = torch.empty_like(x), torch.empty_like(x)
    for _ in range(20):
        plan.spmv_sym(x, y)
        plan.spmv_sym(y, z)
        plan.spmv_sym(x, y, alpha=2.0, beta=-1.0)
    s = oracle.spmv(F, x.cpu().numpy())
    t = oracle.spmv(F, s)
    absum = oracle.spmv(dict(F, val=np.abs(F["val"])), np.ones(A["n"]))
    assert np.all(np.abs(y.cpu().numpy() - s) <= 1e-11 * (absum + 1))
    assert np.all(np.abs(z.cpu().numpy() - t) <= 1e-11 * (absum * absum.max() + 1))
