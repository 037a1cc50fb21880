"""The byte and memory counts of a solve (bytes_alg, mem_bytes): what one more
Arnoldi step of a cycle adds is its SpMV, each basis row twice and w in and out
(n is small enough for the CTAs to hold w) and one more row in x's update; an
ILU(0) adds what its arrays hold, and its path's traffic."""
import numpy as np
import pytest

import oracle
from paper_2405_01599_gb300 import gen
from tests._gpu import lib_and_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return lib_and_device()


def _solve(xb, plan, b, steps, **kw):
    import torch
    x = torch.zeros_like(b)
    info = plan.gmres(b, x, m=40, tol=1e-300, maxiter=steps, small_n=0, **kw)
    assert info["iters"] == steps
    return info


@pytest.mark.parametrize("ortho,rounds", [(0, 1), (1, 1), (2, 2), (3, 1)])
def test_bytes_of_a_step(env, ortho, rounds):
    xb, dev = env
    import torch
    A = gen.convdiff3d(N=20, dims=(23, 21, 20))
    n, nnz = A["n"], A["nnz"]
    b = torch.tensor(oracle.spmv(A, np.ones(n)), device=dev)
    plan = xb.Plan.from_host(A, dev)
    infos = [_solve(xb, plan, b, k, ortho=ortho) for k in (8, 9, 10)]
    spmv = 12 * nnz + 4 * (n + 1) + 16 * n
    for k, (a, c) in zip((9, 10), zip(infos, infos[1:])):
        assert c["bytes_alg"] - a["bytes_alg"] == spmv + 8 * n * (2 * rounds * k + 2) + 8 * n


def test_ilu_counts(env):
    xb, dev = env
    import torch
    A = gen.convdiff3d(N=20, dims=(23, 21, 20))
    n, nnz = A["n"], A["nnz"]
    b = torch.tensor(oracle.spmv(A, np.ones(n)), device=dev)
    plain = _solve(xb, xb.Plan.from_host(A, dev), b, 5)
    got = {}
    for mode in (1, 0):
        plan = xb.Plan.from_host(A, dev)
        plan.ilu0_config(mode)
        got[mode] = _solve(xb, plan, b, 5, precond=xb.PRECOND_ILU0)
    # factors, diagonal positions and a vector; the flow path's entries, rows,
    # pivots twice and published values of both triangles
    least = 8 * nnz + 12 * n + 12 * (nnz - n) + 8 * n + 16 * n + 32 * n
    for mode in (1, 0):
        assert got[mode]["mem_bytes"] - plain["mem_bytes"] >= least, mode
    # the graph path's ELL copies of both triangles, its rows, pivots and result
    assert got[0]["mem_bytes"] - got[1]["mem_bytes"] >= 12 * (nnz - n) + 8 * n + 16 * n
    applied = {m: got[m]["bytes_alg"] - plain["bytes_alg"] for m in got}
    # six applications (five steps and the update of x): entries, rows, r, z,
    # pivots, published values
    assert 6 * (12 * (nnz - n) + 88 * n) <= applied[1] <= 6 * (16 * nnz + 200 * n) + 200 * n
    assert applied[0] != applied[1]
