"""The flow substitution of ILU(0) (one launch in which every row waits for the
values it needs) against the oracle and against the graph of level launches, at
the shapes where its layout changes: one row, no off-diagonal entries, a chain
of n levels, rows longer than a lane's share and than a warp's group, a row and
a column that hold everything, blocks of one and of many CTAs, a block whose
values shared memory does not hold, overlapping operands, NaN and infinity.

Tolerance: the factors are the same bits on both paths; a substitution's rows
are sums of k terms in FP64, so the two paths differ by rounding: 1e-12 of
max |z| on these diagonally dominant systems (the oracle tests' own bound is
1e-10)."""
import numpy as np
import pytest

import oracle
from paper_2405_01599_gb300 import gen
from tests._gpu import lib_and_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return lib_and_device()


def _crs(n, rows, cols, vals):
    o = np.lexsort((cols, rows))
    rp = np.zeros(n + 1, np.int32)
    np.cumsum(np.bincount(rows, minlength=n), out=rp[1:])
    return dict(n=n, nnz=int(rp[-1]), rowptr=rp, col=np.asarray(cols, np.int32)[o],
                val=np.asarray(vals, np.float64)[o], sym_upper=False)


def _arrow(n):
    """A full first and last row and column."""
    i = np.arange(1, n - 1)
    r = np.concatenate([np.zeros(n, int), np.full(n, n - 1), i, i, i])
    c = np.concatenate([np.arange(n), np.arange(n), np.zeros(n - 2, int), i, np.full(n - 2, n - 1)])
    v = np.where(r == c, 4.0 * n, np.cos(r + 3.0 * c))
    return _crs(n, r, c, v)


def _banded(n, width):
    """Every row has min(i, width) entries left and right of the diagonal."""
    off = np.arange(-width, width + 1)
    r = np.repeat(np.arange(n), off.size)
    c = r + np.tile(off, n)
    ok = (c >= 0) & (c < n)
    r, c = r[ok], c[ok]
    return _crs(n, r, c, np.where(r == c, 4.0 * width, np.sin(1.0 + r * 0.1 + c)))


MATS = [
    ("one", lambda: _crs(1, np.array([0]), np.array([0]), [2.0])),
    ("diagonal", lambda: _crs(5000, np.arange(5000), np.arange(5000), np.arange(5000) + 1.0)),
    ("chain", lambda: gen.toeplitz3(9000, -1.0, 4.0, -2.0)),
    ("arrow", lambda: _arrow(3000)),
    ("band3", lambda: _banded(3000, 3)),
    ("band5", lambda: _banded(3000, 5)),
    ("band32", lambda: _banded(2500, 32)),
    ("band33", lambda: _banded(2500, 33)),
    ("band300", lambda: _banded(1500, 300)),
    ("box", lambda: gen.convdiff3d(N=20, dims=(31, 17, 23))),
    ("plane2049", lambda: gen.convdiff3d(N=20, dims=(683, 3, 1))),
    ("powerlaw", lambda: gen.powerlaw(n=30000, seed=4)),
]


@pytest.mark.parametrize("name,make", MATS)
def test_flow_matches_graph_and_oracle(env, name, make):
    xb, dev = env
    import torch
    A = make()
    plan = xb.Plan.from_host(A, dev)
    r = np.random.default_rng(1).standard_normal(A["n"])
    rt = torch.tensor(r, device=dev)
    z = {}
    for mode in (1, 0, -1):
        plan.ilu0_config(mode)
        z[mode] = plan.ilu0_apply(rt, torch.empty_like(rt)).cpu().numpy()
        again = plan.ilu0_apply(rt, torch.empty_like(rt)).cpu().numpy()
        assert np.array_equal(z[mode], again)
    zo = oracle.ilu0_solve(A, oracle.ilu0(A)[0], r)
    scale = np.max(np.abs(zo))
    assert np.max(np.abs(z[1] - zo)) <= 1e-12 * scale
    assert np.max(np.abs(z[0] - zo)) <= 1e-12 * scale
    assert np.array_equal(z[1], z[-1])


def test_blocks_too_large_for_shared_memory(env):
    xb, dev = env
    import torch
    A = gen.convdiff3d(N=20, dims=(2100, 2200, 1))  # 4.6M rows: more than a CTA's share holds
    plan = xb.Plan.from_host(A, dev)
    g = torch.Generator(device=dev)
    g.manual_seed(3)
    r = torch.randn(A["n"], dtype=torch.float64, generator=g, device=dev)
    z = []
    for mode in (1, 0):
        plan.ilu0_config(mode)
        z.append(plan.ilu0_apply(r, torch.empty_like(r)))
    assert float((z[0] - z[1]).abs().max()) <= 1e-12 * float(z[1].abs().max())


def test_operands(env):
    """Overlapping r and z, several right-hand sides in turn, and non-finite
    values, which reach the rows that depend on them and no others."""
    xb, dev = env
    import torch
    A = gen.convdiff3d(N=12, dims=(13, 12, 11))
    n = A["n"]
    lu, _ = oracle.ilu0(A)
    plan = xb.Plan.from_host(A, dev)
    rng = np.random.default_rng(5)
    for _ in range(3):
        r = rng.standard_normal(n)
        buf = torch.zeros(n + 7, dtype=torch.float64, device=dev)
        buf[7:] = torch.tensor(r, device=dev)
        z = plan.ilu0_apply(buf[7:], buf[:n]).cpu().numpy()
        zo = oracle.ilu0_solve(A, lu, r)
        assert np.max(np.abs(z - zo)) <= 1e-12 * np.max(np.abs(zo))
    D = _crs(4, np.arange(4), np.arange(4), [2.0, 4.0, 8.0, 1e-300])
    pd = xb.Plan.from_host(D, dev)
    z = pd.ilu0_apply(torch.tensor([np.nan, np.inf, 1.0, 1e-300], dtype=torch.float64, device=dev),
                      torch.empty(4, dtype=torch.float64, device=dev)).cpu().numpy()
    assert np.isnan(z[0]) and z[1] == np.inf and z[2] == 0.125 and z[3] == 1.0
    bits = torch.tensor([-1, 0, 0, 0], device=dev).view(torch.float64)  # the NaN of all ones
    z = pd.ilu0_apply(bits, torch.empty(4, dtype=torch.float64, device=dev)).cpu().numpy()
    assert np.isnan(z[0]) and z[2] == 0.0
