"""ILU(0) substitution with rows spread over 1 to 32 lanes (four entries a lane
at most), against the oracle and the graph of level launches: triangle rows at
the edges of every number of lanes (4, 8, 16, 32, 64, 128 entries) in one
matrix, with columns of the row's own block, of other blocks and of both, in
one block and in several; and blocks large enough that items are halved.

Tolerance: both paths and the oracle sum a row's terms in FP64 in some order on
diagonally dominant rows: 1e-12 of max |z|, as for the other shapes."""
import numpy as np
import pytest

import oracle
from paper_2405_01599_gb300 import gen
from tests._gpu import lib_and_device

pytestmark = pytest.mark.gpu
LENS = (0, 1, 2, 3, 4, 5, 8, 9, 16, 17, 32, 33, 64, 65, 128, 129, 300)


@pytest.fixture(scope="module")
def env():
    return lib_and_device()


def _mixed(n, near):
    """Row i has LENS[i mod 17] entries on either side of the diagonal (as far as
    there are columns), a share `near` of them among the nearest."""
    rng = np.random.default_rng(n)
    cols = []
    for i in range(n):
        k = LENS[i % len(LENS)]
        c = [i]
        for lo, hi in ((0, i), (i + 1, n)):
            have = min(k, hi - lo)
            close = int(near * have)
            edge = np.arange(hi - close, hi) if hi == i else np.arange(lo, lo + close)
            rest = rng.choice(hi - lo, have, replace=False) + lo
            c.extend(np.unique(np.concatenate([edge, rest]))[:have] if hi > i else
                     np.unique(np.concatenate([edge, rest]))[::-1][:have])
        cols.append(np.sort(np.unique(c)))
    rp = np.cumsum([0] + [len(c) for c in cols]).astype(np.int32)
    col = np.concatenate(cols).astype(np.int32)
    row = np.repeat(np.arange(n), np.diff(rp))
    val = np.where(row == col, 4.0 * np.diff(rp)[row], np.sin(1.0 + row + 3.0 * col))
    return dict(n=n, nnz=int(rp[-1]), rowptr=rp, col=col, val=val, sym_upper=False)


def _both(env, A, r):
    import torch
    xb, dev = env
    plan = xb.Plan.from_host(A, dev)
    z = []
    for mode in (1, 0):
        plan.ilu0_config(mode)
        z.append(plan.ilu0_apply(r, torch.empty_like(r)))
        assert torch.equal(z[-1], plan.ilu0_apply(r, torch.empty_like(r)))
    return z


@pytest.mark.parametrize("n", [40, 700, 9000])
@pytest.mark.parametrize("near", [0.0, 0.5, 1.0])
def test_rows_of_every_number_of_lanes(env, n, near):
    import torch
    A = _mixed(n, near)
    r = np.random.default_rng(2).standard_normal(n)
    flow, graph = _both(env, A, torch.tensor(r, device=env[1]))
    zo = oracle.ilu0_solve(A, oracle.ilu0(A)[0], r)
    for z in (flow, graph):
        assert np.max(np.abs(z.cpu().numpy() - zo)) <= 1e-12 * np.max(np.abs(zo))


def test_large_blocks(env):
    import torch
    A = gen.convdiff3d(N=20, dims=(160, 160, 160))
    g = torch.Generator(device=env[1])
    g.manual_seed(3)
    flow, graph = _both(env, A, torch.randn(A["n"], dtype=torch.float64, generator=g, device=env[1]))
    assert float((flow - graph).abs().max()) <= 1e-12 * float(graph.abs().max())
