"""Batched MGS on both sides of the line from which a CTA takes the basis a vector
at a time instead of in corrected blocks of 4 (1.5 m (m + 100) rows on one CTA,
2.4 m (m + 100) a CTA in a cluster), and around the 512 and 2048 rows that a
CTA's threads have on their way, against the oracle's one-at-a-time GMRES: x
after a full cycle and three steps of the next.

Tolerance: as for the blocks, 32 (m + 3) 2.7^2 eps ||x|| for both sides, with
cond(A) <= 2.7 (I plus four cyclic diagonals)."""
import numpy as np
import pytest

import oracle
from paper_2405_01599_gb300 import gen
from tests._gpu import lib_and_device
from tests.test_gpu_gmres_blocks import _close, _matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("coop_min,m,sizes", [
    ("1000000000", 3, (463, 464, 511, 512, 513)),
    ("1000000000", 5, (787, 788, 2047, 2048, 2049, 2560, 2561)),
    ("1000000000", 10, (1649, 1650, 4097)),
    ("1", 3, (5928, 5929)),
    ("1", 5, (10_080, 10_081)),
    ("", 3, (463, 464, 5929)),
])
def test_both_sides_match_oracle(coop_min, m, sizes, monkeypatch):
    xb, dev = lib_and_device()
    import torch
    if coop_min:
        monkeypatch.setenv("XB_BATCH_COOP_MIN_N", coop_min)
    mats = [_matrix(n, 10 * m + n) for n in sizes]
    for mode in (0, 1):
        systems = [dict(rowptr=torch.as_tensor(A["rowptr"], device=dev), col=torch.as_tensor(A["col"], device=dev),
                        val=torch.as_tensor(A["val"], device=dev), b=torch.as_tensor(b, device=dev),
                        x=torch.zeros(A["n"], dtype=torch.float64, device=dev), m=m, mode=mode) for A, b in mats]
        xb.Batch(systems, tol=1e-15, maxiter=m + 3, ortho=0).run()
        for s, (A, b) in zip(systems, mats):
            _close(s["x"].cpu().numpy(), oracle.gmres(A, b, m=m, tol=1e-15, maxiter=m + 3, ortho=0)[0], m)


def test_restart_length_that_grows():
    """The choice is made for the first length; the restart rule may pass the line."""
    xb, dev = lib_and_device()
    import torch
    A = gen.poisson2d(24)  # 576 rows: singly from m = 3 on down, in blocks beyond
    b = oracle.spmv(A, np.ones(A["n"]))
    systems = [dict(rowptr=torch.as_tensor(A["rowptr"], device=dev), col=torch.as_tensor(A["col"], device=dev),
                    val=torch.as_tensor(A["val"], device=dev), b=torch.as_tensor(b, device=dev),
                    x=torch.zeros(A["n"], dtype=torch.float64, device=dev), m=3, mode=0)]
    bt = xb.Batch(systems, tol=1e-10, maxiter=6000, ortho=0, dafrt=1, m_max=40)
    bt.run()
    info = bt.results()[0]
    assert info["m"] > 3, info
    r = b - oracle.spmv(A, systems[0]["x"].cpu().numpy())
    assert info["status"] == 0, info
    assert np.linalg.norm(r) <= 1e-9 * np.linalg.norm(b)
