"""A batch created on a stream on which its systems' arrays are still being
written: the tiles of mode 1 are cut from the row pointers as they stand there,
so the solve is bit for bit that of a batch whose arrays were complete."""
import numpy as np
import pytest

import oracle
from paper_2405_01599_gb300 import gen
from tests._gpu import lib_and_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [40, 3000, 40_000])  # 40,000: a whole cluster's
def test_row_pointers_still_on_their_way(n):
    xb, dev = lib_and_device()
    import torch
    A = gen.powerlaw(n=n, seed=5) if n > 100 else gen.laplace1d(n)
    t = {k: torch.as_tensor(A[k], device=dev) for k in ("rowptr", "col", "val")}
    b = torch.as_tensor(oracle.spmv(A, np.ones(n)), device=dev)

    def solve(rowptr, s):
        x = torch.zeros(n, dtype=torch.float64, device=dev)
        batch = xb.Batch([dict(t, rowptr=rowptr, b=b, x=x, m=30, mode=1)], stream=s, tol=1e-10, maxiter=90)
        batch.run(stream=s)
        return x, batch.results(stream=s)[0]["iters"]

    want, steps = solve(t["rowptr"], torch.cuda.current_stream())
    late = torch.zeros_like(t["rowptr"])  # until it is written, no row has an entry
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        torch.cuda._sleep(1_000_000_000)
        late.copy_(t["rowptr"], non_blocking=True)
        x, got = solve(late, s)
    torch.cuda.synchronize()
    assert got == steps and torch.equal(x, want)
