"""The bounded waits of the ILU(0) flow substitution, by the kinds of item it
has (a lane a row, a few lanes a row, the warp for a long row, values from
shared memory and from other CTAs): with one poll a wait, a warp gives up as a
whole, the application reports XB_ETIMEOUT (a bounded wait, no fault), and the
next one, on another stream too, returns what another plan does, bit for bit."""
import numpy as np
import pytest

from paper_2405_01599_gb300 import gen
from tests._gpu import lib_and_device

pytestmark = pytest.mark.gpu


def _banded(n, width):
    off = np.arange(-width, width + 1)
    r = np.repeat(np.arange(n), off.size)
    c = r + np.tile(off, n)
    ok = (c >= 0) & (c < n)
    r, c = r[ok], c[ok]
    rp = np.zeros(n + 1, np.int32)
    np.cumsum(np.bincount(r, minlength=n), out=rp[1:])
    return dict(n=n, nnz=int(rp[-1]), rowptr=rp, col=c.astype(np.int32),
                val=np.where(r == c, 4.0 * width, np.sin(1.0 + r * 0.1 + c)), sym_upper=False)


@pytest.mark.parametrize("make", [lambda: gen.poisson2d(80), lambda: gen.powerlaw(n=20_000, seed=4),
                                  lambda: gen.toeplitz3(9000, -1.0, 4.0, -2.0), lambda: _banded(3000, 20),
                                  lambda: _banded(1500, 300)])
def test_gives_up_and_recovers(make):
    xb, dev = lib_and_device()
    import torch
    A = make()
    r = torch.tensor(np.random.default_rng(2).standard_normal(A["n"]), device=dev)
    plan, other = (xb.Plan.from_host(A, dev) for _ in range(2))
    for p in (plan, other):
        p.ilu0_config(1)
        p.ilu0_setup()
    want = other.ilu0_apply(r, torch.empty_like(r))
    torch.cuda.synchronize()
    streams = [torch.cuda.current_stream(), torch.cuda.Stream()]
    for i in range(6):
        plan.ilu0_config(1, barrier_polls=1)
        with pytest.raises(xb.XbError) as e:
            plan.ilu0_apply(r, torch.empty_like(r))
        assert e.value.code == xb.XB_ETIMEOUT
        plan.ilu0_config(1, barrier_polls=0)
        got = plan.ilu0_apply(r, torch.empty_like(r), stream=streams[i % 2])
        torch.cuda.synchronize()
        assert torch.equal(got, want)
