"""The launch shapes that the symmetric tile variant takes and refuses are the
same for short rows (read straight from memory) and longer ones (staged)."""
import numpy as np
import pytest

import oracle
from paper_2405_01599_gb300 import gen
from tests._gpu import assert_rows_close, lib_and_device, row_bound

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_row", [3, 40])
def test_items_per_thread(per_row):
    xb, dev = lib_and_device()
    import torch
    A = gen.random_sym_upper(300, per_row=per_row, seed=2)
    plan = xb.Plan.from_host(A, dev)
    x = np.random.default_rng(1).uniform(-1, 1, A["n"])
    yo = oracle.spmv(A, x)
    bound = row_bound(A, x)
    xt = torch.tensor(x, device=dev)
    for ipt in (1, 2, 4, 8, 16):
        y = plan.spmv(xt, torch.empty_like(xt), variant=xb.VAR_SYM_TILE, block=256, ipt=ipt).cpu().numpy()
        assert_rows_close(y, yo, bound, what=f"ipt {ipt}")
    for ipt in (3, 5, 12, 32):
        with pytest.raises(xb.XbError) as e:
            plan.spmv(xt, torch.empty_like(xt), variant=xb.VAR_SYM_TILE, block=256, ipt=ipt)
        assert e.value.code == xb.XB_EINVAL
