"""Retraining the SpMV heads alone: they learn the new timings, and the layers below
and the head for the restart length keep every bit."""
import numpy as np
import pytest

from tests._gpu import lib_and_device

pytestmark = pytest.mark.gpu


def test_other_parameters_keep_their_bits():
    xb, dev = lib_and_device()
    import torch
    from paper_2405_01599_gb300 import tuner
    D = dict(np.load(tuner.DATA_DIR + "/tuner_sweep_s101.npz"))
    model = xb.Mlp.load(tuner.MODEL_PATH)
    X = torch.tensor(D["feat"].astype(np.float32), device=dev)
    old, before = model.get_params(), model.predict(X)
    best = np.nanargmin(D["times"], axis=1)
    D["times"] = np.array(D["times"])
    for i, k in enumerate(best):  # another variant wins now
        other = (k + 5) % 21 if k < 21 else 21 + (k - 21 + 5) % 12
        D["times"][i, other] = 0.5 * D["times"][i, k]
    model, _ = tuner.retrain_spmv(model, D, steps=300)
    new, after = model.get_params(), model.predict(X)
    d_in, h1, h2, heads = model.dims
    w3, o, s = h1 * d_in + h1 + h2 * h1 + h2, sum(heads), sum(heads[:3])
    assert np.array_equal(old[:w3], new[:w3])
    assert np.array_equal(old[w3 + s * h2:w3 + o * h2], new[w3 + s * h2:w3 + o * h2])
    assert np.array_equal(old[w3 + o * h2 + s:], new[w3 + o * h2 + s:])
    assert np.array_equal(before[:, 3], after[:, 3]) and not np.array_equal(before[:, 0], after[:, 0])
