"""Predictions of more cells than one tile of 16 rows per warp: every warp takes several, the
last of them ragged. Bound and reference are those of the prediction test at the tiles' edges."""
import numpy as np
import pytest
import torch

from test_gpu_cost_model_tiles import _model, _problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [5, 54])
def test_several_tiles_per_warp(K):
    import paper_2112_05834_gb300 as pkg

    n = 2 * 256 * torch.cuda.get_device_properties(0).multi_processor_count + 77
    T, p, Y, _, _, norm, params, buf = _problem(K, n, 300 + K)
    model = pkg.CostModel(K)
    model.set_params(buf)
    got = model.predict(*(torch.tensor(a, device="cuda") for a in (T, p, Y)))
    got = torch.stack(got, 1).cpu().numpy().astype(np.float64)
    *_, H2, out = _model(T, p, Y, norm, params)
    tol = 4 * 2.0 ** -8 * np.abs(params["W3"]).max() * np.abs(H2).max() + 1e-5
    err = np.abs((got - norm[2]) / norm[3] - out)
    print("max error", err.max(), "tolerance", tol)
    assert np.all(err <= tol)
