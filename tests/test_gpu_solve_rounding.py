"""Mixed-form solves without refinement: the FP32 matrix is the nearest one.

x v of a diagonal system v x = 1 has, beside the reciprocal's and the product's unbiased
roundings, the relative error of the FP32 matrix entry. Rounded to nearest that is uniform
in +-2^-24 at most, and its mean over 4,096 entries stays below 6 sd = 6 2^-24 / sqrt(3 4096)
< 0.06 2^-24; an entry cut to 24 bits is low by a half unit on average, 2^-24 ln 2 relative."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [1, 32, 64, 128])
def test_matrix_entries_are_rounded_to_nearest(dim):
    import paper_2112_05834_gb300 as pkg

    v = np.random.default_rng(dim).uniform(1.0, 2.0, (4096 // dim, dim))
    A = torch.diag_embed(torch.tensor(v, device="cuda"))
    x, info = pkg.lu_solve_batched(A, torch.ones_like(A[:, 0]), precision=1, ir_sweeps=0)
    assert not info.any()
    mean = float(np.mean(x.cpu().numpy() * v - 1.0)) * 2.0 ** 24
    print("mean error in 2^-24:", mean)
    assert abs(mean) < 0.25
