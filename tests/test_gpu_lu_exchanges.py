"""FP64 solves whose every pivot needs a row interchange, at the threads per matrix of small
and of large batches.

The bounds: 1e-13 times the condition number (the solver's parity test), and equal bits from
equal calls: a pivot read before or after its row's interchange would differ between them."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_mat", [5, 700])
@pytest.mark.parametrize("dim", [2, 31, 32, 33, 55, 64, 65, 128])
def test_row_interchanges(dim, n_mat):
    import paper_2112_05834_gb300 as pkg

    rng = np.random.default_rng(dim + n_mat)
    A = 0.25 / dim ** 0.5 * rng.standard_normal((n_mat, dim, dim))
    rows = np.arange(dim)
    for s in range(n_mat):
        # a cyclic shift: column k's pivot row is never row k at its step
        A[s, (rows + 1 + s % (dim - 1)) % dim, rows] += rng.choice([-1.0, 1.0], dim) * rng.uniform(1.0, 3.0, dim)
    x = rng.standard_normal((n_mat, dim))
    b = np.einsum("sij,sj->si", A, x)
    dev = [torch.tensor(a, device="cuda") for a in (A, b)]
    got = [pkg.lu_solve_batched(*dev, precision=0) for _ in range(4)]
    assert not got[0][1].any()
    assert all(torch.equal(got[0][0], g[0]) for g in got[1:])
    err = np.abs(got[0][0].cpu().numpy() - x).max(axis=1) / np.abs(x).max(axis=1)
    print("max error", err.max(), "condition", np.linalg.cond(A[:5]).max())
    assert np.all(err <= 1e-13 * np.linalg.cond(A))
