"""Batched solves at the matrix sizes where the threads per matrix, the register layout of
the inverse or the last loads of a matrix change.

The bounds are those of the solver's parity test: 1e-13 (FP64) and 1e-12 (FP32 inverse and
refinement) times the condition number.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 11, 31, 32, 33, 56, 57, 63, 64, 65, 96, 97, 127, 128]


@pytest.mark.parametrize("dim", SIZES)
def test_solve_sizes(dim, oracle_lib):
    import paper_2112_05834_gb300 as pkg

    rng = np.random.default_rng(100 + dim)
    n_mat, cond = 5, 1e3
    A = np.empty((n_mat, dim, dim))
    for s in range(n_mat):
        U, _ = np.linalg.qr(rng.standard_normal((dim, dim)))
        V, _ = np.linalg.qr(rng.standard_normal((dim, dim)))
        A[s] = U @ np.diag(np.logspace(0, -np.log10(cond), dim)) @ V.T
    b = rng.standard_normal((n_mat, dim))
    for precision, tol in ((0, 1e-13), (1, 1e-12), (2, 1e-12)):
        M = A.astype(np.float32).astype(np.float64) if precision == 2 else A
        ref = np.stack([oracle_lib.lu_solve(*oracle_lib.lu_factor(M[s])[:2], b[s]) for s in range(n_mat)])
        x, info = pkg.lu_solve_batched(torch.tensor(A, device="cuda"), torch.tensor(b, device="cuda"),
                                       precision=precision, ir_sweeps=3)
        assert np.all(info.cpu().numpy() == 0)
        err = np.abs(x.cpu().numpy() - ref).max(axis=1) / np.abs(ref).max(axis=1)
        assert err.max() <= tol * cond, (precision, err.max())


@pytest.mark.parametrize("dim", [32, 64, 65, 128])
def test_zero_pivot_sizes(dim):
    import paper_2112_05834_gb300 as pkg

    A = torch.eye(dim, dtype=torch.float64, device="cuda").repeat(3, 1, 1)
    A[1, dim - 1, dim - 1] = 0.0
    A[2, 1, 1] = 0.0
    for precision in (0, 1, 2):
        x, info = pkg.lu_solve_batched(A, torch.ones((3, dim), dtype=torch.float64, device="cuda"), precision=precision)
        assert info.tolist() == [0, dim, 2]
        assert torch.isnan(x[1:]).all() and (x[0] == 1.0).all()
