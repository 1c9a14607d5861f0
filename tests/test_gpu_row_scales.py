"""Mixed-form solves of systems whose rows differ in size by up to 40 decades.

The bound is what the textbook algorithm reaches on the same system: an FP32 Gauss-Jordan
inverse with partial pivoting and pivot rows scaled to a unit pivot, and the same number of
refinement sweeps, computed here; ten times its error, and 1e-12 (the solver's parity bound
at condition 1) for systems that it solves to rounding."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _refined(A, b, sweeps):
    """x by an FP32 inverse of normalised pivot rows and refinement in 64 bits."""
    n = len(b)
    f = np.float32
    w, used, piv = A.astype(f), np.zeros(n, bool), np.zeros(n, int)
    for k in range(n):
        p = int(np.argmax(np.where(used, f(-1.0), np.abs(w[:, k]))))
        used[p], piv[k] = True, p
        row, mult = w[p] / w[p, k], w[:, k].copy()
        row[k] = f(1.0) / w[p, k]
        w[:, k] = 0.0
        mult[p] = 0.0
        w = w - mult[:, None] * row[None, :]
        w[p] = row
    inv = np.empty_like(w)
    inv[:, piv] = w[piv]
    x = (inv @ b.astype(f)).astype(np.float64)
    for _ in range(sweeps):
        x += (inv @ (b - A @ x).astype(f)).astype(np.float64)
    return x


@pytest.mark.parametrize("decades", [30, 40])
@pytest.mark.parametrize("dim", [16, 32, 55, 64, 101, 128])
def test_row_scales(dim, decades):
    import paper_2112_05834_gb300 as pkg

    rng = np.random.default_rng(1000 * decades + dim)
    n_mat, sweeps = 6, 3
    A, x = np.empty((n_mat, dim, dim)), rng.standard_normal((n_mat, dim))
    for s in range(n_mat):
        B = rng.standard_normal((dim, dim)) / dim ** 0.5 + 2.0 * np.eye(dim)
        d = np.linspace(decades / 2, -decades / 2, dim)
        A[s] = 10.0 ** (d if s == 0 else d[::-1] if s == 1 else rng.permutation(d))[:, None] * B
    A = A.astype(np.float32).astype(np.float64)  # the same system for both forms
    b = np.einsum("sij,sj->si", A, x)
    model = np.stack([_refined(A[s], b[s], sweeps) for s in range(n_mat)])
    scale = np.abs(x).max(axis=1)
    bound = np.maximum(10.0 * np.abs(model - x).max(axis=1) / scale, 1e-12)
    print("model error", np.abs(model - x).max(axis=1) / scale)
    for precision in (1, 2):
        got, info = pkg.lu_solve_batched(torch.tensor(A, device="cuda"), torch.tensor(b, device="cuda"),
                                         precision=precision, ir_sweeps=sweeps)
        err = np.abs(got.cpu().numpy() - x).max(axis=1) / scale
        print("precision", precision, "error", err)
        assert info.tolist() == [0] * n_mat
        assert np.all(err <= bound), (precision, err, bound)
