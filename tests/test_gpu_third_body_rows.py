"""The mixed forms' third-body sums at every remainder of the species count by the batch in
which they load the efficiencies.

The bound is that of the right-hand side's parity test: 1e-11 of a species' gross rate."""
import numpy as np
import pytest
import torch

from paper_2112_05834_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", list(range(14, 23)))
@pytest.mark.parametrize("precision", [1, 2])
def test_third_body_sums(K, precision):
    import oracle as orc
    import paper_2112_05834_gb300 as pkg

    m = synth.gen_mechanism(K, ("C", "H", "O", "N"), K, 34, n_third_body=28, n_troe=3, n_lindemann=3)
    n = 5
    st = synth.gen_states(m, n, seed=K, p=40e5, classes=synth.MIXED_CLASSES)
    Y = st.Y + 1e-2 * np.random.default_rng(K).dirichlet(np.ones(K), n)
    Y /= Y.sum(axis=1, keepdims=True)
    f = pkg.Integrator(m, precision=precision).eval_rhs(*(torch.tensor(a, device="cuda") for a in (st.T, st.p, Y)))
    f = f.cpu().numpy()
    M, nu = orc.Mech(m), np.abs(m.net_stoich())
    for c in range(n):
        y = np.concatenate([[st.T[c]], Y[c]])
        fr, q = orc.rhs(M, st.p[c], y), orc.rates(M, st.p[c], y)[2]
        rho = st.p[c] / (8.31446261815324e7 * st.T[c] * np.sum(Y[c] / m.W))
        gross = np.concatenate([[np.abs(fr[0])], m.W * (nu @ np.abs(q)) / rho])
        assert np.all(np.abs(f[c] - fr) <= 1e-11 * (np.abs(fr) + gross) + 1e-300), (K, c)
