"""Rates and an integration with species of a large fuel molecule's thermodynamics.

The bounds are those of the right-hand side's parity test, 1e-11 of a species' gross rate, and
of the integrator's, |dT| <= 1e-6 T and |dY| <= 1e-8 + 1e-5 Y."""
import copy

import numpy as np
import pytest
import torch

from fuels import fuel_like
from paper_2112_05834_gb300 import synth

pytestmark = pytest.mark.gpu


def _mechanism(a1, T_mid):
    m = copy.deepcopy(synth.gen_mechanism(3, ("C", "H", "O", "N"), 37, 130, n_third_body=20, n_troe=14, n_lindemann=9))
    m.reversible[::7] = 0
    for k in (20, 27):
        fuel_like(m, k, a1, T_mid)
    return m


def _cells(m, n, classes=synth.MIXED_CLASSES):
    st = synth.gen_states(m, n, seed=4, p=40e6, classes=classes)
    Y = st.Y + 1e-3 * np.random.default_rng(11).dirichlet(np.ones(m.n_species), n)
    return st.T, st.p, Y / Y.sum(axis=1, keepdims=True)


@pytest.mark.parametrize("a1,T_mid", [(38.5, 1000.0), (60.0, 1000.0), (100.0, 1391.0), (20.0, 2500.0), (5.0, 5000.0)])
@pytest.mark.parametrize("precision", [0, 1])
def test_rates(precision, a1, T_mid):
    import oracle as orc
    import paper_2112_05834_gb300 as pkg

    m = _mechanism(a1, T_mid)
    T = np.array([300.0, 450.0, 777.7, 999.999, 1000.0, 1390.999, 1391.0, 2047.99, 2048.0, 2499.999, 2500.0, 4095.9, 4096.0,
                  4999.99, 5000.0, 5999.0])
    _, p, Y = _cells(m, len(T))
    f = pkg.Integrator(m, precision=precision).eval_rhs(*(torch.tensor(a, device="cuda") for a in (T, p, Y)))
    f = f.cpu().numpy()
    M, nu = orc.Mech(m), np.abs(m.net_stoich())
    for c, t in enumerate(T):
        y = np.concatenate([[t], Y[c]])
        fr, q = orc.rhs(M, p[c], y), orc.rates(M, p[c], y)[2]
        rho = p[c] / (8.31446261815324e7 * t * np.sum(Y[c] / m.W))
        gross = np.concatenate([[np.abs(fr[0])], m.W * (nu @ np.abs(q)) / rho])
        assert np.all(np.abs(f[c] - fr) <= 1e-11 * (np.abs(fr) + gross) + 1e-300), t


@pytest.mark.parametrize("precision", [0, 1])
def test_integration(precision):
    import oracle as orc
    import paper_2112_05834_gb300 as pkg

    m, dt = _mechanism(60.0, 1391.0), 1e-7
    T, p, Y = _cells(m, 16, ((1.0, "unreacted", 700.0, 1500.0),))
    ref = orc.integrate(m, T, p, Y, dt, rtol=1e-8, atol=1e-12)
    integ = pkg.Integrator(m, precision=precision)
    Tg, pg, Yg = (torch.tensor(a, device="cuda") for a in (T, p, Y))
    integ.integrate(Tg, pg, Yg, dt, 1e-8, 1e-12)
    assert integ.totals()["failed"] == 0
    assert np.all(np.abs(Tg.cpu().numpy() - ref["T"]) <= 1e-6 * ref["T"])
    assert np.all(np.abs(Yg.cpu().numpy() - ref["Y"]) <= 1e-8 + 1e-5 * np.abs(ref["Y"]))
