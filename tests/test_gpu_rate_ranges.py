"""The rate evaluation at the ends of its fixed-point range, and the FP64 path beyond it.

The bounds are those of the right-hand side's and Jacobian's parity tests: 1e-11 of a
species' gross rate and 1e-10 of a row's largest entry.
"""
import copy

import numpy as np
import pytest
import torch

from paper_2112_05834_gb300 import synth

pytestmark = pytest.mark.gpu


def _mechanism(wide):
    """Every reaction kind, some irreversible reactions; ``wide``: an activation
    temperature whose Arrhenius argument leaves the fixed-point format."""
    m = copy.deepcopy(synth.gen_mechanism(3, ("C", "H", "O", "N"), 37, 130, n_third_body=20, n_troe=14, n_lindemann=9,
                                          Ea_R_max=40000.0))
    m.reversible[::7] = 0
    if wide:
        m.Ea_R[126] = 3.0e5  # elementary, irreversible: 0 x inf appears nowhere in FP64
    return m


# below 200 K, at its edge, T_mid = 1000 K from both sides, the oxidation range, and both
# sides of 8192 K
TEMPERATURES = [150.0, 199.999, 200.0, 200.001, 511.7, 999.999, 1000.0, 1000.001, 1500.0, 2047.99, 2048.0, 4096.0,
                5999.0, 8191.999, 8192.0, 9000.0]


@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("precision", [0, 1])
def test_rates_over_the_temperature_range(precision, wide):
    import oracle as orc
    import paper_2112_05834_gb300 as pkg

    m = _mechanism(wide)
    T = np.array(TEMPERATURES)
    n = len(T)
    rng = np.random.default_rng(11)
    st = synth.gen_states(m, n, seed=4, p=40e5, classes=synth.MIXED_CLASSES)
    Y = st.Y + 1e-3 * rng.dirichlet(np.ones(m.n_species), n)
    Y /= Y.sum(axis=1, keepdims=True)
    integ = pkg.Integrator(m, precision=precision)
    dev = [torch.tensor(a, device="cuda") for a in (T, st.p, Y)]
    f, J = integ.eval_rhs(*dev).cpu().numpy(), integ.eval_jacobian(*dev).cpu().numpy()
    M = orc.Mech(m)
    nu = np.abs(m.net_stoich())
    for c in range(n):
        y = np.concatenate([[T[c]], Y[c]])
        fr, Jr = orc.rhs(M, st.p[c], y), orc.jac(M, st.p[c], y)
        q = orc.rates(M, st.p[c], y)[2]
        rho = st.p[c] / (8.31446261815324e7 * T[c] * np.sum(Y[c] / m.W))
        gross = np.concatenate([[np.abs(fr[0])], m.W * (nu @ np.abs(q)) / rho])
        assert np.all(np.abs(f[c] - fr) <= 1e-11 * (np.abs(fr) + gross) + 1e-300), (T[c], precision)
        row = np.abs(Jr).max(axis=1, keepdims=True) + 1e-300
        floor = 64 * 2.0 ** -126 if precision == 1 else 0.0  # the float-float form's exponent range
        err = np.maximum(np.abs(J[c] - Jr) - floor, 0.0) / (np.abs(Jr) + row)
        assert err.max() <= 1e-10, (T[c], precision, err.max())


def test_negative_third_body_concentration_is_not_a_valid_rate():
    """A Troe reaction whose [M] is negative has no broadening factor: its rate is NaN on
    the fixed-point path as on the FP64 path, and the integrator rejects such a step."""
    import paper_2112_05834_gb300 as pkg

    for wide in (False, True):
        m = _mechanism(wide)
        i = np.flatnonzero(m.rxn_type == synth.RXN_TROE)[0]
        lo, hi = np.argmin(m.eff[i]), np.argmax(m.eff[i])
        assert m.eff[i, hi] > 1.3 * m.eff[i, lo]
        Y = np.zeros((1, m.n_species))
        Y[0, lo], Y[0, hi] = 0.012 * m.W[lo], -0.01 * m.W[hi]  # sum Y/W > 0, sum eff Y/W < 0
        T, p = np.array([1200.0]), np.array([40e5])
        f = pkg.Integrator(m).eval_rhs(*[torch.tensor(a, device="cuda") for a in (T, p, Y)]).cpu().numpy()
        assert np.isnan(f).any()
