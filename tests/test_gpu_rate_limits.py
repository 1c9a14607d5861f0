"""Rates whose exponents are large, alone or in parts that cancel.

The bounds are those of the right-hand side's parity tests: 1e-11 of a species' gross rate."""
import math

import numpy as np
import pytest
import torch

import mechs

pytestmark = pytest.mark.gpu
RC, P0 = 8.31446261815324e7, 1.01325e6


def _gibbs(a, T):
    h = a[0] + a[1] * T / 2 + a[2] * T ** 2 / 3 + a[3] * T ** 3 / 4 + a[4] * T ** 4 / 5 + a[5] / T
    s = a[0] * math.log(T) + a[1] * T + a[2] * T ** 2 / 2 + a[3] * T ** 3 / 3 + a[4] * T ** 4 / 4 + a[6]
    return h - s


def _four_isomers(a6, **rxn):
    """N2 and A + B <=> C + D of one formula, with heats of formation +-a6."""
    base = [3.5, 1e-4, 0.0, 0.0, 0.0, -1000.0, 4.0]
    nasa = [base] + [[3.8, 2e-4, 1e-8, 0.0, 0.0, s * a6, 6.0] for s in (-1, -1, 1, 1)]
    r = {"reac": [(1, 1), (2, 1)], "prod": [(3, 1), (4, 1)], "b": 0.0, **rxn}
    return mechs.build(["N2", "A", "B", "C", "D"], [{"N": 2}] + 4 * [{"C": 1, "H": 2, "O": 1}], nasa, [r])


def _rhs(m, T, Y, p, **options):
    import paper_2112_05834_gb300 as pkg

    dev = [torch.tensor(np.asarray(a), device="cuda") for a in (T, np.full(len(T), p), np.tile(Y, (len(T), 1)))]
    return pkg.Integrator(m, **options).eval_rhs(*dev).cpu().numpy()


@pytest.mark.parametrize("precision", [0, 1])
def test_reverse_rate_arguments_that_cancel(precision):
    """ln kf near -1000 and dG/RT near +1050 at 200 K: kr is the exponential of their sum."""
    A, E = 1e13, 206000.0
    m = _four_isomers(52400.0, A=A, Ea_R=E)
    T = np.array([200.0, 201.0, 203.0, 207.0, 215.0, 230.0, 260.0, 300.0, 600.0])
    Y, p = np.array([0.9, 0.02, 0.03, 0.04, 0.01]), 10e6
    f = _rhs(m, T, Y, p, precision=precision)
    for c, t in enumerate(T):
        g = [_gibbs(a, t) for a in m.nasa_lo]
        ka = math.log(A) - E / t
        dg = g[3] + g[4] - g[1] - g[2]
        rho = p / (RC * t * np.sum(Y / m.W))
        C = rho * Y / m.W
        qf, qr = math.exp(ka) * C[1] * C[2], math.exp(ka + dg) * C[3] * C[4]
        want = np.array([0.0, -1.0, -1.0, 1.0, 1.0]) * m.W * (qf - qr) / rho
        assert np.all(np.abs(f[c, 1:] - want) <= 1e-11 * np.abs(want)), (t, ka, dg)


@pytest.mark.parametrize("precision", [0, 1])
def test_rate_constants_near_the_largest_double(precision):
    A, E = 1e300, -3000.0  # ln kf: 705.8 at 200 K, 690.8 in the limit
    m = _four_isomers(1000.0, A=A, Ea_R=E, reversible=0)
    T = np.array([200.0, 210.0, 300.0, 1000.0])
    Y, p = np.array([0.9, 0.02, 0.03, 0.04, 0.01]), 10e6
    f = _rhs(m, T, Y, p, precision=precision)
    for c, t in enumerate(T):
        rho = p / (RC * t * np.sum(Y / m.W))
        C = rho * Y / m.W
        want = m.W[1] * math.exp(math.log(A) - E / t) * (C[1] * C[2] / rho)
        assert abs(f[c, 1 + 1] + want) <= 1e-11 * want, (t, f[c, 1 + 1], want)  # [dT/dt, N2, A, ...]
