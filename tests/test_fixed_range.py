"""The temperatures for which rates are evaluated in fixed point: every argument fits there."""
import copy
import ctypes as C
import math

import numpy as np
import pytest

import mechs
from fuels import fuel_like
from paper_2112_05834_gb300 import synth


@pytest.fixture(scope="module")
def fixed_range():
    from paper_2112_05834_gb300 import _build

    _build.build()
    import paper_2112_05834_gb300 as pkg

    lib = pkg.load()

    def call(mech):
        d, keep = pkg.MechanismDesc(), mech.arrays()
        d.n_species, d.n_reactions, d.n_elements = mech.n_species, mech.n_reactions, mech.n_elements
        for name, a in keep.items():
            setattr(d, name, a.ctypes.data)
        out = (C.c_double * 2)()
        lib.chem_internal_fixed_point_range.restype = None
        lib.chem_internal_fixed_point_range(C.byref(d), out)
        return out[0], out[1]

    return call


@pytest.mark.parametrize("preset", ["h2_10", "c_32", "c_54", "c_100"])
def test_presets_take_the_whole_range(fixed_range, preset):
    assert fixed_range(synth.mechanism_preset(preset)) == (200.0, 8192.0)


def _one_reaction(a6, A, E):
    """N2 and A + B <=> C + D of one formula, with heats of formation +-a6; ln kf and ln kr."""
    base = [3.5, 1e-4, 0.0, 0.0, 0.0, -1000.0, 4.0]
    nasa = [base] + [[3.8, 2e-4, 1e-8, 0.0, 0.0, s * a6, 6.0] for s in (-1, -1, 1, 1)]
    r = {"reac": [(1, 1), (2, 1)], "prod": [(3, 1), (4, 1)], "b": 0.0, "A": A, "Ea_R": E}
    m = mechs.build(["N2", "A", "B", "C", "D"], [{"N": 2}] + 4 * [{"C": 1, "H": 2, "O": 1}], nasa, [r])
    return m, lambda T: math.log(A) - E / T, lambda T: math.log(A) + (4 * a6 - E) / T


@pytest.mark.parametrize("a6,A,E", [
    (52400.0, 1e13, 206000.0),   # ln kf -1000 and dG/RT +1048 at 200 K: their sum is what counts
    (80000.0, 1e13, 5000.0),     # ln kr 1605 at 200 K
    (90000.0, 1e13, 5000.0),     # and G/RT of two species 450
    (1000.0, 1e13, 250000.0),    # ln kf -1220
])
def test_arguments_stay_inside_their_bounds(fixed_range, a6, A, E):
    m, ln_kf, ln_kr = _one_reaction(a6, A, E)
    lo, end = fixed_range(m)
    T = np.linspace(lo, end, 20001)
    worst = lambda t: max(abs(ln_kf(t)), abs(ln_kr(t)))
    assert end == 8192.0 and max(map(worst, T)) <= 1000.0
    # and no temperature is given away beyond the grid and what it allows for the changes on it
    assert lo == 200.0 or worst(lo - 12.0) > 970.0


def test_a_mechanism_beyond_every_bound_has_no_range(fixed_range):
    m, _, _ = _one_reaction(1000.0, 1e13, 5000.0)
    m.nasa_lo[1, 6] = m.nasa_hi[1, 6] = 5000.0
    lo, end = fixed_range(m)
    assert not lo < end


@pytest.mark.parametrize("a1,T_mid", [(38.5, 1000.0), (60.0, 1000.0), (100.0, 1391.0), (20.0, 2500.0), (5.0, 5000.0)])
def test_large_fuel_molecules_have_a_range(fixed_range, a1, T_mid):
    m = copy.deepcopy(synth.mechanism_preset("c_54"))
    for k in (40, 47):
        fuel_like(m, k, a1, T_mid)
    lo, end = fixed_range(m)
    assert lo == 200.0 and end >= 6000.0


@pytest.mark.parametrize("b", [-40.0, 40.0])
def test_large_temperature_exponents_have_a_range(fixed_range, b):
    m, _, _ = _one_reaction(1000.0, math.exp(-b * 7.0), 5000.0)
    m.b[0] = b
    assert fixed_range(m) == (200.0, 8192.0)
