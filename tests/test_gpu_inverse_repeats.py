"""Integrations of 101 equations on 64 and 128 threads (the in-place FP32 inverse in shared
memory) and of the FP64 form on 256: equal calls give equal bits, and the results those of
the other block sizes within the integrator's parity bound."""
import pytest
import torch

from paper_2112_05834_gb300 import synth

pytestmark = pytest.mark.gpu


def _integrate(precision, block):
    import paper_2112_05834_gb300 as pkg

    m = synth.mechanism_preset("c_100")
    st = synth.gen_states(m, 24, seed=6, p=40 * synth.BAR, classes=synth.MIXED_CLASSES)
    integ = pkg.Integrator(m, precision=precision, block=block)
    T, p, Y = (torch.tensor(a, device="cuda") for a in (st.T, st.p, st.Y))
    integ.integrate(T, p, Y, 1e-6, 1e-8, 1e-12)
    assert integ.totals()["failed"] == 0
    return T, Y


@pytest.mark.parametrize("precision,block", [(1, 64), (1, 128), (0, 256)])
def test_100_species_repeat(precision, block):
    runs = [_integrate(precision, block) for _ in range(3)]
    for T, Y in runs[1:]:
        assert torch.equal(T, runs[0][0]) and torch.equal(Y, runs[0][1])
    T, Y = runs[0]
    Tr, Yr = _integrate(0, 128)
    assert bool(((T - Tr).abs() <= 1e-6 * Tr).all())
    assert bool(((Y - Yr).abs() <= 1e-8 + 1e-5 * Yr.abs()).all())
