"""A mechanism whose shared-memory layout ends at the last bytes of what a CTA may have."""
import numpy as np
import pytest
import torch

import mechs

pytestmark = pytest.mark.gpu


def test_last_bytes():
    """88 species and 2,336 reactions in FP64: 230,400 bytes, 232,448 with the exponential's
    table, which with the kernel's own 16 is more than a CTA's 232,448."""
    import oracle as orc
    import paper_2112_05834_gb300 as pkg

    K, I = 88, 2336
    rng = np.random.default_rng(5)
    iso = [[3.8 + 0.001 * k, 2e-4, 1e-8, 0.0, 0.0, -5000.0 - 3.0 * k, 6.0] for k in range(K - 1)]
    rx = []
    for i in range(I):
        a, b = 1 + rng.choice(K - 1, 2, replace=False)
        rx.append({"reac": [(int(a), 1)], "prod": [(int(b), 1)], "A": 1e3 * (1.0 + i / I), "b": 0.1, "Ea_R": 2000.0})
    m = mechs.build(["N2"] + [f"A{k}" for k in range(1, K)], [{"N": 2}] + (K - 1) * [{"C": 1, "H": 2, "O": 1}],
                    [[3.5, 1e-4, 0.0, 0.0, 0.0, -1000.0, 4.0]] + iso, rx)
    n = 3
    T, p, Y = np.array([900.0, 1200.0, 1500.0]), np.full(n, 1e6), rng.dirichlet(np.ones(K), n)
    ref = orc.integrate(m, T, p, Y, 1e-4, rtol=1e-8, atol=1e-12)
    integ = pkg.Integrator(m, precision=0)
    Tg, pg, Yg = (torch.tensor(a, device="cuda") for a in (T, p, Y))
    integ.integrate(Tg, pg, Yg, 1e-4, 1e-8, 1e-12)
    assert integ.totals()["failed"] == 0
    assert np.all(np.abs(Tg.cpu().numpy() - ref["T"]) <= 1e-6 * ref["T"])
    assert np.all(np.abs(Yg.cpu().numpy() - ref["Y"]) <= 1e-8 + 1e-5 * np.abs(ref["Y"]))
