"""Species with the thermodynamics of large alkanes."""
import math

import numpy as np


def _h_s(a, T):
    h = a[0] + a[1] * T / 2 + a[2] * T ** 2 / 3 + a[3] * T ** 3 / 4 + a[4] * T ** 4 / 5 + a[5] / T
    return h, a[0] * math.log(T) + a[1] * T + a[2] * T ** 2 / 2 + a[3] * T ** 3 / 3 + a[4] * T ** 4 / 4 + a[6]


def fuel_like(m, k, a1, T_mid=1000.0):
    """Gives species k of mechanism m heat capacities of an alkane's size: a1 is the constant
    above T_mid (38.5 for 12 carbons), with another polynomial below; the enthalpy and entropy
    at 1000 K stay, and are continuous at T_mid >= 1000 K."""
    s = a1 / 38.5
    hi = s * np.array([38.5, 5.6e-2, -1.9e-5, 3.0e-9, -1.7e-13, 0.0, 0.0])
    lo = s * np.array([-3.0, 0.15, -9.4e-5, 2.5e-8, -1.0e-12, 0.0, 0.0])
    for a, like, T in ((lo, m.nasa_lo[k].copy(), 1000.0), (hi, lo, T_mid)):
        (h, sr), (h0, s0) = _h_s(like, T), _h_s(a, T)
        a[5], a[6] = (h - h0) * T, sr - s0
    m.T_mid[k], m.T_hi[k] = T_mid, max(3000.0, 2.0 * T_mid)
    m.nasa_lo[k], m.nasa_hi[k] = lo, hi
