"""The sums of the chemical-potential solve."""
import math
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_node_weights_lose_nothing_between_lanes():
    """One weight alone: at a temperature far below the spacing of the nodes, with mu between the two lowest,
    N = 2 rho at the lowest one.  rho M = mu_0 + 2 sum_k mu_k cos(k pi / 2M) over even k; mu_0 = 1 and fifteen terms of
    about 2^-54, each on a lane of its own, add 3.7 units of the last place of 1 that additions one after
    the other lose in part.  The sum is good to one rounding (2^-53) of a value below 2; M = 256."""
    import torch
    from paper_1812_05264_gb300 import api
    ctx = api.Context()
    p, M = 64, 256
    mom = np.zeros(p)
    mom[0] = 1.0
    mom[2:32:2] = 2.0 ** -55
    emin, emax = -1.0, 1.0
    e = np.cos(np.pi * (np.arange(M) + 0.5) / M)
    mu = 0.5 * (e[M - 1] + e[M - 2])
    out = api.fermi_level(ctx, torch.as_tensor(mom, device="cuda"), emin, emax, None, 1e-8, mu=mu)
    exact = 1 + 2 * sum(Fraction(2.0 ** -55) * Fraction(math.cos(k * math.pi / (2 * M))) for k in range(2, 32, 2))
    assert abs(Fraction(float(out[3])) * M / 2 - exact) <= Fraction(2.0 ** -53) * Fraction(101, 100)
