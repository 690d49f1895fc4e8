"""The sums of the chemical-potential solve: their accuracy, and that a problem's result does not depend on
the problems solved with it."""
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


def _moments(n, p, emin, emax, seed):
    rng = np.random.default_rng(seed)
    e = rng.uniform(emin + 0.3, emax - 0.3, size=n)
    t = np.arccos((2 * e - emin - emax) / (emax - emin))
    return np.cos(np.arange(p)[:, None] * t[None]).sum(axis=1)


@pytest.mark.parametrize("n_batch", [2, 16, 150, 700])
def test_a_problem_alone_and_in_batches_gives_the_same_bits(n_batch):
    """mu, Omega, E and N of problems of several orders, each alone and among others that change the launch: how
    many lanes, CTAs and midpoints at a time a problem would get."""
    import torch
    from paper_1812_05264_gb300 import api
    ctx = api.Context()
    emin, emax = -3.0, 5.0
    kinds = [(1, 2.0), (63, 0.5), (126, 0.2), (700, 0.05), (2476, 0.025)]
    jobs = [(_moments(40 + 3 * i, p, emin, emax, i), kT, 1.1 * (40 + 3 * i)) for i, (p, kT) in enumerate(kinds)]
    dev = [torch.as_tensor(m, device="cuda") for m, _, _ in jobs]
    alone = [api.fermi_level(ctx, d, emin, emax, ne, kT) for d, (_, kT, ne) in zip(dev, jobs)]
    for sel in ([0, 1, 2], [2, 3], [4, 2, 1, 3, 0]):
        pick = [sel[i % len(sel)] for i in range(n_batch)]
        out = api.batched_fermi_level(ctx, [dev[i] for i in pick], [emin] * n_batch, [emax] * n_batch,
                                      [jobs[i][2] for i in pick], [jobs[i][1] for i in pick])
        for row, i in zip(out, pick):
            assert tuple(row) == tuple(alone[i]), (i, row, alone[i])
