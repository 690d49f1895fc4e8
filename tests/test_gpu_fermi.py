"""The chemical-potential solve in every launch shape: 31 to 1 midpoints at a time, one or
several CTAs per midpoint, one or many problems, against the oracle's bisection."""
import numpy as np
import pytest

from oracle import chebyshev as och

pytestmark = pytest.mark.gpu


def _moments(n, p, emin, emax, seed):
    rng = np.random.default_rng(seed)
    e = rng.uniform(emin + 0.3, emax - 0.3, size=n)
    t = np.arccos((2 * e - emin - emax) / (emax - emin))
    return np.cos(np.arange(p)[:, None] * t[None]).sum(axis=1)


# mu: the bracket ends below 1e-13 W and N(mu) carries rounding of ~1e-13 of its value over a slope of
# at least ~0.1 states/eV per electron here; observables are sums of M terms, relative rounding 1e-12
@pytest.mark.parametrize("n_jobs", [1, 5, 40, 150, 1300])
@pytest.mark.parametrize("jackson", [False, True])
def test_fermi_level_in_every_launch_shape(n_jobs, jackson):
    import torch
    from paper_1812_05264_gb300 import api
    ctx = api.Context()
    orders = [(1, 2, 3, 63, 126, 257, 700)[i % 7] for i in range(n_jobs)] if n_jobs > 1 else [1201]
    emin, emax = -3.0, 5.0
    moms, kTs, nes = [], [], []
    for i, p in enumerate(orders):
        n = 40 + 3 * (i % 50)
        moms.append(_moments(n, p, emin, emax, i))
        kTs.append((0.05, 0.2, 1.0)[i % 3] if p > 60 else 2.0)
        nes.append(1.1 * n)
    dev = [torch.as_tensor(m, device="cuda") for m in moms]
    out = api.batched_fermi_level(ctx, dev, [emin] * n_jobs, [emax] * n_jobs, nes, kTs, jackson)
    for i in sorted({0, 1, 2, 3, 4, n_jobs // 2, n_jobs - 1} & set(range(n_jobs))):
        mu = och.estimator_mu(moms[i], emin, emax, nes[i], kTs[i], jackson)
        ref = (mu, *och.estimator_observables(moms[i], emin, emax, mu, kTs[i], jackson))
        assert abs(out[i, 0] - ref[0]) < 1e-10
        assert np.allclose(out[i, 1:], ref[1:], rtol=1e-11, atol=1e-9)
        one = api.fermi_level(ctx, dev[i], emin, emax, nes[i], kTs[i], jackson)
        assert np.allclose(one, ref, rtol=1e-11, atol=1e-9)
