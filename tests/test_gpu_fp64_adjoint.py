"""The FP64 adjoint of the doubled moments with 1x1 blocks (plain step kernel with the adjoint's own-row terms)
against the oracle's gradient, all panels stored and replayed."""
import numpy as np
import pytest

import workloads as wl
from gpu_common import blocks_of, oracle_estimator, oracle_H
from oracle import chebyshev as och

pytestmark = pytest.mark.gpu


# FP64 rounding of p steps: 1e-11 of the largest entry
@pytest.mark.parametrize("order", [1, 2, 3, 4, 5, 14, 41])
@pytest.mark.parametrize("s", [8, 260])
def test_one_orbital_gradient_vs_oracle(order, s):
    import torch
    from paper_1812_05264_gb300 import api
    wk = wl.sc_disorder(L=4, n_probes=s)
    ctx = api.Context()
    pos = torch.as_tensor(wk.positions, dtype=torch.float64, device="cuda")
    H = api.assemble_H(ctx, api.Model.from_workload(wk, "cuda"), pos, api.build_neighbors(ctx, pos, wk.cutoff))
    lo, hi, mu, kT = -9.0, 9.0, 0.3, 0.8
    rp, col, Hd = oracle_H(wk)
    wk.kT = kT
    est = oracle_estimator(wk, Hd, lo, hi, order)
    ref = blocks_of(och.estimator_gradient(est["w"], est["V"], est["R"], lo, hi, mu, kT, False, p=order), rp, col, 1)
    args = (ctx, H, None, None, None, lo, hi, wk.probe_seed, s, order, mu, kT)
    G, _ = api.density_and_forces(*args, fp64=True, want_forces=False)
    assert np.abs(G.cpu().numpy() - ref).max() <= 1e-11 * max(1.0, np.abs(ref).max())
    if order == 41:
        G2, _ = api.density_and_forces(*args, fp64=True, want_forces=False, max_panel_bytes=20 * 64 * s * 8)
        assert torch.equal(G, G2)
