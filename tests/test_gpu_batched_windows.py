"""Windowed outer products of a batch at every remainder of K = order / 2 by the window's four steps: the largest
K of a batch is where the sweep starts, also on the first step of a window."""
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


# G of the two schedules to FP32 summation order (2e-6 of the largest entry, as in the other tests of the schedules)
@pytest.mark.parametrize("orders", [(2, 3), (4, 2), (7, 5), (8, 9), (10, 4), (11, 11), (18, 7), (19, 10), (20, 19),
                                    (126, 90), (130, 61)])
@pytest.mark.parametrize("s", [128, 256])
def test_windowed_batch_matches_fused(orders, s):
    import torch
    from paper_1812_05264_gb300 import api
    ctx = api.Context()
    Hs, pos, lo, hi = [], [], [], []
    for n in (24, 13):
        wk = wl.fcc_cu(n, kT=0.5, n_probes=s, jitter=0.05)
        pos.append(torch.as_tensor(wk.positions, dtype=torch.float64, device="cuda"))
        model = api.Model.from_workload(wk, "cuda")
        Hs.append(api.assemble_H(ctx, model, pos[-1], api.build_neighbors(ctx, pos[-1], wk.cutoff)))
        e = api.spectral_bounds(ctx, Hs[-1])
        lo.append(e[0])
        hi.append(e[1])
    args = (ctx, Hs, model, pos, lo, hi, [5, 6], s, list(orders), [6.0, 6.0], [0.5, 0.5])
    G0, F0 = api.batched_density_and_forces(*args, want_G=True)
    G1, F1 = api.batched_density_and_forces(*args, want_G=True, windowed=True)
    for a, b, fa, fb in zip(G0, G1, F0, F1):
        assert torch.allclose(a, b, rtol=0, atol=2e-6 * a.abs().max().item())
        assert torch.allclose(fa, fb, rtol=0, atol=1e-5)
