"""The self-fed step kernel at sizes that take it (128-probe and narrower tasks, more than 17 warps of 32 probes per
SM): isolated atoms and two distant clusters, whose rows are short or hold the diagonal block alone."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s", [128, 100])
@pytest.mark.parametrize("direct", [False, True])
def test_isolated_atoms_and_separate_clusters(s, direct):
    import torch
    from paper_1812_05264_gb300 import api
    wk = wl.fcc_cu(700, kT=0.5, n_probes=s, jitter=0.05)
    far = wl.fcc_sphere(53, jitter=0.05, seed=3) + np.array([90.0, 0.0, 0.0])
    iso = np.array([[0.0, 90.0, 0.0], [0.0, 0.0, 90.0], [-90.0, 0.0, 0.0]])
    pos = torch.as_tensor(np.vstack([iso[:1], wk.positions, iso[1:2], far, iso[2:]]), dtype=torch.float64, device="cuda")
    ctx = api.Context()
    H = api.assemble_H(ctx, api.Model.from_workload(wk, "cuda"), pos, api.build_neighbors(ctx, pos, wk.cutoff))
    lo, hi = api.spectral_bounds(ctx, H)
    args = (ctx, H, lo, hi, 41, s, 23, False, direct)
    mom, per = api.chebyshev_probe_moments(*args)
    mom_p, per_p = api.chebyshev_probe_moments(*args, plain=True)
    # per-probe moments come from the panels: the same bits; the sums within FP64 rounding of n s terms
    assert torch.equal(per, per_p)
    assert (mom - mom_p).abs().max().item() <= 1e-13 * 9 * len(pos)


# Few probes on many rows take the plain kernel (more than 5,472 atoms on 152 SMs), more the narrow task
@pytest.mark.parametrize("n_atoms,s", [(5472, 16), (5473, 16), (5473, 20), (5600, 4)])
def test_few_probes_on_many_rows(n_atoms, s):
    import torch
    from paper_1812_05264_gb300 import api
    wk = wl.fcc_cu(n_atoms, kT=0.5, n_probes=s, jitter=0.05)
    pos = torch.as_tensor(wk.positions, dtype=torch.float64, device="cuda")
    ctx = api.Context()
    H = api.assemble_H(ctx, api.Model.from_workload(wk, "cuda"), pos, api.build_neighbors(ctx, pos, wk.cutoff))
    lo, hi = api.spectral_bounds(ctx, H, 20)
    args = (ctx, H, lo - 1.0, hi + 1.0, 41, s, 9)
    _, per = api.chebyshev_probe_moments(*args)
    _, per_p = api.chebyshev_probe_moments(*args, plain=True)
    assert torch.equal(per, per_p)
