"""The one-launch Lanczos (cluster, grid, transposed and plain blocks) against the batched one, which
runs a kernel per phase with the same sums: the bounds are equal to the bit."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


def _both(wk, steps):
    import torch
    from paper_1812_05264_gb300 import api
    ctx = api.Context()
    pos = torch.as_tensor(wk.positions, dtype=torch.float64, device="cuda")
    model = api.Model.from_workload(wk, "cuda")
    box = None if wk.box is None else [float(x) for x in wk.box]
    H = api.assemble_H(ctx, model, pos, api.build_neighbors(ctx, pos, wk.cutoff, box), box)
    one = api.spectral_bounds(ctx, H, steps)
    lo, hi = api.batched_spectral_bounds(ctx, [H], steps)
    return one, (lo[0], hi[0])


# 32-row units: 96 fill the cluster (341 atoms), 8 per SM end the loads ahead (4,323 atoms), and past
# 207,126 blocks (12,000 atoms) the blocks are read untransposed
@pytest.mark.parametrize("n_atoms,steps", [(1, 64), (2, 3), (28, 64), (29, 64), (57, 1), (341, 64), (342, 64),
                                           (1000, 40), (4323, 8), (4340, 8), (12300, 6)])
def test_bounds_equal_the_batched_ones(n_atoms, steps):
    one, ref = _both(wl.fcc_cu(n_atoms, kT=0.5, n_probes=8, jitter=0.05), steps)
    assert one == ref


@pytest.mark.parametrize("L,steps", [(1, 4), (6, 64), (14, 64), (15, 64), (34, 16)])
def test_bounds_equal_the_batched_ones_one_orbital(L, steps):
    one, ref = _both(wl.sc_disorder(L=L), steps)
    assert one == ref


def test_periodic_bounds_equal_the_batched_ones():
    one, ref = _both(wl.sc9_periodic(L=8, n_probes=8), 32)
    assert one == ref
    assert np.isfinite(one).all() and one[0] < one[1]


# the last operator of a cluster (455 atoms) and the first of the grid after it, one to four 32-row units per
# SM, and rows longer than the shared memory that a thread's row of H gets (cutoff 7)
@pytest.mark.parametrize("n_atoms,cutoff,steps", [(147, None, 64), (455, None, 40), (456, None, 40), (541, None, 20),
                                                  (1081, None, 20), (1300, None, 20), (2161, None, 12),
                                                  (2162, None, 12), (200, 7.0, 20), (700, 7.0, 20), (1500, 7.0, 10)])
def test_bounds_equal_the_batched_ones_between_cluster_and_grid(n_atoms, cutoff, steps):
    wk = wl.fcc_cu(n_atoms, kT=0.5, n_probes=8, jitter=0.05)
    if cutoff:
        wk.cutoff = cutoff
    one, ref = _both(wk, steps)
    assert one == ref
