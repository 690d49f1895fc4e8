"""The step kernels for small operators, narrow panels and FP64 against the plain kernel: the same
additions in the same order per element, so each probe's moments, taken from the panels, are equal to
the bit; the moments, summed by other threads, agree to FP64 rounding of a sum of n * s terms."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


def _check(n_atoms, s, fp64, direct, order=9):
    import torch
    from paper_1812_05264_gb300 import api
    wk = wl.fcc_cu(n_atoms, kT=0.5, n_probes=s, jitter=0.05)
    ctx = api.Context()
    pos = torch.as_tensor(wk.positions, dtype=torch.float64, device="cuda")
    H = api.assemble_H(ctx, api.Model.from_workload(wk, "cuda"), pos, api.build_neighbors(ctx, pos, wk.cutoff))
    lo, hi = api.spectral_bounds(ctx, H)
    args = (ctx, H, lo, hi, 41, s, order, fp64, direct)
    mom, per = api.chebyshev_probe_moments(*args)
    mom_p, per_p = api.chebyshev_probe_moments(*args, plain=True)
    assert torch.equal(per, per_p)
    n = 9 * n_atoms
    # FP32: products of four probes are rounded alike; FP64: one rounding per product and addition
    assert (mom - mom_p).abs().max().item() <= 1e-13 * n
    one = api.chebyshev_moments(*args)
    assert torch.equal(one, mom)
    assert np.isfinite(mom.cpu().numpy()).all()


# lane kernel: 1 to 4 warps, lanes past the end, 8- and 16-warp chunks, several chunks past 512 probes;
# 700 atoms take the self-fed kernel with a narrow task
@pytest.mark.parametrize("direct", [False, True])
@pytest.mark.parametrize("n_atoms,s", [(1, 4), (2, 32), (13, 36), (55, 100), (55, 124), (55, 128), (40, 132),
                                       (40, 196), (30, 260), (30, 388), (20, 516), (20, 1028), (650, 128), (651, 128),
                                       (700, 100), (700, 4), (2700, 32)])
def test_fp32_steps_equal_the_plain_kernel(n_atoms, s, direct):
    _check(n_atoms, s, False, direct)


# one row per warp below 608 warps of three rows, three beyond; one to eight row groups per warp
@pytest.mark.parametrize("direct", [False, True])
@pytest.mark.parametrize("n_atoms,s", [(1, 4), (2, 8), (13, 16), (55, 32), (55, 36), (202, 32), (203, 32), (60, 100),
                                       (700, 12), (300, 64)])
def test_fp64_steps_equal_the_plain_kernel(n_atoms, s, direct):
    _check(n_atoms, s, True, direct)


# All steps in one launch (1x1 blocks, FP64) against a launch per step: one site, rows that do not divide over
# the cluster, a share of the blocks beyond shared memory (22^3 at 64 probes) and a cluster beyond the rule
# (23^3).  FP64 rounding of the sums: 1e-12 of mu_0.
@pytest.mark.parametrize("L,s,orders", [(1, 4, (2, 3, 8)), (2, 4, (7,)), (3, 36, (2, 3, 4, 41)), (7, 32, (40,)),
                                        (10, 100, (41,)), (13, 512, (20,)), (22, 64, (12,)), (23, 4, (12,))])
def test_one_launch_sweep_equals_the_steps(L, s, orders):
    import torch
    from paper_1812_05264_gb300 import api
    wk = wl.sc_disorder(L=L, n_probes=s)
    ctx = api.Context()
    pos = torch.as_tensor(wk.positions, dtype=torch.float64, device="cuda")
    model = api.Model.from_workload(wk, "cuda")
    H = api.assemble_H(ctx, model, pos, api.build_neighbors(ctx, pos, wk.cutoff))
    for order in orders:
        got = api.chebyshev_moments(ctx, H, -9.0, 9.0, 5, s, order, fp64=True)
        ref = api.chebyshev_moments(ctx, H, -9.0, 9.0, 5, s, order, fp64=True, plain=True)
        assert (got - ref).abs().max().item() <= 1e-12 * L ** 3


# 256-probe tasks around the line of the denser kernel (more than six tasks per SM: 913 atoms on 152 SMs), and
# grids of less and more than two rounds
@pytest.mark.parametrize("n_atoms,direct", [(912, False), (913, False), (913, True), (1217, True), (1530, False),
                                            (2300, False), (2700, False)])
def test_256_probe_steps_equal_the_plain_kernel(n_atoms, direct):
    _check(n_atoms, 256, False, direct, order=5)
