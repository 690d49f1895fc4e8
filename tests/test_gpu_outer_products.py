"""The outer products of the general adjoint (probe counts that are no multiple of 128, FP64, the plain
kernels) at the edges of their 32-probe runs and of the row lookup, against the oracle's gradient or,
where the cluster is too large for it, against the fused kernel."""
import numpy as np
import pytest

from gpu_common import blocks_of, oracle_estimator, oracle_H, small_fcc
from oracle import chebyshev as och

pytestmark = pytest.mark.gpu


def _setup(n_atoms, s, order, mixed):
    import torch
    from paper_1812_05264_gb300 import api
    wk = small_fcc(n_atoms, n_probes=s, order=order, mixed=mixed)
    ctx = api.Context()
    pos = torch.as_tensor(wk.positions, dtype=torch.float64, device="cuda")
    model = api.Model.from_workload(wk, "cuda")
    H = api.assemble_H(ctx, model, pos, api.build_neighbors(ctx, pos, wk.cutoff))
    lo, hi = api.spectral_bounds(ctx, H)
    return api, wk, ctx, pos, model, H, lo, hi


# mixed: FP32 products of unit-variance panels, the kernel-against-oracle bound of the other G tests
# (2e-5 of the largest entry); FP64: rounding of p steps, 1e-11 of it
@pytest.mark.parametrize("n_atoms,s", [(1, 4), (2, 28), (13, 32), (13, 36), (35, 64), (13, 100), (40, 132), (13, 260)])
@pytest.mark.parametrize("fp64", [False, True])
def test_gradient_vs_oracle(n_atoms, s, fp64):
    order = 14
    api, wk, ctx, pos, model, H, lo, hi = _setup(n_atoms, s, order, not fp64)
    rp, col, Hd = oracle_H(wk)
    est = oracle_estimator(wk, Hd, lo, hi, order)
    ref = blocks_of(och.estimator_gradient(est["w"], est["V"], est["R"], lo, hi, est["mu"], wk.kT, False, p=order),
                    rp, col, 9)
    G, _ = api.density_and_forces(ctx, H, model, pos, None, lo, hi, wk.probe_seed, s, order, est["mu"], wk.kT,
                                  fp64=fp64, want_forces=False)
    tol = (1e-11 if fp64 else 2e-5) * np.abs(ref).max()
    assert np.abs(G.cpu().numpy() - ref).max() <= tol


@pytest.mark.parametrize("n_atoms", [33, 1030])
def test_plain_outer_products_equal_the_fused_ones(n_atoms):
    api, wk, ctx, pos, model, H, lo, hi = _setup(n_atoms, 128, 8, True)
    args = (ctx, H, model, pos, None, lo, hi, 7, 128, 8, 6.0, 0.5)
    G, F = api.density_and_forces(*args)
    Gp, Fp = api.density_and_forces(*args, plain=True)
    assert (G - Gp).abs().max().item() <= 2e-5 * G.abs().max().item()
    assert (F - Fp).abs().max().item() <= 1e-3


# Outer products after several steps against the ones fused into each step (a plan with too few panels to
# store every y_k): the same additions in the same order, so the same bits.  Orders around a full window.
@pytest.mark.parametrize("n_atoms,s,orders", [(1, 128, (36, 150)), (13, 128, (37, 129, 130, 131)), (153, 128, (41,)),
                                              (700, 128, (38,)), (1, 256, (36,)), (13, 256, (37, 131)),
                                              (152, 256, (36,)), (153, 256, (37,)), (1030, 256, (37,))])
def test_deferred_outer_products_have_the_fused_bits(n_atoms, s, orders):
    import torch
    api, wk, ctx, pos, model, H, lo, hi = _setup(n_atoms, s, orders[0], True)
    for order in orders:
        args = (ctx, H, model, pos, None, lo, hi, wk.probe_seed, s, order, 6.0, 0.5)
        G0, F0 = api.density_and_forces(*args)
        G1, F1 = api.density_and_forces(*args, max_panel_bytes=(order // 2 + 3) * 9 * n_atoms * s * 4)
        assert torch.equal(G0, G1) and torch.equal(F0, F1)


# Forces from G: the directional derivative sum_k G_k : dH_k against central differences of the assembled
# blocks (error h^2 H'''/6, below 1e-7 of the sum of magnitudes at h = 1e-4), at the edges of the rows that
# a warp takes (one row up to 608 atoms, two, eight), open and with a single pair.
@pytest.mark.parametrize("n_atoms", [2, 35, 608, 609, 1250, 5000])
def test_forces_are_the_derivative_of_the_blocks(n_atoms):
    import torch
    from paper_1812_05264_gb300 import api as A
    api, wk, ctx, pos, model, H, lo, hi = _setup(n_atoms, 128, 6, True)
    G, F = api.density_and_forces(ctx, H, model, pos, None, lo, hi, 7, 128, 6, 6.0, 0.5)
    v = torch.randn(pos.shape, generator=torch.Generator(device="cuda").manual_seed(1), dtype=torch.float64, device="cuda")
    h = 1e-4
    dH = (A.assemble_H(ctx, model, pos + h * v, H.graph).val - A.assemble_H(ctx, model, pos - h * v, H.graph).val) / (2 * h)
    got, ref = -(F * v).sum().item(), (G * dH).sum().item()
    assert abs(got - ref) <= 1e-6 * (G * dH).abs().sum().item()


# The general adjoint's outer products after several steps against one launch per step (a plan with too few
# panels to store every y_k): sums kept to 2^-47 of their magnitudes either way, which cancel by less than
# 10^3 here: 1e-10 of the largest entry.  Whole windows of 16 and a rest, windows ended by the size (2,500
# atoms), the last probe count of each rule and the first beyond.
@pytest.mark.parametrize("n_atoms,s,order", [(1, 4, 40), (13, 36, 32), (13, 36, 33), (13, 36, 34), (35, 100, 150),
                                             (200, 28, 40), (501, 64, 30), (501, 68, 30), (2500, 36, 30),
                                             (13, 124, 40), (13, 132, 40)])
def test_general_deferred_outer_products(n_atoms, s, order):
    api, wk, ctx, pos, model, H, lo, hi = _setup(n_atoms, s, order, True)
    args = (ctx, H, model, pos, None, lo, hi, wk.probe_seed, s, order, 6.0, 0.5)
    G0, _ = api.density_and_forces(*args)
    G1, _ = api.density_and_forces(*args, max_panel_bytes=(order - 1) * 9 * n_atoms * s * 4)
    assert (G0 - G1).abs().max().item() <= 1e-10 * G0.abs().max().item()


# The same where 16 steps run together whatever the size (up to 96 probes) and at the line for wider ones (501 atoms on
# 152 SMs).
@pytest.mark.parametrize("n_atoms,s,order", [(501, 100, 22), (502, 100, 22), (1003, 96, 22), (4000, 64, 20),
                                             (9000, 12, 19)])
def test_general_deferred_outer_products_of_large_panels(n_atoms, s, order):
    test_general_deferred_outer_products(n_atoms, s, order)
