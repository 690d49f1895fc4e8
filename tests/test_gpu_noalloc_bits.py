"""The allocation-free moments have the bits of the regular ones: the same kernels on the same grids."""
import ctypes as C

import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


def _both(wk, s, order, flags):
    import torch
    from paper_1812_05264_gb300 import _lib as L, api
    ctx = api.Context()
    pos = torch.as_tensor(wk.positions, dtype=torch.float64, device="cuda")
    H = api.assemble_H(ctx, api.Model.from_workload(wk, "cuda"), pos, api.build_neighbors(ctx, pos, wk.cutoff))
    lo, hi = api.spectral_bounds(ctx, H)
    out = [torch.empty(order, dtype=torch.float64, device="cuda") for _ in range(2)]
    for name, o in zip(("tbk_chebyshev_moments", "tbk_chebyshev_moments_noalloc"), out):
        L.call(name, ctx.handle, C.byref(H.struct()), lo, hi, C.c_uint64(7), s, order, flags, o.data_ptr())
    assert torch.isfinite(out[0]).all()
    return out


# one launch for all steps (one, 16, 17, 32 and more of them, few and many probes), a launch each, both kernels and forms
@pytest.mark.parametrize("size,s,orders", [(10, 32, (1, 2, 32, 34, 64, 131)), (3, 4, (40,)), (13, 512, (400,)),
                                           (22, 8, (90,)), (23, 8, (20,))])
@pytest.mark.parametrize("flags", [1, 1 + 2, 1 + 4, 0])
def test_one_orbital(size, s, orders, flags):
    import torch
    for order in orders:
        a, b = _both(wl.sc_disorder(L=size, n_probes=s), s, order, flags)
        assert torch.equal(a, b), order


# 1,000 x 256 of order 5,000 and 700 x 100 of order 4,000: the partial sums of all steps do not fit the array together
@pytest.mark.parametrize("n_atoms,s,order,flags", [(1000, 256, 5000, 0), (1000, 256, 60, 0), (700, 100, 4001, 0),
                                                   (333, 100, 101, 0), (200, 64, 60, 1), (90, 512, 61, 2),
                                                   (90, 512, 61, 4), (90, 388, 33, 4)])
def test_nine_orbitals(n_atoms, s, order, flags):
    import torch
    a, b = _both(wl.fcc_cu(n_atoms, kT=0.5, n_probes=s, jitter=0.05), s, order, flags)
    assert torch.equal(a, b)


# FP64 around the line between the step by rows and the plain one (two rounds of 608 CTAs on 152 SMs), against the
# plain kernel to FP64 rounding of a sum of n s terms
@pytest.mark.parametrize("n_atoms,s", [(607, 260), (608, 260), (700, 512)])
def test_fp64_steps_around_the_line(n_atoms, s):
    import torch
    a, b = _both(wl.fcc_cu(n_atoms, kT=0.5, n_probes=s, jitter=0.05), s, 13, 1)
    assert torch.equal(a, b)
    p, _ = _both(wl.fcc_cu(n_atoms, kT=0.5, n_probes=s, jitter=0.05), s, 13, 1 + 4)
    assert (a - p).abs().max().item() <= 1e-13 * 9 * n_atoms


def test_fp64_gradient_of_a_large_panel_has_the_steps_terms():
    """1,300 x 256 in FP64: plain forward steps, backward steps by rows; the gradient against mixed precision."""
    import torch
    from paper_1812_05264_gb300 import api
    wk = wl.fcc_cu(1300, kT=0.5, n_probes=256, jitter=0.05)
    ctx = api.Context()
    pos = torch.as_tensor(wk.positions, dtype=torch.float64, device="cuda")
    H = api.assemble_H(ctx, api.Model.from_workload(wk, "cuda"), pos, api.build_neighbors(ctx, pos, wk.cutoff))
    lo, hi = api.spectral_bounds(ctx, H)
    args = (ctx, H, None, None, None, lo, hi, 3, 256, 20, 6.0, 0.5)
    G, _ = api.density_and_forces(*args, fp64=True, want_forces=False)
    Gm, _ = api.density_and_forces(*args, want_forces=False)
    assert (G - Gm).abs().max().item() <= 2e-5 * G.abs().max().item()
