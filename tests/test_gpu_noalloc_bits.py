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
