"""The bounded waits of every TMA-fed kernel: a launch whose producer copies nothing gives up after 2 s, the call
returns TBK_ERR_TIMEOUT, and the context then computes what it did before."""
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


def _system(n_atoms, s):
    import torch
    from paper_1812_05264_gb300 import api
    wk = wl.fcc_cu(n_atoms, kT=0.5, n_probes=s, jitter=0.05)
    ctx = api.Context()
    pos = torch.as_tensor(wk.positions, dtype=torch.float64, device="cuda")
    H = api.assemble_H(ctx, api.Model.from_workload(wk, "cuda"), pos, api.build_neighbors(ctx, pos, wk.cutoff))
    return api, ctx, H, *api.spectral_bounds(ctx, H)


def _check(ctx, hook, call):
    import torch
    from paper_1812_05264_gb300 import _lib as L
    before = call()
    L.call(hook, ctx.handle)
    with pytest.raises(L.TbkError) as e:
        call()
    assert e.value.code == L.TBK_ERR_TIMEOUT
    assert torch.equal(call(), before)      # the hook is used up, the context usable


# self-fed kernel with whole and with narrow tasks, one probe per lane with 4, 8 and 16 warps, producer warp with two
# consumer warps and its denser form
@pytest.mark.parametrize("n_atoms,s", [(700, 128), (700, 100), (40, 100), (40, 132), (40, 260), (40, 256), (1000, 256)])
def test_recurrence_step(n_atoms, s):
    api, ctx, H, lo, hi = _system(n_atoms, s)
    _check(ctx, "tbk_test_stall_next_step", lambda: api.chebyshev_moments(ctx, H, lo, hi, 3, s, 12))


# one probe per lane (with the adjoint's source terms; general form), self-fed, two and four consumer warps without
# outer products
@pytest.mark.parametrize("n_atoms,s,schedule", [(40, 128, "fused"), (40, 100, "fused"), (700, 100, "fused"),
                                                (700, 128, "fused"), (40, 128, "windowed"), (40, 256, "fused"),
                                                (40, 512, "windowed")])
def test_adjoint_step(n_atoms, s, schedule):
    api, ctx, H, lo, hi = _system(n_atoms, s)
    _check(ctx, "tbk_test_stall_next_adjoint", lambda: api.density_and_forces(
        ctx, H, None, None, None, lo, hi, 3, s, 12, 6.0, 0.5, want_forces=False, windowed=schedule)[0])


# twelve and four warps per block row
@pytest.mark.parametrize("n_atoms", [40, 200])
def test_outer_products(n_atoms):
    api, ctx, H, lo, hi = _system(n_atoms, 256)
    _check(ctx, "tbk_test_stall_next_outer", lambda: api.density_and_forces(
        ctx, H, None, None, None, lo, hi, 3, 256, 12, 6.0, 0.5, want_forces=False)[0])
