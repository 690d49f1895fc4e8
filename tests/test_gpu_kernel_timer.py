"""What the kernel timer books as adjoint: the steps of every form of it, and their outer products."""
import math

import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


# order 30, K = 15.  128 probes: 14 steps and one launch of outer products; 256 probes at 1,500 atoms: as many steps
# together as half of L2 holds (one); FP64: 14 steps, 15 products; ragged: 28 steps of the general form, 29 products
# after up to 16 of them or (1,500 atoms) each
@pytest.mark.parametrize("n_atoms,s,fp64,step,backward", [(40, 128, False, 15, 14 + 1), (1500, 256, False, 15, 14 + 15),
                                                          (40, 512, False, 15, 15), (40, 64, True, 15, 14 + 15),
                                                          (40, 100, False, 28, 28 + 2), (1500, 100, False, 28, 28 + 29)])
def test_adjoint_launches(n_atoms, s, fp64, step, backward):
    import torch
    from paper_1812_05264_gb300 import api
    wk = wl.fcc_cu(n_atoms, kT=0.5, n_probes=s, jitter=0.05)
    ctx = api.Context()
    pos = torch.as_tensor(wk.positions, dtype=torch.float64, device="cuda")
    H = api.assemble_H(ctx, api.Model.from_workload(wk, "cuda"), pos, api.build_neighbors(ctx, pos, wk.cutoff))
    lo, hi = api.spectral_bounds(ctx, H)
    ctx.time_kernels("step", "backward", "window")
    api.density_and_forces(ctx, H, None, None, None, lo, hi, 3, s, 30, 6.0, 0.5, fp64=fp64, want_forces=False)
    got = {f: ctx.kernel_time(f) for f in ("step", "backward", "window")}
    ctx.time_kernels()
    assert {f: n for f, (_, n) in got.items()} == {"step": step, "backward": backward, "window": 0}
    assert got["step"][0] > 0 and got["backward"][0] > 0
