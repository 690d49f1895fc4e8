"""FP64 moments of 1x1 operators with longer rows than the lattice's: all steps in one launch where the rule says
so, some or all blocks of a share in shared memory, against a launch per step."""
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


def _operator(ctx, size, r, ragged=False):
    import torch
    from paper_1812_05264_gb300 import api
    g0 = torch.Generator().manual_seed(3)
    pos = torch.as_tensor(wl.sc_disorder(L=size).positions, dtype=torch.float64)
    if ragged:  # the last eighth of the sites closer together: their rows hold most of the blocks
        pos[-len(pos) // 8:] *= 0.4
    pos = pos.cuda()
    g = api.build_neighbors(ctx, pos, r)
    rows = torch.repeat_interleave(torch.arange(len(pos)), (g.row_ptr[1:] - g.row_ptr[:-1]).cpu())
    cols = g.col.cpu().long()
    # a symmetric value per pair, small beside the bounds of -9 .. 9
    lo, hi = torch.minimum(rows, cols), torch.maximum(rows, cols)
    val = (0.02 * torch.cos((lo * 7919 + hi * 104729).double()) + 2.0 * (lo == hi) * torch.rand(1, generator=g0).double())
    return api.BSR(g, 1, val.reshape(-1, 1, 1).cuda())


# FP64 rounding of the sums: 1e-12 of mu_0.  Blocks that fit with room, to the last, in part (ragged rows), and not
@pytest.mark.parametrize("size,r,s,ragged", [(6, 2.5, 4, False), (6, 3.5, 4, False), (10, 2.5, 32, False),
                                             (10, 3.0, 32, False), (10, 1.5, 512, False), (14, 1.5, 32, False),
                                             (14, 1.8, 32, False), (18, 2.0, 4, False), (10, 2.0, 32, True),
                                             (14, 1.2, 8, True), (22, 1.0, 64, True)])
def test_moments_equal_the_steps(size, r, s, ragged):
    from paper_1812_05264_gb300 import api
    ctx = api.Context()
    H = _operator(ctx, size, r, ragged)
    got = api.chebyshev_moments(ctx, H, -9.0, 9.0, 5, s, 21, fp64=True)
    ref = api.chebyshev_moments(ctx, H, -9.0, 9.0, 5, s, 21, fp64=True, plain=True)
    assert (got - ref).abs().max().item() <= 1e-12 * size ** 3


# launches of a call: one for all steps, or one each (11) and what prepares and finishes them
@pytest.mark.parametrize("size,r,s,one", [(10, 1.0, 32, True), (22, 1.0, 512, True), (10, 2.5, 32, True),
                                          (18, 2.0, 4, False), (14, 1.8, 32, False), (10, 1.5, 512, False)])
def test_one_launch_where_the_blocks_fit(size, r, s, one):
    from paper_1812_05264_gb300 import api
    ctx = api.Context()
    H = _operator(ctx, size, r)
    n0 = ctx.launches
    api.chebyshev_moments(ctx, H, -9.0, 9.0, 5, s, 23, fp64=True)
    assert (ctx.launches - n0 < 8) == one


# The first two steps from a probe panel (FP32 rows of more than eight blocks) or from regenerated probes: the same
# values, so with one operator's values on a shorter and a longer pattern (zeros appended) the same moments.
@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("direct", [False, True])
def test_first_steps_of_one_orbital_operators(fp64, direct):
    import torch
    from paper_1812_05264_gb300 import api
    ctx = api.Context()
    short, wide = _operator(ctx, 9, 1.0), _operator(ctx, 9, 1.5)
    pos = torch.as_tensor(wl.sc_disorder(L=9).positions, dtype=torch.float64).cuda()
    rows = torch.repeat_interleave(torch.arange(729, device="cuda"), wide.graph.row_ptr.diff().long())
    near = (pos[rows] - pos[wide.graph.col.long()]).norm(dim=1) <= 1.0 + 1e-9
    val = torch.zeros_like(wide.val)
    val[near] = short.val
    wide = api.BSR(wide.graph, 1, val)
    assert short.graph.nnzb <= 8 * 729 < wide.graph.nnzb
    args = (-9.0, 9.0, 5, 516, 13, fp64, direct)
    m0, p0 = api.chebyshev_probe_moments(ctx, short, *args)
    m1, p1 = api.chebyshev_probe_moments(ctx, wide, *args)
    assert torch.equal(p0, p1)
    assert (m0 - m1).abs().max().item() <= 1e-12 * 729


# A row without its diagonal entry is found wherever it lies among the rows that share a warp, in the last one too
@pytest.mark.parametrize("row", [0, 1, 2, 3, 7, 124])
@pytest.mark.parametrize("fp64", [False, True])
def test_one_orbital_row_without_its_diagonal_is_rejected(row, fp64):
    import torch
    from paper_1812_05264_gb300 import _lib as L, api
    ctx = api.Context()
    H = _operator(ctx, 5, 1.0)
    api.chebyshev_moments(ctx, H, -9.0, 9.0, 5, 8, 9, fp64=fp64)
    rows = torch.repeat_interleave(torch.arange(125, device="cuda"), H.graph.row_ptr.diff().long())
    keep = ~((rows == row) & (H.graph.col == row))
    rp = H.graph.row_ptr.clone()
    rp[row + 1:] -= 1
    bad = api.BSR(api.Graph(125, H.graph.nnzb - 1, rp, H.graph.col[keep].contiguous()), 1, H.val[keep].contiguous())
    with pytest.raises(L.TbkError) as e:
        api.chebyshev_moments(ctx, bad, -9.0, 9.0, 5, 8, 9, fp64=fp64)
    assert e.value.code == L.TBK_ERR_ARG and "diagonal" in str(e.value)
