"""Slater-Koster assembly by pairs against the oracle's blocks, at the edges of the rows that a warp takes
(one up to 608 atoms, then two), and on a pattern that stores some blocks without their transposes."""
import numpy as np
import pytest

from gpu_common import blocks_of, oracle_H, small_fcc

pytestmark = pytest.mark.gpu


def _operator(n_atoms):
    import torch
    from paper_1812_05264_gb300 import api
    wk = small_fcc(n_atoms, n_probes=8, order=4, mixed=False)
    ctx = api.Context()
    pos = torch.as_tensor(wk.positions, dtype=torch.float64, device="cuda")
    model = api.Model.from_workload(wk, "cuda")
    return api, wk, ctx, pos, model, api.build_neighbors(ctx, pos, wk.cutoff)


@pytest.mark.parametrize("n_atoms", [1, 2, 35, 120])
def test_blocks_vs_oracle(n_atoms):
    api, wk, ctx, pos, model, g = _operator(n_atoms)
    rp, col, Hd = oracle_H(wk)
    got = api.assemble_H(ctx, model, pos, g).val.cpu().numpy()
    # a few rounded products of entries of at most 10: 1e-13
    assert np.abs(got - blocks_of(Hd, rp, col, 9)).max() <= 1e-13


# the transposes are equal to the bit, and one-sided patterns hold the same blocks
@pytest.mark.parametrize("n_atoms", [35, 608, 609, 1300])
def test_transposes_and_one_sided_patterns(n_atoms):
    import torch
    api, wk, ctx, pos, model, g = _operator(n_atoms)
    H = api.assemble_H(ctx, model, pos, g).val
    rp, col = g.row_ptr.cpu().numpy(), g.col.cpu().numpy()
    row = np.repeat(np.arange(n_atoms), np.diff(rp))
    at = {(a, b): k for k, (a, b) in enumerate(zip(row, col))}
    tr = torch.as_tensor([at[(b, a)] for a, b in zip(row, col)], device="cuda")
    assert torch.equal(H, H[tr].transpose(1, 2))
    keep = (row == col) | ((row * 7 + col * 3) % 5 != 0)
    g1 = type(g)(n_atoms, int(keep.sum()), torch.as_tensor(np.concatenate([[0], np.cumsum(np.bincount(row[keep], minlength=n_atoms))]),
                                          dtype=torch.int32, device="cuda"),
                 torch.as_tensor(col[keep], dtype=torch.int32, device="cuda"))
    H1 = api.assemble_H(ctx, model, pos, g1).val
    assert torch.equal(H1, H[torch.as_tensor(np.flatnonzero(keep), device="cuda")])
    # rows in descending order: the same blocks
    order = np.concatenate([np.arange(rp[a], rp[a + 1])[::-1] for a in range(n_atoms)])
    g2 = type(g)(n_atoms, g.nnzb, g.row_ptr, torch.as_tensor(col[order], dtype=torch.int32, device="cuda"))
    H2 = api.assemble_H(ctx, model, pos, g2).val
    assert torch.equal(H2, H[torch.as_tensor(order, device="cuda")])
