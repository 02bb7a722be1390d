"""Scans on both sides of the line between one CTA and tiles (24,576 elements), through the hash grid
of the centers and the neighbour lists: bit-exact lists against a brute-force search by the float32 rule."""
import numpy as np
import pytest
import torch


pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side,n", [(156, 24_575), (157, 24_576), (158, 24_577), (181, 26_624)])
def test_lists_across_scan_paths(side, n):
    from paper_2509_26222_gb300 import native as N
    N.load(build_if_missing=True)
    h, rho = 0.1, 0.15
    c = np.stack([np.tile(np.arange(side) + 0.5, side) * h, np.repeat(np.arange(side) + 0.5, side) * h], 1)
    T = N.Terrain(rho=rho)
    T.set_centers(torch.tensor(c, device="cuda"))
    rng = np.random.default_rng(side)
    p = np.concatenate([rng.uniform(0.0, side * h, (n, 2)), np.zeros((n, 1))], 1).astype(np.float32)
    rp, col = T.neighbors(torch.tensor(p, device="cuda"))
    rp, col = rp.cpu().numpy(), col.cpu().numpy()
    # brute-force on the lattice: the nodes around each point by the float32 rule
    q, c32 = p[:, :2], c.astype(np.float32)
    i0 = np.floor(q[:, 0].astype(np.float64) / h - 0.5).astype(int)
    j0 = np.floor(q[:, 1].astype(np.float64) / h - 0.5).astype(int)
    cand = []
    for dj in range(-2, 4):
        for di in range(-2, 4):
            i, j = i0 + di, j0 + dj
            ok = (i >= 0) & (i < side) & (j >= 0) & (j < side)
            ids = np.where(ok, j * side + i, 0)
            d = q - c32[ids]
            d2 = (d[:, 0] * d[:, 0]).astype(np.float32) + (d[:, 1] * d[:, 1]).astype(np.float32)
            r32 = np.float32(rho)
            cand.append(np.where(ok & (d2.astype(np.float32) < r32 * r32), ids, -1))
    cand = np.sort(np.stack(cand, 1), axis=1)
    counts = (cand >= 0).sum(1)
    assert np.array_equal(np.diff(rp), counts) and rp[-1] == counts.sum()
    assert np.array_equal(col, cand[cand >= 0])
