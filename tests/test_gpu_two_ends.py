"""Factorization of a band from both ends (no explicit inverse, long narrow blocks): odd and even
numbers of 64-row blocks, ragged and full last blocks, the substitution with it, and the covariance
of the centers that leave the block in the next update."""
import numpy as np
import pytest
import torch

from oracle import rbf_oracle as O

pytestmark = pytest.mark.gpu

F64_TOL = 1e-5  # the update's float64 parity tolerance


@pytest.mark.parametrize("nx,ny", [(1, 700), (6, 200), (6, 203), (5, 256), (7, 183), (12, 171)])
def test_two_ends(nx, ny):
    from paper_2509_26222_gb300 import native as N
    N.load(build_if_missing=True)
    h, rho, M = 0.2, 0.6, nx * ny
    c = np.stack([np.tile(np.arange(nx) + 0.5, ny) * h, np.repeat(np.arange(ny) + 0.5, nx) * h], 1)
    T = N.Terrain(rho=rho, lam=1e-2, update_precision=N.UPDATE_MIXED, inverse_max=-1)
    T.set_centers(torch.tensor(c, device="cuda"))
    st = O.BlockState(c, 1e-2, O.WENDLAND, rho=rho)
    rng = np.random.default_rng(M)
    for y1 in (ny * h, 0.97 * ny * h):  # then the last few rows leave
        n = 6 * M
        x, y = rng.uniform(0.0, nx * h, n), rng.uniform(0.0, y1, n)
        z = 0.1 * np.sin(2 * x) * np.cos(1.5 * y) + rng.normal(0, 0.02, n)
        p = np.stack([x, y, z], 1).astype(np.float32)
        T.update(torch.tensor(p, device="cuda"), noise=0.02)
        A = O.block_update(st, p.astype(np.float64))
        assert np.array_equal(T.active().cpu().numpy(), A)
        assert np.max(np.abs(T.weights().cpu().numpy() - st.w)) < F64_TOL * np.max(np.abs(st.w))
        ids = np.unique(np.r_[rng.choice(M, 40, replace=False), np.arange(M - 8, M)])
        ref = st.P.block(ids)
        assert np.max(np.abs(T.cov(ids).cpu().numpy() - ref)) < F64_TOL * np.max(np.abs(ref))
