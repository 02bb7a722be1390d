"""Updates that drop an exact number of centers: one, less than, equal to and more than a 16-column panel, and both
sides of the 128 where the float64 path goes from the one-CTA inverse to a partial factorization; then all of
them come back.  The number that left is asserted, the state compared with the oracle."""
import numpy as np
import pytest
import torch

from oracle import rbf_oracle as O

pytestmark = pytest.mark.gpu

F64_TOL = 1e-5  # the update's parity tolerance


# columns, rows, columns that leave: 1, 5, 15, 16, 17, 127, 128, 129 and 150 centers
@pytest.mark.parametrize("nx,ny,cols", [(40, 1, 1), (12, 5, 1), (12, 5, 3), (12, 16, 1), (12, 17, 1), (10, 127, 1),
                                        (12, 32, 4), (12, 43, 3), (30, 10, 15)])
@pytest.mark.parametrize("prec", [0, 1])
def test_leaving(nx, ny, cols, prec):
    from paper_2509_26222_gb300 import native as N
    N.load(build_if_missing=True)
    h, rho, M = 0.25, 0.6, nx * ny
    c = np.stack([np.tile(np.arange(nx) + 0.5, ny) * h, np.repeat(np.arange(ny) + 0.5, nx) * h], 1)
    T = N.Terrain(rho=rho, lam=1e-2, update_precision=prec)
    T.set_centers(torch.tensor(c, device="cuda"))
    st = O.BlockState(c, 1e-2, O.WENDLAND, rho=rho)
    rng = np.random.default_rng(M)
    # a raster of points up to x1: a center is touched if it lies within rho of it, and the first column
    # that leaves is half a spacing farther than that
    stay = (nx - cols) * h - rho
    for x1, active in ((nx * h, M), (stay, M - cols * ny), (nx * h, M)):
        gx, gy = np.meshgrid(np.linspace(0.0, x1, int(x1 / 0.1) + 2), np.linspace(0.0, ny * h, 10 * ny // 4 + 2))
        z = 0.1 * np.sin(2 * gx) * np.cos(1.5 * gy) + rng.normal(0, 0.02, gx.shape)
        p = np.stack([gx.ravel(), gy.ravel(), z.ravel()], 1).astype(np.float32)
        T.update(torch.tensor(p, device="cuda"), noise=0.02)
        A = O.block_update(st, p.astype(np.float64))
        assert len(A) == active and np.array_equal(T.active().cpu().numpy(), A)
        assert np.max(np.abs(T.weights().cpu().numpy() - st.w)) < F64_TOL * np.max(np.abs(st.w))
        ids = np.unique(np.r_[rng.choice(M, min(30, M), replace=False), np.arange(M - min(8, M), M)])
        ref = st.P.block(ids)
        assert np.max(np.abs(T.cov(ids).cpu().numpy() - ref)) < F64_TOL * np.max(np.abs(ref))
