"""The float64 factorization and solves at the edges of their blocks: 16-column panels,
32 x 32 trailing tiles, 32-row solve blocks, chunks of 4 and 8 right-hand sides, and the
partial factorization that drops more than 128 centers at once."""
import numpy as np
import pytest
import torch

from oracle import rbf_oracle as O

pytestmark = pytest.mark.gpu

F64_TOL = 1e-5  # the update's float64 parity tolerance


def rel_inf(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300))


def cloud(rng, n, x0, x1, y1):
    x, y = rng.uniform(x0, x1, n), rng.uniform(0.0, y1, n)
    z = 0.1 * np.sin(2 * x) * np.cos(1.5 * y) + rng.normal(0, 0.02, n)
    return np.stack([x, y, z], 1).astype(np.float32)


# (lattice, share of the width that the second scan covers): 1, 2, 15, 16, 17, 31 ... centers;
# the last ones drop 1, 5 and about 170 centers
@pytest.mark.parametrize("nx,ny,keep", [(1, 1, 1.0), (2, 1, 1.0), (5, 3, 1.0), (4, 4, 1.0), (17, 1, 1.0), (31, 1, 0.5),
                                        (8, 4, 0.4), (11, 3, 0.4), (7, 7, 0.3), (16, 15, 0.6), (19, 17, 0.25)])
def test_fp64_blocks(nx, ny, keep):
    from paper_2509_26222_gb300 import native as N
    N.load(build_if_missing=True)
    h, rho = 0.25, 0.6
    c = np.stack([np.tile(np.arange(nx) + 0.5, ny) * h, np.repeat(np.arange(ny) + 0.5, nx) * h], 1)
    T = N.Terrain(rho=rho, lam=1e-2, update_precision=N.UPDATE_FP64)
    T.set_centers(torch.tensor(c, device="cuda"))
    st = O.BlockState(c, 1e-2, O.WENDLAND, rho=rho)
    rng = np.random.default_rng(nx * 100 + ny)
    w = nx * h
    for x1 in (w, max(w * keep - rho, 0.3 * h), w):
        p = cloud(rng, 40 + 6 * nx * ny, 0.0, x1, ny * h)
        T.update(torch.tensor(p, device="cuda"), noise=0.02)
        A = O.block_update(st, p.astype(np.float64))
        assert np.array_equal(T.active().cpu().numpy(), A)
        assert rel_inf(T.weights().cpu().numpy(), st.w) < F64_TOL
        for k in (1, 4, 5, 64, 65):
            ids = np.sort(rng.choice(nx * ny, min(k, nx * ny), replace=False))
            assert rel_inf(T.cov(ids).cpu().numpy(), st.P.block(ids)) < F64_TOL
