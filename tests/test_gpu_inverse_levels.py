"""The explicit inverse of the float32 factor where its largest level changes kernel (half-size
1024) and where that level is ragged: blocks of 1,025 to 2,070 centers, not multiples of 4, 64 or
128, against the ridge solution and its covariance."""
import numpy as np
import pytest
import torch

from oracle import rbf_oracle as O

pytestmark = pytest.mark.gpu

F64_TOL = 1e-5  # the update's float64 parity tolerance


@pytest.mark.parametrize("nx,ny", [(32, 32), (41, 25), (13, 79), (48, 24), (45, 46)])
def test_inverse_levels(nx, ny):
    from paper_2509_26222_gb300 import native as N
    N.load(build_if_missing=True)
    h, rho, M = 0.2, 0.6, nx * ny
    c = np.stack([np.tile(np.arange(nx) + 0.5, ny) * h, np.repeat(np.arange(ny) + 0.5, nx) * h], 1)
    rng = np.random.default_rng(M)
    n = 6 * M
    x, y = rng.uniform(0.0, nx * h, n), rng.uniform(0.0, ny * h, n)
    z = 0.1 * np.sin(2 * x) * np.cos(1.5 * y) + rng.normal(0, 0.02, n)
    p = np.stack([x, y, z], 1).astype(np.float32)
    T = N.Terrain(rho=rho, lam=1e-2, update_precision=N.UPDATE_MIXED)
    T.set_centers(torch.tensor(c, device="cuda"))
    T.update(torch.tensor(p, device="cuda"), noise=0.02)
    ids = np.sort(rng.choice(M, 40, replace=False))
    st = O.BlockState(c, 1e-2, O.WENDLAND, rho=rho)
    A = O.block_update(st, p.astype(np.float64))
    assert np.array_equal(T.active().cpu().numpy(), A)
    w, P = T.weights().cpu().numpy(), T.cov(ids).cpu().numpy()
    assert np.max(np.abs(w - st.w)) < F64_TOL * np.max(np.abs(st.w))
    ref = st.P.block(ids)
    assert np.max(np.abs(P - ref)) < F64_TOL * np.max(np.abs(ref))
