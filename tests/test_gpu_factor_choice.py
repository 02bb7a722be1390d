"""The choice between the two factorizations of the mixed update is kept for dense and banded blocks apart:
a dense block that follows a banded one of the same size takes the launch chain (its tensor-core trailing
updates are three times faster at this size), whatever the banded one took."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_dense_block_after_banded():
    from paper_2509_26222_gb300 import native as N
    N.load(build_if_missing=True)
    side, h = 87, 0.2  # 7,569 centers, and 7,482 without the last column: one size bucket (7,424 to 7,679)
    i = np.arange(side * side)
    C = torch.tensor(np.stack([(i % side + 0.5) * h, (i // side + 0.5) * h], 1), device="cuda")
    rng = np.random.default_rng(3)

    def scan(x1):
        x, y = rng.uniform(0.0, x1, 30_000), rng.uniform(0.0, side * h, 30_000)
        z = 0.1 * np.sin(2 * x) * np.cos(1.5 * y) + rng.normal(0, 0.02, x.size)
        return torch.tensor(np.stack([x, y, z], 1).astype(np.float32), device="cuda")

    T = N.Terrain(rho=0.6, lam=1e-2, update_precision=N.UPDATE_MIXED)
    T.set_centers(C)
    T.update(scan(side * h), noise=0.02)              # banded
    T.update(scan((side - 0.6) * h - 0.6), noise=0.02)  # the last column leaves: dense from here on
    T.profile(True)
    T.update(scan((side - 0.6) * h - 0.6), noise=0.02)
    st = T.profile_read()
    assert 7424 <= len(T.active()) < 7569 and st["trailing"][2] > 0  # the chain: one interval per trailing update
