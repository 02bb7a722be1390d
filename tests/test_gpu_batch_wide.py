"""Batched patches whose band has more tiles than the substitution loads ahead (six): 64 to 150 columns, one
to nine tiles in groups of four, against the ridge solution of the oracle."""
import numpy as np
import pytest
import torch

from oracle import rbf_oracle as O

pytestmark = pytest.mark.gpu

F64_TOL = 1e-5  # the update's float64 parity tolerance


def test_wide_patches():
    from paper_2509_26222_gb300 import native as N
    N.load(build_if_missing=True)
    T = N.Terrain(rho=0.6, lam=1e-2, update_precision=N.UPDATE_MIXED)
    h, rng = 0.2, np.random.default_rng(2)
    patches, refs = [], []
    for nx, rows in ((64, 17), (76, 14), (100, 12), (115, 9), (128, 14), (150, 13)):
        M = nx * rows - 3
        ids = np.arange(M)
        c = np.stack([(ids % nx + 0.5) * h, (ids // nx + 0.5) * h], 1)
        xy = rng.uniform(0.0, 1.0, (5 * M, 2)) * (nx * h, rows * h)
        p = np.concatenate([xy, np.sin(2 * xy[:, :1]) + rng.normal(0, 0.02, (5 * M, 1))], 1).astype(np.float32)
        t = torch.tensor(p, device="cuda")
        patches.append(dict(x0=0.0, y0=0.0, spacing=h, nx=nx, M=M, pts=t, q=t[:64, :2].contiguous()))
        refs.append(O.batch_ridge(p.astype(np.float64), c, 1e-2, O.WENDLAND, rho=0.6))
    for (w, _, _), ref in zip(T.batch_update_eval(patches), refs):
        assert np.max(np.abs(w.cpu().numpy() - ref)) < F64_TOL * np.max(np.abs(ref))
