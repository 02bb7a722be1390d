"""The Gram accumulation at the edges of its rules: neighbour lists of 31, 32 and 33 entries
(folded pairs against rows of 32) and 1,023 / 1,024 points (where the units of the sum let one
fused multiply-add form a product), against the ridge solution of the oracle."""
import numpy as np
import pytest
import torch

from oracle import rbf_oracle as O

pytestmark = pytest.mark.gpu

F64_TOL = 1e-5  # the update's float64 parity tolerance


@pytest.mark.parametrize("entries", [1, 2, 30, 31, 32, 33, 65])
@pytest.mark.parametrize("n", [1023, 1024])
@pytest.mark.parametrize("prec", [0, 1])
def test_gram_list_lengths(entries, n, prec):
    from paper_2509_26222_gb300 import native as N
    N.load(build_if_missing=True)
    # every center lies within the support of every point: all lists hold all centers
    c = np.stack([0.05 * (np.arange(entries) % 8), 0.05 * (np.arange(entries) // 8)], 1).astype(np.float64)
    rng = np.random.default_rng(entries * 7 + n)
    xy = rng.uniform(0.0, 0.4, (n, 2))
    p = np.concatenate([xy, 0.1 * np.sin(5 * xy[:, :1]) + rng.normal(0, 0.02, (n, 1))], 1).astype(np.float32)
    T = N.Terrain(rho=1.5, lam=1.0, update_precision=prec)
    T.set_centers(torch.tensor(c, device="cuda"))
    T.update(torch.tensor(p, device="cuda"), noise=0.02)
    ref = O.batch_ridge(p.astype(np.float64), c, 1.0, O.WENDLAND, rho=1.5)
    w = T.weights().cpu().numpy()
    assert len(T.active()) == entries
    assert np.max(np.abs(w - ref)) < F64_TOL * np.max(np.abs(ref))
