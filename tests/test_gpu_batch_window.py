"""The batched patches at the edges of their Gram and evaluation: windows of 2 to 8 nodes (up to 50
neighbours, past one pass of a warp), points outside the lattice, heights of both signs and of very
different sizes, far and non-finite queries, against the ridge solution and evaluation of the oracle."""
import numpy as np
import pytest
import torch

from oracle import rbf_oracle as O

pytestmark = pytest.mark.gpu

F64_TOL, EVAL_TOL = 1e-5, 1e-3  # the update's and the evaluation's parity tolerances


@pytest.mark.parametrize("kernel,spacing,zscale", [("w", 0.62, 1.0), ("w", 0.31, -1e5), ("w", 0.2, 1e-6), ("w", 0.155, 1.0),
                                                   ("w", 0.151, 3.0), ("g", 0.2, -1.0), ("g", 0.155, 1e5)])
def test_batch_windows(kernel, spacing, zscale):
    from paper_2509_26222_gb300 import native as N
    N.load(build_if_missing=True)
    h = spacing
    kw = dict(rho=0.6) if kernel == "w" else dict(sigma=0.15)
    kind = O.WENDLAND if kernel == "w" else O.GAUSSIAN
    T = (N.Terrain(rho=0.6, lam=1e-2, update_precision=N.UPDATE_MIXED) if kernel == "w" else
         N.Terrain(kernel=N.KERNEL_GAUSSIAN, sigma=0.15, cutoff_mult=4.0, lam=1e-2, update_precision=N.UPDATE_MIXED))
    rng = np.random.default_rng(5)
    patches, refs = [], []
    for nx, M, n in ((1, 1, 3), (3, 8, 40), (9, 65, 300), (23, 500, 2500), (40, 1290, 5000)):
        rows = -(-M // nx)
        ids = np.arange(M)
        c = np.stack([-0.3 + (ids % nx + 0.5) * h, 0.7 + (ids // nx + 0.5) * h], 1)
        lo, hi = c.min(0) - 1.2 * h, c.max(0) + 1.2 * h  # some points lie outside the lattice
        xy = rng.uniform(lo, hi, (n, 2))
        z = zscale * (0.3 + np.sin(2 * xy[:, :1]) + rng.normal(0, 0.02, (n, 1)))
        z[::7] *= 1e-4
        p = np.concatenate([xy, z], 1).astype(np.float32)
        q = np.concatenate([xy[:200].astype(np.float32), np.float32([[1e30, 0], [-50, 3], [np.nan, 1], [1, np.inf]])])
        patches.append(dict(x0=-0.3, y0=0.7, spacing=h, nx=nx, M=M, pts=torch.tensor(p, device="cuda"),
                            q=torch.tensor(q, device="cuda")))
        refs.append((c, O.batch_ridge(p.astype(np.float64), c, 1e-2, kind, **kw), q))
    for (w, hh, g), (c, ref, q) in zip(T.batch_update_eval(patches), refs):
        assert np.max(np.abs(w.cpu().numpy() - ref)) < F64_TOL * np.max(np.abs(ref))
        k = len(q) - 4
        ho, gx, gy, ah, ax, ay = O.eval_h(q[:k].astype(np.float64), c, ref, kind, **kw)
        hh, g = hh.cpu().double().numpy(), g.cpu().double().numpy()
        assert np.all(np.abs(hh[:k] - ho) <= EVAL_TOL * (ah + 1e-12))
        assert np.all(np.abs(g[:k, 0] - gx) <= EVAL_TOL * (ax + 1e-12))
        assert np.all(np.abs(g[:k, 1] - gy) <= EVAL_TOL * (ay + 1e-12))
        assert np.all(hh[k:k + 2] == 0) and np.all(np.isnan(hh[k + 2:])) and np.all(np.isnan(g[k + 2:]))
