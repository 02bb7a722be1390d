"""Recorded graphs of batches that outlive a larger batch of the same context: a batch three times
(run, record, replay), a larger one that needs more workspace, then the first again, bit for bit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def batch(N, patches, M, nx, n, seed):
    """A prepared descriptor array (its buffers stay where they are) and its outputs."""
    h = 0.2
    rng = np.random.default_rng(seed)
    arr, keep, out = (N.RbfPatch * patches)(), [], []
    for d in arr:
        x, y = rng.uniform(0.0, nx * h, n), rng.uniform(0.0, (M // nx) * h, n)
        p = np.stack([x, y, 0.1 * np.sin(2 * x) + 0.05 * np.cos(y) + rng.normal(0, 0.02, n)], 1).astype(np.float32)
        pts = torch.tensor(p, device="cuda")
        q = pts[:, :2].contiguous()
        w = torch.empty(M, dtype=torch.float64, device="cuda")
        hq, g = torch.empty(n, device="cuda"), torch.empty(n, 2, device="cuda")
        d.x0, d.y0, d.spacing, d.nx, d.M, d.n, d.Q = 0.0, 0.0, h, nx, M, n, n
        d.pts, d.q, d.w, d.h, d.grad = pts.data_ptr(), q.data_ptr(), w.data_ptr(), hq.data_ptr(), g.data_ptr()
        keep += [pts, q]
        out += [w, hq, g]
    return arr, keep, out


# mixed: one-column patches have 2,048 or 4,096 chunks each (edges of 8 or 4 nodes), so that the first
# batch's scans are tiled (from 24,577 chunks on) and the second's tile sums outgrow 64 words (131,072)
@pytest.mark.parametrize("prec,small,large", [(1, (13, 16384, 1, 40), (64, 16384, 1, 40)),
                                              (0, (9, 130, 10, 400), (9, 1100, 25, 3000))])
def test_graph_outlives_larger_batch(prec, small, large):
    from paper_2509_26222_gb300 import native as N
    N.load(build_if_missing=True)
    T = N.Terrain(rho=0.6, lam=1e-2, update_precision=prec)
    first = batch(N, *small, seed=1)
    ref = None
    for _ in range(3):
        T.batch_update_eval_into(first[0], small[0])
        got = [t.clone() for t in first[2]]
        assert ref is None or all(torch.equal(a, b) for a, b in zip(ref, got))
        ref = got
    second = batch(N, *large, seed=2)
    for _ in range(3):
        T.batch_update_eval_into(second[0], large[0])
    filler = torch.full((1 << 20,), 7, dtype=torch.int32, device="cuda")  # may take the place of what was freed
    for t in first[2]:
        t.zero_()
    for _ in range(3):
        T.batch_update_eval_into(first[0], small[0])
        assert all(torch.equal(a, b) for a, b in zip(ref, first[2]))
    assert bool((filler == 7).all())
    assert all(bool(torch.isfinite(t).all()) for t in second[2])
