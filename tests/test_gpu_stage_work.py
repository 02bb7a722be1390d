"""The work that the stage timing reports for a factorization: within its band, and of a partial one the columns
that it eliminates, counted here column by column."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def work(n, columns, bw):
    r = np.minimum(n - 1 - np.arange(columns, dtype=np.float64), bw)
    return float(np.sum(r * r + 2.0 * r))


def scan(rng, n, x1, y1):
    x, y = rng.uniform(0.0, x1, n), rng.uniform(0.0, y1, n)
    return torch.tensor(np.stack([x, y, 0.1 * np.sin(2 * x)], 1).astype(np.float32), device="cuda")


@pytest.mark.parametrize("prec", [0, 1])
def test_factorization_work(prec):
    from paper_2509_26222_gb300 import native as N
    N.load(build_if_missing=True)
    nx, ny, h = 8, 100, 0.2
    i = np.arange(nx * ny)
    T = N.Terrain(rho=0.6, lam=1e-2, update_precision=prec)
    T.set_centers(torch.tensor(np.stack([(i % nx + 0.5) * h, (i // nx + 0.5) * h], 1), device="cuda"))
    rng = np.random.default_rng(0)
    p = scan(rng, 6000, nx * h, ny * h)
    T.update(p, noise=0.02)  # (the mixed path times its two factorizations in the first block of a kind)
    T.set_centers(T.centers())
    T.profile(True)
    T.update(p, noise=0.02)
    st = T.profile_read()
    a = len(T.active())
    local = np.full(nx * ny, -1)
    local[T.active().cpu().numpy()] = np.arange(a)
    rp, col = (t.cpu().numpy() for t in T.neighbors(p, noise=0.02))
    lists = np.split(local[col], rp[1:-1])
    bw = max(int(v.max() - v.min()) for v in lists if len(v))
    assert 3 * bw < a
    if prec == 0 or st["trailing"][2] == 0:  # (the mixed path's launch chain reports its launches one by one)
        assert np.isclose(st["panel"][1], work(a, a, bw), rtol=1e-12) and st["trailing"][2] == 0
    if prec == 0:  # more than 128 centers leave: a partial factorization, then a dense one
        T.update(scan(rng, 6000, nx * h, ny * h - 5.0), noise=0.02)
        part = T.profile_read()["panel"][1] - work(len(T.active()), len(T.active()), a)
        d = a - len(T.active())
        assert d > 128 and any(np.isclose(part, work(d + k, d, a), rtol=1e-9) for k in range(1, a - d + 1))
