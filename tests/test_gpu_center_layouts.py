"""Layouts of centers at the edges of the search for a lattice: scattered ones (given up early), single rows and
columns, long strips, more distinct coordinates than the hash set holds, repeated coordinates off a lattice;
heights against the float64 oracle."""
import numpy as np
import pytest
import torch

from oracle import rbf_oracle as O

pytestmark = pytest.mark.gpu

EVAL_TOL = 1e-3  # the evaluation's parity tolerance


def lattice(nx, ny):
    i = np.arange(nx * ny)
    return np.stack([(i % nx + 0.5) * 0.2, (i // nx + 0.5) * 0.2], 1)


def scattered(n, seed):
    return np.random.default_rng(seed).uniform(0.0, 0.2 * np.sqrt(n), (n, 2))


@pytest.mark.parametrize("c", [scattered(65, 1), scattered(700, 2), scattered(5000, 3), lattice(1, 3000), lattice(3000, 1),
                               lattice(2, 1500), lattice(1500, 2), lattice(5000, 1), lattice(40, 70)[::-1],
                               np.concatenate([lattice(30, 30), scattered(900, 4)]),
                               np.concatenate([scattered(900, 5), lattice(30, 30)]),
                               np.repeat(scattered(60, 6), 20, 0) * [1.0, 0.5] + [[0.0, 0.1]]],
                         ids=lambda c: str(len(c)))
def test_layouts(c):
    from paper_2509_26222_gb300 import native as N
    N.load(build_if_missing=True)
    c = np.ascontiguousarray(c)
    rng = np.random.default_rng(len(c))
    w = rng.normal(0.0, 0.3, len(c))
    q = (c[rng.integers(0, len(c), 400)] + rng.uniform(-0.4, 0.4, (400, 2))).astype(np.float32)
    T = N.Terrain(rho=0.6)
    T.set_centers(torch.tensor(c, device="cuda"))
    T.set_weights(torch.tensor(w, device="cuda"))
    h, g = (t.cpu().double().numpy() for t in T.eval(torch.tensor(q, device="cuda")))
    ho, gx, gy, ah, ax, ay = O.eval_h(q.astype(np.float64), c, w, O.WENDLAND, rho=0.6)
    assert np.all(np.abs(h - ho) <= EVAL_TOL * (ah + 1e-12))
    assert np.all(np.abs(g[:, 0] - gx) <= EVAL_TOL * (ax + 1e-12))
    assert np.all(np.abs(g[:, 1] - gy) <= EVAL_TOL * (ay + 1e-12))
