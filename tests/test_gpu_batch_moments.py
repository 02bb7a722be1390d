"""The batched patches' m~ z where m is small: a center that its points meet near the edge of the support,
w = m z / (lambda + m^2), with m of 1e-14 to 1e-9.  m z has all bits of m (the sum's unit of 2^-64 is 5e-10 of
the smallest product here); m in units of 2^-52 is off by 3e-7 (Wendland) and up to 6e-3 (Gaussian).  (Coordinates near 64, where
the offset of a point from its node is exact.)"""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

TOL = 1e-7


@pytest.mark.parametrize("kernel,z", [("w", 1000.0), ("w", -30.0), ("g", 1000.0), ("g", -250.0)])
def test_small_entries(kernel, z):
    from paper_2509_26222_gb300 import native as N
    N.load(build_if_missing=True)
    kw = (dict(rho=0.6) if kernel == "w" else dict(kernel=N.KERNEL_GAUSSIAN, sigma=0.075, cutoff_mult=8.0))
    T = N.Terrain(lam=1e-2, update_precision=N.UPDATE_MIXED, **kw)
    patches, refs = [], []
    for k, far in enumerate((0.5994, 0.598, 0.59)):
        x0 = 64.0 + 0.37 * k
        c = x0 + 0.1
        p = np.float32([[c + far, c, z]])
        t = torch.tensor(p, device="cuda")
        patches.append(dict(x0=x0, y0=x0, spacing=0.2, nx=1, M=1, pts=t, q=t[:, :2].contiguous()))
        d = math.hypot(float(p[0, 0]) - (x0 + 0.5 * 0.2), float(p[0, 1]) - (x0 + 0.5 * 0.2))
        m = (1.0 - d / 0.6) ** 4 * (4.0 * d / 0.6 + 1.0) if kernel == "w" else math.exp(-d * d / (2.0 * 0.075 ** 2))
        refs.append(m * float(p[0, 2]) / (1e-2 + m * m))
    for (w, _, _), ref in zip(T.batch_update_eval(patches), refs):
        assert abs(float(w[0]) - ref) <= TOL * abs(ref)
