"""Pivots of the float64 factorization over their whole range: the reciprocal against CUDA's division,
and ridges that are subnormal, huge or infinite."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

F64_TOL = 1e-5  # the update's float64 parity tolerance

KERNEL = r"""
#include "recip.cuh"
__global__ void k(const double* d, double* r, double* r0, int* in, long n) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  r[i] = rbf::rcp_pos(d[i]);
  r0[i] = 1.0 / d[i];
  in[i] = rbf::rcp_pos_range(d[i]) ? 1 : 0;
}
extern "C" int run(const double* d, double* r, double* r0, int* in, long n) {
  k<<<(unsigned)((n + 255) / 256), 256>>>(d, r, r0, in, n);
  return (int)cudaDeviceSynchronize();
}
"""


def test_reciprocal_against_division(tmp_path):
    from paper_2509_26222_gb300 import build as B
    src, lib = tmp_path / "k.cu", tmp_path / "k.so"
    src.write_text(KERNEL)
    subprocess.run([B.nvcc(), *B.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", B.CSRC, str(src),
                    "-o", str(lib)], check=True, cwd=tmp_path)
    rng = np.random.default_rng(0)
    n = 1 << 20
    mant = np.concatenate([1.0 + np.arange(4096) / 4096, 2.0 - np.arange(1, 4097) * 2.0**-52, rng.uniform(1.0, 2.0, n)])
    d = np.ldexp(mant, rng.integers(-1000, 1000, mant.size).astype(np.int32))
    wide = np.concatenate([d, [5e-324, 1e-310, 2.0**-1022, 2.0**-1001, 2.0**1000, 2.0**1023, 1.79e308, np.inf]])
    t = [torch.tensor(wide, device="cuda")] + [torch.empty(wide.size, dtype=dt, device="cuda")
                                               for dt in (torch.float64, torch.float64, torch.int32)]
    torch.cuda.synchronize()
    assert ctypes.CDLL(os.fspath(lib)).run(*(ctypes.c_void_p(a.data_ptr()) for a in t), ctypes.c_long(wide.size)) == 0
    r, r0, inside = (a.cpu().numpy() for a in t[1:])
    k = d.size
    assert np.all(np.abs(r[:k] - r0[:k]) <= np.spacing(r0[:k]))  # one unit in the last place
    assert np.all(inside[:k] == 1) and np.all(inside[k:] == 0)


@pytest.mark.parametrize("lam", [1e-310, 2.5e-308])
def test_tiny_ridge(lam):
    """A center that a point meets only at the edge of its support: m^2 vanishes in the sum, w = m z / lambda."""
    from paper_2509_26222_gb300 import native as N
    N.load(build_if_missing=True)
    T = N.Terrain(rho=1.0, lam=lam, update_precision=N.UPDATE_FP64)
    T.set_centers(torch.tensor([[0.0, 0.0], [5.0, 0.0]], dtype=torch.float64, device="cuda"))
    x, z = np.float32(0.999), np.float32(0.75)
    T.update(torch.tensor([[x, 0.0, z]], dtype=torch.float32, device="cuda"), noise=0.02)
    s = float(x)
    ref = (1.0 - s) ** 4 * (4.0 * s + 1.0) * float(z) / lam
    w = T.weights().cpu().numpy()
    assert abs(w[0] - ref) <= F64_TOL * ref and w[1] == 0.0


@pytest.mark.parametrize("lam", [1e300, 1e308, np.inf])
def test_huge_ridge(lam):
    from paper_2509_26222_gb300 import native as N
    N.load(build_if_missing=True)
    c = np.stack([np.tile(np.arange(6) + 0.5, 6) * 0.25, np.repeat(np.arange(6) + 0.5, 6) * 0.25], 1)
    T = N.Terrain(rho=0.6, lam=lam, update_precision=N.UPDATE_FP64)
    T.set_centers(torch.tensor(c, device="cuda"))
    rng = np.random.default_rng(1)
    p = np.concatenate([rng.uniform(0.0, 1.5, (300, 2)), rng.normal(1.0, 0.1, (300, 1))], 1).astype(np.float32)
    T.update(torch.tensor(p, device="cuda"), noise=0.02)
    w = T.weights().cpu().numpy()
    ref = np.zeros(len(c))
    if np.isfinite(lam):  # H' is lambda I to float64 rounding: w = m z / lambda
        for q in p.astype(np.float64):
            s = np.hypot(q[0] - c[:, 0], q[1] - c[:, 1]) / 0.6
            ref += np.clip(1.0 - s, 0.0, None) ** 4 * (4.0 * s + 1.0) * q[2] / lam
    assert np.all(np.isfinite(w)) and np.max(np.abs(w - ref)) <= F64_TOL * np.max(np.abs(ref))
