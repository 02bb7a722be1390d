"""A NaN in the factor stays visible in the levels of the explicit inverse that run on the tensor cores: the rows
that depend on it are NaN, those that do not are not."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("row,col", [(1500, 700), (1024, 0), (2047, 1023)])
def test_nan_in_the_factor(row, col):
    from paper_2509_26222_gb300 import native as N
    lib = N.load(build_if_missing=True)
    f = lib._ZN3rbf11trtri_mixedEPNS_3CtxEPKfllS3_PflP11CUstream_st  # rbf::trtri_mixed
    P, I = ctypes.c_void_p, ctypes.c_int64
    f.argtypes, f.restype = [P, P, I, I, P, P, I, P], ctypes.c_int
    T = N.Terrain(update_precision=N.UPDATE_MIXED)
    n = 2048  # one level of half-size 1,024: Z21 = -Z22 (L21 Z11)
    g = torch.Generator(device="cuda").manual_seed(1)
    W = torch.tril(0.02 * torch.randn(n, n, generator=g, device="cuda"), -1)
    W.diagonal().fill_(1.0)
    Zd = torch.stack([torch.linalg.inv(W[k:k + 64, k:k + 64].double()).float() for k in range(0, n, 64)]).contiguous()
    nan = (torch.zeros((), device="cuda") - torch.inf) + torch.inf  # the GPU's own
    W[row, col] = nan
    Z = torch.zeros(2 * n, n, device="cuda")
    assert f(T._h, W.data_ptr(), n, n, Zd.data_ptr(), Z.data_ptr(), n, torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    assert bool(torch.isnan(Z[row:n, :col + 1]).all())
    first = 1024 + (row - 1024) // 128 * 128  # (a tile's rows share their range of K)
    assert bool(torch.isfinite(Z[:first]).all()) and bool(torch.isfinite(Z[:n, 1024:]).all())
