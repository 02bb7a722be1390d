"""The levels of the explicit inverse that run on the tensor cores (half-size 1,024 and more), each against
64 bits: the block Z21 = -Z22 (L21 Z11) must be no further off (2-norm) than with float32 multiply-adds in
order, the arithmetic of the other levels.  One level and several, ragged ones, and the whole-K form that
serves blocks above 4,096 rows."""
import ctypes
import math

import pytest
import torch

pytestmark = pytest.mark.gpu

F64, F32 = torch.float64, torch.float32


def factor(n):
    """Float32 Cholesky factor of the information matrix of a lattice patch with 6 points a center."""
    g = torch.Generator(device="cuda").manual_seed(n)
    nx, h, rho = int(math.sqrt(n)), 0.2, 0.6
    x = torch.rand(6 * n, 2, generator=g, device="cuda", dtype=F64) * (math.sqrt(n) * h)
    ids = torch.arange(n, device="cuda")
    c = torch.stack([(ids % nx).to(F64) + 0.5, (ids // nx).to(F64) + 0.5], 1) * h
    H = 1e-2 * torch.eye(n, device="cuda", dtype=F64)
    for q in x.split(4096):
        s = torch.cdist(q, c) / rho
        m = torch.clamp(1 - s, min=0) ** 4 * (4 * s + 1)
        H += m.T @ m
    return torch.linalg.cholesky(H).to(F32)


def in_order(A, B):
    """A B by float32 multiply-adds, k ascending."""
    acc = torch.zeros(A.shape[0], B.shape[1], device=A.device, dtype=F32)
    for k in range(A.shape[1]):
        acc = (acc.to(F64) + A[:, k:k + 1].to(F64) * B[k:k + 1].to(F64)).to(F32)
    return acc


@pytest.mark.parametrize("n", [1500, 2048, 3333, 4096, 5000])
def test_tensor_core_levels(n):
    from paper_2509_26222_gb300 import native as N
    lib = N.load(build_if_missing=True)
    f = lib._ZN3rbf11trtri_mixedEPNS_3CtxEPKfllS3_PflP11CUstream_st  # rbf::trtri_mixed
    P, I = ctypes.c_void_p, ctypes.c_int64
    f.argtypes, f.restype = [P, P, I, I, P, P, I, P], ctypes.c_int
    T = N.Terrain(update_precision=N.UPDATE_MIXED)
    L, ld = factor(n), (n + 3) & ~3
    W = torch.zeros(n, ld, device="cuda", dtype=F32)
    W[:, :n] = L
    Zd = torch.zeros((n + 63) // 64, 64, 64, device="cuda", dtype=F32)
    for b in range(len(Zd)):
        d = L[64 * b:64 * b + 64, 64 * b:64 * b + 64].to(F64)
        Zd[b, :len(d), :len(d)] = torch.linalg.inv(d).to(F32)
    Z = torch.zeros(2 * n, ld, device="cuda", dtype=F32)
    assert f(T._h, W.data_ptr(), ld, n, Zd.data_ptr(), Z.data_ptr(), ld, torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    h = 1024
    while h < n:
        for r1 in range(0, n - h, 2 * h):
            r2 = r1 + h
            e2 = min(r2 + h, n)
            Z11, Z22, L21 = Z[r1:r2, r1:r2], Z[r2:e2, r2:e2], L[r2:e2, r1:r2]
            ref = -(Z22.to(F64) @ (L21.to(F64) @ Z11.to(F64)))
            plain = -in_order(Z22, in_order(L21, Z11))
            off, off32 = (Z[r2:e2, r1:r2].to(F64) - ref).norm(), (plain.to(F64) - ref).norm()
            assert off <= off32, (h, r1, float(off / ref.norm()), float(off32 / ref.norm()))
        h *= 2
