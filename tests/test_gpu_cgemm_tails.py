"""Tensor-core slice products with operands contiguous along K, odd pitches and odd batch strides: rows
of one operand alternate between 8- and 16-byte alignment and batch entry 1 starts 8 bytes off, so
the paired copies and loads and the single ones meet every tail of K.  The bounds are each
engine's in test_gpu_cgemm.py, relative to || |A| |B| ||_F against the FP64 product."""
import numpy as np
import pytest

from test_gpu_cgemm import crandn, op

pytestmark = pytest.mark.gpu


def check(prec, tol, k, transa, transb, m, n):
    import torch
    from paper_1407_1785_gb300 import libtsvd
    batch = 3
    ra, ca = (m, k) if transa == 0 else (k, m)
    rb, cb = (k, n) if transb == 0 else (n, k)
    lda, ldb = ra + 1 - ra % 2, rb + 1 - rb % 2          # odd pitches
    sa, sb = lda * ca + 1 - lda * ca % 2, ldb * cb + 1 - ldb * cb % 2   # odd strides
    A = np.ascontiguousarray(crandn(5, 0, (batch, sa)), np.complex64)
    B = np.ascontiguousarray(crandn(5, 2, (batch, sb)), np.complex64)
    Ad = torch.from_numpy(A.view(np.float32)).cuda()
    Bd = torch.from_numpy(B.view(np.float32)).cuda()
    Cd = torch.full((2 * m * n * batch,), 7.0, device="cuda")
    with libtsvd.Context(device=0, stream=torch.cuda.current_stream().cuda_stream,
                         precision=prec) as ctx:
        ctx.cgemm(transa, transb, m, n, k, Ad, lda, sa, Bd, ldb, sb, Cd, m, m * n, batch)
        torch.cuda.synchronize()
    C = Cd.cpu().numpy().view(np.complex64).reshape(batch, n, m).transpose(0, 2, 1)
    for b in range(batch):
        a = op(A[b, :lda * ca].reshape((lda, ca), order="F")[:ra].astype(np.complex128), transa)
        c = op(B[b, :ldb * cb].reshape((ldb, cb), order="F")[:rb].astype(np.complex128), transb)
        err = np.linalg.norm(C[b] - a @ c) / np.linalg.norm(np.abs(a) @ np.abs(c))
        assert err <= tol, f"entry {b}: {err:.3e}"


@pytest.mark.parametrize("m,n", [(7, 5), (129, 65)])
@pytest.mark.parametrize("transa,transb", [(2, 0), (1, 1), (0, 0)])
@pytest.mark.parametrize("k", [1, 2, 15] + [32 + t for t in range(16)])
def test_tails_of_k_on_odd_strides(k, transa, transb, m, n):
    check(3, 4e-6, k, transa, transb, m, n)


# a chunk of K is 32 entries in TF32 and 64 in BF16, an instruction takes 8 or 16 of them
@pytest.mark.parametrize("prec,tol", [(1, 2e-3), (2, 1.6e-2)], ids=["tf32", "bf16"])
@pytest.mark.parametrize("transa,transb", [(2, 0), (0, 2)])
@pytest.mark.parametrize("k", [1, 7, 8, 9, 16, 17, 31, 63, 64, 65, 73, 95])
def test_tails_of_k_through_registers(k, transa, transb, prec, tol):
    check(prec, tol, k, transa, transb, 133, 67)
