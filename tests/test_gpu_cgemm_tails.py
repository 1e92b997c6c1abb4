"""3xTF32 slice products with operands contiguous along K, odd pitches and odd batch strides: rows of
one operand alternate between 8- and 16-byte alignment and batch entry 1 starts 8 bytes off, so the
paired copies and the single ones meet every tail of K.  The bound is that engine's in
test_gpu_cgemm.py: 4e-6 of || |A| |B| ||_F against the FP64 product."""
import numpy as np
import pytest

from test_gpu_cgemm import crandn, op

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(7, 5), (129, 65)])
@pytest.mark.parametrize("transa,transb", [(2, 0), (1, 1), (0, 0)])
@pytest.mark.parametrize("k", [1, 2, 15] + [32 + t for t in range(16)])
def test_tails_of_k_on_odd_strides(k, transa, transb, m, n):
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
                         precision=3) as ctx:
        ctx.cgemm(transa, transb, m, n, k, Ad, lda, sa, Bd, ldb, sb, Cd, m, m * n, batch)
        torch.cuda.synchronize()
    C = Cd.cpu().numpy().view(np.complex64).reshape(batch, n, m).transpose(0, 2, 1)
    for b in range(batch):
        a = op(A[b, :lda * ca].reshape((lda, ca), order="F")[:ra].astype(np.complex128), transa)
        c = op(B[b, :ldb * cb].reshape((ldb, cb), order="F")[:rb].astype(np.complex128), transb)
        err = np.linalg.norm(C[b] - a @ c) / np.linalg.norm(np.abs(a) @ np.abs(c))
        assert err <= 4e-6, f"entry {b}: {err:.3e}"
