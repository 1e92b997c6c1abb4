"""The FP32 slice products at the edges of their tiles.

Every real part of C is a sum of 2K products accumulated by fused multiply-adds, so an entry is
off by at most about 2 K u (|A| |B|) with u = 2^-24, entry by entry (|.| the complex moduli,
which bound each |re re| + |im im|); 1.05 covers the second-order terms at these K.
"""
import numpy as np
import pytest

from test_gpu_cgemm import crandn, op

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("transa,transb", [(0, 0), (2, 0), (1, 2), (0, 1)])
@pytest.mark.parametrize("m,n,k,batch", [
    (1, 1, 1, 1),
    (31, 16, 15, 2),        # one short tile, K below a tile of it
    (33, 17, 17, 3),        # one entry past the smallest tile and past a tile of K
    (48, 48, 16, 2),        # exact tiles of 48
    (49, 65, 33, 2),
    (64, 64, 32, 200),      # exact tiles of 64, a grid above the SM count
    (65, 63, 31, 160),
    (130, 7, 40, 5),        # narrow
    (5, 200, 40, 5),        # flat
])
def test_products_at_tile_edges(transa, transb, m, n, k, batch):
    import torch
    from paper_1407_1785_gb300 import libtsvd
    ra, ca = (m, k) if transa == 0 else (k, m)
    rb, cb = (k, n) if transb == 0 else (n, k)
    lda, ldb, ldc = ra + 1, rb + 2, m + 1
    A = crandn(11, 0, (lda, ca * batch)).astype(np.complex64)
    B = crandn(11, 2, (ldb, cb * batch)).astype(np.complex64)
    Ad = torch.from_numpy(A.ravel(order="F").view(np.float32).copy()).cuda()
    Bd = torch.from_numpy(B.ravel(order="F").view(np.float32).copy()).cuda()
    Cd = torch.full((2 * ldc * n * batch,), 7.0, device="cuda")
    with libtsvd.Context(device=0, stream=torch.cuda.current_stream().cuda_stream) as ctx:
        ctx.cgemm(transa, transb, m, n, k, Ad, lda, lda * ca, Bd, ldb, ldb * cb, Cd, ldc, ldc * n,
                  batch)
        torch.cuda.synchronize()
    C = Cd.cpu().numpy().view(np.complex64).reshape((ldc, n * batch), order="F")
    assert np.all(C[m:] == 7 + 7j)   # rows past m are not written
    for b in range(batch):
        a = op(A[:ra, b * ca:(b + 1) * ca].astype(np.complex128), transa)
        c = op(B[:rb, b * cb:(b + 1) * cb].astype(np.complex128), transb)
        d = C[:m, b * n:(b + 1) * n].astype(np.complex128) - a @ c
        bound = 1.05 * 2 * k * 2.0 ** -24 * (np.abs(a) @ np.abs(c))
        assert np.all(np.abs(d.real) <= bound) and np.all(np.abs(d.imag) <= bound)
