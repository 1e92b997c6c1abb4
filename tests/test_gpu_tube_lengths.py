"""The tube pass at every length from 1 to 260 of the last mode (512 entries a tube), with a mode 3 of
up to 5 entries, through the t-product: the compiled DFT tables against numpy's FFT in FP64 (2e-5 relative, the bound of
the other FP32 t-product tests)."""
import numpy as np
import pytest

from helpers import colmajor, relerr, uncolmajor
from paper_1407_1785_gb300 import libtsvd, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nf", [1, 2, 3, 4, 5])
def test_every_tube_length(nf):
    import torch
    with libtsvd.Context(device=0, stream=torch.cuda.current_stream().cuda_stream) as ctx:
        for nh in range(1, min(260, 512 // nf) + 1):
            rest = (nh,) if nf == 1 else (nf, nh)
            sa, sb, sc = (3, 2) + rest, (2, 4) + rest, (3, 4) + rest
            A = synth.normal(7, nh, int(np.prod(sa))).reshape(sa, order="F").astype(np.float32)
            B = synth.normal(8, nh, int(np.prod(sb))).reshape(sb, order="F").astype(np.float32)
            a = torch.from_numpy(colmajor(A)).cuda()
            b = torch.from_numpy(colmajor(B)).cuda()
            c = torch.empty(int(np.prod(sc)), device="cuda")
            ctx.tproduct(a, b, c, sa, 4)
            torch.cuda.synchronize()
            axes = tuple(range(2, len(sa)))
            Ah = np.fft.fftn(A.astype(np.float64), axes=axes)
            Bh = np.fft.fftn(B.astype(np.float64), axes=axes)
            C = np.real(np.fft.ifftn(np.einsum("ik...,kj...->ij...", Ah, Bh), axes=axes))
            assert relerr(uncolmajor(c.cpu().numpy(), sc), C) <= 2e-5, (nf, nh)
