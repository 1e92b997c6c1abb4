"""Slice SVTs whose blocks are exchanged between CTAs: the rounds that keep one vector of a pair in
registers, at vector counts that leave padding in the last block or whole blocks of it, for every
lane count, with and without accumulated rotations, against the FP64 oracle (2e-5 of the result,
or of 1e-3 ||Y|| for a nearly empty one, as in the other t-SVT tests)."""
import numpy as np
import pytest

import oracle
from paper_1407_1785_gb300 import libtsvd, synth
from helpers import colmajor, relerr, uncolmajor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vform", [0, 1])
@pytest.mark.parametrize("shape,ctas,lanes", [
    ((20, 17, 3), 2, 8),       # 17 vectors in 4 blocks of 5: 3 short
    ((9, 17, 3), 8, 8),        # 16 blocks of 1 vector, 7 of them padding
    ((70, 61, 3), 4, 16),
    ((61, 75, 4), 8, 16),
    ((129, 40, 3), 2, 32),     # 3 chunks a lane, the last nearly empty
    ((260, 33, 2), 2, 16),     # more chunks than stay in registers with V
    ((100, 96, 3), 1, 8),      # one CTA, several passes a round
])
def test_exchanged_blocks_match_oracle(shape, ctas, lanes, vform):
    import torch
    Y = synth.normal(41, 0, int(np.prod(shape))).reshape(shape, order="F").astype(np.float32)
    Yh = np.fft.fft(Y.astype(np.float64), axis=2)
    sv = np.sort(np.concatenate([np.linalg.svd(Yh[:, :, k], compute_uv=False)
                                 for k in range(shape[2])]))
    tau = float(0.5 * (sv[sv.size // 2 - 1] + sv[sv.size // 2]))
    with libtsvd.Context(device=0, stream=torch.cuda.current_stream().cuda_stream, autotune=0,
                         ctas_per_slice=ctas, lanes_per_pair=lanes, accumulate_v=vform) as ctx:
        y = torch.from_numpy(colmajor(Y)).cuda()
        z = torch.empty_like(y)
        ctx.tsvt(y, z, shape, tau)
        torch.cuda.synchronize()
    Zo = oracle.tsvt(Y.astype(np.float64), tau)
    assert relerr(uncolmajor(z.cpu().numpy(), shape), Zo, floor=1e-3 * np.linalg.norm(Y)) <= 2e-5
