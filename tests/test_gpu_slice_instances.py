"""Every way a slice-SVT launch runs its local rounds, one plan each, with and without accumulated
rotations, against the FP64 oracle (2e-5 of the result, or of 1e-3 ||Y|| for a nearly empty one, as
in the other t-SVT tests).  The plan comes from a saved-plan file, which alone can ask for two
pairs in flight; the file stays as written, so the plan was taken and nothing was timed."""
import numpy as np
import pytest

import oracle
from paper_1407_1785_gb300 import libtsvd, synth
from helpers import colmajor, relerr, uncolmajor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vform", [0, 1])
@pytest.mark.parametrize("shape,ctas,lanes,pairs", [
    # x in registers: two pairs in flight, blocks short of vectors; V in registers (2 chunks) or not
    ((33, 60, 3), 2, 16, 2),
    ((61, 75, 3), 2, 16, 2),
    ((45, 90, 3), 4, 8, 2),
    ((17, 64, 3), 8, 16, 2),     # blocks of 2 vectors, 7 blocks of padding
    ((38, 300, 3), 2, 32, 1),    # 3 chunks, the most with which V stays too
    # several passes a round after the first
    ((70, 400, 2), 2, 32, 1),    # 4 chunks, one instance
    ((100, 90, 2), 1, 32, 1),    # three passes rather than two
    # more warps, no resident x: one pass instead of two, a wave of CTAs fewer, 3 chunks on one CTA
    ((80, 100, 2), 2, 32, 1),
    ((96, 100, 3), 1, 16, 1),
    ((40, 100, 200), 8, 32, 1),
    ((61, 75, 3), 1, 8, 1),
])
def test_rounds_match_oracle(tmp_path, shape, ctas, lanes, pairs, vform):
    import torch
    Y = synth.normal(43, 0, int(np.prod(shape))).reshape(shape, order="F").astype(np.float32)
    Yh = np.fft.fft(Y.astype(np.float64), axis=2)
    sv = np.sort(np.concatenate([np.linalg.svd(Yh[:, :, k], compute_uv=False)
                                 for k in range(shape[2])]))
    tau = float(0.5 * (sv[sv.size // 2 - 1] + sv[sv.size // 2]))
    plans = tmp_path / "plans.txt"
    line = (f"{torch.cuda.get_device_name(0).replace(' ', '_')} {shape[0]} {shape[1]} "
            f"{shape[2] // 2 + 1} {vform} {ctas} {lanes} {pairs} 0\n")
    plans.write_text(line)
    with libtsvd.Context(device=0, stream=torch.cuda.current_stream().cuda_stream, autotune=1,
                         autotune_cache=str(plans), accumulate_v=vform) as ctx:
        y = torch.from_numpy(colmajor(Y)).cuda()
        z = torch.empty_like(y)
        ctx.tsvt(y, z, shape, tau)
        torch.cuda.synchronize()
    assert plans.read_text() == line
    Zo = oracle.tsvt(Y.astype(np.float64), tau)
    assert relerr(uncolmajor(z.cpu().numpy(), shape), Zo, floor=1e-3 * np.linalg.norm(Y)) <= 2e-5
