"""MI on both sides of the sizes where its kernels change form (one voxel per
thread in blocks of 512 with four histogram copies; the gradient's one- and
four-voxel forms) against the oracle.  Bar, as on the other grids: 1e-5 of the
loss and, max-abs over max-abs, of dL/dJ."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def fa():
    from paper_2404_01249_gb300 import build, fa
    build.build()
    assert torch.cuda.is_available()
    fa.load()
    return fa


# 512 x 152 voxels and one plane on either side; 2^20 and one plane above; odd
@pytest.mark.parametrize("shape", [(7, 9, 11), (152, 16, 32), (153, 16, 32), (64, 128, 128),
                                   (65, 128, 128), (31, 33, 77)])
@pytest.mark.parametrize("bins", [8, 32, 64])
def test_mi_at_the_lines(fa, orc, shape, bins):
    rng = np.random.Generator(np.random.PCG64(5))
    I = rng.random(shape).astype(np.float32)
    J = (0.5 * I + 0.5 * rng.random(shape)).astype(np.float32)
    r = fa.fa_mi_fwd_bwd(torch.from_numpy(I).cuda(), torch.from_numpy(J).cuda(), bins)
    ref = orc.mi(I, J, bins)
    assert abs(float(r["loss"]) - ref["loss"]) <= TOL * max(1.0, abs(ref["loss"]))
    d = r["dJ"].cpu().double().numpy()
    assert np.abs(d - ref["dJ"]).max() <= TOL * np.abs(ref["dJ"]).max()
