"""Smoothing of volumes with few rows, on both sides of the height from which
the one-launch kernel takes over, against the FP64 oracle.

Tolerance: 1e-5 of the largest value, as on the other grids."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fa():
    from paper_2404_01249_gb300 import build, fa
    build.build()
    assert torch.cuda.is_available()
    fa.load()
    return fa


@pytest.mark.parametrize("sigma", [0.3, 1.0, 2.0])
@pytest.mark.parametrize("shape", [(40, 1, 70), (33, 2, 35), (9, 5, 33), (9, 6, 33)])
def test_few_rows(fa, orc, sigma, shape):
    x = np.random.Generator(np.random.PCG64(shape[1])).normal(size=(3,) + shape).astype(np.float32)
    xt = torch.from_numpy(x).cuda()
    y = fa.fa_gauss_smooth(xt, sigma)
    for c in range(3):
        ref = orc.gauss_smooth(x[c], float(np.float32(sigma)))
        assert np.abs(y[c].cpu().double().numpy() - ref).max() <= 1e-5 * np.abs(x).max()
    z = xt.clone()
    fa.fa_gauss_smooth(z, sigma, out=z)
    assert torch.equal(z, y)
