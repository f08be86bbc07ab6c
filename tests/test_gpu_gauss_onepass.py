"""The one-launch Gaussian at the edges of its 32 x 32 tiles and slabs, every
radius it takes (1..6) and the first it does not (7), one to four channels,
against the FP64 oracle; a result over its input or overlapping it equals the
separate one bit for bit.

Tolerance: 1e-5 of the largest value (three FP32 sums of at most 15 products
each: below 3e-6)."""
import ctypes

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


@pytest.mark.parametrize("sigma", [0.3, 0.5, 1.0, 1.3, 1.6, 2.0, 2.3])
@pytest.mark.parametrize("C,shape", [(1, (1, 1, 1)), (3, (5, 31, 33)), (2, (40, 32, 32)),
                                     (4, (9, 33, 65)), (3, (70, 7, 40))])
def test_edges(fa, orc, sigma, C, shape):
    x = np.random.Generator(np.random.PCG64(int(10 * sigma) + C)).normal(
        size=(C,) + shape).astype(np.float32)
    xt = torch.from_numpy(x).cuda()
    y = fa.fa_gauss_smooth(xt, sigma)
    for c in range(C):
        ref = orc.gauss_smooth(x[c], float(np.float32(sigma)))
        assert np.abs(y[c].cpu().double().numpy() - ref).max() <= 1e-5 * np.abs(x).max()
    z = xt.clone()
    fa.fa_gauss_smooth(z, sigma, out=z)
    assert torch.equal(z, y)
    # input and output overlap by all but four elements
    n = xt.numel()
    buf = torch.zeros(n + 4, device="cuda")
    buf[4:] = xt.reshape(-1)
    lib = fa.load()
    vol = lambda p: ctypes.byref(fa.Vol(p, 0, C, *shape))  # noqa: E731
    ws = fa.workspace(lib.fa_gauss_workspace_size(C, *shape))
    fa._check(lib.fa_gauss_smooth(vol(buf.data_ptr() + 16), vol(buf.data_ptr()),
                                  ctypes.c_float(sigma), fa._ptr(ws), ws.numel(), fa._stream()))
    assert torch.equal(buf[:n].reshape(xt.shape), y)
