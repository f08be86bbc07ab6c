"""The two update kernels of the fused iteration (smoothing with Adam, compose
with smoothing) at every radius they take, at the edges of their 32 x 8 and
32 x 16 tiles and of their slabs, with row lengths that tile copies take and
row lengths they do not, against the one-kernel-per-step schedule; and the
loops that borrow them: symmetric registration against its per-step calls,
the inverse against the oracle.

The two schedules form the same products and add them in the same order, so the
fields are equal bit for bit."""
import numpy as np
import pytest
import torch

from paper_2404_01249_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fa():
    from paper_2404_01249_gb300 import build, fa
    build.build()
    assert torch.cuda.is_available()
    fa.load()
    return fa


def pair(shape):
    f, m, _ = synth.blobs_pair(shape=shape, sigma=2.5, max_disp=1.5)
    return torch.from_numpy(f).cuda(), torch.from_numpy(m).cuda()


# radii 0..6 of both filters: sigma = R / 3
@pytest.mark.parametrize("rg,rw", [(0, 0), (1, 2), (2, 1), (3, 2), (4, 3), (5, 6), (6, 4), (3, 5)])
@pytest.mark.parametrize("shape", [(8, 8, 8), (9, 17, 33), (21, 15, 32), (12, 32, 65), (70, 9, 36)])
def test_fused_equals_plain(fa, rg, rw, shape):
    f, m = pair(shape)
    kw = dict(scales=(1,), iters=(4,), sigma_grad=rg / 3, sigma_warp=rw / 3)
    a = fa.fa_register(f, m, fa.RegParams(mode="plain", **kw), sync=True)
    b = fa.fa_register(f, m, fa.RegParams(mode="fused", **kw), sync=True)
    assert torch.isfinite(b["u"]).all() and b["u"].abs().max() > 0
    assert torch.equal(a["u"], b["u"])


@pytest.mark.parametrize("loss", ["lncc", "mse"])
@pytest.mark.parametrize("shape", [(11, 17, 33), (9, 14, 36)])
def test_symmetric_iteration(fa, loss, shape):
    """One iteration against its per-step calls, whose bias corrections are
    formed on the device: the directions differ by a few ulps (below 1e-6)."""
    f, m = pair(shape)
    p = fa.RegParams(scales=(1,), iters=(1,), loss=loss)
    r = fa.fa_register_symmetric(f, m, p, fa.RegParams(scales=(1,), iters=(1,)))
    zero = torch.zeros((3,) + shape, device="cuda")
    _, gF, gM = fa.fa_symmetric_loss_grad(f, m, zero, zero, 5, loss)
    for g, name in ((gF, "uF"), (gM, "uM")):
        t = torch.zeros(1, dtype=torch.int32, device="cuda")
        u, _ = fa.fa_radam_step(zero, zero.clone(), zero.clone(),
                                fa.fa_gauss_smooth(g, p.sigma_grad), t, p)
        u = fa.fa_gauss_smooth(u, p.sigma_warp)
        assert u.abs().max() > 0
        assert (r[name] - u).abs().max() <= 1e-5 * u.abs().max()


@pytest.mark.parametrize("shape", [(11, 17, 33), (9, 14, 36)])
def test_inverse(fa, orc, shape):
    u = synth.random_field(shape, 3.0, 1.2, seed=5).astype(np.float32)
    r = fa.fa_inverse(torch.from_numpy(u).cuda(), fa.RegParams(scales=(2, 1), iters=(20, 10)))
    d = np.sqrt(((r["w"].cpu().double().numpy() - orc.inverse(u, [2, 1], [20, 10])["w"]) ** 2).sum(0))
    assert d.mean() <= 0.01 and d.max() <= 0.05  # as on the grids of test_gpu_inverse.py
