"""The two update kernels of the fused iteration (smoothing with Adam, compose
with smoothing) at every radius they take, at the edges of their 32 x 8 and
32 x 16 tiles and of their slabs, with row lengths that tile copies take and
row lengths they do not, against the one-kernel-per-step schedule.

The two schedules form the same products and add them in the same order, so the
fields are equal bit for bit."""
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
