"""Steps of a voxel and more: the fused schedule's compose gathers u from
global memory, all three channels of a position at once, inside and across the
grid's faces, on padded rows.  It equals the plain schedule's bit for bit."""
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


# radii 0..6 of the compose's smoothing, on 32 x 8 and 32 x 16 tiles; steps of
# up to 1.25 voxels (some below one: both rules for the cell) and 6
@pytest.mark.parametrize("rw", [0, 1, 2, 3, 5, 6])
@pytest.mark.parametrize("lr", [2.5, 12.0])
@pytest.mark.parametrize("shape", [(9, 10, 12), (12, 18, 33), (40, 17, 35)])
def test_fused_equals_plain(fa, rw, lr, shape):
    f, m, _ = synth.blobs_pair(shape=shape, sigma=2.5, max_disp=1.5)
    f, m = torch.from_numpy(f).cuda(), torch.from_numpy(m).cuda()
    kw = dict(scales=(1,), iters=(4,), sigma_warp=rw / 3, lr=lr)
    a = fa.fa_register(f, m, fa.RegParams(mode="plain", **kw))
    b = fa.fa_register(f, m, fa.RegParams(mode="fused", **kw))
    assert torch.isfinite(b["u"]).all() and b["u"].abs().max() > 0
    assert torch.equal(a["u"], b["u"])
