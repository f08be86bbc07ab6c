"""Registrations whose levels have rows of an odd length: the fused schedule
pads them (to a multiple of 4) for every loss, direction and width of the
Gaussians.  It equals the plain schedule, which runs on dense rows, bit for
bit; the padding never reaches a result."""
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


@pytest.mark.parametrize("kw", [dict(loss="mse"), dict(loss="mi"), dict(loss="lncc", use_jac=True),
                                dict(loss="mse", use_jac=True), dict(loss="mi", use_jac=True),
                                dict(loss="mse", sigma_grad=2.5), dict(loss="mi", sigma_warp=2.5),
                                dict(loss="lncc", sigma_grad=2.5, sigma_warp=2.5),
                                dict(loss="mse", state="bf16"), dict(loss="mi", lr=2.5)])
@pytest.mark.parametrize("shape", [(12, 18, 33), (9, 13, 6), (10, 17, 35)])
def test_padded_fused_equals_dense_plain(fa, kw, shape):
    f, m, _ = synth.blobs_pair(shape=shape, sigma=2.5, max_disp=1.5)
    # images far from zero: a padding element taken for a voxel would show in
    # the range, the histogram and the maxima
    f, m = (torch.from_numpy(x).cuda() * 3 + 7 for x in (f, m))
    kw = dict(scales=(2, 1), iters=(4, 3), mi_bins=16, **kw)
    a = fa.fa_register(f, m, fa.RegParams(mode="plain", **kw), sync=True)
    b = fa.fa_register(f, m, fa.RegParams(mode="fused", **kw), sync=True)
    assert torch.isfinite(b["u"]).all() and b["u"].abs().max() > 0
    assert torch.equal(a["u"], b["u"])
    assert a["final_loss"] == b["final_loss"]


@pytest.mark.parametrize("loss", ["mse", "mi"])
def test_padded_start_from_a_field(fa, loss):
    shape = (11, 14, 27)
    f, m, _ = synth.blobs_pair(shape=shape, sigma=2.5, max_disp=1.5)
    f, m = (torch.from_numpy(x).cuda() for x in (f, m))
    u0 = torch.from_numpy(synth.random_field(shape, 3.0, 1.0, seed=4)).float().cuda()
    kw = dict(scales=(2, 1), iters=(3, 3), loss=loss, mi_bins=16)
    a = fa.fa_register(f, m, fa.RegParams(mode="plain", **kw), u_init=u0)
    b = fa.fa_register(f, m, fa.RegParams(mode="fused", **kw), u_init=u0)
    assert torch.equal(a["u"], b["u"]) and a["final_loss"] == b["final_loss"]
