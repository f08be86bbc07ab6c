"""The LNCC window kernels on volumes of one plane, and of one row per plane
(the same memory): every window against the oracle, loss and both gradients,
at the edges of the kernels' tiles; a registration of such images against the
plain schedule's bits.  Bar: 1e-5, as on the other grids."""
import numpy as np
import pytest
import torch

from paper_2404_01249_gb300 import synth

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def fa():
    from paper_2404_01249_gb300 import build, fa
    build.build()
    assert torch.cuda.is_available()
    fa.load()
    return fa


def rel(a, b):
    d = np.abs(a.cpu().double().numpy().reshape(b.shape) - b).max()
    return float(d / max(np.abs(b).max(), 1e-300))


@pytest.mark.parametrize("window", [1, 3, 5, 7, 9, 11, 13, 15])
@pytest.mark.parametrize("hw", [(1, 1), (8, 32), (17, 33), (40, 70)])
def test_one_plane(fa, orc, window, hw):
    rng = np.random.Generator(np.random.PCG64(window))
    I = rng.random((1,) + hw).astype(np.float32)
    J = (0.5 * I + 0.5 * rng.random((1,) + hw)).astype(np.float32)
    f, m = torch.from_numpy(I).cuda(), torch.from_numpy(J).cuda()
    r = fa.fa_lncc_fwd_bwd(f, m, window, 1e-5, True, True)
    rows = (hw[0], 1, hw[1])
    q = fa.fa_lncc_fwd_bwd(f.view(rows), m.view(rows), window, 1e-5, True, True)
    for k in ("loss", "dJ", "dI"):
        assert torch.equal(r[k].reshape(-1), q[k].reshape(-1)), k
    ref = orc.lncc(I, J, window, np.float32(1e-5), want_dJ=True, want_dI=True)
    assert abs(float(r["loss"]) - ref["loss"]) <= TOL * max(1.0, abs(ref["loss"]))
    if window > 1 and hw != (1, 1):
        assert rel(r["dJ"], ref["dJ"]) <= TOL and rel(r["dI"], ref["dI"]) <= TOL


@pytest.mark.parametrize("window", [3, 9, 13])
@pytest.mark.parametrize("shape", [(1, 34, 41), (34, 1, 40)])
def test_registration(fa, window, shape):
    f, m, _ = synth.blobs_pair(shape=(1, 34, shape[2]), sigma=3.0, max_disp=1.5)
    f, m = (torch.from_numpy(x).cuda().reshape(shape) for x in (f, m))
    kw = dict(scales=(2, 1), iters=(4, 4), window=window)
    a = fa.fa_register(f, m, fa.RegParams(mode="plain", **kw))
    b = fa.fa_register(f, m, fa.RegParams(mode="fused", **kw))
    assert torch.equal(a["u"], b["u"]) and a["final_loss"] == b["final_loss"]
    assert b["u"].abs().max() > 0
