"""Symmetric registration over several iterations and levels whose updates run
as the fused update kernels, as one kernel per step, or change between the two
from level to level (rows that are no multiple of 4 with MSE or the Jacobian
direction) and on padded rows (LNCC at an odd width),
against the oracle: both maps, the composed map and both losses."""
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


def mean_disp(a, b):
    d = a.cpu().double().numpy() - b
    return float(np.sqrt((d ** 2).sum(0)).mean())


@pytest.mark.parametrize("shape,kw", [
    ((12, 15, 21), dict()),                        # padded rows on both levels
    ((15, 12, 23), dict(window=7, scales=(3, 1))),
    ((14, 13, 20), dict(loss="mse")),              # 10: one kernel per step, 20: fused
    ((13, 14, 26), dict(loss="mse")),              # both one kernel per step
    ((12, 14, 24), dict(use_jac=True)),            # both fused, dense rows
    ((14, 12, 20), dict(use_jac=True)),            # per step, then fused
    ((12, 13, 40), dict(loss="mse", use_jac=True, scales=(5, 2, 1), iters=(6, 6, 4))),
])
def test_matches_oracle(fa, orc, shape, kw):
    f, m, _ = synth.blobs_pair(shape=shape, sigma=2.5, max_disp=1.5)
    kw = dict(dict(scales=(2, 1), iters=(12, 8)), **kw)
    inv = dict(scales=(2, 1), iters=(10, 6))
    r = fa.fa_register_symmetric(torch.from_numpy(f).cuda(), torch.from_numpy(m).cuda(),
                                 fa.RegParams(**kw), fa.RegParams(**inv))
    okw = {k: v for k, v in kw.items() if k not in ("scales", "iters")}
    ref = orc.register_symmetric(f, m, list(kw["scales"]), list(kw["iters"]),
                                 inv_scales=inv["scales"], inv_iters=inv["iters"], **okw)
    # the bars of the other whole registrations
    assert abs(r["final_loss"] - ref["final_loss"]) < 1e-3
    assert abs(r["final_mid_loss"] - ref["mid_loss"]) < 1e-3
    for k in ("uF", "uM", "u"):
        assert np.abs(ref[k]).max() > 0
        assert mean_disp(r[k], ref[k]) < 0.05, k
