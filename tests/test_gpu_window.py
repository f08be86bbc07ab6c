"""The LNCC window-sum kernels at the edges of their tiles (32 x 16 outputs,
32 x 8 for windows above 7): grids one voxel below, at and above a tile, rows
of odd and even length (single and paired accesses), one-plane grids, every
window's tile and ring, against the FP64 oracle.

Tolerance: 1e-5 of the largest value, as for every kernel (FP32 rounding of
O(100) operations on exact sums is below 1e-6 of it)."""
import ctypes

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


def rel(a, b):
    a, b = a.detach().cpu().double().numpy(), np.asarray(b, np.float64)
    return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-300))


def pair(shape, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    f = rng.uniform(-0.5, 1.0, shape).astype(np.float32)
    m = (0.6 * f + 0.4 * rng.uniform(0.0, 1.0, shape)).astype(np.float32)
    return f, m


@pytest.mark.parametrize("shape,window", [
    ((1, 16, 32), 5), ((4, 15, 31), 5), ((5, 17, 33), 5), ((23, 33, 34), 3), ((2, 3, 2), 5),
    ((9, 16, 64), 1), ((12, 17, 35), 7), ((3, 40, 36), 9), ((11, 9, 33), 11), ((30, 8, 40), 13),
    ((17, 18, 37), 15)])
def test_tile_edges(fa, orc, shape, window):
    f, m = pair(shape, 7 + window)
    ft, mt = torch.from_numpy(f).cuda(), torch.from_numpy(m).cuda()
    out = fa.fa_lncc_fwd_bwd(ft, mt, window, 1e-3, want_dJ=True, want_dI=True)
    ref = orc.lncc(f, m, window, np.float32(1e-3), want_dI=True)
    assert abs(float(out["loss"]) - ref["loss"]) <= TOL * max(abs(ref["loss"]), 1e-6)
    assert rel(out["dJ"], ref["dJ"]) < TOL
    assert rel(out["dI"], ref["dI"]) < TOL
    # one gradient alone and the loss alone give the same bits
    one = fa.fa_lncc_fwd_bwd(ft, mt, window, 1e-3, want_dJ=False, want_dI=True)
    none = fa.fa_lncc_fwd_bwd(ft, mt, window, 1e-3, want_dJ=False)
    assert torch.equal(one["dI"], out["dI"])
    assert float(none["loss"]) == float(out["loss"]) == float(one["loss"])


def test_gradient_written_over_an_input(fa):
    """dL/dJ may be written over the warped image also where dL/dI, which
    still reads that image, is asked for in the same call."""
    f, m = pair((9, 21, 45), 3)
    ft, mt = torch.from_numpy(f).cuda(), torch.from_numpy(m).cuda()
    ref = fa.fa_lncc_fwd_bwd(ft, mt, 5, 1e-5, want_dJ=True, want_dI=True)
    lib = fa.load()
    ws = fa.workspace(lib.fa_lncc_workspace_size(*ft.shape))
    dI = torch.empty_like(ft)
    over = mt.clone()
    fa._check(lib.fa_lncc_fwd_bwd(fa._vol(ft, 1), fa._vol(over, 1), 5, ctypes.c_float(1e-5), None,
                                  fa._vol(over, 1), fa._vol(dI, 1), fa._ptr(ws), ws.numel(),
                                  fa._stream()))
    assert torch.equal(over, ref["dJ"]) and torch.equal(dI, ref["dI"])
