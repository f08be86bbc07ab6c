"""Outputs that share memory with inputs: a result laid over an image or a
field that the call still reads is the same as one kept apart."""
import ctypes

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


@pytest.mark.parametrize("shape", [(12, 16, 40), (9, 17, 33)])
@pytest.mark.parametrize("channel", [0, 1, 2])
def test_adjoint_field_gradient_over_the_fixed_image(fa, shape, channel):
    f, m, _ = synth.voronoi_pair(shape=shape, seed=321)
    f, m = torch.from_numpy(f).cuda(), torch.from_numpy(m).cuda()
    u = torch.from_numpy(synth.random_field(shape, 3.0, 2.5, seed=9)).float().cuda()
    ref = fa.fa_warp_lncc_adjoint(f, m, u, 5)
    lib = fa.load()
    ws = fa.workspace(lib.fa_warp_lncc_adjoint_workspace_size(*shape))
    # the image's 16-byte aligned place inside the gradient's buffer
    n = f.numel()
    du = torch.empty((3,) + shape, device="cuda")
    fixed = du.view(-1)[channel * n:(channel + 1) * n].view(shape)
    assert fixed.data_ptr() % 16 == 0 or channel  # odd grids: channel 0 only
    if fixed.data_ptr() % 16:
        pytest.skip("an image must start on 16 bytes")
    fixed.copy_(f)
    dI, dM, loss = torch.empty_like(f), torch.empty_like(f), torch.empty((), device="cuda")
    fa._check(lib.fa_warp_lncc_adjoint(fa._vol(fixed, 1), fa._vol(m, 1), fa._vol(u, 3), 5,
                                       ctypes.c_float(1e-5), fa._ptr(loss), fa._vol(du, 3),
                                       fa._vol(dI, 1), fa._vol(dM, 1), fa._ptr(ws), ws.numel(),
                                       fa._stream()))
    assert float(loss) == float(ref["loss"])
    assert torch.equal(du, ref["dL_du"])
    assert torch.equal(dI, ref["dL_dfixed"])
    assert torch.equal(dM, ref["dL_dmoving"])


@pytest.mark.parametrize("steps", [0, 3])
@pytest.mark.parametrize("shift", [0, 0.5])  # u_out starts this much of a field behind v
def test_svf_displacement_over_the_velocity(fa, steps, shift):
    shape = (40, 52, 64)
    n3 = 3 * shape[0] * shape[1] * shape[2]
    f, m, _ = synth.blobs_pair(shape=shape, sigma=3.0)
    f, m = torch.from_numpy(f).cuda(), torch.from_numpy(m).cuda()
    v = torch.from_numpy(synth.random_field(shape, 4.0, 1.5, seed=6)).float().cuda()
    L, g, u = fa.fa_svf_loss_grad(f, m, v, steps)
    off = int(shift * n3)
    buf = torch.empty(n3 + off, device="cuda")
    # early elements of u_out go where late ones of v are
    vo, uo = buf[:n3].view((3,) + shape), buf[off:].view((3,) + shape)
    vo.copy_(v)
    lib, p = fa.load(), fa.RegParams(scales=(1,), iters=(0,)).to_c()
    ws = fa.workspace(lib.fa_register_svf_workspace_size(*shape, ctypes.byref(p), steps))
    go, loss = torch.empty_like(v), torch.empty((), device="cuda")
    fa._check(lib.fa_svf_loss_grad(fa._vol(f, 1), fa._vol(m, 1), fa._vol(vo, 3), ctypes.byref(p),
                                   steps, fa._ptr(loss), fa._vol(go, 3), fa._vol(uo, 3),
                                   fa._ptr(ws), ws.numel(), fa._stream()))
    assert float(loss) == float(L)
    assert torch.equal(go, g) and torch.equal(uo, u)
