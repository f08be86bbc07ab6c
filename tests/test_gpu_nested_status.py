"""What the kernels of the post-hoc inverse and of symmetric registration
record reaches the caller: the nested inverse's status word is part of the
symmetric call's, and a bounded wait that gave up raises.  Nothing waits for
long here: the timeout is the library's own self-test, run on the call's
workspace."""
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


def pair(shape):
    f, m, _ = synth.blobs_pair(shape=shape, sigma=2.5, max_disp=1.5)
    return torch.from_numpy(f).cuda(), torch.from_numpy(m).cuda()


@pytest.mark.parametrize("shape", [(10, 10, 10), (10, 12, 8)])  # per-step kernels, fused update
def test_nested_inverse_status_is_the_calls(fa, shape):
    """The inverse's directions overflow |d|^2 (reported as non-finite) while
    its field stays finite: one step of +-a per component, a = 1.75e-20 * voxels,
    gives the inverse a gradient of +-4a / voxels = 7e-20, whose square
    (times 1 - beta2 = 2^-24) underflows, so d = 7e-20 / adam_eps = 2.3e19 at
    every voxel that moves; no finite maximum is left and the step is 0."""
    f, m = pair(shape)
    n = shape[0] * shape[1] * shape[2]
    a = 7e-20 * n / 4
    plain = dict(scales=(1,), iters=(1,), sigma_grad=0.0, sigma_warp=0.0)
    P = fa.RegParams(lr=a * 2 * 3 ** 0.5, adam_eps=1e-30, **plain)
    Pi = fa.RegParams(adam_eps=3e-39, beta2=1 - 2.0 ** -24, **plain)
    p, pi = P.to_c(), Pi.to_c()
    ws = fa.workspace(fa.load().fa_register_symmetric_workspace_size(
        *shape, ctypes.byref(p), ctypes.byref(pi)))
    r = fa.fa_register_symmetric(f, m, P, Pi, sync=False, ws=ws)
    assert torch.isfinite(r["u"]).all() and torch.isfinite(r["loss"]) and r["uF"].abs().max() > 0
    wi = fa.workspace(fa.load().fa_inverse_workspace_size(*shape, ctypes.byref(pi)))
    fa.fa_inverse(r["uF"], Pi, sync=False, ws=wi)
    for w in (wi, ws):
        with pytest.raises(fa.FAError) as e:
            fa.fa_ws_status(w)
        assert e.value.status == fa.FA_ERR_NONFINITE


class TimedOut:
    """The library, with the named call's workspace left as after a timeout."""

    def __init__(self, lib, name):
        self.lib, self.name = lib, name

    def __getattr__(self, k):
        real = getattr(self.lib, k)
        if k != self.name:
            return real

        def call(*args):
            st = real(*args)
            ws, nbytes, stream = args[-3:]
            assert self.lib.fa_selftest_wait_timeout(ws, nbytes, 1 << 12, stream) == 0
            return st
        return call


def test_timeout_raises(fa, monkeypatch):
    f, m = pair((9, 10, 12))
    P = fa.RegParams(scales=(1,), iters=(1,))
    u = torch.zeros((3, 9, 10, 12), device="cuda")
    calls = (("fa_inverse", lambda **kw: fa.fa_inverse(u, P, **kw)),
             ("fa_register_symmetric", lambda **kw: fa.fa_register_symmetric(f, m, P, P, **kw)))
    lib = fa.load()
    for name, call in calls:
        call()
        monkeypatch.setattr(fa, "load", lambda path=None, n=name: TimedOut(lib, n))
        with pytest.raises(fa.FAError) as e:
            call()
        assert e.value.status == fa.FA_ERR_TIMEOUT
        call(sync=False)
        torch.cuda.synchronize()
        monkeypatch.undo()
