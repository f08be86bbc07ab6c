"""Run by test_gpu_device_reset.py in a process of its own: losses, their
gradients and a registration through the C ABI on raw device memory, then
cudaDeviceReset (which ends this process' context), then the same again.
Prints OK when every output has the same bytes."""
import ctypes
import os
import sys

import numpy as np
import torch  # noqa: F401  (loads the CUDA runtime the library links against)

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
from paper_2404_01249_gb300 import fa, synth  # noqa: E402

SHAPE = (20, 24, 28)
N = SHAPE[0] * SHAPE[1] * SHAPE[2]


def outputs(rt, lib, f, m):
    def check(st, what):
        assert st == 0, (what, st, lib.fa_last_error())

    def dev(nbytes):
        p = ctypes.c_void_p()
        check(rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(max(nbytes, 256))), "cudaMalloc")
        return p

    def vol(p, C):
        return ctypes.byref(fa.Vol(p.value, 0, C, *SHAPE))

    I, J, loss = dev(4 * N), dev(4 * N), dev(4)
    for d, h in ((I, f), (J, m)):
        check(rt.cudaMemcpy(d, h.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(4 * N), 1), "copy")
    res = []

    def take(*ps_n):
        check(rt.cudaDeviceSynchronize(), "synchronize")
        for p, n in ps_n:
            h = np.empty(n, np.float32)
            check(rt.cudaMemcpy(h.ctypes.data_as(ctypes.c_void_p), p, ctypes.c_size_t(4 * n), 2), "copy")
            res.append(h.tobytes())

    dJ, dI = dev(4 * N), dev(4 * N)
    n = lib.fa_lncc_workspace_size(*SHAPE)
    check(lib.fa_lncc_fwd_bwd(vol(I, 1), vol(J, 1), 5, 1e-5, loss, vol(dJ, 1), vol(dI, 1), dev(n), n,
                              None), "lncc")
    take((loss, 1), (dJ, N), (dI, N))
    check(lib.fa_lncc_fwd_bwd_noalloc(vol(I, 1), vol(J, 1), 5, 1e-5, loss, vol(dJ, 1), vol(dI, 1),
                                      None), "lncc without a workspace")
    take((loss, 1), (dJ, N), (dI, N))
    n = lib.fa_mi_workspace_size(32)
    check(lib.fa_mi_fwd_bwd(vol(I, 1), vol(J, 1), 32, None, loss, vol(dJ, 1), dev(n), n, None), "mi")
    take((loss, 1), (dJ, N))
    for mode in ("plain", "fused", "persistent"):
        p = fa.RegParams(scales=(2, 1), iters=(3, 2), mode=mode, graph=False).to_c()
        u = dev(12 * N)
        n = lib.fa_register_workspace_size(*SHAPE, ctypes.byref(p))
        check(lib.fa_register(vol(I, 1), vol(J, 1), ctypes.byref(p), vol(u, 3), loss, None, dev(n), n,
                              None), mode)
        take((loss, 1), (u, 3 * N))
    return res


def main():
    lib, rt = fa.load(), ctypes.CDLL("libcudart.so.13")
    f, m, _ = synth.blobs_pair(shape=SHAPE, sigma=3.0)
    f, m = (np.ascontiguousarray(x, dtype=np.float32) for x in (f, m))
    before = outputs(rt, lib, f, m)
    assert rt.cudaDeviceReset() == 0
    assert before == outputs(rt, lib, f, m)
    print("OK")


if __name__ == "__main__":
    main()
