"""A tile table may ask for slabs of any depth: the loss stays exact.  Images
that are constant along z add the same terms plane after plane, the fastest
way for a thread's partial sums to grow."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fa():
    from paper_2404_01249_gb300 import build, fa
    build.build()
    assert torch.cuda.is_available()
    fa.load()
    yield fa
    fa.fa_autotune_reset()


@pytest.mark.parametrize("depth", [1024, 2048, 4096])
def test_loss_does_not_depend_on_the_slab(fa, depth):
    D, H, W = 4096, 8, 8
    rng = np.random.default_rng(5)  # 14 of 32 pairs of terms sum beyond 2^31 over 4096 planes
    f, m = (torch.from_numpy(rng.random((H, W)).astype(np.float32)).cuda().expand(D, H, W)
            .contiguous() for _ in range(2))
    p = fa.RegParams(scales=(1,), iters=(0,))
    fa.fa_autotune_reset()
    ref = fa.fa_register(f, m, p)["final_loss"]
    fa.fa_autotune_set(0, 2, 0, D, H, W, 0, depth)
    assert fa.fa_register(f, m, p)["final_loss"] == ref
