"""A block of warps whose stack overflows leaves the kernel as a whole and reports it.

The stack's bound keeps an overflow from happening, so the library is linked
once more with the neighbour search's blocks held to 24 entries: one of a
block's warps overflows, the others have nothing to walk."""
import os
import subprocess

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def small_stack(tmp_path_factory):
    import paper_1112_4539_gb300 as bh
    from paper_1112_4539_gb300 import _build as b
    b.build()
    d = tmp_path_factory.mktemp("small_stack")
    obj, lib = str(d / "bh_sph.o"), str(d / "libbhtree_small_stack.so")
    subprocess.run([b.NVCC] + b.FLAGS + ["-DBH_SPH_TEAM_STACK=24", "-c", os.path.join(b.CSRC, "bh_sph.cu"), "-o", obj],
                   check=True, capture_output=True)
    rest = [os.path.join(b.OUT, f[:-3] + ".o") for f in b.sources() if f != "bh_sph.cu"]
    subprocess.run([b.NVCC] + b.ARCH + ["-shared", "-o", lib, obj] + rest + ["--cudart", "shared"], check=True,
                   capture_output=True)
    with pytest.MonkeyPatch.context() as m:
        m.setattr(bh, "LIB_PATH", lib)
        m.setattr(bh, "_lib", None)
        yield bh


@pytest.mark.parametrize("G", [32, 256])
@pytest.mark.parametrize("far", [1, 4])
def test_overflow_ends_the_search(small_stack, G, far):
    """6000 particles fill one node of level 4 and `far` single ones are leaves of level 1, so that the node's
    index is 4 + far: warp 5 of 8 (1 of 4) walks it, or warp 0.  Its pushes: 1 range, 8, then 32 beside 4."""
    bh = small_stack
    rng = np.random.default_rng(3)
    pos = np.full((6000 + far, 4), 1e-3, np.float32)
    pos[:6000, :3] = rng.uniform(0.0, 1.0 / 17.0, (6000, 3))
    pos[0, :3] = 0.0
    pos[6000:, :3] = np.array([[1, 1, 1], [1, 0, 0], [0, 1, 0], [1, 1, 0]])[:far]
    pos = torch.from_numpy(pos).cuda()
    ctx = bh.Context(6000 + far, leaf_size=4, group_size=G)
    ref = ctx.evaluate(pos, 0.5, 0.01).cpu().numpy()
    level = ctx.export("node_level")
    assert (level == 4).sum() == 1 and level[4 + far] == 4
    ctx.neighbors(pos, 0.2)
    assert ctx.status() == bh.BH_ERR_CAPACITY
    assert ctx.status() == bh.BH_OK
    np.testing.assert_array_equal(ctx.evaluate(pos, 0.5, 0.01).cpu().numpy(), ref)
    assert ctx.status() == bh.BH_OK
    ctx.close()
