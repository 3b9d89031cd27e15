"""The index build gives its temporary memory back: after builds whose bricks have to
be split (a brick of more fascicles than its table holds, several times over), the
device's stream-ordered pool holds no more than before them."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

USED_MEM_CURRENT = 7  # CU_MEMPOOL_ATTR_USED_MEM_CURRENT


@pytest.fixture(scope="module")
def life():
    import paper_1905_06234_gb300 as L
    L.load(build_if_missing=True)
    return L


def pool_used():
    """Bytes allocated from the default memory pool of the current device."""
    cu = ctypes.CDLL("libcuda.so.1")
    dev, pool, used = ctypes.c_int(), ctypes.c_void_p(), ctypes.c_uint64()
    assert cu.cuDeviceGet(ctypes.byref(dev), torch.cuda.current_device()) == 0
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), dev) == 0
    assert cu.cuMemPoolGetAttribute(pool, USED_MEM_CURRENT, ctypes.byref(used)) == 0
    return used.value


def build(life, nf, autotune=False):
    """32^3 voxels, one entry per fascicle: a brick of 16^3 voxels touches nf / 8 fascicles."""
    rng = np.random.default_rng(5)
    v = rng.integers(0, 32 ** 3, nf).astype(np.int32)
    k, j, i = np.unravel_index(np.arange(32 ** 3), (32, 32, 32))
    ijk = np.stack([i, j, k], 1).astype(np.int32).reshape(-1)
    dev = lambda t: torch.from_numpy(t).cuda()
    idx = life.life_build_index(dev(rng.integers(0, 20, nf).astype(np.int32)), dev(v), dev(np.arange(nf, dtype=np.int32)),
                                dev(np.ones(nf, np.float32)), 8, 20, 32 ** 3, nf, voxel_ijk=dev(ijk),
                                precision=life.LIFE_BF16, algo=life.LIFE_ALGO_TC, brick_dim=16, autotune=autotune)
    edge = idx.info()["brick_edge"]
    idx.close()
    return edge


@pytest.mark.parametrize("autotune", [False, True])
def test_split_bricks_leave_no_temporaries(life, autotune):
    build(life, 1000)
    torch.cuda.synchronize()
    before = pool_used()
    for _ in range(3):
        edge = build(life, 600000, autotune)
        assert autotune or edge < 16        # 75000 fascicles a 16^3 brick: split until 15872 or fewer are left
    torch.cuda.synchronize()
    assert pool_used() == before
