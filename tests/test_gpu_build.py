"""The device-side index build at the edges of its tiles: the radix sort (8192 pairs a
block), the merge (2048 keys a block) and the tile layout's counting sorts, bit for bit
against the oracle's restructured orders and a host re-derivation."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def life():
    import paper_1905_06234_gb300 as L
    L.load(build_if_missing=True)
    return L


def raw_list(n, na, nv, nf, seed, by_fascicle):
    """n raw entries, a fifth of them repeats of others, in fascicle order or none."""
    rng = np.random.default_rng(seed)
    a, v, f = (rng.integers(0, k, n).astype(np.int32) for k in (na, nv, nf))
    src, dst = rng.integers(0, n, n // 5), rng.integers(0, n, n // 5)
    a[dst], v[dst], f[dst] = a[src], v[src], f[src]
    x = rng.uniform(0.5, 1.0, n).astype(np.float32)
    if by_fascicle:
        o = np.argsort(f, kind="stable")
        a, v, f, x = a[o], v[o], f[o], x[o]
    return a, v, f, x


@pytest.mark.parametrize("by_fascicle", [True, False])
@pytest.mark.parametrize("n", [1, 2, 3, 2047, 2048, 2049, 8191, 8192, 8193, 70001])
@pytest.mark.parametrize("dims", [(360, 500, 2000), (1, 1, 65537), (5, 40000, 3)])
def test_orders_bit_exact(life, n, dims, by_fascicle):
    na, nv, nf = dims
    a, v, f, x = raw_list(n, na, nv, nf, n + na, by_fascicle)
    idx = life.index_from_arrays(a, v, f, x, 8, na, nv, nf)
    for layout, order in ((life.LIFE_LAYOUT_VOXEL, oracle.ORDER_VOXEL), (life.LIFE_LAYOUT_FIBER, oracle.ORDER_FIBER),
                          (life.LIFE_LAYOUT_ATOM, oracle.ORDER_ATOM)):
        ref = oracle.canon(a, v, f, x, na, nv, nf, order)
        got = [t.cpu().numpy() for t in life.life_index_export(idx, layout)]
        for g, r in zip(got, (ref.atom, ref.voxel, ref.fasc, ref.val)):
            assert np.array_equal(g, r), (layout, n)
    ptr = life.life_index_export_voxel_streams(idx)[0].cpu().numpy()
    assert np.array_equal(ptr, np.searchsorted(oracle.canon(a, v, f, x, na, nv, nf).voxel, np.arange(nv + 1)))


def test_unaligned_input_arrays(life):
    """Input arrays that start off a 16-byte boundary are read entry by entry."""
    a, v, f, x = raw_list(5001, 50, 300, 700, 3, False)
    t = [torch.from_numpy(np.concatenate([y[:1], y])).cuda()[1:] for y in (a, v, f, x)]
    idx = life.life_build_index(*t, 8, 50, 300, 700)
    ref = oracle.canon(a, v, f, x, 50, 300, 700)
    got = [y.cpu().numpy() for y in life.life_index_export(idx)]
    assert all(np.array_equal(g, r) for g, r in zip(got, (ref.atom, ref.voxel, ref.fasc, ref.val)))
