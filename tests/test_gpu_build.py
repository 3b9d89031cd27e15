"""The device-side index build at the edges of its tiles: the radix sort (6144 pairs a
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
@pytest.mark.parametrize("n", [1, 2, 3, 2047, 2048, 2049, 6143, 6144, 6145, 70001])
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


# one voxel-id brick and several; a fascicle range of more than one bitmap window
# (2^19 ids); Na = 512 (four chunks); a tile of more entries a pass than are staged at
# once (19456); single-entry and empty voxels
@pytest.mark.parametrize("precision", ["bf16", "fp32"])
@pytest.mark.parametrize("dims", [(360, 700, 3000, 60000), (129, 1025, 600000, 30000), (512, 300, 2000, 40000),
                                  (20, 60, 9000, 90000), (384, 127, 4000, 1), (1, 640, 15000, 20000)])
def test_tile_layout_bit_exact(life, dims, precision):
    from test_gpu_tc import expected_tiles
    na, nv, nf, n = dims
    if precision == "fp32" and na > 384:
        pytest.skip("FP32 storage on the tensor cores needs Na <= 384")
    a, v, f, x = raw_list(n, na, nv, nf, n + nv, False)
    v[n // 3:n // 2] = nv // 2        # one very full voxel
    prec = life.LIFE_BF16 if precision == "bf16" else life.LIFE_FP32
    idx = life.index_from_arrays(a, v, f, x, 16, na, nv, nf, precision=prec, algo=life.LIFE_ALGO_TC, brick_dim=6)
    phi = oracle.canon(a, v, f, x, na, nv, nf)
    info, m = idx.info(), idx.nnz
    got = {k: t.cpu().numpy() for k, t in life.life_index_export_tiles(idx).items()}
    exp = expected_tiles(phi, got["tile_vox"], got["brick_tile_ptr"], nv, info["n_sub"])
    for k in ("chunk_ptr", "brick_fasc_ptr"):
        assert np.array_equal(got[k], exp[k]), k
    assert np.array_equal(got["va"][:m].view(np.uint16), exp["va"])
    assert np.array_equal(got["fl"][:m].view(np.uint16), exp["fl"])
    assert np.array_equal(got["brick_fasc"][:info["n_brick_fasc"]], exp["brick_fasc"])
    val = got["val"][:m] if precision == "bf16" else torch.from_numpy(got["val"][:m]).bfloat16().float().numpy()
    assert np.array_equal(val, exp["val"])
    assert np.array_equal(np.sort(got["tile_vox"][got["tile_vox"] >= 0]), np.arange(nv))
