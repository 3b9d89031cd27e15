"""The tile layout where it is built by sorting instead of by counting: few, very full
tiles, and more fascicles than are worth walking a brick's entries for.  Bit for bit
against the host re-derivation (FP32 values unrounded), both SpMVs exactly in whole
numbers (every entry of both streams at its place), on both sides of the rule; and the
time: such an index builds about as fast as one whose entries are spread out."""
import time

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


def entries(na, nv, nf, n, seed, one_voxel=0.0):
    rng = np.random.default_rng(seed)
    a, v, f = (rng.integers(0, k, n).astype(np.int32) for k in (na, nv, nf))
    v[:int(one_voxel * n)] = nv // 2
    keep = np.unique((v.astype(np.int64) * na + a) * nf + f, return_index=True)[1]  # no repeats: values stay 1
    return a[keep], v[keep], f[keep]


def check_exact(life, idx, a, v, f, nt, na, nv, nf, seed):
    """DSC and WC in whole numbers small enough that every rounding on the way is exact."""
    rng = np.random.default_rng(seed)
    D, r, w = rng.integers(-2, 3, (na, nt)), rng.integers(-3, 4, (nv, nt)), rng.integers(0, 2, nf)
    dev = lambda x: torch.from_numpy(x.astype(np.float32).reshape(-1)).cuda()
    S = np.zeros((nv, na), np.int64)
    np.add.at(S, (v, a), w[f])
    assert S.max() <= 2048                                  # exact as an FP16 operand
    g = np.zeros(nf, np.int64)
    np.add.at(g, f, (r @ D.T)[v, a])
    y = life.life_dsc(idx, dev(D), dev(w))[0].cpu().numpy()
    got = life.life_wc(idx, dev(D), dev(r))[0].cpu().numpy()
    life.life_check_device_status()
    assert np.array_equal(y, (S @ D).reshape(-1).astype(np.float32))
    assert np.array_equal(got, g.astype(np.float32))


# sorted: full tiles, one full voxel, Na = 512 (four chunks), a few voxels; counted: a pass
# of more entries than are staged at once (19456), ordinary tiles
SHAPES = [(360, 100, 3000, 200000, 0.0), (20, 60, 9000, 120000, 0.0), (360, 700, 3000, 150000, 0.6),
          (512, 130, 5000, 300000, 0.0), (40, 3, 2000, 90000, 0.0), (384, 1, 15000, 200000, 0.0),
          (128, 128, 3000, 26000, 0.0), (129, 1025, 6000, 30000, 0.0)]


@pytest.mark.parametrize("precision", ["bf16", "fp32"])
@pytest.mark.parametrize("dims", SHAPES)
def test_layout_and_products(life, dims, precision):
    from test_gpu_tc import expected_tiles
    na, nv, nf, n, one = dims
    if precision == "fp32" and na > 384:
        pytest.skip("FP32 storage on the tensor cores needs Na <= 384")
    prec = life.LIFE_BF16 if precision == "bf16" else life.LIFE_FP32
    a, v, f = entries(na, nv, nf, n, n + nv, one)
    x = np.random.default_rng(n).uniform(0.5, 1.0, len(a)).astype(np.float32)
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
    if precision == "fp32":     # the values in stream order, all 32 bits
        tile, row = np.zeros(nv, np.int64), np.zeros(nv, np.int64)
        at = np.flatnonzero(got["tile_vox"] >= 0)
        tile[got["tile_vox"][at]], row[got["tile_vox"][at]] = at // 128, at % 128
        t, r, q = tile[phi.voxel], row[phi.voxel], phi.atom.astype(np.int64)
        cell = ((q >> 7) << 14) | ((r >> 3) << 10) | (((q >> 3) & 15) << 6) | ((r & 7) << 3) | (q & 7)
        assert np.array_equal(got["val"][:m].view(np.uint32), phi.val[np.lexsort((phi.fasc, cell, t))].view(np.uint32))
    else:
        assert np.array_equal(got["val"][:m], exp["val"])
    one_idx = life.index_from_arrays(a, v, f, np.ones(len(a), np.float32), 16, na, nv, nf, precision=prec,
                                     algo=life.LIFE_ALGO_TC, brick_dim=6)
    check_exact(life, one_idx, a, v, f, 16, na, nv, nf, n)


@pytest.mark.parametrize("precision", ["bf16", "fp32"])
def test_split_bricks(life, precision):
    """One 8^3 brick of 40000 fascicles, far above a table's 15872: split several times, the
    full tiles of the first attempts sorted and the small ones of the last counted."""
    na, nv, nf = 60, 512, 40000
    a, v, f = entries(na, nv, nf, 400000, 7)
    k, j, i = np.unravel_index(np.arange(nv), (8, 8, 8))
    prec = life.LIFE_BF16 if precision == "bf16" else life.LIFE_FP32
    idx = life.index_from_arrays(a, v, f, np.ones(len(a), np.float32), 8, na, nv, nf,
                                 voxel_ijk=np.stack([i, j, k], 1).astype(np.int32), precision=prec,
                                 algo=life.LIFE_ALGO_TC, brick_dim=8)
    assert idx.info()["n_bricks"] > 8
    check_exact(life, idx, a, v, f, 8, na, nv, nf, 3)


@pytest.mark.parametrize("precision", ["bf16", "fp32"])
def test_batch_of_full_tiles(life, precision):
    prec = life.LIFE_BF16 if precision == "bf16" else life.LIFE_FP32
    na, ps = 90, [(100, 4000, 150000), (130, 3000, 90000)]
    raw = [entries(na, nv, nf, n, n) for nv, nf, n in ps]
    idx = [life.index_from_arrays(a, v, f, np.ones(len(a), np.float32), 16, na, p[0], p[1], precision=prec,
                                  algo=life.LIFE_ALGO_TC) for (a, v, f), p in zip(raw, ps)]
    batch = life.life_batch_create(idx, algo=life.LIFE_ALGO_TC)
    a = np.concatenate([t[0] for t in raw])
    v = np.concatenate([raw[0][1], raw[1][1] + ps[0][0]])
    f = np.concatenate([raw[0][2], raw[1][2] + ps[0][1]])
    check_exact(life, batch.index, a, v, f, 16, na, ps[0][0] + ps[1][0], ps[0][1] + ps[1][1], 11)


def test_many_fascicles_bit_exact(life):
    """10^8 fascicle ids, few of them used: 191 windows of 2^19 ids a brick if counted."""
    from test_gpu_tc import expected_tiles
    na, nv, nf = 30, 20000, 100_000_000
    a, v, f = entries(na, nv, nf, 30000, 2)
    idx = life.index_from_arrays(a, v, f, np.ones(len(a), np.float32), 8, na, nv, nf, precision=life.LIFE_BF16,
                                 algo=life.LIFE_ALGO_TC)
    info, m = idx.info(), idx.nnz
    got = {k: t.cpu().numpy() for k, t in life.life_index_export_tiles(idx).items()}
    exp = expected_tiles(oracle.canon(a, v, f, np.ones(len(a), np.float32), na, nv, nf), got["tile_vox"],
                         got["brick_tile_ptr"], nv, info["n_sub"])
    assert np.array_equal(got["brick_fasc_ptr"], exp["brick_fasc_ptr"])
    assert np.array_equal(got["brick_fasc"][:info["n_brick_fasc"]], exp["brick_fasc"])
    assert np.array_equal(got["fl"][:m].view(np.uint16), exp["fl"])


def build_s(life, n, nv, nf, seed=1):
    """Shortest build time of n random entries (sorted by fascicle), BF16 on the tensor cores."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    ints = lambda k: torch.randint(0, k, (n,), generator=g, device="cuda", dtype=torch.int32)
    a, v, f = ints(360), ints(nv), ints(nf).sort()[0]
    x, t = torch.rand(n, generator=g, device="cuda") + 0.5, []
    for _ in range(6):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        life.life_build_index(a, v, f, x, 16, 360, nv, nf, precision=life.LIFE_BF16, algo=life.LIFE_ALGO_TC).close()
        t.append(time.perf_counter() - t0)
    return min(t[1:])


def test_full_tiles_build_as_fast(life):
    """2M entries in 128 voxels against 2M in 262144: no more than five times as long."""
    assert build_s(life, 2_000_000, 128, 10000) <= 5 * build_s(life, 2_000_000, 64 ** 3, 500000)


def test_many_fascicles_build_as_fast(life):
    """1M entries in 4M voxels: 10^8 fascicle ids take no more than twice as long as 500000."""
    assert build_s(life, 1_000_000, 4_000_000, 100_000_000) <= 2 * build_s(life, 1_000_000, 4_000_000, 500000)
