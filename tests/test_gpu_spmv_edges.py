"""DSC and WC of the tensor-core forms at the shapes where a launch's division of the
work changes: Nθ at the 4-, 8- and 16-value steps of the loaders and epilogues, one
to many tiles and bricks, tiles with far fewer entries than the producer warps take
at once.  Tolerances are those of the existing parity tests (FP32 form 1e-5 relative
L2, BF16 form the rounding-model bounds of test_gpu_tc)."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_tc import rel, rounding_bounds

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def life():
    import paper_1905_06234_gb300 as L
    L.load(build_if_missing=True)
    return L


def problem(nt, na, nv, nf, n, seed):
    rng = np.random.default_rng(seed)
    a, v, f = (rng.integers(0, k, n).astype(np.int32) for k in (na, nv, nf))
    x = rng.uniform(0.5, 1.0, n).astype(np.float32)
    D = rng.standard_normal((na, nt)).astype(np.float32)
    return a, v, f, x, (D - D.mean(1, keepdims=True)).astype(np.float32).reshape(-1)


def check(life, form, nt, na, nv, nf, n, brick_dim, seed=5):
    a, v, f, x, D = problem(nt, na, nv, nf, n, seed)
    prec = life.LIFE_BF16 if form == "bf16" else life.LIFE_FP32
    idx = life.index_from_arrays(a, v, f, x, nt, na, nv, nf, precision=prec, algo=life.LIFE_ALGO_TC,
                                 brick_dim=brick_dim)
    phi = oracle.canon(a, v, f, x, na, nv, nf)
    rng = np.random.default_rng(seed + 1)
    w, r, b = (rng.standard_normal(k).astype(np.float32) for k in (nf, nt * nv, nt * nv))
    dev = lambda t: torch.from_numpy(t).cuda()
    e, ss = life.life_dsc(idx, dev(D), dev(w), b=dev(b), sumsq=True)
    y, _ = life.life_dsc(idx, dev(D), dev(w))
    g, _ = life.life_wc(idx, dev(D), dev(r))
    torch.cuda.synchronize()
    life.life_check_device_status()
    y_ref, g_ref = oracle.dsc(phi, D, w, nt, nv), oracle.wc(phi, D, r, nt, nf)
    e, y, g = (t.cpu().numpy().astype(np.float64) for t in (e, y, g))
    assert abs(float(ss) - e @ e) <= 1e-5 * (e @ e)
    if form == "bf16":
        yb, gb = rounding_bounds(phi, D, w, r, nt, nv, nf)
        # the subtraction of b rounds once more to float32
        assert (np.abs(y - y_ref) <= yb + 1e-30).all()
        assert (np.abs(e - (y_ref - b)) <= yb + 2.0 ** -23 * np.abs(y_ref - b) + 1e-30).all()
        assert (np.abs(g - g_ref) <= gb + 1e-30).all()
    else:
        assert rel(y, y_ref) <= 1e-5 and rel(e, y_ref - b) <= 1e-5 and rel(g, g_ref) <= 1e-5


@pytest.mark.parametrize("form", ["bf16", "fp32"])
@pytest.mark.parametrize("nt", [1, 4, 12, 16, 17, 20, 36, 60, 100, 127, 128])
def test_direction_counts(life, form, nt):
    check(life, form, nt, 40, 700, 500, 30000, 8)


@pytest.mark.parametrize("form", ["bf16", "fp32"])
@pytest.mark.parametrize("nv,n,brick_dim", [(1, 50, 8), (127, 3000, 8), (129, 3000, 8), (1025, 500, 8), (4096, 120000, 8),
                                            (20000, 9000, 8), (40000, 300000, 4), (5000, 0, 8), (2048, 200000, 16)])
def test_tile_and_brick_counts(life, form, nv, n, brick_dim):
    check(life, form, 96, 200, nv, 3000, n, brick_dim)


@pytest.mark.parametrize("form", ["bf16", "fp32"])
@pytest.mark.parametrize("edge", [31, 32, 33, 64, 127, 128, 129, 256, 257, 600])
def test_thin_and_thick_segments(life, form, edge):
    """WC segments (32 voxels x 32 atoms) of `edge` entries and of none among thin ones."""
    nt, na, nv, nf = 32, 96, 384, 900
    rng = np.random.default_rng(edge)
    n = 3000
    a, v, f = (rng.integers(0, k, n).astype(np.int32) for k in (na, nv, nf))
    f2 = rng.permutation(nf)[:edge].astype(np.int32)            # one segment gets exactly `edge` distinct entries
    keep = ~((a // 32 == 1) & (v // 32 == 3))
    a = np.concatenate([a[keep], np.full(edge, 32 + 5, np.int32)])
    v = np.concatenate([v[keep], (96 + rng.integers(0, 32, edge)).astype(np.int32)])
    f = np.concatenate([f[keep], f2])
    x = rng.uniform(0.5, 1.0, len(a)).astype(np.float32)
    D, r = (rng.standard_normal(k).astype(np.float32) for k in (nt * na, nt * nv))
    prec = life.LIFE_BF16 if form == "bf16" else life.LIFE_FP32
    idx = life.index_from_arrays(a, v, f, x, nt, na, nv, nf, precision=prec, algo=life.LIFE_ALGO_TC)
    phi = oracle.canon(a, v, f, x, na, nv, nf)
    g, _ = life.life_wc(idx, torch.from_numpy(D).cuda(), torch.from_numpy(r).cuda())
    life.life_check_device_status()
    g, g_ref = g.cpu().numpy(), oracle.wc(phi, D, r, nt, nf)
    if form == "bf16":
        assert (np.abs(g - g_ref) <= rounding_bounds(phi, D, np.zeros(nf, np.float32), r, nt, nv, nf)[1] + 1e-30).all()
    else:
        assert rel(g, g_ref) <= 1e-5
