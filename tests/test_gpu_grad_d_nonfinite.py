"""dL/dD with infinite and NaN upstream gradients: the non-finite results are those of
the sum over the entries, val·w·gy each, also where one (atom, voxel) run holds zero
weights or weights of both signs (inf·0 and inf − inf are NaN, not the inf that
inf · Σ val·w would give).  Runs within a 32-entry window, across windows and across
chunks; the finite results keep the 1e-5 of the other dL/dD tests."""
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


def by_entries(phi, w, gy, nt, na):
    ref = np.zeros((na, nt))
    with np.errstate(invalid="ignore"):
        np.add.at(ref, phi.atom, (phi.val.astype(np.float64) * w[phi.fasc])[:, None] *
                  gy.astype(np.float64).reshape(-1, nt)[phi.voxel])
    return ref.reshape(-1)


def check(got, ref):
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    inf = np.isinf(ref)
    assert np.array_equal(np.isinf(got), inf) and np.array_equal(got[inf], ref[inf].astype(np.float32))
    ok = np.isfinite(ref)
    assert np.linalg.norm(got[ok] - ref[ok]) <= 1e-5 * max(np.linalg.norm(ref[ok]), 1e-300)


@pytest.mark.parametrize("w", [(0.0, 1.0), (2.0, -1.0), (1.0, 1.0), (-1.0, -2.0), (0.0, 0.0), (3.0, -3.0)])
def test_one_run(life, w):
    a, v, f = (np.array(t, np.int32) for t in ([0, 0], [0, 0], [0, 1]))
    idx = life.index_from_arrays(a, v, f, np.ones(2, np.float32), 4, 1, 1, 2)
    w, gy = np.array(w, np.float32), np.array([np.inf, -np.inf, np.nan, 2.0], np.float32)
    got = life.life_dsc_grad_D(idx, torch.from_numpy(gy).cuda(), torch.from_numpy(w).cuda()).cpu().numpy()
    check(got, by_entries(oracle.canon(a, v, f, np.ones(2, np.float32), 1, 1, 2), w, gy, 4, 1))


@pytest.mark.parametrize("nt,run", [(1, 2), (33, 5), (96, 31), (96, 33), (150, 300)])
def test_runs_of_mixed_weights(life, nt, run):
    rng = np.random.default_rng(nt + run)
    na, nv, nf = 7, 24, 400
    v, a = (x.astype(np.int32) for x in np.divmod(np.arange(nv * na), na))
    lens = rng.integers(1, run + 1, nv * na)
    v, a = np.repeat(v, lens), np.repeat(a, lens)
    f = np.concatenate([rng.permutation(nf)[:k] for k in lens]).astype(np.int32)
    x = rng.uniform(0.5, 1.0, len(v)).astype(np.float32)
    gy = rng.standard_normal(nt * nv).astype(np.float32)
    gy[rng.integers(0, nt * nv, max(1, nt * nv // 40))] = np.inf
    gy[rng.integers(0, nt * nv, max(1, nt * nv // 80))] = -np.inf
    gy[rng.integers(0, nt * nv, max(1, nt * nv // 200))] = np.nan
    phi = oracle.canon(a, v, f, x, na, nv, nf)
    idx = life.index_from_arrays(a, v, f, x, nt, na, nv, nf)
    for w in (rng.uniform(0.1, 1.0, nf), np.where(rng.random(nf) < 0.3, 0.0, rng.uniform(0.1, 1.0, nf)),
              rng.choice([-1.0, 1.0, 2.0], nf)):
        w = w.astype(np.float32)
        got = life.life_dsc_grad_D(idx, torch.from_numpy(gy).cuda(), torch.from_numpy(w).cuda()).cpu().numpy()
        check(got, by_entries(phi, w, gy, nt, na))
