"""FP32 storage on the tensor cores with Nθ off a multiple of 4, whose rows of b and y
are read and written value by value: the DSC with b is exact in whole numbers at every
remainder, and costs little more than with aligned rows of the next multiple of 4."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def life():
    import paper_1905_06234_gb300 as L
    L.load(build_if_missing=True)
    return L


def problem(life, nt, na, nv, nf, n):
    rng = np.random.default_rng(7)
    a, v, f = (rng.integers(0, k, n).astype(np.int32) for k in (na, nv, nf))
    idx = life.index_from_arrays(a, v, f, np.ones(n, np.float32), nt, na, nv, nf, algo=life.LIFE_ALGO_TC)
    D, w, b = rng.integers(-2, 3, (na, nt)), rng.integers(0, 2, nf), rng.integers(-9, 10, (nv, nt))
    return idx, (a, v, f), (D, w, b), [torch.from_numpy(x.astype(np.float32).reshape(-1)).cuda() for x in (D, w, b)]


@pytest.mark.parametrize("nt", [1, 7, 31, 33, 39, 41, 65, 95, 98, 127])
def test_exact(life, nt):
    na, nv = 40, 700
    idx, (a, v, f), (D, w, b), dev = problem(life, nt, na, nv, 500, 20000)
    S = np.zeros((nv, na), np.int64)
    np.add.at(S, (v, a), w[f])
    e = life.life_dsc(idx, dev[0], dev[1], b=dev[2])[0].cpu().numpy()
    assert np.array_equal(e, (S @ D - b).reshape(-1).astype(np.float32))


def test_time_against_aligned_rows(life):
    us = {}
    for nt in (33, 36):
        idx, _, _, (D, w, b) = problem(life, nt, 181, 64000, 10000, 960000)
        run = lambda: life.life_dsc(idx, D, w, b=b)
        for _ in range(20):
            run()
        t = []
        for _ in range(7):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            for _ in range(20):
                run()
            e1.record()
            torch.cuda.synchronize()
            t.append(e0.elapsed_time(e1) * 50)
        us[nt] = min(t)
    assert us[33] <= 1.7 * us[36], us
