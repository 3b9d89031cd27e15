"""The host-side rules that shape the tensor-core launches, compiled here with the host
compiler: how a launch's tiles are shared out to the CTAs, and the form of a BF16 DSC."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1905_06234_gb300", "csrc")
WRAP = r"""
#include "launch_rules.cuh"
extern "C" int share(const int* order, const int* btile, const int* base, const int* bfasc, int nb, int sms, int batch,
                     int fp32, int* cta_unit, int* brick, int* t0, int* t1) {
    auto vec = [](const int* p, int n) { return std::vector<int32_t>(p, p + n); };
    const auto W = life::share_out(vec(order, nb), vec(btile, nb + 1), vec(base, btile[nb] + 1), vec(bfasc, nb + 1), sms,
                                   batch != 0, fp32 != 0);
    std::copy(W.cta_unit.begin(), W.cta_unit.end(), cta_unit);
    std::copy(W.brick.begin(), W.brick.end(), brick);
    std::copy(W.t0.begin(), W.t0.end(), t0);
    std::copy(W.t1.begin(), W.t1.end(), t1);
    return W.grid();
}
extern "C" int form(long long nnz, long long tiles, long long bricks, int n_c, int can, int max_stages) {
    const auto F = life::dsc_form(nnz, tiles, bricks, n_c, can != 0, [&](int stages) { return stages <= max_stages; });
    return F.y_tile ? F.stages : -F.stages;
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    cxx = shutil.which("g++") or pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("rules")
    (d / "w.cpp").write_text(WRAP)
    so = str(d / "w.so")
    subprocess.run([cxx, "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, "-o", so, str(d / "w.cpp")], check=True)
    return ctypes.CDLL(so)


def layout(rng, nb, tiles, entries, slots, spread):
    """Bricks of `tiles` tiles (spread: of 1 to 2·tiles - 1), their entries and table sizes."""
    nt = rng.integers(1, 2 * tiles, nb) if spread else np.full(nb, tiles)
    btile = np.concatenate([[0], np.cumsum(nt)]).astype(np.int32)
    e = rng.integers(0, 2 * entries + 1, btile[-1]) if spread else np.full(btile[-1], entries)
    f = rng.integers(0, 2 * slots + 1, nb) if spread else np.full(nb, slots)
    base = np.concatenate([[0], np.cumsum(e)]).astype(np.int32)
    bfasc = np.concatenate([[0], np.cumsum(f)]).astype(np.int32)
    order = np.argsort(-(base[btile[1:]] - base[btile[:-1]]), kind="stable").astype(np.int32)
    return order, btile, base, bfasc


def share(rules, lay, sms, batch, fp32):
    order, btile, base, bfasc = (np.ascontiguousarray(x) for x in lay)
    nt = int(btile[-1])
    out = [np.zeros(max(nt, sms) + 1, np.int32) for _ in range(4)]
    p = lambda x: x.ctypes.data_as(ctypes.c_void_p)
    grid = rules.share(p(order), p(btile), p(base), p(bfasc), len(btile) - 1, sms, int(batch), int(fp32), *(p(x) for x in out))
    n = int(out[0][grid])
    return out[0][:grid + 1], [x[:n] for x in out[1:]]


def makespan(lay, cta_unit, units):
    """The most loaded CTA, in the rule's own costs (a tile 50000, a unit 14000, a slot 6, an entry 1)."""
    _, btile, base, bfasc = lay
    cost = [14000 + 6 * (bfasc[b + 1] - bfasc[b]) + 50000 * (t1 - t0) + base[t1] - base[t0] for b, t0, t1 in zip(*units)]
    return max(sum(cost[cta_unit[c]:cta_unit[c + 1]]) for c in range(len(cta_unit) - 1))


def whole_bricks(lay, sms):
    order, btile = lay[0], lay[1]
    nb = len(order)
    g = min(sms, nb)
    mine = [[order[k] for r in range(nb // g + 1) for k in [r * g + (g - 1 - c if r & 1 else c)] if k < nb] for c in range(g)]
    units = [np.array([f(b) for m in mine for b in m]) for f in (int, lambda b: btile[b], lambda b: btile[b + 1])]
    return makespan(lay, np.concatenate([[0], np.cumsum([len(m) for m in mine])]), units)


@pytest.mark.parametrize("batch,fp32", [(False, False), (False, True), (True, False), (True, True)])
@pytest.mark.parametrize("spread", [False, True])
@pytest.mark.parametrize("nb", [1, 7, 64, 125, 128, 152, 153, 250, 300, 303, 304, 305, 700])
@pytest.mark.parametrize("entries,slots", [(1300, 280), (2200, 1000), (10000, 4000), (29000, 9000), (0, 0)])
def test_share(rules, nb, entries, slots, spread, batch, fp32):
    lay = layout(np.random.default_rng(nb + entries), nb, 4, entries, slots, spread)
    for sms in (152, 148, 1):
        cta_unit, (brick, t0, t1) = share(rules, lay, sms, batch, fp32)
        btile = lay[1]
        assert cta_unit[0] == 0 and (np.diff(cta_unit) > 0).all() and len(cta_unit) - 1 <= sms
        # every tile once, every unit inside its brick
        assert (t0 < t1).all() and (btile[brick] <= t0).all() and (t1 <= btile[brick + 1]).all()
        seen = np.zeros(btile[-1], int)
        for a, b in zip(t0, t1):
            seen[a:b] += 1
        assert (seen == 1).all()
        # never a worse share than whole bricks (10 % in the batches of FP32 storage, which measure better)
        assert makespan(lay, cta_unit, (brick, t0, t1)) <= (1.1 if batch and fp32 else 1.0) * whole_bricks(lay, sms)


# the form measured fastest (4, 3, 2: with the tile of Y and so many stages; -2: general), by entries
# per tile and chunk, chunks a tile, tiles a brick, stages that fit
@pytest.mark.parametrize("epc,n_c,per_brick,fit,best", [
    (339, 3, 4, 3, 3), (3812, 3, 4, 3, 2), (7621, 3, 4, 2, 2), (255, 4, 4, 4, 4), (2864, 4, 4, 4, 4), (7481, 4, 4, 4, 2),
    (1005, 1, 4, 4, -2), (7536, 1, 4, 4, -2), (22635, 1, 4, 4, 2), (29545, 1, 4, 4, 2), (1893, 2, 4, 4, 2),
    (12525, 2, 2, 4, 2), (1270, 3, 1, 2, 2), (4756, 3, 1, 2, -2), (8603, 3, 1, 2, -2), (339, 3, 4, 1, -2)])
def test_dsc_form(rules, epc, n_c, per_brick, fit, best):
    tiles = 1000 * per_brick
    args = lambda can: [ctypes.c_longlong(x) for x in (epc * tiles * n_c, tiles, 1000)] + [n_c, can, fit]
    assert rules.form(*args(1)) == best
    assert rules.form(*args(0)) == -2       # FP32 storage, or rows off a 16-byte boundary


def test_dsc_form_of_an_empty_index(rules):
    assert rules.form(ctypes.c_longlong(0), ctypes.c_longlong(1), ctypes.c_longlong(1), 1, 1, 4) == -2
