"""Exports cost a few passes over the entries, also those of fields that the index does
not hold as such: the voxel of an entry (from the voxels' offsets) and the row and atom
of the tensor-core stream (from its offsets and the chunks')."""
import time

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def life():
    import paper_1905_06234_gb300 as L
    L.load(build_if_missing=True)
    return L


def best_s(f):
    t = []
    for _ in range(12):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        f()
        torch.cuda.synchronize()
        t.append(time.perf_counter() - t0)
    return min(t[2:])


@pytest.mark.parametrize("nv", [1_000_000, 512, 1])
def test_against_the_stored_streams(life, nv):
    """The stored streams are copied out as they lie, 12 bytes an entry; 16 and 8 here."""
    g = torch.Generator(device="cuda").manual_seed(3)
    n, nf = (20_000_000, 500_000) if nv > 512 else (8_000_000, 15000)
    ints = lambda k: torch.randint(0, k, (n,), generator=g, device="cuda", dtype=torch.int32)
    if nv > 512:     # runs along the voxel ids, as a fascicle makes
        f = torch.arange(nf, device="cuda", dtype=torch.int32).repeat_interleave(n // nf)
        v = (ints(1)[:1] + torch.randint(0, nv, (nf,), generator=g, device="cuda", dtype=torch.int32)
             .repeat_interleave(n // nf) + torch.arange(n // nf, device="cuda", dtype=torch.int32).repeat(nf)).clamp_(max=nv - 1)
    else:
        f, v = ints(nf), ints(nv)
    idx = life.life_build_index(ints(360), v, f, torch.ones(n, device="cuda"), 16, 360, nv, nf, precision=life.LIFE_BF16,
                                algo=life.LIFE_ALGO_TC)
    streams = best_s(lambda: life.life_index_export_voxel_streams(idx))
    assert best_s(lambda: life.life_index_export(idx)) <= 1.7 * streams
    assert best_s(lambda: life.life_index_export_tiles(idx)) <= 3.0 * streams
    a, voxel, _, _ = life.life_index_export(idx)
    ptr = life.life_index_export_voxel_streams(idx)[0].long()
    assert torch.equal(voxel, torch.repeat_interleave(torch.arange(nv, device="cuda", dtype=torch.int32), ptr.diff()))
