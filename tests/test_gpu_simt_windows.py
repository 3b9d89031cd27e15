"""The windowed CUDA-core kernels (32 entries a window, runs compacted, dots in
eights and sixteens) and dL/dD against the FP64 oracle at 1e-5: voxels whose entries
end at, before and after the edges of windows and of 8- and 16-run groups, empty
voxels between them, runs that cross windows, more and fewer voxels than warps."""
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


def rel(a, b):
    b = np.asarray(b, np.float64)
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("kernels", [0, 1, 2])
@pytest.mark.parametrize("nt,na,scale", [(96, 360, 1), (1, 3, 1), (33, 40, 1), (150, 61, 1), (256, 20, 1), (96, 700, 1),
                                         (96, 40, 40)])
def test_window_edges(life, kernels, nt, na, scale):
    lens = [0, 1, 7, 8, 9, 15, 16, 17, 0, 0, 31, 32, 33, 63, 64, 65, 100, 0, 1] * scale
    nv, nf = len(lens), 120
    rng = np.random.default_rng(nt + na)
    v = np.repeat(np.arange(nv), lens).astype(np.int32)
    a, f = (rng.integers(0, k, len(v)).astype(np.int32) for k in (na, nf))
    a[v % 3 == 0] %= 2                # long runs of equal atoms
    x = rng.uniform(0.5, 1.0, len(v)).astype(np.float32)
    D, w, r, b = (rng.standard_normal(k).astype(np.float32) for k in (nt * na, nf, nt * nv, nt * nv))
    w[::7] = 0.0
    dev = lambda t: torch.from_numpy(t).cuda()
    idx = life.index_from_arrays(a, v, f, x, nt, na, nv, nf, simt_kernels=kernels)
    phi = oracle.canon(a, v, f, x, na, nv, nf)
    e, ss = life.life_dsc(idx, dev(D), dev(w), b=dev(b), sumsq=True)
    y, _ = life.life_dsc(idx, dev(D), dev(w))
    g, _ = life.life_wc(idx, dev(D), dev(r))
    gD = life.life_dsc_grad_D(idx, dev(r), dev(w))
    y_ref = oracle.dsc(phi, D, w, nt, nv)
    assert rel(y.cpu().numpy(), y_ref) <= 1e-5 and rel(e.cpu().numpy(), y_ref - b) <= 1e-5
    assert abs(float(ss) - (y_ref - b) @ (y_ref - b)) <= 2e-5 * ((y_ref - b) @ (y_ref - b))
    assert rel(g.cpu().numpy(), oracle.wc(phi, D, r, nt, nf)) <= 1e-5
    gd_ref = np.zeros((na, nt))
    np.add.at(gd_ref, phi.atom, (phi.val.astype(np.float64) * w[phi.fasc])[:, None] * r.reshape(nv, nt)[phi.voxel])
    assert rel(gD.cpu().numpy(), gd_ref.reshape(-1)) <= 1e-5


def test_non_finite_gradient_reaches_zero_weights(life):
    """A NaN of gy reaches dL/dD through entries whose val·w is zero, as in the oracle's sum."""
    a, v, f = (np.array(t, np.int32) for t in ([0, 0, 1], [0, 0, 1], [0, 1, 1]))
    idx = life.index_from_arrays(a, v, f, np.ones(3, np.float32), 2, 2, 2, 2)
    w, gy = torch.tensor([1.0, -1.0]).cuda(), torch.tensor([float("nan"), 2.0, 3.0, float("inf")]).cuda()
    gD = life.life_dsc_grad_D(idx, gy, w).cpu().numpy()
    assert np.isnan(gD[0]) and gD[1] == 0.0 and gD[2] == -3.0 and np.isneginf(gD[3])
