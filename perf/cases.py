"""The measured cases: what a LiFE program asks of this library, from the smallest
calls (latency and launches) to the paper-scale connectome.

The inputs are persistent random walks through a voxel grid, made on the GPU from
the seed alone, with the shapes of the workloads the tests and the benchmark use
(`tiny`, `medium`, `paper_small`, `paper` and the batch): every walk step is one
raw Phi entry (atom nearest to the step's direction, voxel, fascicle, step length).
"""
import math

import numpy as np
import torch

import paper_1905_06234_gb300 as life

BVAL, LAM = 2.0, 1.7            # ms/µm², µm²/ms
FORMS = {                        # storage and kernels of an index, by the names used below
    "fp32": dict(precision=life.LIFE_FP32, algo=life.LIFE_ALGO_AUTO),    # the default: CUDA cores
    "fp32tc": dict(precision=life.LIFE_FP32, algo=life.LIFE_ALGO_TC),
    "bf16": dict(precision=life.LIFE_BF16, algo=life.LIFE_ALGO_AUTO),
}


def _case(name, op, form, grid, mask, nf, steps, nt=96, na=360, **more):
    c = dict(op=op, form=form, nx=grid[0], ny=grid[1], nz=grid[2], mask=mask, nf=nf, lo=steps[0], hi=steps[1],
             nt=nt, na=na, **more)
    return dict(c, name=name) if name else c


TINY = ((16, 16, 16), False, 2000, (40, 80))
MEDIUM = ((64, 64, 64), False, 50000, (30, 150))
SMALL = ((64, 64, 48), True, 150000, (20, 300))
PAPER = ((96, 96, 72), True, 500000, (20, 300))


def listed():
    return [
        # one signal prediction of a small region of interest: the smallest call there is
        _case("tiny_dsc_fp32", "dsc", "fp32", *TINY),
        # a short fit of a region of interest, all of it launches and latency
        _case("tiny_solve_bf16", "solve", "bf16", *TINY, iters=4),
        # the dictionary's diffusivity, the dictionary and the weights learned by gradient descent: forward and backward
        _case("medium_grad_fp32", "grad", "fp32", *MEDIUM),
        # a sparse whole-brain connectome fitted at FP32 accuracy on the tensor cores
        _case("medium_solve_fp32tc", "solve", "fp32tc", *MEDIUM, iters=4),
        # another scanner's scheme: odd numbers of directions, atoms, voxels and fascicles; residual, then gradient
        _case("odd_gradient_bf16", "gradient", "bf16", (41, 35, 27), True, 30011, (25, 170), nt=33, na=181),
        # the two SpMVs of the default form (FP32, CUDA cores) at the paper's density
        _case("small_dsc_fp32", "dsc", "fp32", *SMALL),
        _case("small_wc_fp32", "wc", "fp32", *SMALL),
        # residual and gradient of the FP32 tensor-core form at the paper's density
        _case("small_gradient_fp32tc", "gradient", "fp32tc", *SMALL),
        # the two SpMVs of the fastest form at the paper's scale: nearly all of a fit's time
        _case("paper_dsc_bf16", "dsc", "bf16", *PAPER),
        _case("paper_wc_bf16", "wc", "bf16", *PAPER),
        # a new connectome arrives: its index is built and the first prediction and gradient taken
        _case("paper_build_bf16", "build", "bf16", *PAPER),
        # several subjects of uneven sizes fitted together
        _case("batch_solve_bf16", "batch", "bf16", (24, 48, 0), False, 12000, (30, 150), n=8, mix=5, iters=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: region of interest to whole brain, every form and operation."""
    op = rng.choice(["dsc", "wc", "gradient", "solve", "grad", "build", "batch"])
    form = rng.choice(["fp32", "fp32tc", "bf16", "bf16"])
    edge = _log_int(rng, 12, 96 if op not in ("grad",) else 64)
    grid = [max(8, min(96, int(edge * rng.uniform(0.7, 1.15)))) for _ in range(3)]
    mask = rng.random() < 0.5
    steps = rng.choice([(40, 80), (30, 150), (20, 300), (25, 170)])
    vox = grid[0] * grid[1] * grid[2] * (0.52 if mask else 1.0)
    # entries per voxel from sparse (medium) to the paper's density, at most 60M of them
    entries = min(vox * math.exp(rng.uniform(math.log(15.0), math.log(235.0))), 6e7 if op != "grad" else 5e6)
    nf = max(500, int(entries / (0.5 * (steps[0] + steps[1]))))
    # Nθ and Na: the shell and dictionary sizes the tests use, odd ones among them
    nt = rng.choice([96, 96, 33, 64, 80, rng.randint(17, 128)])
    na = rng.choice([360, 360, 181, rng.randint(64, 384)])
    if form == "fp32tc":
        na = min(na, 384)
    if op == "batch":
        return _case(None, op, form, (rng.randint(16, 24), rng.randint(30, 48), 0), False, _log_int(rng, 2000, 16000),
                     (30, 150), nt=nt, na=na, n=rng.randint(2, 9),
                     mix=rng.randint(0, 999), iters=rng.randint(2, 4))
    more = dict(iters=rng.randint(2, 4)) if op == "solve" else {}
    return _case(None, op, form, grid, mask, nf, steps, nt=nt, na=na, **more)


# ------------------------------------------------------------------- inputs

def _fibonacci(n, hemisphere):
    i = np.arange(n, dtype=np.float64)
    z = 1.0 - (i + 0.5) / n if hemisphere else 1.0 - (2.0 * i + 1.0) / n
    r, ph = np.sqrt(np.maximum(0.0, 1.0 - z * z)), i * math.pi * (3.0 - math.sqrt(5.0))
    return np.stack([r * np.cos(ph), r * np.sin(ph), z], axis=1)


def _dictionary(nt, na, lam):
    """(D, dD/dλ) in 64 bits, [Na, Nθ]: columns exp(-bλ(g·u)²), demeaned over the directions."""
    c2 = torch.from_numpy((_fibonacci(na, True) @ _fibonacci(nt, False).T) ** 2).cuda()
    e = torch.exp(-BVAL * lam * c2)
    d = -BVAL * c2 * e
    return e - e.mean(1, keepdim=True), d - d.mean(1, keepdim=True)


def _walks(g, grid, mask, nf, lo, hi, na):
    """Raw Phi of persistent random walks: (atom, voxel, fascicle, value) in walk order, Nv, voxel coordinates."""
    dims = torch.tensor(grid, dtype=torch.float32, device="cuda")
    nx, ny, nz = grid
    k, j, i = torch.meshgrid(*(torch.arange(n, device="cuda") for n in (nz, ny, nx)), indexing="ij")
    ijk = torch.stack([i, j, k], -1).reshape(-1, 3)
    inside = torch.ones(len(ijk), dtype=torch.bool, device="cuda")
    if mask:
        inside = (((ijk + 0.5 - dims / 2) / (dims / 2)) ** 2).sum(1) <= 1.0
    vid = torch.where(inside, torch.cumsum(inside.int(), 0, dtype=torch.int32) - 1, -1)
    ijk = ijk[inside].to(torch.int32)
    nv = len(ijk)
    stride = torch.tensor([1.0, nx, nx * ny], device="cuda")

    def voxel(p):
        q = torch.floor(p)
        ok = ((q >= 0) & (q < dims)).all(1)
        return torch.where(ok, vid[(torch.where(ok[:, None], q, 0.0) @ stride).long()], -1)

    length = torch.randint(lo, hi + 1, (nf,), generator=g, device="cuda")
    length, order = torch.sort(length, descending=True)
    live = (length[None, :] > torch.arange(hi, device="cuda")[:, None]).sum(1).tolist()
    # inside a voxel of the domain (short of its far faces, where the sum could round into the next)
    p = ijk[torch.randint(0, nv, (nf,), generator=g, device="cuda")] + 0.999 * torch.rand(nf, 3, generator=g, device="cuda")
    t = torch.nn.functional.normalize(torch.randn(nf, 3, generator=g, device="cuda"))
    u = torch.from_numpy(_fibonacci(na, True)).to("cuda", torch.float32)
    out = [torch.empty(hi, nf, dtype=dt, device="cuda") for dt in (torch.int16, torch.int32, torch.float32)]
    for s in range(hi):
        n = live[s]              # walks are held longest first: those still going are the first n
        if n == 0:
            break
        p, t = p[:n], t[:n]
        t = torch.nn.functional.normalize(t + 0.3 * torch.randn(n, 3, generator=g, device="cuda"))
        ell = 0.5 + 0.5 * torch.rand(n, 1, generator=g, device="cuda")
        q = p + ell * t
        off = voxel(q) < 0
        box = ((q < 0) | (q >= dims)).any(1, keepdim=True)
        nrm = torch.nn.functional.normalize((p - dims / 2) / (dims / 2) ** 2)
        t2 = torch.where(box, torch.where((q < 0) | (q >= dims), -t, t), t - 2 * (t * nrm).sum(1, keepdim=True) * nrm)
        t = torch.where(off[:, None], t2, t)
        q = p + ell * t
        vq = voxel(q)
        q = torch.where((vq < 0)[:, None], p, q)     # nowhere to go: the step stays in place
        m = voxel(0.5 * (p + q))
        out[0][s, :n] = (t @ u.T).abs_().argmax(1).to(torch.int16)
        out[1][s, :n] = torch.where(m >= 0, m, voxel(q))
        out[2][s, :n] = ell[:, 0]
        p = q
    # back to fascicle order, each walk's steps together
    back = torch.argsort(order)
    keep = (length[None, :] > torch.arange(hi, device="cuda")[:, None])[:, back].T
    atom, vox, val = (x[:, back].T[keep] for x in out)
    fasc = torch.arange(nf, device="cuda", dtype=torch.int32)[:, None].expand(nf, hi)[keep]
    return (atom.to(torch.int32).contiguous(), vox.contiguous(), fasc.contiguous(), val.contiguous()), nv, \
        ijk.contiguous()


class _Exact:
    """M and its transpose in 64 bits: S = Phi w scattered, then the dictionary."""

    def __init__(self, phi, nv, nf, D):      # D [Na, Nθ], 64 bits
        self.nv, self.nf, self.na, self.nt, self.D = nv, nf, D.shape[0], D.shape[1], D
        self.va = phi[1].long() * self.na + phi[0].long()
        self.f, self.x = phi[2].long(), phi[3].double()

    def s(self, w):
        return torch.zeros(self.nv * self.na, dtype=torch.float64, device="cuda").index_add_(
            0, self.va, self.x * w.double()[self.f]).view(self.nv, self.na)

    def dsc(self, w):
        return (self.s(w) @ self.D).reshape(-1)

    def wc(self, r):
        z = r.double().view(self.nv, self.nt) @ self.D.T
        return torch.zeros(self.nf, dtype=torch.float64, device="cuda").index_add_(
            0, self.f, self.x * z.reshape(-1)[self.va])


def _weights(g, nf):
    """Uniform in (0, 1), a third of them zero, as a fit's iterates have them."""
    w = torch.rand(nf, generator=g, device="cuda")
    return torch.where(torch.rand(nf, generator=g, device="cuda") < 0.3, 0.0, w)


def _inputs(case, seed, grid=None, nf=None):
    """Phi, the dictionary, a measured signal b = M w_true + noise, and other weights w."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    grid = grid or (case["nx"], case["ny"], case["nz"])
    nf = nf or case["nf"]
    phi, nv, ijk = _walks(g, grid, case["mask"], nf, case["lo"], case["hi"], case["na"])
    D = _dictionary(case["nt"], case["na"], LAM)[0].float()
    w_true, w = _weights(g, nf), _weights(g, nf)
    b = _Exact(phi, nv, nf, D.double()).dsc(w_true).float()
    b += 0.01 * torch.randn(len(b), generator=g, device="cuda")
    return dict(phi=phi, nv=nv, nf=nf, ijk=ijk.reshape(-1), D=D.reshape(-1), b=b, w=w)


def _batch_shapes(case):
    """Uneven problems: grid edges between nx and ny, numbers of fascicles from a quarter of nf to four times it."""
    r = np.random.RandomState(case["mix"])
    return [((int(r.randint(case["nx"], case["ny"] + 1)),) * 3,
             int(case["nf"] * math.exp(r.uniform(-math.log(4.0), math.log(4.0))))) for _ in range(case["n"])]


def _problems(case, seed):
    if case["op"] != "batch":
        return [_inputs(case, seed)]
    return [_inputs(case, int(seed) * 64 + k, grid, nf) for k, (grid, nf) in enumerate(_batch_shapes(case))]


def _index(case, p):
    return life.life_build_index(*p["phi"], case["nt"], case["na"], p["nv"], p["nf"], voxel_ijk=p["ijk"],
                                 **FORMS[case["form"]])


def prepare(case, seed):
    op, ps = case["op"], _problems(case, seed)
    s = dict(case=case, op=op)
    if op == "batch":
        s["indices"] = [_index(case, p) for p in ps]
        s["batch"] = life.life_batch_create(s["indices"])
        s.update(D=ps[0]["D"], b=[p["b"] for p in ps], w=[torch.empty_like(p["w"]) for p in ps],
                 st0=life.new_batch_states(len(ps)), work=life.new_batch_workspace(s["batch"]))
        s["st"] = torch.empty_like(s["st0"])
        return s
    p = ps[0]
    s.update({k: p[k] for k in ("D", "b", "w")}, r=p["b"])
    if op == "build":
        return dict(s, p=p)
    s["index"] = _index(case, p)
    if op == "solve":
        s.update(st=life.new_sbb_state(), work=life.new_sbb_workspace(s["index"]))
    if op == "grad":
        s.update(lam=torch.tensor([1.5], device="cuda", requires_grad=True), w=p["w"].requires_grad_(),
                 gdirs=torch.from_numpy(_fibonacci(case["nt"], False)).cuda(),
                 adirs=torch.from_numpy(_fibonacci(case["na"], True)).cuda())
    return s


def run(s):
    op = s["op"]
    if op == "dsc":
        return life.life_dsc(s["index"], s["D"], s["w"], b=s["b"])[0]
    if op == "wc":
        return life.life_wc(s["index"], s["D"], s["r"])[0]
    if op == "gradient":
        e = life.life_dsc(s["index"], s["D"], s["w"], b=s["b"])[0]
        return e, life.life_wc(s["index"], s["D"], e)[0]
    if op == "build":
        index = _index(s["case"], s["p"])
        y = life.life_dsc(index, s["D"], s["w"])[0]
        g = life.life_wc(index, s["D"], s["r"])[0]
        index.close()
        return y, g
    if op == "solve":            # a fit from w = 1
        s["w"].fill_(1.0)
        life.life_sbb_state_init(s["st"])
        life.life_sbbnnls_solve(s["index"], s["D"], s["b"], s["w"], s["case"]["iters"], s["st"], s["work"])
        return s["w"], s["st"][:8].view(torch.int64), s["st"][8:40].view(torch.float64).float()
    if op == "batch":
        for w in s["w"]:
            w.fill_(1.0)
        s["st"].copy_(s["st0"])
        life.life_batch_solve(s["batch"], s["D"], s["b"], s["w"], s["case"]["iters"], s["st"], s["work"])
        return s["w"], s["st"].view(len(s["w"]), -1)[:, :8].contiguous().view(torch.int64)
    D = life.dictionary(s["lam"], s["gdirs"], s["adirs"], BVAL)
    y = life.dsc(s["index"], D, s["w"])
    e = y - s["b"]
    gD, gw, glam = torch.autograd.grad(0.5 * (e * e).sum(), (D, s["w"], s["lam"]))
    return y.detach(), gD, gw, glam


# ---------------------------------------------------------------- work, exact

def _spmv_work(case, entries, nv, nf, vectors):
    """Compact Phi (2 B atom, 4 B fascicle, 4 or 2 B value; CSR pointers), the signal vectors, w or g, D; a
    multiply-add per entry and the dense contraction of the occupied part (at most one cell per entry)."""
    phi = entries * (8 if case["form"] == "bf16" else 10) + 4 * nv
    cells = min(entries, nv * case["na"])
    return (phi + 4 * (vectors * case["nt"] * nv + nf + case["nt"] * case["na"]),
            2 * entries + 2 * cells * case["nt"])


def work(case):
    op = case["op"]
    dims = [(case["nx"], case["ny"], case["nz"], case["nf"])]
    if op == "batch":
        dims = [(*grid, nf) for grid, nf in _batch_shapes(case)]
    B = F = 0.0
    for nx, ny, nz, nf in dims:
        nv = nx * ny * nz * (math.pi / 6 if case["mask"] else 1.0)
        entries = nf * 0.5 * (case["lo"] + case["hi"])
        dsc, dscb, wc = (_spmv_work(case, entries, nv, nf, v) for v in (1, 2, 1))
        if op == "build":        # the COO list is read; then a DSC and a WC's vectors
            B += 16 * entries + 8 * case["nt"] * nv + 8 * nf + 12 * nv
            F += dsc[1] + wc[1]
            continue
        n = {"dsc": (1, 0, 0), "wc": (0, 0, 1), "gradient": (1, 0, 1), "grad": (0, 2, 1),
             "solve": (1, 1, 1.5), "batch": (1, 1, 1.5)}[op]
        n = [x * case.get("iters", 1) for x in n]
        for k, w in zip(n, (dscb, dsc, wc)):
            B += k * w[0]
            F += k * w[1]
    return {"bytes": B, "flops": F}


def _exact_solve(M, b, iters):
    """SBB-NNLS in 64 bits from w = 1: step sizes <g,g>/<Mg,Mg> and <Mg,Mg>/<MᵀMg,MᵀMg> in turn."""
    w = torch.ones(M.nf, dtype=torch.float64, device="cuda")
    b, gg0 = b.double(), None
    for it in range(iters):
        e = M.dsc(w) - b
        g = M.wc(e)
        g = torch.where((w == 0) & (g > 0), 0.0, g)
        gg, obj = g @ g, 0.5 * (e @ e)
        gg0 = gg if gg0 is None else gg0
        v = M.dsc(g)
        if it % 2 == 0:
            alpha = gg / (v @ v)
        else:
            u = M.wc(v)
            alpha = (v @ v) / (u @ u)
        w = torch.clamp_min(w - alpha * g, 0.0)
    return w, torch.tensor([iters], device="cuda"), torch.stack([alpha, obj, gg, gg0])


def exact(case, seed):
    op, ps = case["op"], _problems(case, seed)
    D = ps[0]["D"].double().view(case["na"], case["nt"])
    if op == "batch":
        got = [_exact_solve(_Exact(p["phi"], p["nv"], p["nf"], D), p["b"], case["iters"]) for p in ps]
        return [g[0] for g in got], torch.stack([g[1] for g in got])
    p = ps[0]
    if op == "grad":
        D, dD = _dictionary(case["nt"], case["na"], 1.5)
    M = _Exact(p["phi"], p["nv"], p["nf"], D)
    if op == "dsc":
        return M.dsc(p["w"]) - p["b"].double()
    if op == "wc":
        return M.wc(p["b"])
    if op == "gradient":
        e = M.dsc(p["w"]) - p["b"].double()
        return e, M.wc(e)
    if op == "build":
        return M.dsc(p["w"]), M.wc(p["b"])
    if op == "solve":
        return _exact_solve(M, p["b"], case["iters"])
    y = M.dsc(p["w"])
    e = y - p["b"].double()
    gD = M.s(p["w"]).T @ e.view(p["nv"], case["nt"])
    return y, gD.reshape(-1), M.wc(e), (gD * dD).sum().reshape(1)
