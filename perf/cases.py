"""Performance cases: the work that users of the library have it do, through
its public entry points, from the smallest calls to the 4M-cell step.

Kinds of case
  residual  cams_residual_norm_noalloc on a caller's own 7-point system
  assemble  cams_assemble and the read-back of A and f (a caller with a linear
            solver of its own)
  basis     cams_update_basis with every local entity rebuilt, and the read-back
            of P, R A P and the ILU(0) pivots
  iterate   one linearisation's assembly and a fixed number of C-AMS iterations
            with the operators built before
  solve     implicit time steps on a new permeability field (a handle is kept
            per grid; realisations go through it one after the other)
  ensemble  one implicit step of several independent realisations at once
  train     one Adam step of the learned basis surrogate
  infer     the surrogate network on the tensor cores

Fields are seeded log-normal permeabilities (circulant embedding, exponential
covariance) with the statistics of the repository's workloads.  exact() has
plain 64-bit torch versions of the same definitions.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_1705_05783_gb300 import cams, surrogate

DEV = "cuda"
F64 = dict(dtype=torch.float64, device=DEV)

# what a problem case carries unless it says otherwise: the 4M-cell
# workload's fluid and solver options (Dirichlet west/east, (B4), MSFE, 5
# ILU(0) post-smoothing steps)
DEFAULTS = dict(bc="dirichlet", sigma=2.0, cx=0.1, cz=0.1, kz_ratio=1.0, alpha=1.0, law=0, coef=0.1,
                dt_star=0.01, basis=4, restriction=0, n_post=5, precision=0, nl_tol=1e-8, steps=1,
                iters=0)


def _case(name, kind, nx=0, ny=0, nz=0, b=(1, 1, 1), **kw):
    c = dict(kind=kind)
    if nx:
        c.update(DEFAULTS, nx=nx, ny=ny, nz=nz, bx=b[0], by=b[1], bz=b[2])
    c.update(kw)
    if name:
        c["name"] = name
    return c


WELLS = dict(bc="wells", sigma=3.0, cx=0.2, cz=0.02, kz_ratio=0.1, coef=0.2, basis=1)
LINES = dict(bc="lines", sigma=2.0, cx=0.125, cz=0.125, alpha=5.0, law=1, coef=1.0, dt_star=0.4, nl_tol=1e-6)
MIXED = dict(sigma=3.0, precision=1)


def listed():
    return [
        # a service call on a small 2D system: launch and read-back latency
        _case("residual-2d-40x40", "residual", 40, 40, 1),
        # the same service on the largest Test Case 1 grid
        _case("residual-256x256x256", "residual", 256, 256, 256, cx=0.125, cz=0.125),
        # one linearisation of the 4M-cell workload handed to the caller
        _case("assemble-200x200x100", "assemble", 200, 200, 100, (10, 10, 10), sigma=3.0),
        # a full operator build of the wells workload with the MSFV restriction
        _case("basis-wells-100x100x50-msfv", "basis", 100, 100, 50, (10, 10, 5), **dict(WELLS, restriction=1)),
        # FP64 iterations on a grid that no tile divides
        _case("iterate-135x117x63-fp64", "iterate", 135, 117, 63, (9, 9, 9), iters=4),
        # five steps of the smallest workload
        _case("solve-2d-40x40", "solve", 40, 40, 1, (5, 5, 1), n_post=1, steps=5, nl_tol=1e-6),
        # one step of the wells workload in FP64 (at the tolerance that it meets)
        _case("solve-wells-100x100x50-fp64", "solve", 100, 100, 50, (10, 10, 5), nl_tol=1e-5, **WELLS),
        # Test Case 2: two prescribed columns, stretched cells, flat coarse blocks
        _case("solve-lines-64x64x64-a5", "solve", 64, 64, 64, (2, 8, 8), **LINES),
        # the headline: the 4M-cell step with the FP32 preconditioner
        _case("solve-200x200x100-mixed", "solve", 200, 200, 100, (10, 10, 10), **MIXED),
        # uneven realisations at once (the ensemble workload's ladder of grids)
        _case("ensemble-16-mixed", "ensemble", members=16, smallest=32768, largest=1048576),
        # one training step on a batch of 11^3 patches
        _case("train-64x11", "train", B=64, S=11),
        # the network over one chunk of 11^3 patches
        _case("infer-1024x11", "infer", B=1024, S=11),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, lo, hi, blocks):
    """Grid sizes of lo to hi cells in all, whole coarse blocks of the given
    edge choices per direction (three of them at least)."""
    while True:
        b = tuple(rng.choice(blocks) for _ in range(3))
        edge = _logint(rng, lo, hi) ** (1 / 3)
        n = tuple(v * max(3, int(round(edge * rng.uniform(0.6, 1.6) / v))) for v in b)
        if lo <= n[0] * n[1] * n[2] <= hi:
            return n, b


def draw(rng):
    kind = rng.choice(["residual", "residual", "assemble", "basis", "basis", "iterate", "iterate", "solve2d",
                       "solve", "solve", "mixed", "mixed", "ensemble", "train", "infer"])
    sigma = round(rng.uniform(1.0, 3.0), 2)
    if kind == "residual":
        edge = [_logint(rng, 20, 256) for _ in range(3)]
        return _case("", "residual", edge[0], edge[1], rng.choice([1, edge[2]]), sigma=sigma)
    if kind in ("assemble", "basis"):
        n, b = _grid(rng, 20000, 4000000 if kind == "assemble" else 600000, [5, 6, 7, 8, 10])
        kw = dict(WELLS if rng.random() < 0.5 else {}, sigma=sigma)
        if kind == "basis":
            kw.update(basis=rng.choice([1, 2, 3, 4]), restriction=rng.choice([0, 1]))
        return _case("", kind, *n, b, **kw)
    if kind == "iterate":
        n, b = _grid(rng, 20000, 1200000, [5, 6, 7, 8, 9, 10])
        return _case("", "iterate", *n, b, sigma=sigma, restriction=rng.choice([0, 0, 1]), iters=rng.randint(1, 5),
                     n_post=rng.choice([1, 3, 5]))
    if kind == "solve2d":
        b = rng.choice([4, 5, 7])
        return _case("", "solve", b * rng.randint(5, 20), b * rng.randint(5, 20), 1, (b, b, 1), sigma=sigma, n_post=rng.choice([1, 2, 5]),
                     steps=rng.randint(1, 5), nl_tol=1e-6)
    if kind in ("solve", "mixed"):
        n, b = _grid(rng, 30000, 500000 if kind == "solve" else 3000000, [7, 8, 9, 10])
        return _case("", "solve", *n, b, sigma=sigma, precision=int(kind == "mixed"), nl_tol=1e-8 if kind == "mixed" else 1e-7)
    if kind == "ensemble":
        return _case("", "ensemble", members=rng.randint(3, 16), smallest=32768, largest=_logint(rng, 100000, 1048576))
    return _case("", kind, B=_logint(rng, 8, 64 if kind == "train" else 2048), S=rng.randint(6, 11))


# ------------------------------------------------------------- inputs ---

class Handle:
    """A solver handle released with its state."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        try:
            cams.cams_destroy(self.h)
        except Exception:
            pass


def _field(nx, ny, nz, sigma, cx, cz, gen):
    """Log-normal permeability with correlation lengths cx (x, y) and cz (z)
    in units of the x extent, by circulant embedding."""
    n = (nz, ny, nx)
    emb = [2 * s if s > 1 else 1 for s in n]
    lag = [torch.minimum(torch.arange(m, device=DEV), m - torch.arange(m, device=DEV)).float() for m in emb]
    ell = (cz * nx, cx * nx, cx * nx)
    h2 = sum(((a / c) ** 2).reshape([-1 if d == e else 1 for e in range(3)]) for d, (a, c) in enumerate(zip(lag, ell)))
    lam = torch.fft.fftn(torch.exp(-torch.sqrt(h2)).to(torch.complex64)).real.clamp_min(0)
    z = torch.complex(torch.randn(emb, generator=gen, device=DEV), torch.randn(emb, generator=gen, device=DEV))
    y = torch.fft.fftn(torch.sqrt(lam / float(np.prod(emb))) * z).real[:nz, :ny, :nx]
    return torch.exp(sigma * y.double()).reshape(-1).contiguous()


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _problem(c, seed):
    """Permeabilities, spacings, time step, sources and prescribed cells of a
    case (the time scale and the well rates as in the workloads)."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    k = _field(nx, ny, nz, c["sigma"], c["cx"], c["cz"], _gen(seed))
    pr = dict(c, k=k, kz=k * c["kz_ratio"] if c["kz_ratio"] != 1.0 else k, N=nx * ny * nz, h=1.0 / nx)
    pr["d"] = (c["alpha"] * pr["h"], pr["h"], pr["h"])
    pr["dt"] = c["dt_star"] * 0.1 * c["alpha"] ** 2 / math.exp(float(k.log().mean()))
    z = torch.arange(nz, device=DEV) * (nx * ny)
    ends = torch.cat([z, z + nx * ny - 1]).to(torch.int32)
    pr["src"] = pr["fix"] = (None, None)
    if c["bc"] == "wells":
        t = _trans(pr)
        tsum = sum(a + _up(pr, a, e) for e, a in enumerate(t))[ends.long()]
        pr["src"] = (ends, torch.where(torch.arange(2 * nz, device=DEV) < nz, 0.02, -0.02).double() * tsum)
    if c["bc"] == "lines":
        pr["fix"] = (ends, (torch.arange(2 * nz, device=DEV) < nz).double())
    return pr


def _bc(pr):
    return cams.make_bc(pr["bc"] == "dirichlet", 1.0, 0.0, *pr["src"], *pr["fix"])


def _setup(pr):
    g = cams.cams_grid(pr["nx"], pr["ny"], pr["nz"], *pr["d"])
    fl = cams.cams_fluid(pr["law"], pr["coef"], 1.0, 1.0, 0.1)
    opt = cams.make_options((pr["bx"], pr["by"], pr["bz"]), basis=pr["basis"], restriction=pr["restriction"],
                            n_post=pr["n_post"], nl_tol=pr["nl_tol"], memspace=cams.CAMS_DEVICE, precision=pr["precision"])
    return Handle(cams.cams_setup(g, fl, opt, pr["k"], pr["k"], pr["kz"]))


def _pressures(pr, seed):
    """An iterate and a previous time level as they stand inside a run: a
    front moving in from the west, and the iterate a little ahead of it."""
    g = _gen(seed + 7919)
    x = (torch.arange(pr["N"], device=DEV) % pr["nx"]).double() / pr["nx"]
    wob = 1.0 + 0.1 * torch.rand(pr["N"], generator=g, **F64)
    return torch.exp(-6.0 * x) * wob, torch.exp(-8.0 * x) * wob


# grids of an ensemble: whole 8^3 blocks, as uneven as the workload's ladder
LADDER = ((32, 32, 32), (48, 48, 32), (64, 48, 32), (64, 64, 32), (64, 64, 64), (96, 64, 48), (96, 96, 48), (128, 96, 64), (128, 128, 64))


def _members(c, seed):
    """The members' shapes belong to the case, their fields to the seed."""
    fit = [s for s in LADDER if c["smallest"] <= s[0] * s[1] * s[2] <= c["largest"]]
    out = []
    for m in range(c["members"]):
        kw = dict(MIXED, sigma=1.0 + 2.0 * ((7 * m) % 16) / 16)
        out.append(_problem(_case("", "solve", *fit[(5 * m) % len(fit)], (8, 8, 8), **kw), seed * 1000 + m))
    return out


def _patches(B, S, seed):
    """Network inputs as the engine cuts them: log couplings and relative
    accumulation of a heterogeneous patch, and corner functions' deviations
    on the patch boundary; targets and mask live on the interior cells."""
    g = _gen(seed)

    def rn(ch):
        return torch.randn((B, ch, S, S, S), generator=g, device=DEV)

    inner = torch.zeros((S, S, S), device=DEV)
    inner[1:-1, 1:-1, 1:-1] = 1.0
    lnk = F.avg_pool3d(F.pad(2.0 * rn(1), (1,) * 6, mode="replicate"), 3, 1) * 3.0
    x = torch.cat([lnk + 0.3 * rn(3), 0.01 * rn(1).abs(), 0.2 * rn(8) * (1.0 - inner)], 1)
    t = 0.1 * F.avg_pool3d(F.pad(rn(8), (1,) * 6), 3, 1) * inner
    m = inner.expand(B, 8, S, S, S)
    return [v.reshape(B, -1, S ** 3).contiguous() for v in (x, t, m)]


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "residual":
        pr = _problem(c, seed)
        p, pn = _pressures(pr, seed)
        A, f, _ = _linearise(pr, p, pn)
        return dict(kind=kind, pr=pr, A=A, f=f, p=p, r=torch.empty_like(p))
    if kind in ("assemble", "basis", "iterate"):
        pr = _problem(c, seed)
        p, pn = _pressures(pr, seed)
        h = _setup(pr)
        bc, keep = _bc(pr)
        s = dict(kind=kind, pr=pr, h=h, bc=bc, keep=keep, p=p, pn=pn)
        nc = (c["nx"] // c["bx"]) * (c["ny"] // c["by"]) * (c["nz"] // c["bz"])
        if kind == "assemble":
            s["out"] = [(cams.CAMS_Q_MATRIX, torch.empty(4 * pr["N"], **F64)), (cams.CAMS_Q_RHS, torch.empty(pr["N"], **F64))]
        elif kind == "basis":
            cams.cams_assemble(h.h, p, pn, pr["dt"], bc)
            s["out"] = [(cams.CAMS_Q_PROLONG, torch.empty(8 * pr["N"], **F64)), (cams.CAMS_Q_COARSE, torch.empty(27 * nc, **F64)),
                        (cams.CAMS_Q_ILU_DIAG, torch.empty(pr["N"], **F64))]
        else:
            cams.cams_assemble(h.h, p, pn, pr["dt"], bc)
            cams.cams_update_basis(h.h, True)
            s["out"] = [(cams.CAMS_Q_PRESSURE, torch.empty(pr["N"], **F64))]
        return s
    if kind == "solve":
        pr = _problem(c, seed)
        bc, keep = _bc(pr)
        return dict(kind=kind, pr=pr, h=_setup(pr), bc=bc, keep=keep)
    if kind == "ensemble":
        prs = _members(c, seed)
        bcs = [_bc(pr) for pr in prs]
        return dict(kind=kind, prs=prs, hs=[_setup(pr) for pr in prs], bcs=[b for b, _ in bcs], keep=bcs,
                    p0=[torch.zeros(pr["N"], **F64) for pr in prs])
    B, S = c["B"], c["S"]
    x, t, m = _patches(B, S, seed)
    if kind == "train":
        tr = surrogate.Trainer(surrogate.init_params(seed), B, S, torch.device(DEV, 0))
        g = _gen(seed + 1)
        # the moments of a run that has been going for a while
        tr.m.copy_(1e-3 * torch.randn(tr.p.numel(), generator=g, device=DEV))
        tr.v.copy_(1e-5 * (0.5 + torch.rand(tr.p.numel(), generator=g, device=DEV)))
        return dict(kind=kind, tr=tr, start=[tr.p.clone(), tr.m.clone(), tr.v.clone()], x=x, t=t, m=m)
    nb = cams.cams_net_tc_work_bytes(B, S)
    return dict(kind=kind, B=B, S=S, x=x, params=torch.from_numpy(surrogate.load_params()).to(DEV),
                y=torch.empty((B, cams.CAMS_NET_OUT, S ** 3), device=DEV),
                work=torch.empty(nb, dtype=torch.uint8, device=DEV), nb=nb)


# --------------------------------------------------------------- a pass ---

def run(s):
    kind = s["kind"]
    if kind == "residual":
        pr, N = s["pr"], s["pr"]["N"]
        A = s["A"]
        code, norm = cams.cams_residual_norm_noalloc(pr["nx"], pr["ny"], pr["nz"], A[0], A[1], A[2], A[3], s["f"], s["p"], s["r"],
                                                     torch.cuda.current_stream().cuda_stream)
        if code != cams.CAMS_OK:
            raise cams.CamsError(code, cams.cams_last_error())
        return dict(norm=norm, r=s["r"])
    if kind in ("assemble", "basis", "iterate"):
        h, pr = s["h"].h, s["pr"]
        out = {}
        if kind == "basis":
            out["rebuilt"] = cams.cams_update_basis(h, True)
        else:
            out["eps"] = cams.cams_assemble(h, s["p"], s["pn"], pr["dt"], s["bc"])
            if kind == "iterate":
                out["norms"] = cams.cams_iterate(h, pr["iters"])
        for q, dst in s["out"]:
            out["q%d" % q] = cams.cams_get(h, q, dst)
        return out
    if kind == "solve":
        h, pr = s["h"].h, s["pr"]
        cams.cams_set_permeability(h, pr["k"], pr["k"], pr["kz"])
        p, steps = torch.zeros(pr["N"], **F64), []
        for _ in range(pr["steps"]):
            pn, p = p, p.clone()
            cams.cams_solve(h, pn, pr["dt"], s["bc"], p, allow_noconv=True)
            steps.append(p)
        return steps
    if kind == "ensemble":
        for h, pr in zip(s["hs"], s["prs"]):
            cams.cams_set_permeability(h.h, pr["k"], pr["k"], pr["kz"])
        ps = [p.clone() for p in s["p0"]]
        torch.cuda.current_stream().synchronize()   # the members run on streams of their own
        cams.cams_ensemble_solve([h.h for h in s["hs"]], s["p0"], [pr["dt"] for pr in s["prs"]], s["bcs"], ps)
        return ps
    if kind == "train":
        tr = s["tr"]
        for dst, src in zip((tr.p, tr.m, tr.v), s["start"]):   # the same step of the same run
            dst.copy_(src)
        tr.t = 99
        loss = tr.step(s["x"], s["t"], s["m"])
        return dict(loss=loss, g=tr.g, p=tr.p, m=tr.m, v=tr.v)
    code = cams.cams_net_forward_tc(s["B"], s["S"], s["x"], s["params"], s["y"], s["work"], s["nb"],
                                    torch.cuda.current_stream().cuda_stream)
    if code != cams.CAMS_OK:
        raise cams.CamsError(code, cams.cams_last_error())
    return s["y"]


# ------------------------------------------------------------------ work ---

NET = surrogate.LAYERS
# typical counts of a step from p = 0 (the 4M-cell step: 5 linearisations and
# 45 iterations)
NEWTON, ITERATIONS = 5, 45


def _iteration_bytes(c):
    """Per cell: a coarse correction reads P, A, f, p and writes p; a
    smoothing step reads A, its pivots, f, p and writes p (half of the
    preconditioner's in FP32)."""
    w = 4 if c["precision"] else 8
    return (8 + 4) * w + 24 + c["n_post"] * 8 * w


def _basis_flops(c):
    """Banded factorisations and solves of the full dual-block interiors."""
    l = sorted(max(v - 1, 1) for v in (c["bx"], c["by"], c["bz"]))
    n, m = l[0] * l[1] * l[2], l[0] * l[1]
    nrhs = 2 ** sum(v > 1 for v in (c["bx"], c["by"], c["bz"]))
    return (n * m * m + 4.0 * n * m * nrhs) * (c["nx"] * c["ny"] * c["nz"]) / (c["bx"] * c["by"] * c["bz"])


def _step_work(c):
    N = c["nx"] * c["ny"] * c["nz"]
    w = 4 if c["precision"] else 8
    return dict(bytes=N * (NEWTON * 80.0 + 8 * w + 32 + ITERATIONS * _iteration_bytes(c)),
                flops=_basis_flops(c) + N * (NEWTON * 60.0 + ITERATIONS * (60.0 + 30.0 * c["n_post"])))


def work(case):
    c, kind = case, case["kind"]
    if kind in ("train", "infer"):
        cells = c["B"] * c["S"] ** 3
        mac = 27.0 * sum(a * b for a, b in NET)
        first = 27.0 * NET[0][0] * NET[0][1]
        if kind == "infer":
            return dict(bytes=cells * 4.0 * (12 + 8) + 4 * cams.CAMS_NET_PARAMS, flops=2 * cells * mac)
        return dict(bytes=cells * 4.0 * (12 + 16) + 4 * 6 * cams.CAMS_NET_PARAMS, flops=2 * cells * (3 * mac - first))
    if kind == "ensemble":
        fit = [s for s in LADDER if c["smallest"] <= s[0] * s[1] * s[2] <= c["largest"]]
        ws = [_step_work(_case("", "solve", *fit[(5 * m) % len(fit)], (8, 8, 8), **MIXED)) for m in range(c["members"])]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    N = c["nx"] * c["ny"] * c["nz"]
    if kind == "residual":
        return dict(bytes=56.0 * N, flops=15.0 * N)
    if kind == "assemble":
        return dict(bytes=80.0 * N, flops=60.0 * N)
    if kind == "basis":
        return dict(bytes=136.0 * N, flops=_basis_flops(c) + 300.0 * N)
    if kind == "iterate":
        return dict(bytes=N * (80.0 + c["iters"] * _iteration_bytes(c)), flops=N * (60.0 + c["iters"] * (60.0 + 30.0 * c["n_post"])))
    w = _step_work(c)
    return {k: v * c["steps"] for k, v in w.items()}


# ------------------------------------------- the definitions in 64 bits ---
# Arrays over the cells, x fastest.  A coupling along direction e is stored at
# the upper cell of its face, 0 on the low side of the grid.

def _stride(pr, e):
    return (1, pr["nx"], pr["nx"] * pr["ny"])[e]


def _low(pr, v, e):
    """The value at each cell's lower neighbour (0 outside)."""
    a = v.reshape(pr["nz"], pr["ny"], pr["nx"])
    out = torch.zeros_like(a)
    ax = 2 - e
    out.narrow(ax, 1, a.shape[ax] - 1).copy_(a.narrow(ax, 0, a.shape[ax] - 1))
    return out.reshape(-1)


def _up(pr, v, e):
    """The value at each cell's upper neighbour (0 outside)."""
    a = v.reshape(pr["nz"], pr["ny"], pr["nx"])
    out = torch.zeros_like(a)
    ax = 2 - e
    out.narrow(ax, 0, a.shape[ax] - 1).copy_(a.narrow(ax, 1, a.shape[ax] - 1))
    return out.reshape(-1)


def _trans(pr):
    """Transmissibilities of the lower faces: half-cell conductances in series."""
    d = pr["d"]
    V = d[0] * d[1] * d[2]
    out = []
    for e, k in enumerate((pr["k"], pr["k"], pr["kz"])):
        r = d[e] / (2.0 * k)
        t = (V / d[e]) / (r + _low(pr, r, e))
        inside = _low(pr, torch.ones_like(t), e)
        out.append(t * inside)
    return out


def _rho(pr, p):
    return torch.exp(pr["coef"] * p) if pr["law"] == 0 else 1.0 + pr["coef"] * p


def _drho(pr, p):
    return pr["coef"] * torch.exp(pr["coef"] * p) if pr["law"] == 0 else torch.full_like(p, pr["coef"])


def _linearise(pr, p, pn):
    """(A as [diagonal, x, y, z couplings], f, norm of the nonlinear error)."""
    d, phi, dt = pr["d"], 0.1, pr["dt"]
    V = d[0] * d[1] * d[2]
    rho, rhon = _rho(pr, p), _rho(pr, pn)
    C = V * phi * rhon * _drho(pr, p) / (dt * rho)
    q = torch.zeros_like(p)
    if pr["src"][0] is not None:
        q.index_add_(0, pr["src"][0].long(), pr["src"][1])
    w = [t * 0.5 * (rho + _low(pr, rho, e)) for e, t in enumerate(_trans(pr))]
    diag = C + sum(a + _up(pr, a, e) for e, a in enumerate(w))
    flux = sum(a * (p - _low(pr, p, e)) - _up(pr, a * (p - _low(pr, p, e)), e) for e, a in enumerate(w))
    f = V * rho * (-phi / dt + phi * rhon / (dt * rho) + q / V) + C * p
    if pr["bc"] == "dirichlet":
        x = torch.arange(pr["N"], device=DEV) % pr["nx"]
        tb = (V / d[0]) / (d[0] / (2.0 * pr["k"]))
        for at, pb in ((0, 1.0), (pr["nx"] - 1, 0.0)):
            wb = torch.where(x == at, tb * float(_rho(pr, torch.tensor(pb, dtype=torch.float64))), 0.0)
            diag, f, flux = diag + wb, f + wb * pb, flux + wb * (p - pb)
    eps = q / V - phi / dt + phi / dt * rhon / rho - flux / (V * rho)
    return [diag] + [-a for a in w], f, float(torch.linalg.vector_norm(eps))


def _apply(pr, A, p):
    out = A[0] * p
    for e in range(3):
        out = out + A[1 + e] * _low(pr, p, e) + _up(pr, A[1 + e] * p, e)
    return out


def _basis_matrix(pr, p, pn):
    """The basis operator of the case's basis equation: [diagonal, couplings]
    (internal faces only)."""
    rho, rhon = _rho(pr, p), _rho(pr, pn)
    w, kind = _trans(pr), pr["basis"]
    V = pr["d"][0] * pr["d"][1] * pr["d"][2]
    if kind in (1, 2):
        w = [t * 0.5 * (rho + _low(pr, rho, e)) for e, t in enumerate(w)]
    diag = sum(a + _up(pr, a, e) for e, a in enumerate(w))
    if kind == 1:
        diag = diag + V * 0.1 * rhon * _drho(pr, p) / (pr["dt"] * rho)
    if kind == 3:
        diag = diag + V * 0.1 * _drho(pr, pn) / (pr["dt"] * rhon)
    return [diag] + [-a for a in w]


def _pieces(n, b):
    """(first cell, cells, free) of the vertex planes and of the runs between
    them along one direction."""
    if n == 1:
        return [(0, 1, False)]
    nodes = list(range(b // 2, n, b))
    cuts = [-1] + nodes + [n]
    return [(v, 1, False) for v in nodes] + [(lo + 1, hi - lo - 1, True) for lo, hi in zip(cuts, cuts[1:]) if hi - lo > 1]


def _prolongation(pr, Ab):
    """P slot-major (8, N) and the coarse column of every slot (-1: none):
    slot bit e = the lower or upper coarse node along e of the cell's dual
    block.  Vertices, edges, faces and interiors in turn, each entity's
    system with its higher-level neighbours lumped on the diagonal."""
    n, b, N = (pr["nx"], pr["ny"], pr["nz"]), (pr["bx"], pr["by"], pr["bz"]), pr["N"]
    i = torch.arange(N, device=DEV)
    xyz = (i % n[0], i // n[0] % n[1], i // (n[0] * n[1]))
    free = [torch.zeros(N, dtype=torch.bool, device=DEV) if n[e] == 1 else (xyz[e] - b[e] // 2) % b[e] != 0 for e in range(3)]
    level = free[0].int() + free[1].int() + free[2].int()
    lower = [torch.div(xyz[e] - b[e] // 2, b[e], rounding_mode="floor") if n[e] > 1 else torch.zeros_like(i) for e in range(3)]
    nc = [n[e] // b[e] for e in range(3)]
    col = torch.zeros((8, N), dtype=torch.int64, device=DEV)
    for s in range(8):
        ok, J = torch.ones(N, dtype=torch.bool, device=DEV), torch.zeros(N, dtype=torch.int64, device=DEV)
        for e in (2, 1, 0):
            bit = s >> e & 1
            at = lower[e] + bit
            ok &= (at >= 0) & (at < nc[e]) & (free[e] if bit else torch.ones_like(ok))
            J = J * nc[e] + at
        col[s] = torch.where(ok, J, -1)
    P = torch.zeros((8, N), **F64)
    P[0, level == 0] = 1.0
    lumped = Ab[0].clone()
    for e in range(3):
        for nb, a in ((_low, Ab[1 + e]), (_up, _up(pr, Ab[1 + e], e))):
            lumped += torch.where(nb(pr, level, e) == level + 1, a, 0.0)
    per = [_pieces(n[e], b[e]) for e in range(3)]
    for lev in (1, 2, 3):
        groups = {}
        for cz in per[2]:
            for cy in per[1]:
                for cx in per[0]:
                    if cx[2] + cy[2] + cz[2] == lev:
                        key = ((cx[1], cy[1], cz[1]), (cx[2], cy[2], cz[2]))
                        groups.setdefault(key, []).append(cx[0] + n[0] * (cy[0] + n[1] * cz[0]))
        for (L, fr), org in groups.items():
            m = L[0] * L[1] * L[2]
            j = torch.arange(m, device=DEV)
            at = (j % L[0], j // L[0] % L[1], j // (L[0] * L[1]))
            off = at[0] + n[0] * (at[1] + n[1] * at[2])
            for part in torch.tensor(org, device=DEV).split(max(1, int(2e8) // (m * m))):
                cell = part[:, None] + off[None, :]
                M = torch.zeros((len(part), m, m), **F64)
                M[:, j, j] = lumped[cell]
                rhs = torch.zeros((len(part), m, 8), **F64)
                for e in range(3):
                    if not fr[e]:
                        continue
                    st, lst = _stride(pr, e), (1, L[0], L[0] * L[1])[e]
                    hi = j[at[e] > 0]
                    v = Ab[1 + e][cell[:, hi]]
                    M[:, hi, hi - lst] = v
                    M[:, hi - lst, hi] = v
                    for edge, side in ((0, 0), (L[e] - 1, 1)):
                        q = j[at[e] == edge]
                        mine = cell[:, q]
                        x = mine[0, 0] // st % n[e]
                        # partial dual blocks have no plane on the grid's side
                        here = (mine[:, 0] // st % n[e] > 0) if side == 0 else (mine[:, 0] // st % n[e] < n[e] - 1)
                        if not bool(here.any()):
                            continue
                        other = (mine + (st if side else -st)).clamp(0, N - 1)
                        a = Ab[1 + e][other if side else mine] * here[:, None]
                        for s in range(8):
                            if s >> e & 1 == side:
                                rhs[:, q, s] -= a * P[s & ~(1 << e)][other]
                sol = torch.linalg.solve(M, rhs)
                for s in range(8):
                    P[s, cell.reshape(-1)] = sol[:, :, s].reshape(-1)
    P = torch.where(col >= 0, P, 0.0)
    return P, col


def _coarse(pr, A, P, col):
    """R A P as a 27-point stencil per coarse row (MSFE: R = P^T; MSFV: sums
    over the primal blocks)."""
    n, b = (pr["nx"], pr["ny"], pr["nz"]), (pr["bx"], pr["by"], pr["bz"])
    nc = [n[e] // b[e] for e in range(3)]
    Nc = nc[0] * nc[1] * nc[2]
    out = torch.zeros(27 * Nc, **F64)

    def parts(J):
        return J % nc[0], J // nc[0] % nc[1], J // (nc[0] * nc[1])

    i = torch.arange(pr["N"], device=DEV)
    if pr["restriction"] == 1:
        blk = [torch.div(c, b[e], rounding_mode="floor") for e, c in enumerate((i % n[0], i // n[0] % n[1], i // (n[0] * n[1])))]
        rows = [(blk[0] + nc[0] * (blk[1] + nc[1] * blk[2]), torch.ones(pr["N"], **F64))]
    else:
        rows = [(col[s], P[s]) for s in range(8)]
    nbr = [(i, A[0])]
    for e in range(3):
        st = _stride(pr, e)
        nbr += [((i - st).clamp_min(0), A[1 + e]), ((i + st).clamp_max(pr["N"] - 1), _up(pr, A[1 + e], e))]
    for I, wt in rows:
        Ip = parts(I.clamp_min(0))
        for j, a in nbr:
            for s in range(8):
                J, v = col[s][j], wt * a * P[s][j]
                keep = (I >= 0) & (J >= 0) & (v != 0)
                Jp = parts(J.clamp_min(0))
                t = (Jp[0] - Ip[0] + 1) + 3 * (Jp[1] - Ip[1] + 1) + 9 * (Jp[2] - Ip[2] + 1)
                out.index_add_(0, (27 * I + t)[keep], v[keep])
    return out


def _planes(pr):
    """The cells of every hyperplane x + y + z = const."""
    i = torch.arange(pr["N"], device=DEV)
    s = i % pr["nx"] + i // pr["nx"] % pr["ny"] + i // (pr["nx"] * pr["ny"])
    order = torch.argsort(s, stable=True)
    return order.split(torch.bincount(s).tolist())


def _wave(pr, planes, start, couplings, step):
    """Visits the hyperplanes in order: v = step(cells, neighbours' values)."""
    v = torch.zeros(pr["N"] + 1, **F64)
    for cells in planes:
        got = []
        for e in range(3):
            at = cells + start * _stride(pr, e)
            a = couplings[e][cells]
            got.append((a, v[torch.where(a != 0, at, pr["N"])]))
        v[cells] = step(cells, got)
    return v[:-1]


def _pivots(pr, A, planes):
    return 1.0 / _wave(pr, planes, -1, A[1:], lambda c, g: 1.0 / (A[0][c] - sum(a * a * v for a, v in g)))


def _iterate(pr, A, f, p, P, col, n):
    """n C-AMS iterations; the residual norms before and after each."""
    planes = _planes(pr)
    back = planes[::-1]
    d = _pivots(pr, A, planes)
    low = [a / d for a in A[1:]]
    high = [_up(pr, a, e) / d for e, a in enumerate(A[1:])]
    st = _coarse(pr, A, P, col).reshape(-1, 27)
    Nc, nc = st.shape[0], [pr[a] // pr[b] for a, b in (("nx", "bx"), ("ny", "by"), ("nz", "bz"))]
    K = torch.zeros((Nc, Nc), **F64)
    I = torch.arange(Nc, device=DEV)
    for t in range(27):
        at = (I % nc[0] + t % 3 - 1, I // nc[0] % nc[1] + t // 3 % 3 - 1, I // (nc[0] * nc[1]) + t // 9 - 1)
        ok = sum(((at[e] >= 0) & (at[e] < nc[e])).int() for e in range(3)) == 3
        J = at[0] + nc[0] * (at[1] + nc[1] * at[2])
        K[I[ok], J[ok]] = st[ok, t]
    LU = torch.linalg.lu_factor(K)
    i = torch.arange(pr["N"], device=DEV)
    blk = i % pr["nx"] // pr["bx"] + nc[0] * (i // pr["nx"] % pr["ny"] // pr["by"] + nc[1] * (i // (pr["nx"] * pr["ny"]) // pr["bz"]))
    norms = []
    for k in range(n + 1):
        r = f - _apply(pr, A, p)
        norms.append(float(torch.linalg.vector_norm(r)))
        if k == n:
            break
        rc = torch.zeros(Nc, **F64)
        if pr["restriction"] == 1:
            rc.index_add_(0, blk, r)
        else:
            for s in range(8):
                rc.index_add_(0, col[s].clamp_min(0), P[s] * r)
        pc = torch.linalg.lu_solve(*LU, rc[:, None])[:, 0]
        p = p + sum(P[s] * pc[col[s].clamp_min(0)] for s in range(8))
        for _ in range(pr["n_post"]):
            rd = (f - _apply(pr, A, p)) / d
            w = _wave(pr, planes, -1, low, lambda c, g: rd[c] - sum(a * v for a, v in g))
            p = p + _wave(pr, back, 1, high, lambda c, g: w[c] - sum(a * v for a, v in g))
    return np.array(norms), p


def _dense_step(pr, pn):
    """The implicit step's root by Newton steps with dense solves."""
    p, N = pn.clone(), pr["N"]
    i = torch.arange(N, device=DEV)
    for _ in range(60):
        A, f, _ = _linearise(pr, p, pn)
        M = torch.diag(A[0])
        for e in range(3):
            hi = i[A[1 + e] != 0]
            M[hi, hi - _stride(pr, e)] = A[1 + e][hi]
            M[hi - _stride(pr, e), hi] = A[1 + e][hi]
        new = torch.linalg.solve(M, f)
        done = float((new - p).abs().max()) < 1e-14
        p = new
        if done:
            break
    return p


def _network(w, x, S):
    a, o = x.reshape(x.shape[0], -1, S, S, S), 0
    for k, (ci, co) in enumerate(NET):
        wt, bias = w[o:o + co * ci * 27].reshape(co, ci, 3, 3, 3), w[o + co * ci * 27:o + co * ci * 27 + co]
        o += co * ci * 27 + co
        pad = F.pad(a, (1,) * 6)
        # one product per tap: plain matrix products in 64 bits
        y = bias.reshape(1, -1, 1) + sum(
            torch.matmul(wt[:, :, t // 9, t // 3 % 3, t % 3],
                         pad[:, :, t // 9:t // 9 + S, t // 3 % 3:t // 3 % 3 + S, t % 3:t % 3 + S].reshape(a.shape[0], ci, -1))
            for t in range(27))
        a = y.clamp_min(0).reshape(-1, co, S, S, S) if k < len(NET) - 1 else y
    return a


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "infer":
        s = prepare(c, seed)
        w = s["params"].double()
        return torch.cat([_network(w, x.double(), c["S"]) for x in s["x"].split(256)])
    if kind == "train":
        s = prepare(c, seed)
        S = c["S"]
        w0, m0, v0 = (a.double() for a in s["start"])
        w = w0.clone().requires_grad_(True)
        e = (s["m"].double() * (_network(w, s["x"].double(), S) - s["t"].double())).reshape(c["B"], 8, S, S, S)
        wt = torch.exp(s["x"].double()).reshape(c["B"], -1, S, S, S)
        loss = 0.0
        for d in range(3):
            ax = 4 - d
            hi, lo = e.narrow(ax, 1, S - 1), e.narrow(ax, 0, S - 1)
            loss = loss + (wt[:, d:d + 1].narrow(ax, 1, S - 1) * (hi - lo) ** 2).sum()
        loss = (loss / s["m"].double().sum())
        loss.backward()
        g = w.grad
        m, v = 0.9 * m0 + 0.1 * g, 0.999 * v0 + 0.001 * g * g
        p = w0 - 1e-3 * (m / (1 - 0.9 ** 100)) / (torch.sqrt(v / (1 - 0.999 ** 100)) + 1e-8)
        return dict(loss=loss.detach().reshape(1), g=g, p=p, m=m, v=v)
    if kind == "ensemble":
        return None   # no closed values short of solving every member to its root
    pr = _problem(c, seed)
    if kind == "solve":
        # the root of each step, where dense solves do it
        if pr["N"] > 3000 or pr["bc"] != "dirichlet":
            return None
        p, steps = torch.zeros(pr["N"], **F64), []
        for _ in range(pr["steps"]):
            p = _dense_step(pr, p)
            steps.append(p)
        return steps
    p, pn = _pressures(pr, seed)
    A, f, eps = _linearise(pr, p, pn)
    if kind == "residual":
        r = f - _apply(pr, A, p)
        return dict(norm=float(torch.linalg.vector_norm(r)), r=r)
    if kind == "assemble":
        return dict(eps=eps, q2=torch.cat(A), q3=f)
    P, col = _prolongation(pr, _basis_matrix(pr, p, pn))
    if kind == "basis":
        return dict(rebuilt=None, q6=P.reshape(-1), q8=_coarse(pr, A, P, col), q9=_pivots(pr, A, _planes(pr)))
    norms, p = _iterate(pr, A, f, p, P, col, c["iters"])
    return dict(eps=eps, norms=norms, q5=p)

