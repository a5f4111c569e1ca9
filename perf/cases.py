"""Performance cases: what a user of the library has it do, through its public Python entry points.

A pass is one call of a user's program: the set-up of a hierarchy and its PCG solve (one problem in, its
solution out), further PCG or GMRES solves on a hierarchy that the program keeps, or a batch of independent
problems.  Every pass returns the whole solution vectors.  The solves run to a tight tolerance, as a program
that differentiates or post-processes the solution asks for: the solution is then determined by the problem
and not by where the iteration stopped.
"""
import math

import numpy as np
import torch

import paper_2106_06404_gb300 as msdd

ETA = 0.3                                  # the eigenvalue threshold of every workload of this repository
DRAWN_KINDS = ("setup_solve", "setup_solve", "setup_solve", "solve", "gmres", "batch")


def _case(name, kind, n, parts, levels, nev, precision, field, contrast, tol, overlap=2, group=(1, 1, 1), faces=1,
          count=1):
    n, parts, group = [tuple(v) + (1,) * (3 - len(v)) for v in (n, parts, group)]
    c = dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], px=parts[0], py=parts[1], pz=parts[2], levels=levels, gx=group[0],
             gy=group[1], gz=group[2], overlap=overlap, nev=nev, precision=precision, field=field, contrast=contrast,
             tol=tol, faces=faces, count=count)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest problems (a parameter study's inner solve): latency of some hundred small launches
        _case("channels_64_small", "setup_solve", (64, 64), (4, 4), 2, 8, 1, "channels", 1e4, 1e-10),
        # a ragged rectangle with three levels in the default FP64 form, Dirichlet on two faces
        _case("ragged_104x88_fp64", "setup_solve", (104, 88), (6, 5), 3, 6, 0, "grf", 1e3, 1e-10, group=(2, 2),
              faces=0b0110),
        # anisotropic tensors on a mid-size mesh, uneven subdomains, two levels
        _case("tensor_250x190", "setup_solve", (250, 190), (9, 7), 2, 10, 1, "tensor", 1e2, 1e-10),
        # the ordinary call: 512^2, three levels, FP32 local factors
        _case("grf_512_3lvl", "setup_solve", (512, 512), (16, 16), 3, 12, 1, "grf", 1e1, 1e-10, group=(4, 4)),
        # the same kind of problem in the default form, all FP64
        _case("grf_384_fp64", "setup_solve", (384, 384), (12, 12), 3, 12, 0, "grf", 1e2, 1e-10, group=(4, 4)),
        # more subdomains than one wave of the GPU, wide coarse spaces
        _case("grf_1000_3lvl", "setup_solve", (1000, 1000), (31, 31), 3, 12, 1, "grf", 1e1, 1e-10, group=(4, 4)),
        # 3D, the default FP64 form on a small layered box
        _case("layers_30_fp64", "setup_solve", (30, 30, 30), (3, 3, 3), 2, 10, 0, "layers", 1e2, 1e-10, overlap=1),
        # 3D, FP32 local factors, uneven boxes
        _case("layers_50x44x38", "setup_solve", (50, 44, 38), (4, 4, 3), 2, 12, 1, "layers", 1e2, 1e-10, overlap=1),
        # 3D, the layered anisotropic composite at 16^3 elements a subdomain: the largest call
        _case("composite_96", "setup_solve", (96, 96, 96), (6, 6, 6), 3, 16, 1, "composite", 1e2, 1e-10, overlap=1,
              group=(2, 2, 2)),
        # the next right-hand side on a hierarchy that the program keeps: PCG, then the hybrid form in GMRES
        _case("pcg_512_kept", "solve", (512, 512), (16, 16), 3, 12, 1, "grf", 1e1, 1e-10, group=(4, 4)),
        _case("gmres_300_kept_fp64", "gmres", (300, 300), (9, 9), 2, 10, 0, "grf", 1e3, 1e-10),
        # independent problems of uneven size on concurrent streams
        _case("batch_16", "batch", (128, 128), (4, 4), 2, 8, 1, "channels", 1e4, 1e-10, count=16),
    ]


def draw(rng):
    kind = rng.choice(DRAWN_KINDS)
    precision = rng.choice((0, 1, 1))
    contrast = 10.0 ** rng.uniform(0.5, 3.0)
    if kind == "batch":
        n = rng.randint(96, 200)
        return _case(None, kind, (n, n), (4, 4), 2, 8, precision, rng.choice(("channels", "grf")), contrast, 1e-10,
                     count=rng.randint(4, 16))
    if kind == "setup_solve" and rng.random() < 0.35:                     # 3D boxes
        parts = rng.randint(2, 5) if precision else rng.randint(2, 3)
        n = [rng.randint(5 * parts, 16 * parts if precision else 10 * parts) for _ in range(3)]
        return _case(None, kind, n, (parts,) * 3, 2, rng.randint(6, 16), precision, rng.choice(("layers", "composite")),
                     min(contrast, 1e2), 1e-10, overlap=1)
    side = math.exp(rng.uniform(math.log(48), math.log(700 if precision else 320)))
    n = (int(side * rng.uniform(0.8, 1.2)), int(side * rng.uniform(0.8, 1.2)))
    parts = [max(2, int(v / rng.uniform(18.0, 36.0))) for v in n]
    levels = 3 if min(parts) >= 4 and rng.random() < 0.5 else 2
    if levels == 3:
        contrast = min(contrast, 20.0)            # the coefficient's own scatter comes on top
    return _case(None, kind, n, parts, levels, rng.randint(6, 14), precision, rng.choice(("channels", "grf", "tensor")),
                 contrast, 1e-10, overlap=rng.randint(1, 3), group=(2, 2) if levels == 3 else (1, 1),
                 faces=rng.choice((0b1, 0b0110, 0b0011)))


# ------------------------------------------------------------------ inputs
def _dim(c):
    return 3 if c["nz"] > 1 else 2


def _shape(c):
    return tuple(c[k] for k in ("nx", "ny", "nz")[:_dim(c)])


def _gaussian_field(nx, ny, gen, corr_len=0.05, variance=2.0):
    """Stationary field with covariance variance * exp(-r / corr_len), by circulant embedding; (ny, nx)."""
    big = 2 * max(nx, ny)
    h = 2.0 / big
    i = torch.arange(big, device="cuda", dtype=torch.float64)
    d = torch.minimum(i, big - i) * h
    cov = variance * torch.exp(-torch.sqrt(d[:, None] ** 2 + d[None, :] ** 2) / corr_len)
    lam = torch.fft.fft2(cov).real.clamp_min(0.0)
    eps = torch.randn((big, big, 2), generator=gen, device="cuda", dtype=torch.float64)
    return torch.fft.fft2(torch.sqrt(lam / (big * big)) * torch.view_as_complex(eps)).real[:ny, :nx]


def _coefficient(c, seed):
    """The element coefficients: (elements,) scalar or (elements, 3 | 6) tensor, x fastest."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    f64 = dict(device="cuda", dtype=torch.float64)
    if c["field"] in ("channels", "tensor"):
        # conducting one-element channels in a background of 1 with some scatter
        rows = torch.tensor(rng.choice(ny, max(2, ny // 8), replace=False), device="cuda")
        k = torch.exp(0.2 * torch.randn((ny, nx), generator=gen, **f64))
        k[rows] *= c["contrast"]
        if c["field"] == "channels":
            return k.reshape(-1)
        # principal axes rotated by an angle of each element, anisotropy 1 : 1e-1
        a = math.pi * torch.rand((ny, nx), generator=gen, **f64)
        co, si = torch.cos(a), torch.sin(a)
        return torch.stack([k * (co * co + 0.1 * si * si), k * (si * si + 0.1 * co * co), k * 0.9 * co * si],
                           dim=-1).reshape(-1, 3).contiguous()
    if c["field"] == "grf":
        # log-normal background, channels and square inclusions of higher conductivity
        k = torch.exp(_gaussian_field(nx, ny, gen))
        mask = torch.zeros((ny, nx), dtype=torch.bool, device="cuda")
        for r in rng.choice(ny - 1, max(2, ny // 32), replace=False):
            mask[r:r + 2] = True
        for _ in range(max(2, min(nx, ny) // 16)):
            s = int(rng.integers(3, max(4, min(24, nx // 8)) + 1))
            x0, y0 = int(rng.integers(0, nx - s)), int(rng.integers(0, ny - s))
            mask[y0:y0 + s, x0:x0 + s] = True
        k[mask] *= c["contrast"]
        return k.reshape(-1)
    scatter = torch.exp(0.3 * torch.randn((nz, ny, nx), generator=gen, **f64))
    if c["field"] == "layers":
        thick = np.sort(rng.choice(np.arange(1, nz), max(1, nz // 4), replace=False))
        layer = torch.tensor(np.searchsorted(thick, np.arange(nz), side="right") % 2, device="cuda")
        return (scatter * torch.where(layer == 1, c["contrast"], 1.0)[:, None, None]).reshape(-1)
    # plies diag(1, a, a) rotated by +-45 degrees about z, a = 1 / contrast, with thin isotropic resin layers between
    plies = max(2, min(9, nz // 6))
    cut = np.sort(rng.choice(np.arange(2, nz - 1), plies - 1, replace=False))
    ply = np.searchsorted(cut, np.arange(nz), side="right")
    resin = np.isin(np.arange(nz), cut)
    a, sign = 1.0 / c["contrast"], rng.choice((-1.0, 1.0))
    t = torch.zeros((nz, ny, nx, 6), **f64)
    for z in range(nz):
        s = sign * (1.0 if ply[z] % 2 else -1.0)
        v = [0.1, 0.1, 0.1, 0.0, 0.0, 0.0] if resin[z] else [(1 + a) / 2, (1 + a) / 2, a, 0.0, 0.0, s * (1 - a) / 2]
        t[z] = torch.tensor(v, **f64)
    return (t * scatter[..., None]).reshape(-1, 6).contiguous()


def _problems(c, seed):
    """The problems of a batch: sides spread over [side, 2 side), subdomains of about 24 elements a side."""
    rng = np.random.default_rng(seed + 77)
    out = []
    for k in range(c["count"]):
        # one element shape, and sizes that depend on the case alone: the same work for every seed
        n = c["nx"] + (k * c["nx"]) // max(1, c["count"])
        p = max(c["px"], n // 24)
        out.append(dict(c, nx=n, ny=n, px=p, py=p, seed=int(rng.integers(1 << 30))))
    return out


def _arguments(c):
    d = _dim(c)
    return dict(n=_shape(c), parts=(c["px"], c["py"], c["pz"])[:d], overlap=c["overlap"], levels=c["levels"],
                group=(c["gx"], c["gy"], c["gz"])[:d], nev_max=c["nev"], eta=ETA, dirichlet_faces=c["faces"],
                precision=c["precision"], allow_eig_unconverged=True)


def prepare(case, seed):
    if case["kind"] == "batch":
        problems = []
        for p in _problems(case, seed):
            a = _arguments(p)
            problems.append(dict(n=a["n"], parts=a["parts"], overlap=a["overlap"], levels=a["levels"], group=a["group"],
                                 kappa=_coefficient(p, p["seed"]), b=msdd.assemble_rhs(a["n"])))
        return dict(case=case, problems=problems)
    kappa, args = _coefficient(case, seed), _arguments(case)
    b = msdd.assemble_rhs(args["n"], args["dirichlet_faces"])
    state = dict(case=case, kappa=kappa, args=args, b=b)
    if case["kind"] != "setup_solve":
        state["hierarchy"] = msdd.Hierarchy(coeff=kappa, **args)
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        return msdd.batch_run(state["problems"], case["nev"], ETA, tol=case["tol"], maxit=4000,
                              precision=case["precision"], allow_fail=True)[0]
    if case["kind"] == "setup_solve":
        h = msdd.Hierarchy(coeff=state["kappa"], **state["args"])
        x, _, _ = h.solve(state["b"], tol=case["tol"], maxit=4000)
        h.close()
        return x
    if case["kind"] == "solve":
        return state["hierarchy"].solve(state["b"], tol=case["tol"], maxit=4000)[0]
    return state["hierarchy"].solve_gmres(state["b"], tol=case["tol"], maxit=4000)[0]


# ------------------------------------------------------------------ work
def _boxes(c):
    """(nodes, half-bandwidth) of every subdomain's box."""
    d = _dim(c)
    axes = []
    for n, p in zip(_shape(c), (c["px"], c["py"], c["pz"])):
        base, rem = divmod(n, p)
        at, w = 0, []
        for k in range(p):
            e = base + (k < rem)
            w.append(min(n, at + e + c["overlap"]) - max(0, at - c["overlap"]) + 1)
            at += e
        axes.append(w)
    if d == 2:
        return [(x * y, x + 1) for y in axes[1] for x in axes[0]]
    return [(x * y * z, x * y + x + 1) for z in axes[2] for y in axes[1] for x in axes[0]]


def work(case):
    if case["kind"] == "batch":
        w = [work(dict(p, kind="setup_solve")) for p in _problems(case, 0)]
        return {k: sum(v[k] for v in w) for k in ("bytes", "flops")}
    n, d, size = math.prod(_shape(case)), _dim(case), 4 if case["precision"] else 8
    comps = {"tensor": 3, "composite": 6}.get(case["field"], 1)
    boxes = _boxes(case)
    factor = sum(m * (b + 1) for m, b in boxes)
    steps = 40                                   # CG or GMRES steps that a well-preconditioned solve takes at least
    solve_bytes = steps * (factor * size + 10 * 8 * n)
    solve_flops = steps * (4.0 * factor + 2.0 * 3 ** d * n + 10 * n)
    if case["kind"] != "setup_solve":
        return {"bytes": solve_bytes + 16 * n, "flops": solve_flops}
    # two factorisations, and ten subspace iterations on nev + 4 columns with one solve, the stencil products of
    # both forms, two Gram products and the update each
    q = min(case["nev"] + 4, 32)
    eig = sum(10.0 * (4.0 * m * b * q + 4.0 * 3 ** d * m * q + 6.0 * m * q * q) for m, b in boxes)
    eig_bytes = sum(10.0 * (2.0 * m * (b + 1) * size + 6.0 * 8 * m * q) for m, b in boxes)
    return {"bytes": 8.0 * n * (comps + 2) + 2.0 * factor * size + eig_bytes + solve_bytes,
            "flops": 2.0 * sum(m * b * b for m, b in boxes) + eig + solve_flops}


# ------------------------------------------------------------------ exact
def _assemble(c, kappa):
    """Q1 stiffness over all nodes as lines (2D) or planes (3D): diagonal and upper off-diagonal dense blocks."""
    d, n = _dim(c), _shape(c)
    h = [1.0 / v for v in n]
    g = 0.5 / math.sqrt(3.0)
    pts = (0.5 - g, 0.5 + g)
    nloc = 1 << d
    ref = torch.zeros((d, d, nloc, nloc), dtype=torch.float64)
    for q in range(nloc):
        xi = [pts[(q >> k) & 1] for k in range(d)]
        grad = torch.zeros((nloc, d), dtype=torch.float64)
        for a in range(nloc):
            for e in range(d):
                v = (1.0 if (a >> e) & 1 else -1.0) / h[e]
                for k in range(d):
                    if k != e:
                        v *= xi[k] if (a >> k) & 1 else 1.0 - xi[k]
                grad[a, e] = v
        ref += math.prod(h) / nloc * torch.einsum("ae,bf->efab", grad, grad)
    ref = ref.cuda()
    ne = math.prod(n)
    k = kappa.reshape(ne, -1)
    full = torch.zeros((ne, d, d), dtype=torch.float64, device="cuda")
    if k.shape[1] == 1:
        for e in range(d):
            full[:, e, e] = k[:, 0]
    else:
        order = [(0, 0), (1, 1), (0, 1)] if d == 2 else [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)]
        for s, (e, f) in enumerate(order):
            full[:, e, f] = k[:, s]
            full[:, f, e] = k[:, s]
    ke = torch.einsum("nef,efab->nab", full, ref)
    m = [v + 1 for v in n]
    slab = math.prod(m[:-1])
    layer = math.prod(n[:-1])
    e = torch.arange(layer, device="cuda")
    ex, ey = (e, torch.zeros_like(e)) if d == 2 else (e % n[0], e // n[0])
    half = nloc // 2
    node = torch.stack([(ex + (a & 1)) + (m[0] * (ey + ((a >> 1) & 1)) if d == 3 else 0) for a in range(half)], 1)
    idx = (node[:, :, None] * slab + node[:, None, :]).reshape(-1)
    diag = [torch.zeros(slab * slab, dtype=torch.float64, device="cuda") for _ in range(m[-1])]
    off = []
    ke = ke.reshape(n[-1], layer, nloc, nloc)
    for z in range(n[-1]):
        diag[z].index_add_(0, idx, ke[z, :, :half, :half].reshape(-1))
        diag[z + 1].index_add_(0, idx, ke[z, :, half:, half:].reshape(-1))
        off.append(torch.zeros(slab * slab, dtype=torch.float64, device="cuda").index_add_(
            0, idx, ke[z, :, :half, half:].reshape(-1)).reshape(slab, slab))
    return [v.reshape(slab, slab) for v in diag], off


def _direct(c, kappa):
    """The solution at the unknowns by block elimination over lines or planes, with one step of refinement."""
    d, n = _dim(c), _shape(c)
    diag, off = _assemble(c, kappa)
    m = [v + 1 for v in n]
    free = torch.ones(tuple(reversed(m)), dtype=torch.bool, device="cuda")
    load = torch.ones(tuple(reversed(m)), dtype=torch.float64, device="cuda") * math.prod(1.0 / v for v in n)
    for k in range(d):
        ax = d - 1 - k
        load.select(ax, 0).mul_(0.5)
        load.select(ax, n[k]).mul_(0.5)
        if (c["faces"] >> (2 * k)) & 1:
            free.select(ax, 0).fill_(False)
        if (c["faces"] >> (2 * k + 1)) & 1:
            free.select(ax, n[k]).fill_(False)
    free = free.reshape(m[-1], -1)
    rhs = torch.where(free, load.reshape(m[-1], -1), 0.0)
    for z in range(m[-1]):
        f = free[z].to(torch.float64)
        diag[z].mul_(f[:, None] * f[None, :])
        diag[z].diagonal().add_(1.0 - f)
        if z + 1 < m[-1]:
            off[z].mul_(f[:, None] * free[z + 1].to(torch.float64)[None, :])
    chol, s = [], diag[0]
    for z in range(m[-1]):
        chol.append(torch.linalg.cholesky(s))
        if z + 1 < m[-1]:
            s = diag[z + 1] - off[z].T @ torch.cholesky_solve(off[z], chol[z])

    def solve(b):
        y = [b[0]]
        for z in range(1, m[-1]):
            y.append(b[z] - off[z - 1].T @ torch.cholesky_solve(y[z - 1][:, None], chol[z - 1])[:, 0])
        x = [None] * m[-1]
        for z in reversed(range(m[-1])):
            v = y[z] if z == m[-1] - 1 else y[z] - off[z] @ x[z + 1]
            x[z] = torch.cholesky_solve(v[:, None], chol[z])[:, 0]
        return torch.stack(x)

    x = solve(rhs)
    r = torch.stack([rhs[z] - diag[z] @ x[z] - (off[z] @ x[z + 1] if z + 1 < m[-1] else 0)
                     - (off[z - 1].T @ x[z - 1] if z else 0) for z in range(m[-1])])
    return (x + solve(r))[free]


def exact(case, seed):
    if case["kind"] == "batch":
        ps = _problems(case, seed)
        cost = sum(p["nx"] for p in ps)
        return [_direct(dict(p, faces=1), _coefficient(p, p["seed"])) for p in ps] if cost <= 4000 else None
    n = _shape(case)
    slab = math.prod(v + 1 for v in n[:-1])
    if slab ** 3 * n[-1] > 4e12 or slab * slab * n[-1] * 24 > 6e10:
        return None                                   # too long, or too large, for a dense block elimination
    return _direct(case, _coefficient(case, seed))
