"""The solver's work as its users call it, as timed cases.

A case names one call (or one step of a simulation loop) on one grid:

  solve    new psi or new load, then the multigrid solve from the boundary data
  grad     SIMP density -> solve -> loss -> adjoint gradient (SBMSolve, one training step)
  loop     steps of the staggered topology optimisation
  refine   composite solve on block-structured refinement
  residual FP64 residual of a given displacement (one layer of a custom outer loop)
  source   load vector of the SBM equation from eigenstrain, body force and traction

Inputs are synthetic, drawn on the GPU from the seed; the sizes are those of this
repository's configurations, tests and benchmark, ragged ones among them.  Solves run
to a relative residual of 1e-10 in FP64 and tighter where FP32 V-cycles or refinement
would leave a larger error in the solution, as this repository's tests do.
"""
import math
import random

import torch

import paper_2212_02362_gb300 as sbm

DEV = "cuda"
F8 = torch.float64


def listed():
    return [
        # 2D plate with a hole, load stepping on a fixed geometry: the smallest solve
        dict(name="plate_2d_65", kind="solve", dim=2, nx=65, ny=65, nz=1, precision="fp64"),
        # a plate at the size of the closed-form validation runs, FP64
        dict(name="plate_2d_513", kind="solve", dim=2, nx=513, ny=513, nz=1, precision="fp64"),
        # 2D voids, three refinement levels, colour Gauss-Seidel, FP64
        dict(name="voids_2d_refined", kind="refine", dim=2, n=129, levels=3, count=8, layout=1, precision="fp64"),
        # a damaged crystal on a small ragged box: every step of a damage evolution re-solves with a new psi
        dict(name="damage_3d_ragged", kind="solve", dim=3, nx=41, ny=33, nz=57, precision="mixed"),
        # the same at the benchmark's size: FP32 V-cycles in FP64 defect correction
        dict(name="damage_3d_129", kind="solve", dim=3, nx=129, ny=129, nz=129, precision="mixed"),
        # plain FP64, the precision a grid has by default
        dict(name="damage_3d_65_fp64", kind="solve", dim=3, nx=65, ny=65, nz=65, precision="fp64"),
        # one step of gradient-based design on the full-size cantilever: forward, adjoint, dJ/drho
        dict(name="design_3d_257", kind="grad", dim=3, nx=257, ny=129, nz=129, precision="mixed"),
        # the phase-field topology loop on a half-size cantilever, three steps in one call
        dict(name="topology_3d_129", kind="loop", dim=3, nx=129, ny=65, nz=65, steps=3, precision="mixed"),
        # spherical voids, two refinement levels in several patches, mixed precision
        dict(name="voids_3d_refined", kind="refine", dim=3, n=65, levels=2, count=6, layout=2, precision="mixed"),
        # the FP64 residual on its own
        dict(name="residual_3d_129", kind="residual", dim=3, nx=129, ny=129, nz=129),
        # the load vector on its own
        dict(name="source_3d_129", kind="source", dim=3, nx=129, ny=129, nz=129),
    ]


def draw(rng):
    case = _drawn(rng)
    lo = -3 if case["kind"] == "grad" or (case["kind"] == "refine" and case["dim"] == 3) else -4
    return dict(case, psi_min=float("%.3g" % 10 ** rng.uniform(lo, -2)))


def _drawn(rng):
    def box(lo, hi, ms, dim):
        # cells per axis m 2^k, lo to hi over the logarithm, k common to the axes so that the
        # coarsest multigrid level stays a few cells wide
        want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        k = max(0, min(int(math.log2(want / min(ms))), int(math.log2(hi / min(ms)))))
        return [(rng.choice([m for m in ms if m << k <= hi]) << k) + 1 for _ in range(dim)] + [1] * (3 - dim)

    kind = rng.choice(["solve2", "solve3", "solve3", "grad", "loop", "refine2", "refine3", "residual", "source"])
    if kind == "solve2":
        prec = rng.choice(["fp64", "fp64", "mixed"])
        n = box(16, 512 if prec == "fp64" else 96, (4, 5, 6, 7), 2)
        return dict(kind="solve", dim=2, nx=n[0], ny=n[1], nz=1, precision=prec)
    if kind == "solve3":
        prec = rng.choice(["mixed", "mixed", "fp64"])
        n = box(16, 128 if prec == "mixed" else 64, (4, 5, 6, 7), 3)
        return dict(kind="solve", dim=3, nx=n[0], ny=n[1], nz=n[2], precision=prec)
    if kind in ("grad", "loop"):
        n = box(16, 96 if kind == "grad" else 64, (4, 5), 3)
        c = dict(kind=kind, dim=3, nx=2 * n[0] - 1, ny=n[1], nz=n[2], precision="mixed")
        return c if kind == "grad" else dict(c, steps=rng.randint(1, 4))
    if kind == "refine2":
        return dict(kind="refine", dim=2, n=rng.choice([49, 57, 65, 81, 97, 113]), levels=rng.randint(1, 3),
                    count=rng.randint(3, 8), layout=rng.randint(0, 999), precision="fp64")
    if kind == "refine3":
        return dict(kind="refine", dim=3, n=rng.choice([25, 29, 33, 41, 49, 57]), levels=rng.randint(1, 2),
                    count=rng.randint(2, 6), layout=rng.randint(0, 999), precision="mixed")
    dim = rng.choice([2, 3, 3]) if kind == "residual" else 3
    n = box(12, 160 if dim == 3 else 1024, (5, 6, 7, 8, 9, 10, 11), dim)
    return dict(kind=kind, dim=dim, nx=n[0], ny=n[1], nz=n[2])


# ------------------------------------------------------------------ inputs

def _iso(E, nu):
    lam, mu = E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))
    return lam + 2 * mu, lam, mu


def _axes(dim, n, h, off):
    return [(torch.arange(n[a], dtype=F8, device=DEV) + off) * h if a < dim else torch.zeros(1, dtype=F8, device=DEV)
            for a in range(3)]


def _field(fn, dim, n, h, org=(0, 0, 0)):
    """fn(x, y, z) at the cell centres of a grid whose node (0, 0, 0) is global node org, packed."""
    nc = [n[a] - 1 if a < dim else 1 for a in range(3)]
    x, y, z = [_axes(dim, nc, h, 0.5 + (org[a] if a < dim else 0))[a] for a in range(3)]
    return fn(x[None, None, :], y[None, :, None], z[:, None, None]).expand(nc[2], nc[1], nc[0]).contiguous().reshape(-1)


def _step(d, w):
    return 0.5 * (1 + torch.tanh(d / w))


def _balls(r, count, rmin, rmax, gap, dim):
    out = []
    for _ in range(20000):
        if len(out) == count:
            break
        rad = r.uniform(rmin, rmax)
        c = [r.uniform(rad + gap, 1 - rad - gap) for _ in range(dim)]
        if all(math.dist(c, c2) >= rad + r2 + gap for c2, r2 in out):
            out.append((c, rad))
    return out


def _plate(r, h):
    cx, cy, rad = r.uniform(0.42, 0.58), r.uniform(0.42, 0.58), r.uniform(0.15, 0.25)
    return lambda x, y, z: _step(torch.sqrt((x - cx) ** 2 + (y - cy) ** 2) - rad, 2 * h)


def _damage(r, h, size):
    ells = [([r.uniform(0.2, 0.8) * s for s in size], [r.uniform(0.05, 0.2) * min(size) for _ in range(3)])
            for _ in range(3)]

    def fn(x, y, z):
        d = torch.zeros((), dtype=F8, device=DEV)
        for c, a in ells:
            rho = torch.sqrt(((x - c[0]) / a[0]) ** 2 + ((y - c[1]) / a[1]) ** 2 + ((z - c[2]) / a[2]) ** 2)
            d = torch.maximum(d, 0.5 * (1 - torch.tanh((rho - 1) * min(a) / (2 * h))))
        return 1 - d
    return fn


def _voids(balls, hf):
    def fn(x, y, z):
        v = torch.ones((), dtype=F8, device=DEV)
        for c, rad in balls:
            d2 = (x - c[0]) ** 2 + (y - c[1]) ** 2 + ((z - c[2]) ** 2 if len(c) == 3 else 0)
            v = v * _step(torch.sqrt(d2) - rad, 2 * hf)
        return v
    return fn


def _smooth(rho, n):
    v = rho.reshape(1, 1, n[2] - 1, n[1] - 1, n[0] - 1)
    k = torch.zeros(1, 1, 3, 3, 3, dtype=F8, device=DEV)
    for a in ((1, 1, 1), (0, 1, 1), (2, 1, 1), (1, 0, 1), (1, 2, 1), (1, 1, 0), (1, 1, 2)):
        k[(0, 0) + a] = 1
    ones = torch.nn.functional.conv3d(torch.ones_like(v), k, padding=1)
    for _ in range(3):
        v = torch.nn.functional.conv3d(v, k, padding=1) / ones
    return v.reshape(-1)


def _rand(case, seed, what, n):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 16 + what)
    return torch.rand(n, dtype=F8, device=DEV, generator=g)


def _tip_load(n, h, scale):
    x, y, z = _axes(3, n, h, 0.0)
    d2 = (x[None, None, :] - x[-1]) ** 2 + (y[None, :, None] - y[-1] / 2) ** 2 + (z[:, None, None] - z[-1] / 2) ** 2
    g = torch.exp(-d2 / (2 * (2 * h) ** 2))
    f = torch.zeros(3, *g.shape, dtype=F8, device=DEV)
    f[1] = -scale * g / (h ** 3 * g.sum())
    return f.reshape(-1)


def _stretch(dim):
    """Bottom clamped, top displaced by 0.01 along the last axis."""
    lo, hi = ("-y", "+y") if dim == 2 else ("-z", "+z")
    return [(lo, p, 0.0) for p in range(dim)] + [(hi, p, 0.01 if p == dim - 1 else 0.0) for p in range(dim)]


def _setup(case, seed):
    """Grid shape, spacing, moduli, boundary faces and options of a case."""
    dim = case["dim"]
    n = (case["n"],) * dim + (1,) * (3 - dim) if "n" in case else (case["nx"], case["ny"], case["nz"])
    kind = case["kind"]
    if kind in ("grad", "loop"):
        h, mod, bcs, om = 1.0 / (n[1] - 1), (_iso(1.0, 0.3) if kind == "grad" else _iso(1480.0, 0.22)), \
            [("-x", p, 0.0) for p in range(3)], 0.5
    elif kind == "refine" and dim == 3:
        h, mod, om = 1.0 / (n[0] - 1), _iso(1.0, 0.25), 0.5
        bcs = [(f, p, None) for f in ("-x", "+x", "-y", "+y", "-z", "+z") for p in range(3)]
    elif dim == 2:
        h, mod, bcs, om = 1.0 / (n[0] - 1), _iso(1.0, 0.3), _stretch(2), 2.0 / 3.0
    else:
        h, mod, bcs, om = 1.0 / (n[0] - 1), (1.0, 0.6, 0.5), _stretch(3), 2.0 / 3.0
    opts = dict(omega=om, tol=1e-10, max_cycles=500)
    if case.get("precision") == "mixed":
        opts.update(tol=1e-11, inner_cycles=12, inner_rtol=1e-6)
    if kind == "loop":
        opts.update(tol=1e-8)             # of each warm start's own residual
    if kind == "refine" and dim == 2:
        opts.update(smoother="gs", tol=1e-11)
    elif kind == "refine":
        opts.update(inner_cycles=6, inner_rtol=0.0, tol=1e-12)
    return n, h, mod, bcs, opts


def _grid(case, n, h, mod, bcs):
    g = sbm.Grid(case["dim"], n, h, precision=case.get("precision", "fp64"))
    g.set_moduli(sbm.SBM_CUBIC, mod)
    for face, comp, value in bcs:
        g.set_bc(face, comp, sbm.SBM_DIRICHLET if value is not None else sbm.SBM_DIRICHLET_FROM_U, value or 0.0)
    return g


def prepare(case, seed):
    dim, kind = case["dim"], case["kind"]
    n, h, mod, bcs, opts = _setup(case, seed)
    r = random.Random(seed)
    N, NC = n[0] * n[1] * n[2], (n[0] - 1) * (n[1] - 1) * (n[2] - 1 if dim == 3 else 1)
    g = _grid(case, n, h, mod, bcs)
    s = dict(kind=kind, grid=g, opts=opts, case=case, n=n, h=h, mod=mod, bcs=bcs)
    size = [(n[a] - 1) * h if a < dim else 0.0 for a in range(3)]
    if kind == "solve":
        s["psi"] = _field(_plate(r, h) if dim == 2 else _damage(r, h, size), dim, n, h)
        s["psi_min"] = case.get("psi_min", 1e-3 if dim == 2 else 1e-4)
        s["f"] = (2e-3 * (_rand(case, seed, 1, dim * N) - 0.5)) if dim == 2 else torch.zeros(dim * N, dtype=F8, device=DEV)
        s["u0"] = torch.zeros(dim * N, dtype=F8, device=DEV)
        g.set_psi(s["psi"], s["psi_min"])
        g.set_source(s["f"])
    elif kind == "grad":
        s["rho"] = _smooth(0.05 + 0.95 * _rand(case, seed, 1, NC), n)
        s["psi_min"], s["f"] = case.get("psi_min", 1e-3), _tip_load(n, h, 1.0)
        s["u0"] = torch.zeros(dim * N, dtype=F8, device=DEV)
        g.psi_min, g.q = s["psi_min"], 3.0
        g.set_source(s["f"])
        s["load"] = h ** 3 * s["f"]
    elif kind == "loop":
        s["eta"] = _smooth(0.05 + 0.95 * _rand(case, seed, 1, NC), n).clamp(0.0, 1.0)
        s["u0"] = torch.zeros(dim * N, dtype=F8, device=DEV)
        s["prm"] = dict(alpha=200.0, beta=0.01, zeta=0.01, lam=400.0, lam_rate=0.0,
                        V0=0.25 * size[0] * size[1] * size[2], mobility=1.0, dt=5e-5, psi_min=case.get("psi_min", 1e-4))
        g.set_source(_tip_load(n, h, 0.1))
    elif kind == "refine":
        _prepare_refined(case, s, r)
    elif kind == "residual":
        s["psi"] = _field(_plate(r, h) if dim == 2 else _damage(r, h, size), dim, n, h)
        s["psi_min"] = case.get("psi_min", 1e-4)
        g.set_psi(s["psi"], s["psi_min"])
        # a displacement field as a solve leaves it: smooth stretch, a wave and small noise
        ax = _axes(dim, n, h, 0.0)
        X, Y, Z = ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]
        ph = [r.uniform(0, 6.28) for _ in range(3)]
        top = Y if dim == 2 else Z
        u = [0.01 * (top if p == dim - 1 else 0.0 * top) + 1e-3 * torch.sin(3 * X + ph[p]) * torch.cos(2 * Y + p)
             * torch.cos(Z) for p in range(dim)]
        s["u"] = torch.stack([v.expand(n[2], n[1], n[0]) for v in u]).reshape(-1) \
            + 1e-6 * (_rand(case, seed, 2, dim * N) - 0.5)
        s["f"] = _rand(case, seed, 3, dim * N) - 0.5
    else:
        nv = 6 if dim == 3 else 3
        s["psi"] = _field(_plate(r, h) if dim == 2 else _damage(r, h, size), dim, n, h)
        s["eps0"] = 1e-2 * (_rand(case, seed, 1, nv * NC) - 0.5)
        s["b"] = _rand(case, seed, 2, dim * N) - 0.5
        s["t"] = _rand(case, seed, 3, dim * N) - 0.5
    torch.cuda.synchronize()
    return s


def _prepare_refined(case, s, r):
    dim, levels, g, n, h = case["dim"], case["levels"], s["grid"], s["n"], s["h"]
    rmax = 0.10 if dim == 2 else 0.09
    # the voids, and with them the patches, belong to the case; the body force to the seed
    balls = _balls(random.Random(case["layout"]), case["count"], 0.03 if dim == 2 else 0.05, rmax, 0.05, dim)
    wave = [[r.uniform(2, 9) for _ in range(dim)] + [r.uniform(0, 6.28)] for _ in range(dim)]

    def force(m, hm, org):
        x = _axes(dim, m, hm, 0.0)
        X = [(x[a] + (org[a] * hm if a < dim else 0.0)) for a in range(3)]
        at = [X[0][None, None, :], X[1][None, :, None], X[2][:, None, None]]
        return torch.stack([0.02 * torch.sin(sum(w[a] * at[a] for a in range(dim)) + w[-1]).expand(m[2], m[1], m[0])
                            for w in wave]).reshape(-1)

    hf = h / 2 ** levels
    fn = _voids(balls, hf)
    psi_min = case.get("psi_min", 1e-4 if dim == 2 else 1e-3)
    g.set_psi(_field(fn, dim, n, h), psi_min)
    g.set_source(force(n, h, (0, 0, 0)))
    s["us"] = [_start(case, n, h, (0, 0, 0), n)]
    for lev in range(1, levels + 1):
        hl = h / 2 ** lev
        for lo, hi, a in g.amr_regrid(lev, 0.1, 2):
            pn = tuple(hi[k] - lo[k] + 3 if k < dim else 1 for k in range(3))
            org = tuple(lo[k] - 1 if k < dim else 0 for k in range(3))
            N = tuple((n[k] - 1) * 2 ** lev + 1 if k < dim else 1 for k in range(3))
            g.amr_set_psi(a, _field(fn, dim, pn, hl, org), psi_min)
            g.amr_set_source(a, force(pn, hl, org))
            s["us"].append(_start(case, pn, hl, org, N))


def _start(case, n, h, org, N):
    """Zero inside, the boundary values on nodes of the domain's faces."""
    dim = case["dim"]
    u = torch.zeros(dim, n[2], n[1], n[0], dtype=F8, device=DEV)
    gi = [torch.arange(n[a], device=DEV) + org[a] for a in range(3)]
    idx = [gi[0][None, None, :], gi[1][None, :, None], gi[2][:, None, None]]
    if dim == 2:
        u[1][(idx[1] == N[1] - 1).expand(n[2], n[1], n[0])] = 0.01
        return u.reshape(-1)
    face = torch.zeros(n[2], n[1], n[0], dtype=torch.bool, device=DEV)
    for a in range(3):
        face |= (idx[a] <= 0) | (idx[a] >= N[a] - 1)
    for p in range(3):
        u[p] = torch.where(face, 0.01 * (idx[p] * h - 0.5), torch.zeros((), dtype=F8, device=DEV))
    return u.reshape(-1)


# ------------------------------------------------------------------ the call

def run(s):
    g, kind, opts = s["grid"], s["kind"], s["opts"]
    if kind == "solve":
        if s["case"]["dim"] == 2:
            g.set_source(s["f"])                     # a new load on the same geometry
        else:
            g.set_psi(s["psi"], s["psi_min"])        # a new damage field under the same load
        u = s["u0"].clone()
        g.solve(u, **opts)
        return u
    if kind == "grad":
        rho = s["rho"].detach().requires_grad_(True)
        u = sbm.SBMSolve.apply(rho, g, s["u0"], opts)
        (s["load"] * u).sum().backward()
        return {"u": u.detach(), "drho": rho.grad}
    if kind == "loop":
        eta, u = s["eta"].clone(), s["u0"].clone()
        res = g.topopt_run(eta, u, s["case"]["steps"], **s["prm"], **opts)
        return {"eta": eta, "u": u, "compliance": res["compliance"], "volume": res["volume"]}
    if kind == "refine":
        us = [u.clone() for u in s["us"]]
        g.amr_solve(us, **opts)
        return us
    if kind == "residual":
        r, norm = g.residual(g.finest, s["f"], s["u"])
        return {"r": r, "norm": norm}
    return g.source_terms(s["psi"], s["eps0"], s["b"], s["t"])


# ------------------------------------------------------------------ work and values

def work(case):
    dim = case["dim"]
    n = (case["n"],) * dim + (1,) * (3 - dim) if "n" in case else (case["nx"], case["ny"], case["nz"])
    N, NC = n[0] * n[1] * n[2], (n[0] - 1) * (n[1] - 1) * (n[2] - 1 if dim == 3 else 1)
    cell = 195.0 if dim == 3 else 38.0               # one operator application, per cell
    kind = case["kind"]
    if kind == "source":
        return {"bytes": 8.0 * (NC * (1 + (6 if dim == 3 else 3)) + 3 * dim * N), "flops": 120.0 * N}
    if kind == "residual":
        return {"bytes": 8.0 * (NC + 3 * dim * N), "flops": cell * NC}
    # psi and load in, solution out; a solve applies the operator at least once per V-cycle
    # stage of one cycle: two sweeps before, two after and the residual
    b, f = 8.0 * (NC + 2 * dim * N), 5.0 * cell * NC
    if kind == "grad":
        return {"bytes": 2 * b + 16.0 * NC, "flops": 2 * f}
    if kind == "loop":
        return {"bytes": case["steps"] * (b + 16.0 * NC), "flops": case["steps"] * f}
    return {"bytes": b, "flops": f}


def _unit_cell(dim, h, mod):
    """Cell matrix of the unit indicator by 2-point Gauss quadrature, rows corner * dim + component, over h^dim."""
    c11, c12, c44 = mod
    nc, pts = 1 << dim, [0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0)]
    K = torch.zeros(nc * dim, nc * dim, dtype=F8)
    for q in range(nc):
        xi = [pts[(q >> a) & 1] for a in range(dim)]
        dN = torch.zeros(nc, dim, dtype=F8)
        for c in range(nc):
            for a in range(dim):
                v = (1.0 if (c >> a) & 1 else -1.0) / h
                for m in range(dim):
                    if m != a:
                        v *= xi[m] if (c >> m) & 1 else 1.0 - xi[m]
                dN[c, a] = v
        nv = dim * (dim + 1) // 2
        B = torch.zeros(nv, nc * dim, dtype=F8)
        pairs = [(a, b) for a in range(dim) for b in range(a + 1, dim)]
        for c in range(nc):
            for p in range(dim):
                B[p, c * dim + p] = dN[c, p]
            for v, (a, b) in enumerate(pairs):
                B[dim + v, c * dim + a] = dN[c, b]
                B[dim + v, c * dim + b] = dN[c, a]
        C = torch.zeros(nv, nv, dtype=F8)
        C[:dim, :dim] = c12
        for p in range(nv):
            C[p, p] = c11 if p < dim else c44
        K += B.T @ C @ B / nc
    return K.to(DEV)


def _corner(v, c, dim):
    """The part of a node array (.., z, y, x) that holds corner c of every cell."""
    ix = [slice(1, None) if (c >> a) & 1 else slice(0, -1) for a in range(dim)]
    return v[(Ellipsis, ix[2] if dim == 3 else slice(None), ix[1], ix[0])]


def _apply(K, psi, u, dim):
    """K u by the definition, u (dim, z, y, x), psi (z, y, x)."""
    nc = 1 << dim
    U = torch.stack([_corner(u, c, dim)[p] for c in range(nc) for p in range(dim)])
    F = torch.tensordot(K, U, dims=([1], [0])) * psi
    out = torch.zeros_like(u)
    for c in range(nc):
        _corner(out, c, dim).add_(F[c * dim:(c + 1) * dim])
    return out


def _fixed(s, dim, n):
    m = torch.zeros(dim, n[2], n[1], n[0], dtype=torch.bool, device=DEV)
    val = torch.zeros(dim, n[2], n[1], n[0], dtype=F8, device=DEV)
    at = {"-x": (slice(None), slice(None), 0), "+x": (slice(None), slice(None), -1), "-y": (slice(None), 0),
          "+y": (slice(None), -1), "-z": (0,), "+z": (-1,)}
    for face, comp, value in s["bcs"]:
        m[comp][at[face]] = True
        val[comp][at[face]] = value
    return m, val


def exact(case, seed):
    kind, dim = case["kind"], case["dim"]
    if kind not in ("solve", "residual", "source"):
        return None
    if kind == "solve" and case["nx"] * case["ny"] * case["nz"] > 90000:
        return None
    s = prepare(case, seed)
    n, h = s["n"], s["h"]
    shape, cells = (dim, n[2], n[1], n[0]), (n[2] - 1 if dim == 3 else 1, n[1] - 1, n[0] - 1)
    psi = s["psi"].reshape(cells)
    if kind == "source":
        return _exact_source(s, psi, shape)
    K, psi, f = _unit_cell(dim, h, s["mod"]), torch.clamp(psi, min=s["psi_min"]), s["f"].reshape(shape)
    fixed, value = _fixed(s, dim, n)
    if kind == "residual":
        r = torch.where(fixed, 0.0, f - _apply(K, psi, s["u"].reshape(shape), dim))
        return {"r": r.reshape(-1), "norm": float(r.norm())}
    # conjugate gradients on the free values, scaled by the diagonal
    diag = torch.zeros(shape, dtype=F8, device=DEV)
    for c in range(1 << dim):
        for p in range(dim):
            _corner(diag, c, dim)[p].add_(psi * K[c * dim + p, c * dim + p])
    u = torch.where(fixed, value, 0.0)
    for _ in range(3):                               # restarts take the residual anew
        r = torch.where(fixed, 0.0, f - _apply(K, psi, u, dim))
        z = r / diag
        d, rz, x = z.clone(), (r * z).sum(), torch.zeros_like(u)
        stop, it = 1e-15 * float(rz), 0
        while it < 20000 and float(rz) > stop * 1e-13:
            for _ in range(50):
                q = torch.where(fixed, 0.0, _apply(K, psi, d, dim))
                al = rz / (d * q).sum()
                x += al * d
                r -= al * q
                z = r / diag
                new = (r * z).sum()
                d = z + (new / rz) * d
                rz = new
            it += 50
        u = u + x
    return u.reshape(-1)


def _exact_source(s, psi, shape):
    dim, h = s["case"]["dim"], s["h"]
    c11, c12, c44 = s["mod"]
    e = s["eps0"].reshape((-1,) + tuple(psi.shape))
    tr = e[:dim].sum(0)
    sig = [[None] * dim for _ in range(dim)]
    for a in range(dim):
        for b in range(dim):
            v = a if a == b else (2 if dim == 2 else 6 - a - b)
            sig[a][b] = psi * (c11 * e[a] + c12 * (tr - e[a]) if a == b else 2 * c44 * e[v])
    f = torch.zeros(shape, dtype=F8, device=DEV)
    share = torch.zeros(shape[1:], dtype=F8, device=DEV)
    for c in range(1 << dim):
        _corner(share, c, dim).add_(1.0 / (1 << dim))
        for p in range(dim):
            for q in range(dim):                     # the cell lies below its node along q where the corner's bit is set
                _corner(f, c, dim)[p].add_((1.0 if (c >> q) & 1 else -1.0) * sig[p][q] / (2 ** (dim - 1) * h))
    pad = torch.nn.functional.pad(psi[None, None], (1, 1, 1, 1) + ((1, 1) if dim == 3 else (0, 0)), mode="replicate")[0, 0]
    mean, grad = torch.zeros_like(share), [torch.zeros_like(share) for _ in range(dim)]
    for c in range(1 << dim):
        v = _corner(pad, c, dim)
        mean += v / (1 << dim)
        for a in range(dim):
            grad[a] += (v if (c >> a) & 1 else -v) / (2 ** (dim - 1) * h)
    gn = torch.sqrt(sum(v * v for v in grad))
    return (f - share * (mean * s["b"].reshape(shape) + gn * s["t"].reshape(shape))).reshape(-1)
