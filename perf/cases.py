"""Workloads that the performance of the solver is measured on.

Each case is a pass of work that a program using the solver does through its
public entry points: whole solves at the sizes of ``workloads.py`` (a small
FP64 one, the middle and benchmark sizes, the largest grid), several densities
of one geometry, a serving batch, one rank's modes, and single steps of the
path (transforms of a slab and of a whole grid, a multigrid solve, smoothing).

``listed()`` gives the fixed cases and ``draw(rng)`` more of the same kinds and
ranges.  Grid sides are powers of two (the solver takes no others), so the odd
sizes are the counts a caller chooses freely: rows of a slab, densities, modes.
Inputs are made on the GPU from the seed alone.
"""
import numpy as np
import torch

import paper_2606_17636_gb300 as ps

PI = np.pi

# Grid laws of the workloads: geometry, radial spacing, radial range and
# polar / vertical range; "half": n_tz = n_r / 2, else n_tz = n_r.
GRIDS = {
    # a body on the axis of a cylinder (workload 1)
    "cyl_axis": dict(geometry=ps.CYLINDRICAL, spacing=ps.UNIFORM, r=(0.0, 1.0), t=(-0.5, 0.5), half=False),
    # logarithmic sphere (workload 2) and the benchmark's wider one (workloads 3, 5)
    "sph_log": dict(geometry=ps.SPHERICAL, spacing=ps.LOG, r=(0.1, 10.0), t=(0.0, PI), half=True),
    "sph_wide": dict(geometry=ps.SPHERICAL, spacing=ps.LOG, r=(0.05, 20.0), t=(0.0, PI), half=True),
    # disc in a cylinder with an inner cavity (workload 4) and the serving mix's cylinder (workload 5)
    "cyl_disc": dict(geometry=ps.CYLINDRICAL, spacing=ps.UNIFORM, r=(0.2, 4.0), t=(-1.0, 1.0), half=True),
    "cyl_cavity": dict(geometry=ps.CYLINDRICAL, spacing=ps.UNIFORM, r=(4.0 / 33.0, 4.0), t=(-2.0, 2.0), half=True),
}


def listed():
    return [
        # a small problem in double precision on the axis grid: launches and latency
        dict(name="solve_cyl32_fp64", kind="solve", grid="cyl_axis", n=32, n_phi=32, precision="fp64", tol=1e-10, tuned=False),
        # an ordinary simulation grid, default options
        dict(name="solve_sph128", kind="solve", grid="sph_log", n=128, n_phi=128, precision="mixed", tol=1e-8, tuned=False),
        # the same grid for a user who wants FP64 throughout
        dict(name="solve_sph128_fp64", kind="solve", grid="sph_log", n=128, n_phi=128, precision="fp64", tol=1e-10, tuned=False),
        # the benchmark's grid and tolerance with the schedule its autotuner installs
        dict(name="solve_sph256_tuned", kind="solve", grid="sph_wide", n=256, n_phi=256, precision="mixed", tol=1e-8, tuned=True),
        # the largest grid of the workloads, default options
        dict(name="solve_cyl512", kind="solve", grid="cyl_disc", n=512, n_phi=512, precision="mixed", tol=1e-8, tuned=False),
        # several densities of one geometry in one call (an odd number of them)
        dict(name="multi5_sph128", kind="multi", grid="sph_log", n=128, n_phi=64, precision="mixed", tol=1e-8, count=5),
        # one rank's share of the modes of a mode-sharded solve, every eighth mode
        dict(name="modes_sph256", kind="modes", grid="sph_wide", n=256, n_phi=128, precision="mixed", tol=1e-8, first=0, step=8),
        # a serving batch: independent problems of uneven size in one captured graph
        dict(name="serve4", kind="serve", sizes="sph_wide:64,cyl_cavity:64,cyl_cavity:128,sph_wide:128", precision="mixed", tol=1e-8),
        # the forward transform of one rank's radial slab (an odd number of rows)
        dict(name="forward_slab37", kind="forward", grid="cyl_disc", n=512, n_phi=512, rows=37),
        # the inverse transform of the benchmark's grid
        dict(name="inverse_sph256", kind="inverse", grid="sph_wide", n=256, n_phi=256, rows=256),
        # the multigrid solve alone, zero boundary values
        dict(name="mg_cyl256", kind="mg", grid="cyl_cavity", n=256, n_phi=64, precision="mixed", tol=1e-8),
        # the smoother on the finest level, all modes: two cycles of Algorithm 1
        dict(name="smooth_sph256", kind="smooth", grid="sph_wide", n=256, n_phi=256, precision="mixed", cycles=2),
    ]


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "multi", "modes", "serve", "forward", "inverse", "mg", "smooth"])
    grid = rng.choice(["cyl_axis", "sph_log", "sph_wide", "cyl_cavity"])
    if grid == "cyl_axis":
        n = rng.choice([32, 64, 128])
    else:
        n = rng.choice([64, 128, 256])
    n_phi = 2 ** rng.randint(4, 8)
    case = dict(kind=kind, grid=grid, n=n, n_phi=n_phi)
    if kind in ("solve", "multi", "modes", "mg"):
        case["precision"] = rng.choice(["mixed", "mixed", "fp64"])
        case["tol"] = rng.choice([1e-8, 1e-9, 1e-10])
        if case["precision"] == "fp64" and n == 256:   # no more work than the largest listed solve
            case["n_phi"] = n_phi = min(n_phi, 64)
    if kind == "solve":
        case["tuned"] = rng.random() < 0.3
    elif kind == "multi":
        case["n"], case["n_phi"] = min(n, 128), min(n_phi, 64)
        case["count"] = rng.randint(2, 9)
    elif kind == "modes":
        case["step"] = rng.randint(2, 9)
        case["first"] = rng.randint(0, min(case["step"], n_phi // 2) - 1)
    elif kind == "serve":
        sizes = ["%s:%d" % (rng.choice(["sph_wide", "cyl_cavity"]), rng.choice([64, 64, 128])) for _ in range(rng.randint(2, 5))]
        case = dict(kind=kind, sizes=",".join(sizes), precision="mixed", tol=rng.choice([1e-8, 1e-9]))
    elif kind in ("forward", "inverse"):
        case["n_phi"] = 2 ** rng.randint(4, 9)
        case["rows"] = max(1, min(n, int(round(2 ** rng.uniform(2, 8)))))
    elif kind == "smooth":
        case["precision"] = rng.choice(["mixed", "mixed", "fp64"])
        case["cycles"] = rng.randint(1, 3)
    return case


# ---- inputs ------------------------------------------------------------------

def _spec(grid, n, n_phi):
    g = GRIDS[grid]
    return dict(geometry=g["geometry"], n_r=n, n_tz=n // 2 if g["half"] else n, n_phi=n_phi, spacing=g["spacing"],
                r_in=g["r"][0], r_out=g["r"][1], t_min=g["t"][0], t_max=g["t"][1])


def _faces(spec):
    k = np.arange(spec["n_r"] + 1) / spec["n_r"]
    lo, hi = spec["r_in"], spec["r_out"]
    fr = lo * (hi / lo) ** k if spec["spacing"] == ps.LOG else lo + k * (hi - lo)
    ft = spec["t_min"] + (spec["t_max"] - spec["t_min"]) * np.arange(spec["n_tz"] + 1) / spec["n_tz"]
    return fr, ft


def _density(spec, seed):
    """Four Gaussian clumps over a power-law background with 1 % noise,
    FP64 [n_r][n_tz][n_phi] on the GPU."""
    rng = np.random.default_rng(seed)
    fr, ft = _faces(spec)
    dev = "cuda"
    r = torch.tensor(0.5 * (fr[1:] + fr[:-1]), device=dev)[:, None, None]
    t = torch.tensor(0.5 * (ft[1:] + ft[:-1]), device=dev)[None, :, None]
    ph = (torch.arange(spec["n_phi"], device=dev, dtype=torch.float64) + 0.5)[None, None, :] * (2 * PI / spec["n_phi"])
    sph = spec["geometry"] == ps.SPHERICAL
    R = r * torch.sin(t) if sph else r
    z = r * torch.cos(t) if sph else t
    lo, hi = spec["r_in"], spec["r_out"]
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    rho = 0.05 / (1.0 + (R * R + z * z)) ** 1.5
    rho = rho * (1.0 + 0.01 * torch.randn((spec["n_r"], spec["n_tz"], spec["n_phi"]), generator=gen, device=dev, dtype=torch.float64))
    for _ in range(4):
        rc = np.exp(rng.uniform(np.log(max(0.3, 3 * lo)), np.log(min(5.0, hi / 2)))) if sph else rng.uniform(lo + 0.25 * (hi - lo), lo + 0.75 * (hi - lo))
        zc = rc * rng.uniform(-0.7, 0.7) if sph else rng.uniform(0.5 * spec["t_min"], 0.5 * spec["t_max"])
        Rc = np.sqrt(rc * rc - zc * zc) if sph else rc
        pc, w, amp = rng.uniform(0, 2 * PI), rng.uniform(0.1, 0.4) * min(1.0, hi / 4), rng.uniform(0.5, 2.0)
        rho += amp * torch.exp(-(R * R + Rc * Rc - 2 * R * Rc * torch.cos(ph - pc) + (z - zc) ** 2) / (2 * w * w))
    return rho.contiguous()


def _modes_of(rho):
    """4 pi times the normalised azimuthal modes of a density, [M][n_tz][n_r]."""
    f = torch.fft.rfft(rho, dim=2) * (4 * PI / rho.shape[2])
    return f.permute(2, 1, 0).contiguous()


def _random_planes(shape, dtype, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return torch.randn(shape, generator=gen, device="cuda", dtype=dtype)


def _precision(case):
    return ps.FP64 if case.get("precision") == "fp64" else ps.MIXED


def _solver(case, spec, **kw):
    s = ps.Solver.from_spec(spec, precision=_precision(case), **kw)
    if case.get("tuned"):
        # what the autotuner installs for the benchmark's grid
        s.set_schedule(2, 1, 2, lines_r=4, cols_t=16, nu_pre_fused=3, nu_post_fused=1)
    return s


def _mode_list(case):
    return list(range(case["first"], case["n_phi"] // 2 + 1, case["step"]))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        specs = [_spec(g, int(n), int(n)) for g, n in (x.split(":") for x in case["sizes"].split(","))]
        solvers = [_solver(case, sp) for sp in specs]
        rhos = [_density(sp, seed + 101 * k) for k, sp in enumerate(specs)]
        phis = [torch.empty_like(r) for r in rhos]
        return dict(kind=kind, batch=ps.Batch(solvers, rhos, phis, tol=case["tol"]), phis=phis)
    spec = _spec(case["grid"], case["n"], case["n_phi"])
    st = dict(kind=kind, tol=case.get("tol"))
    if kind == "multi":
        st["solver"] = _solver(case, spec, n_densities=case["count"])
        st["rho"] = torch.stack([_density(spec, seed + 101 * k) for k in range(case["count"])])
        st["phi"] = torch.empty_like(st["rho"])
        return st
    st["solver"] = _solver(case, spec)
    if kind == "solve":
        st["rho"] = _density(spec, seed)
        st["phi"] = torch.empty_like(st["rho"])
    elif kind == "modes":
        st["modes"] = _mode_list(case)
        st["f"] = _modes_of(_density(spec, seed))[st["modes"]].contiguous()
    elif kind == "forward":
        st["rho"] = _density(spec, seed)[: case["rows"]].contiguous()
    elif kind == "inverse":
        st["f"] = _modes_of(_density(spec, seed))[:, :, : case["rows"]].contiguous()
    elif kind == "mg":
        st["f"] = _modes_of(_density(spec, seed))
    elif kind == "smooth":
        shape = (spec["n_phi"] // 2 + 1, spec["n_tz"], spec["n_r"])
        dtype = torch.complex64 if _precision(case) == ps.MIXED else torch.complex128
        st["e"], st["f"] = _random_planes(shape, dtype, seed), _random_planes(shape, dtype, seed + 1)
        st["cycles"] = case["cycles"]
    return st


def run(st):
    kind = st["kind"]
    if kind == "serve":
        st["batch"].run()
        return st["phis"]
    s = st["solver"]
    if kind in ("solve", "multi"):
        s.solve(st["rho"], st["phi"], tol=st["tol"])
        return st["phi"]
    if kind == "modes":
        return s.solve_modes(st["modes"], st["f"], tol=st["tol"])[0]
    if kind == "forward":
        return s.stage_forward_rows(st["rho"])
    if kind == "inverse":
        return s.stage_inverse_rows(st["f"])
    if kind == "mg":
        return s.stage_mg_solve(st["f"], tol=st["tol"])[0]
    return s.stage_smooth(0, st["e"].clone(), st["f"], st["cycles"])


# ---- what a pass cannot do without ----------------------------------------------

def _boundary_points(spec):
    nr, nt = spec["n_r"], spec["n_tz"]
    n = nt * (2 if spec["r_in"] > 0 else 1)
    return n if spec["geometry"] == ps.SPHERICAL else n + 2 * nr


def _work_of(spec, count=1):
    """Whole solves of `count` densities: rho in, phi out, the table of the
    boundary convolution; the two transforms and the convolution."""
    cells = spec["n_r"] * spec["n_tz"] * spec["n_phi"]
    M, nb, n = spec["n_phi"] // 2 + 1, _boundary_points(spec), spec["n_phi"]
    return 16 * cells * count + 8 * M * nb * nb, count * (2 * 2.5 * cells * np.log2(n) + 4 * M * nb * nb)


def work(case):
    kind = case["kind"]
    if kind == "serve":
        parts = [_work_of(_spec(g, int(n), int(n))) for g, n in (x.split(":") for x in case["sizes"].split(","))]
        return dict(bytes=float(sum(p[0] for p in parts)), flops=float(sum(p[1] for p in parts)))
    spec = _spec(case["grid"], case["n"], case["n_phi"])
    plane, M, n = spec["n_r"] * spec["n_tz"], spec["n_phi"] // 2 + 1, spec["n_phi"]
    if kind in ("solve", "multi"):
        b, f = _work_of(spec, case.get("count", 1))
    elif kind == "modes":
        k, nb = len(_mode_list(case)), _boundary_points(spec)
        b, f = 32 * k * plane + 8 * k * nb * nb, k * (4 * nb * nb + 2 * 20 * plane)
    elif kind in ("forward", "inverse"):
        rows = case["rows"] * spec["n_tz"]
        b, f = rows * (8 * n + 16 * M), rows * 2.5 * n * np.log2(n)
    elif kind == "mg":
        b, f = 32 * M * plane, 20 * M * plane
    else:
        v = 8 if _precision(case) == ps.MIXED else 16
        b, f = 3 * v * M * plane, case["cycles"] * 2 * (16 + 16 * 2) * M * plane
    return dict(bytes=float(b), flops=float(f))


# ---- the values in 64 bits ---------------------------------------------------------

def _operator(spec):
    """The finite-volume operator's 1-D factors on the cells and one ghost per
    side: L_m u = aE (u_E - u) + aW (u_W - u) + P (aN (u_N - u) + aS (u_S - u))
    - s_m^2 Q T u, and the cell centres."""
    sph = spec["geometry"] == ps.SPHERICAL
    fr, ft = _faces(spec)
    if spec["spacing"] == ps.LOG:
        q = fr[1] / fr[0]
        fr = np.concatenate([[fr[0] / q], fr, [fr[-1] * q]])
    else:
        d = fr[1] - fr[0]
        fr = np.concatenate([[fr[0] - d], fr, [fr[-1] + d]])
    d = ft[1] - ft[0]
    ft = np.concatenate([[ft[0] - d], ft, [ft[-1] + d]])
    a, b = fr[:-1], fr[1:]
    c, e = ft[:-1], ft[1:]
    if sph:
        xr = 0.75 * (b ** 4 - a ** 4) / (b ** 3 - a ** 3)
        v = b ** 3 - a ** 3
        east, west, P = 3 * b * b / v, 3 * a * a / v, 1.5 / xr * (b * b - a * a) / v
        Q = P
        xt = (np.sin(e) - np.sin(c) + c * np.cos(c) - e * np.cos(e)) / (np.cos(c) - np.cos(e))
        vt = np.cos(c) - np.cos(e)
        face = np.sin(ft)
        face[np.abs(np.sin(ft)) < 1e-12] = 0.0
        north, south, T = face[1:] / vt, face[:-1] / vt, (e - c) / (np.sin(xt) * vt)
    else:
        xr = 2.0 / 3.0 * (b ** 3 - a ** 3) / (b * b - a * a)
        v = b * b - a * a
        east, west, P, Q = 2 * b / v, 2 * a / v, np.ones_like(a), 2.0 / (xr * (a + b))
        xt = 0.5 * (c + e)
        north, south, T = 1 / (e - c), 1 / (e - c), np.ones_like(c)
    mid = slice(1, -1)
    o = dict(aE=east[mid] / (xr[2:] - xr[1:-1]), aW=west[mid] / (xr[1:-1] - xr[:-2]), P=P[mid], Q=Q[mid],
             aN=north[mid] / (xt[2:] - xt[1:-1]), aS=south[mid] / (xt[1:-1] - xt[:-2]), T=T[mid], xr=xr, xt=xt)
    m = np.arange(spec["n_phi"] // 2 + 1)
    o["s2"] = (np.sin(m * PI / spec["n_phi"]) * spec["n_phi"] / PI) ** 2
    return o


def _direct(spec, f):
    """u with L_m u = f per mode (zero ghosts): eigenvectors along theta / z,
    a tridiagonal elimination along r for every eigenvalue.  f: [M][n_tz][n_r]."""
    o = _operator(spec)
    sph = spec["geometry"] == ps.SPHERICAL
    s2 = o["s2"]
    dt = -(o["aN"] + o["aS"])[None, :] - (s2[:, None] * o["T"][None, :] if sph else 0.0) + 0 * s2[:, None]
    off = np.sqrt(o["aN"][:-1] * o["aS"][1:])
    w = np.sqrt(np.concatenate([[1.0], np.cumprod(o["aN"][:-1] / o["aS"][1:])]))
    S = np.zeros((len(s2), len(w), len(w)))
    k = np.arange(len(w))
    S[:, k, k] = dt
    S[:, k[:-1], k[1:]] = S[:, k[1:], k[:-1]] = off
    lam, U = np.linalg.eigh(S)
    z = np.einsum("mjk,mji->mki", U, w[None, :, None] * f, optimize=True)
    dr = -(o["aE"] + o["aW"])[None, :] - (0.0 if sph else s2[:, None] * o["Q"][None, :]) + 0 * s2[:, None]
    n = len(o["aE"])
    c = np.zeros(z.shape)
    for i in range(n):
        den = dr[:, None, i] + lam * o["P"][i] - (o["aW"][i] * c[:, :, i - 1] if i else 0.0)
        c[:, :, i] = o["aE"][i] / den
        z[:, :, i] = (z[:, :, i] - (o["aW"][i] * z[:, :, i - 1] if i else 0.0)) / den
    for i in range(n - 2, -1, -1):
        z[:, :, i] -= c[:, :, i] * z[:, :, i + 1]
    return np.einsum("mjk,mki->mji", U, z, optimize=True) / w[None, :, None]


def _relaxed(spec, e, f, cycles, n_sor=2):
    """`cycles` smoothing cycles (Algorithm 1): zebra lines along r, then along
    theta / z, even lines first, each with n_sor even-odd SOR sweeps on a fixed
    source; omega per line from App. A.  e, f: complex128 [M][n_tz][n_r] on the
    GPU."""
    o = _operator(spec)
    x = {k: torch.tensor(v, device=e.device) for k, v in o.items()}
    s2 = x["s2"][:, None, None]
    P = x["P"][None, None, :]
    aE, aW = x["aE"][None, None, :], x["aW"][None, None, :]
    aN, aS = P * x["aN"][None, :, None], P * x["aS"][None, :, None]
    diag = -(aE + aW) - (aN + aS) - s2 * x["Q"][None, None, :] * x["T"][None, :, None]

    def omega(c, couple, dim):   # per line along dim: [M][n_tz][1] or [M][1][n_r]
        length = c[-1] - c[0]
        shape = [1, 1, 1]
        shape[dim] = -1
        wgt = (torch.sin(PI * (c[1:-1] - c[0]) / length) ** 2).reshape(shape)
        cos = torch.cos(PI * (c[1:-1] - c[:-2]) / length).reshape(shape)
        mu = ((couple * cos * wgt).sum(dim, keepdim=True) / (diag * wgt).sum(dim, keepdim=True)).abs().clamp(max=1.0)
        return 2.0 / (1.0 + torch.sqrt(1.0 - mu * mu))

    om = {2: omega(x["xr"], (aE + aW).expand_as(diag), 2), 1: omega(x["xt"], aN + aS, 1)}

    def shifted(u, dim, by):     # value of the next (by = +1) or previous cell along dim, zero beyond
        v = torch.zeros_like(u)
        n = u.shape[dim]
        v.narrow(dim, 0 if by > 0 else 1, n - 1).copy_(u.narrow(dim, 1 if by > 0 else 0, n - 1))
        return v

    cells = {d: (torch.arange(e.shape[d], device=e.device) % 2).reshape([-1 if k == d else 1 for k in range(3)]) for d in (1, 2)}
    for _ in range(cycles):
        for along, across in ((2, 1), (1, 2)):
            up, dn = (aE, aW) if along == 2 else (aN, aS)
            un, us = (aN, aS) if along == 2 else (aE, aW)
            for color in (0, 1):
                g = f - un * shifted(e, across, 1) - us * shifted(e, across, -1)
                for _ in range(n_sor):
                    for par in (0, 1):
                        new = (g - up * shifted(e, along, 1) - dn * shifted(e, along, -1)) / diag
                        on = (cells[across] == color) & (cells[along] == par)
                        e = torch.where(on, e + om[along] * (new - e), e)
    return e


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "multi", "modes", "serve"):
        # the boundary values of a whole solve come from discrete Green's
        # functions: one 2-D solve per boundary cell and mode, minutes in numpy
        return None
    spec = _spec(case["grid"], case["n"], case["n_phi"])
    if kind == "forward":
        return _modes_of(_density(spec, seed)[: case["rows"]])
    if kind == "inverse":
        f = _modes_of(_density(spec, seed))[:, :, : case["rows"]]
        return torch.fft.irfft(f.permute(2, 1, 0), n=case["n_phi"], dim=2, norm="forward").contiguous()
    if kind == "mg":
        return _direct(spec, _modes_of(_density(spec, seed)).cpu().numpy())
    shape = (spec["n_phi"] // 2 + 1, spec["n_tz"], spec["n_r"])
    dtype = torch.complex64 if _precision(case) == ps.MIXED else torch.complex128
    e, f = _random_planes(shape, dtype, seed), _random_planes(shape, dtype, seed + 1)
    return _relaxed(spec, e.to(torch.complex128), f.to(torch.complex128), case["cycles"])
