"""The work a user of the integrator has it do, case by case, and the exact
results it is held to.

Every case goes through the public binding (`paper_1110_0740_gb300.ctu`,
`amr_advance`).  Inputs are seeded and built on the GPU with the distributions
of `paper_1110_0740_gb300.workloads` (random-phase spectra, a pressure sphere,
a relativistic beam, an expanding spherical shock); `exact` recomputes a case
in float64 from the equations of Mignone et al. (2012) with torch alone.

Kinds of case
  mhd    one periodic patch: ghost fill and one CTU step with the next dt, as a
         time loop runs it (2-D turbulence or the 3-D blast)
  jet    the same loop for the relativistic beam
  level  one batched step of an AMR level's uneven patches, flux registers bound
  amr    a whole subcycled coarse step of a 3-level hierarchy (CUDA graph)
  tag    refinement tagging of a patch
"""
import math

import torch

from paper_1110_0740_gb300 import ctu

NG, NV = 4, 9
GAMMA, GAMMA_SR = 5.0 / 3.0, 4.0 / 3.0
ALPHA = 0.1  # psi damping
PREC = {"fp64": ctu.CTU_FP64, "mixed": ctu.CTU_MIXED}
RECON = {"mc": ctu.CTU_LINEAR_MC, "ppm": ctu.CTU_PPM}


def _mhd(nx, ny, nz, prec, recon, cfl, corner=0, kappa=0.0, nu=0.0, eta=0.0):
    return {"kind": "mhd", "nx": nx, "ny": ny, "nz": nz, "prec": prec, "recon": recon, "cfl": cfl,
            "corner": corner, "kappa": kappa, "nu": nu, "eta": eta}


def listed():
    return [
        # 2-D runs and quick tests: the smallest call, where launches and latency count
        dict(_mhd(128, 128, 1, "fp64", "mc", 0.4), name="turb-128x128-fp64"),
        # a small 3-D run, an ordinary test size
        dict(_mhd(48, 48, 48, "mixed", "ppm", 0.3), name="blast-48-mixed"),
        # a ragged box with the cheaper linear reconstruction
        dict(_mhd(200, 131, 67, "mixed", "mc", 0.3), name="blast-200x131x67-mixed-mc"),
        # production size: the headline benchmark's patch
        dict(_mhd(256, 256, 256, "mixed", "ppm", 0.3), name="blast-256-mixed"),
        # the float64 path, for reference solutions
        dict(_mhd(96, 96, 96, "fp64", "ppm", 0.3), name="blast-96-fp64"),
        # transverse fluxes from the normal predictor states
        dict(_mhd(128, 128, 128, "mixed", "ppm", 0.3, corner=1), name="blast-128-mixed-corner"),
        # conduction, viscosity and resistivity
        dict(_mhd(128, 128, 128, "mixed", "ppm", 0.3, kappa=1e-3, nu=1e-3, eta=1e-3), name="blast-128-mixed-parabolic"),
        # the relativistic beam at production size
        {"name": "jet-256-mixed", "kind": "jet", "nx": 256, "ny": 256, "nz": 256, "prec": "mixed"},
        # and its float64 path at a test size
        {"name": "jet-64-fp64", "kind": "jet", "nx": 64, "ny": 64, "nz": 64, "prec": "fp64"},
        # the finest level of the AMR benchmark: hundreds of uneven patches in one call
        {"name": "level-459-patches-mixed", "kind": "level", "prec": "mixed", "n8": 306, "n16": 82, "n32": 66, "n64": 5},
        # the AMR benchmark's whole coarse step
        {"name": "amr-base128-mixed", "kind": "amr", "prec": "mixed", "base": 128, "width": 0.0157, "layout": 0},
        # tagging before a regrid, sigma = B^2 / rho
        {"name": "tag-256-b2rho", "kind": "tag", "nx": 256, "ny": 256, "nz": 256, "sigma": 2, "chi_r": 0.1},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def box(lo, hi, most):
        while True:
            n = [log(lo, hi) for _ in range(3)]
            if n[0] * n[1] * n[2] <= most:
                return n

    kind = rng.choice(["turb", "blast", "blast", "blast", "jet", "jet", "level", "amr", "tag"])
    if kind == "turb":
        return _mhd(log(32, 1024), log(32, 1024), 1, rng.choice(["fp64", "mixed"]), rng.choice(["mc", "ppm"]), 0.4)
    if kind == "blast":
        prec = rng.choice(["fp64", "mixed", "mixed"])
        n = box(16, 256, 1 << 24 if prec == "mixed" else 1 << 20)
        option = rng.choice(["", "", "corner", "parabolic"])
        par = option == "parabolic"
        return _mhd(n[0], n[1], n[2], prec, rng.choice(["mc", "ppm", "ppm"]), 0.3, corner=int(option == "corner"),
                    kappa=1e-3 * par, nu=1e-3 * par, eta=1e-3 * par)
    if kind == "jet":
        prec = rng.choice(["fp64", "mixed", "mixed"])
        n = box(16, 256, 1 << 23 if prec == "mixed" else 1 << 20)
        return {"kind": "jet", "nx": n[0], "ny": n[1], "nz": n[2], "prec": prec}
    if kind == "level":
        return {"kind": "level", "prec": "mixed", "n8": log(8, 400), "n16": log(4, 120), "n32": log(1, 80),
                "n64": rng.randint(0, 6)}
    if kind == "amr":
        return {"kind": "amr", "prec": "mixed", "base": rng.choice([64, 128]), "width": round(rng.uniform(0.0145, 0.017), 4),
                "layout": rng.randint(0, 99)}
    n = box(16, 256, 1 << 24)
    return {"kind": "tag", "nx": n[0], "ny": n[1], "nz": n[2], "sigma": rng.randint(0, 3), "chi_r": 0.1}


# ------------------------------------------------------------------ inputs

def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed):
    g = torch.Generator(device=_dev())
    g.manual_seed(int(seed))
    return g


def _dims(case):
    n = [case["nx"], case["ny"], case["nz"]]
    return n, 2 if n[2] == 1 else 3, 1.0 / max(n)


def _spectrum(n, g, kmax, grad=False):
    """Real random-phase field on an (nz, ny, nx) periodic box, modes
    0 < |k| <= kmax, max |f| = 1 (with its gradient in box units)."""
    dev = _dev()
    f = [torch.fft.fftfreq(m, d=1.0 / m, device=dev, dtype=torch.float64) for m in (n[2], n[1])]
    kz, ky = f[0][:, None, None], f[1][None, :, None]
    kx = torch.fft.rfftfreq(n[0], d=1.0 / n[0], device=dev, dtype=torch.float64)[None, None, :]
    k2 = kx * kx + ky * ky + kz * kz
    ph = torch.rand(k2.shape, generator=g, device=dev, dtype=torch.float64) * (2.0 * math.pi)
    spec = torch.where((k2 > 0) & (k2 <= kmax * kmax), torch.polar(torch.ones_like(ph), ph), torch.zeros_like(ph))
    s = (n[2], n[1], n[0])
    out = torch.fft.irfftn(spec, s=s)
    top = out.abs().max()
    if not grad:
        return out / top
    return [torch.fft.irfftn(spec * (2j * math.pi * k), s=s) / top for k in (kx, ky, kz)]


def _cons(V, gamma=GAMMA):
    rho, vx, vy, vz, p, bx, by, bz, psi = V
    E = p / (gamma - 1.0) + 0.5 * rho * (vx * vx + vy * vy + vz * vz) + 0.5 * (bx * bx + by * by + bz * bz)
    return torch.stack([rho, rho * vx, rho * vy, rho * vz, E, bx, by, bz, psi])


def _into_ghosted(F, ndim):
    """The interior state F (9, nz, ny, nx) in a ghosted block of zeros."""
    n = list(F.shape[:0:-1])
    N = [n[d] + 2 * NG if d < ndim else n[d] for d in range(3)]
    U = torch.zeros((NV, N[2], N[1], N[0]), dtype=torch.float64, device=F.device)
    _inner(U, ndim).copy_(F)
    return U


def _inner(U, ndim):
    s = [slice(NG, -NG) if d < ndim else slice(None) for d in (2, 1, 0)]
    return U[(Ellipsis, *s)]


def _mhd_state(n, ndim, seed):
    """2-D turbulence (no pressure sphere) or the 3-D blast; psi as a few
    steps of cleaning leave it."""
    g = _gen(seed)
    kmax = min(4 if ndim == 2 else 8, max(1, min(n[:ndim]) // 8))
    rho = 1.0 + 0.2 * _spectrum(n, g, kmax)
    v = [0.5 * _spectrum(n, g, kmax) for _ in range(ndim)]
    psi = 0.02 * _spectrum(n, g, kmax)
    z = torch.zeros_like(rho)
    if ndim == 2:
        a = _spectrum(n, g, kmax, grad=True)
        p = 1.0 + 0.1 * _spectrum(n, g, kmax)
        return _cons([rho, v[0], v[1], z, p, 0.1 * a[1], -0.1 * a[0], z, psi])
    a = [_spectrum(n, g, kmax, grad=True) for _ in range(3)]
    b = [a[2][1] - a[1][2], a[0][2] - a[2][0], a[1][0] - a[0][1]]
    del a
    bmax = (b[0] ** 2 + b[1] ** 2 + b[2] ** 2).max().sqrt()
    c = torch.rand(3, generator=g, device=_dev(), dtype=torch.float64)
    h = 1.0 / max(n)
    r2 = 0.0
    for d in range(3):
        L = n[d] * h
        x = ((torch.arange(n[d], device=_dev(), dtype=torch.float64) + 0.5) * h - c[d] * L).abs()
        x = torch.minimum(x, L - x)
        r2 = r2 + (x * x).reshape([-1 if e == d else 1 for e in (2, 1, 0)])
    p = torch.where(r2 < 0.01, 100.0, 1.0).to(torch.float64)
    return _cons([rho, v[0], v[1], v[2], p, b[0] / bmax, b[1] / bmax, b[2] / bmax, psi])


def _jet_state(n, seed, lorentz=10.0, ratio=0.01, sigma=0.1, p0=0.01, radius=0.1, pert=0.01):
    """The relativistic magnetised beam along z."""
    g, dev, h = _gen(seed), _dev(), 1.0 / max(n)
    c = 0.3 + 0.4 * torch.rand(2, generator=g, device=dev, dtype=torch.float64)
    x = (torch.arange(n[0], device=dev, dtype=torch.float64) + 0.5) * h - c[0] * n[0] * h
    y = (torch.arange(n[1], device=dev, dtype=torch.float64) + 0.5) * h - c[1] * n[1] * h
    r = torch.sqrt(y[:, None] ** 2 + x[None, :] ** 2)
    prof = (0.5 * (1.0 - torch.tanh((r - radius) / (2.0 * h))))[None].expand(n[2], n[1], n[0])

    def noise():
        return pert * (2.0 * torch.rand(prof.shape, generator=g, device=dev, dtype=torch.float64) - 1.0)

    vz = torch.sqrt(1.0 - 1.0 / (1.0 + (lorentz - 1.0) * prof) ** 2)
    rho = (ratio + (1.0 - ratio) * prof) * (1.0 + noise())
    vx, vy = noise() * prof, noise() * prof
    vz = vz * torch.sqrt((1.0 - (vx ** 2 + vy ** 2) / vz.square().clamp_min(1e-300)).clamp_min(0.0))
    z = torch.zeros_like(rho)
    bz = math.sqrt(sigma * (1.0 + 4.0 * p0) * lorentz ** 2)
    return torch.stack(_sr_cons([rho, vx, vy, vz, z + p0, z, z, z + bz, z]))


def _shock_state(x, y, z, c, r0, field=(0.3, 0.4, 0.0)):
    """Expanding spherical shock: a dense shell moving outwards from hot gas."""
    dx, dy, dz = x - c[0], y - c[1], z - c[2]
    r = torch.sqrt(dx * dx + dy * dy + dz * dz) + 1e-12
    shell = torch.exp(-(((r - r0) / 0.02) ** 2))
    p = 1.0 + 9.5 * (1.0 - torch.tanh((r - r0) / 0.01))
    o = torch.zeros_like(r)
    vr = 1.5 * shell / r
    return _cons([1.0 + 3.0 * shell, vr * dx, vr * dy, vr * dz, p, *(o + b for b in field), o])


def _level_groups(case):
    return [(s, case["n%d" % s]) for s in (64, 32, 16, 8) if case["n%d" % s] > 0]


LEVEL_H = 1.0 / 512


def _level_state(case, seed):
    """Pool of the batch: patches of each size at random places on the shock
    shell, ghosts filled; and the shell's centre and radius."""
    g, dev = _gen(seed), _dev()
    c = 0.4 + 0.2 * torch.rand(3, generator=g, device=dev, dtype=torch.float64)
    r0 = 0.18 + 0.07 * torch.rand((), generator=g, device=dev, dtype=torch.float64)
    chunks = []
    for s, count in _level_groups(case):
        d = torch.randn((count, 3), generator=g, device=dev, dtype=torch.float64)
        o = c + r0 * d / d.norm(dim=1, keepdim=True)  # patch centres
        w = (torch.arange(s + 2 * NG, device=dev, dtype=torch.float64) - (s + 2 * NG - 1) / 2.0) * LEVEL_H
        x, y, z = (o[:, k].reshape(-1, 1, 1, 1) for k in range(3))
        U = _shock_state(x + w.reshape(1, 1, 1, -1), y + w.reshape(1, 1, -1, 1), z + w.reshape(1, -1, 1, 1), c, r0)
        chunks.append(U.reshape(NV, -1))
    return torch.cat(chunks, dim=1)


def _level_windows(case):
    """The six faces of every patch, weight +1, one register array."""
    win, i, off = [], 0, 0
    for s, count in _level_groups(case):
        for _ in range(count):
            for d in range(3):
                for plane in (0, s):
                    win.append((i, d, plane, 0, s, 0, s, 1.0, off))
                    off += NV * s * s
            i += 1
    return win, off


def _dt(M, cfl, h):
    """{dt, c_h} of the largest CFL rate M, cell width h."""
    dt = cfl / M
    return torch.stack([dt, cfl * h / dt])


# ------------------------------------------------------------------ the calls

def _config(case, ndim):
    if case["kind"] == "jet":
        return ctu.make_config(ndim=3, gamma=GAMMA_SR, recon=ctu.CTU_LINEAR_MC, precision=PREC[case["prec"]], cfl=0.3,
                               glm_alpha=ALPHA, physics=ctu.CTU_SRMHD, predictor=ctu.CTU_MUSCL_HANCOCK,
                               riemann=ctu.CTU_HLL)
    return ctu.make_config(ndim=ndim, recon=RECON[case["recon"]], precision=PREC[case["prec"]], cfl=case["cfl"],
                           glm_alpha=ALPHA, corner=case["corner"], kappa=case["kappa"], nu=case["nu"], eta=case["eta"])


def _patch_input(case, seed):
    """Interior state and {dt, c_h} of a one-patch case."""
    n, ndim, h = _dims(case)
    if case["kind"] == "jet":
        U = _jet_state(n, seed)
        return U, _dt(_sr_rate(list(U), h), 0.3, h)
    U = _mhd_state(n, ndim, seed)
    if case["kind"] == "tag":
        return U, None
    return U, _dt(_rate(_prim(U), ndim, h, case), case["cfl"], h)


def _amr_levels(case, seed):
    """The hierarchy around the shock: level l + 1 covers the cells of level l
    within case["width"] / (l + 1) of the shock radius with aligned cubes.
    case["layout"] places the shock, the seed turns the field through it and
    sets its strength."""
    import numpy as np
    from paper_1110_0740_gb300 import workloads as W
    rng = np.random.default_rng(case["layout"])
    base = case["base"]
    c, r0 = rng.uniform(0.4, 0.6, size=3), float(rng.uniform(0.18, 0.25))
    g = _gen(seed)
    d = torch.randn(3, generator=g, device=_dev(), dtype=torch.float64)
    field = (0.4 + 0.2 * torch.rand(1, generator=g, device=_dev(), dtype=torch.float64)) * d / d.norm()
    half = base // 2
    cubes, parents = [((k, j, i), half) for k in (0, half) for j in (0, half) for i in (0, half)], []
    levels = []
    for lev in (0, 1, 2):
        h = 1.0 / (base * 2 ** lev)
        if lev:
            plist, parents = [], []
            for pi, (o, s) in enumerate(cubes):
                x = [(np.arange(2 * s) + 2 * o[e] + 0.5) * h - c[2 - e] for e in range(3)]
                rr = np.sqrt(x[0][:, None, None] ** 2 + x[1][None, :, None] ** 2 + x[2][None, None, :] ** 2)
                for lo, size in W._cover(np.abs(rr - r0) < case["width"] / lev):
                    plist.append((tuple(int(lo[e] + 2 * o[e]) for e in range(3)), size))
                    parents.append(pi)
            above, cubes = cubes, plist
        patches, chunks, off = [], [], 0
        for o, s in cubes:
            z, y, x = ((torch.arange(-NG, s + NG, device=_dev(), dtype=torch.float64) + o[e] + 0.5) * h for e in range(3))
            U = _shock_state(x.reshape(1, 1, -1), y.reshape(1, -1, 1), z.reshape(-1, 1, 1), c, r0, field)
            chunks.append(U.reshape(NV, -1))
            patches.append(([s] * 3, [h] * 3, off, lev))
            off += (s + 2 * NG) ** 3
        foot = [(pi, tuple(o[e] // 2 - above[pi][0][e] for e in range(3)), s // 2) for (o, s), pi in zip(cubes, parents)]
        levels.append({"patches": patches, "pool": torch.cat(chunks, dim=1).cpu().numpy(), "origins": cubes,
                       "footprints": foot})
    return levels


def prepare(case, seed):
    if case["kind"] == "amr":
        return _prepare_amr(case, seed)
    dev = _dev()
    if case["kind"] == "level":
        U = _level_state(case, seed)
        specs, off = [], 0
        for s, count in _level_groups(case):
            for _ in range(count):
                specs.append(([s] * 3, [LEVEL_H] * 3, off, 2))
                off += (s + 2 * NG) ** 3
        win, nreg = _level_windows(case)
        reg = torch.zeros(nreg, dtype=torch.float64, device=dev)
        ctx = ctu.Ctx(ctu.make_config(ndim=3, precision=PREC[case["prec"]], cfl=0.3, glm_alpha=ALPHA))
        ctx.flux_registers(reg, win)
        return {"kind": "level", "ctx": ctx, "U": U, "Un": U.clone(), "stride": U.shape[1], "reg": reg,
                "patches": ctu.make_patches(specs), "dt": _level_dt(U)}
    n, ndim, h = _dims(case)
    F, dt = _patch_input(case, seed)
    U = _into_ghosted(F, ndim).reshape(NV, -1)
    del F
    s = {"kind": case["kind"], "U": U, "stride": U.shape[1], "patches": ctu.make_patches([(n, [h] * 3, 0)])}
    if case["kind"] == "tag":
        s.update(ctx=ctu.Ctx(ctu.make_config(ndim=ndim)), sigma=case["sigma"], chi_r=case["chi_r"],
                 tags=torch.zeros(U.shape[1], dtype=torch.uint8, device=dev),
                 count=torch.zeros(1, dtype=torch.int64, device=dev))
        s["ctx"].fill_periodic(U, U.shape[1], s["patches"])
    else:
        s.update(ctx=ctu.Ctx(_config(case, ndim)), Un=torch.zeros_like(U), dt=dt, dtn=torch.zeros_like(dt))
    return s


def _prepare_amr(case, seed):
    from paper_1110_0740_gb300.amr_advance import LevelAdvance
    levels = _amr_levels(case, seed)
    adv = LevelAdvance(levels, case["base"], precision=PREC[case["prec"]], cfl=0.3)
    dt0 = adv.local_dt()
    adv.set_dt(dt0, 0.3 / (case["base"] * dt0))
    snap = [a.clone() for a in adv.A]
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        adv.coarse_step(s)  # binds the patch lists and tables before the capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        for a, b in zip(adv.A, snap):  # the stored state the step starts from
            a.copy_(b)
        adv.coarse_step(s)
    return {"kind": "amr", "adv": adv, "graph": g, "snap": snap, "stream": s}


def run(s):
    k = s["kind"]
    if k in ("mhd", "jet"):
        s["ctx"].fill_periodic(s["U"], s["stride"], s["patches"])
        s["ctx"].step_next_dt(s["U"], s["Un"], s["stride"], s["patches"], s["dt"], s["dtn"])
        return {"U": s["Un"], "dt": s["dtn"]}
    if k == "level":
        s["reg"].zero_()
        s["ctx"].step(s["U"], s["Un"], s["stride"], s["patches"], s["dt"])
        return {"U": s["Un"], "reg": s["reg"]}
    if k == "amr":
        s["graph"].replay()
        return s["adv"].outputs()
    s["ctx"].tag(s["U"], s["stride"], s["patches"], s["sigma"], 0.01, s["chi_r"], s["tags"], s["count"])
    return {"tags": s["tags"], "count": s["count"]}


# Operations of one cell update (the counts of profiles/flops_per_cell.txt).
PRIM, RIEMANN, UPDATE, NEXT = 20.0, 386.1, 37.0, 86.0
PREDICT = {"mc": 1020.2, "ppm": 1240.5}
SR_CELL = 15837.1


def _flops_per_cell(ndim, recon, corner=0, par=False, nxt=True):
    sweep = PREDICT[recon] + RIEMANN + 134.0
    f = PRIM + ndim * (RIEMANN + sweep) + UPDATE + NEXT * nxt
    if corner:
        f += ndim * PREDICT[recon]
    if par:
        f += 2 * ndim * 126.0 + 200.0
    return f


def work(case):
    if case["kind"] == "amr":
        # cells of the covered shells (level l + 1: half-width w / (l + 1)); the cubes hold about 4.3 times the tagged half-shell
        b, w = case["base"], case["width"]
        shell = 4.0 * math.pi * 0.215 ** 2
        cells = [b ** 3, shell * 2.0 * w * 4.3 * (2 * b) ** 3, shell * w * 4.3 * (4 * b) ** 3]
        upd = cells[0] + 2 * cells[1] + 4 * cells[2]
        return {"bytes": 144.0 * upd, "flops": upd * _flops_per_cell(3, "ppm", nxt=False)}
    if case["kind"] == "level":
        g = _level_groups(case)
        ins, ghosted = sum(c * s ** 3 for s, c in g), sum(c * (s + 8) ** 3 for s, c in g)
        return {"bytes": 72.0 * (ins + ghosted) + 72.0 * sum(6 * c * s * s for s, c in g),
                "flops": ins * _flops_per_cell(3, "ppm", nxt=False)}
    n, ndim, _ = _dims(case)
    cells = n[0] * n[1] * n[2]
    if case["kind"] == "tag":
        ring = (n[0] + 2) * (n[1] + 2) * (n[2] + 2)
        return {"bytes": 8.0 * (1, 1, 4, 2)[case["sigma"]] * ring + cells, "flops": 60.0 * cells}
    # the interior in and out once: the ghosts of a periodic box are its own cells
    if case["kind"] == "jet":
        return {"bytes": 144.0 * cells, "flops": SR_CELL * cells}
    par = case["kappa"] > 0 or case["nu"] > 0 or case["eta"] > 0
    return {"bytes": 144.0 * cells, "flops": cells * _flops_per_cell(ndim, case["recon"], case["corner"], par)}


# ------------------------------------------------------------------ exact results
#
# Arrays carry the variable first and (batch,) z, y, x last; `_at` cuts the
# cells [lo, hi) of an array whose first cell has the coordinates `org`.

def _at(F, org, lo, hi):
    return F[..., lo[2] - org[2]:hi[2] - org[2], lo[1] - org[1]:hi[1] - org[1], lo[0] - org[0]:hi[0] - org[0]]


def _moved(v, d, k):
    return [x + (k if e == d else 0) for e, x in enumerate(v)]


# Components (rho, normal, t1, t2, E or p, B normal, B t1, B t2, psi) of a
# sweep along d, and the way back.
PERM = ([0, 1, 2, 3, 4, 5, 6, 7, 8], [0, 2, 1, 3, 4, 6, 5, 7, 8], [0, 3, 1, 2, 4, 7, 5, 6, 8])
BACK = [[p.index(q) for q in range(NV)] for p in PERM]


def _prim(U):
    rho, v = U[0], [U[k] / U[0] for k in (1, 2, 3)]
    p = (GAMMA - 1.0) * (U[4] - 0.5 * (U[1] * v[0] + U[2] * v[1] + U[3] * v[2])
                         - 0.5 * (U[5] * U[5] + U[6] * U[6] + U[7] * U[7]))
    return torch.stack([rho, *v, p, U[5], U[6], U[7], U[8]])


def _fast(V, bn, b1, b2):
    a2 = GAMMA * V[4] / V[0]
    n2, t2 = bn * bn / V[0], (b1 * b1 + b2 * b2) / V[0]
    t = n2 + t2
    return torch.sqrt(0.5 * (a2 + t + torch.sqrt((a2 - t) ** 2 + 4.0 * a2 * t2)))


def _rate(V, ndim, h, case):
    """Largest CFL rate, Eq. (Ca)."""
    m = 0.0
    for d in range(ndim):
        L = V[PERM[d]]
        s = (L[1].abs() + _fast(L, L[5], L[6], L[7])) / h
        m = s if d == 0 else torch.maximum(m, s)
    if case["kappa"] > 0 or case["nu"] > 0 or case["eta"] > 0:
        D = torch.clamp_min((GAMMA - 1.0) * case["kappa"] / V[0], max(4.0 / 3.0 * case["nu"], case["eta"]))
        m = m + ndim * 2.0 * D / (h * h)
    return m.max()


def _hlld(L, R, ch):
    """HLLD (Miyoshi & Kusano 2005) between local states, with the exact
    (B_n, psi) face solve."""
    Bn = 0.5 * (L[5] + R[5]) - 0.5 * (R[8] - L[8]) / ch
    psi = 0.5 * (L[8] + R[8]) - 0.5 * ch * (R[5] - L[5])

    def side(V):
        r, u, v, w, p, y, z = V[0], V[1], V[2], V[3], V[4], V[6], V[7]
        B2 = Bn * Bn + y * y + z * z
        pt = p + 0.5 * B2
        E = p / (GAMMA - 1.0) + 0.5 * r * (u * u + v * v + w * w) + 0.5 * B2
        vB = u * Bn + v * y + w * z
        U = [r, r * u, r * v, r * w, E, y, z]
        F = [r * u, r * u * u + pt - Bn * Bn, r * u * v - Bn * y, r * u * w - Bn * z,
             (E + pt) * u - Bn * vB, u * y - Bn * v, u * z - Bn * w]
        return {"r": r, "u": u, "v": v, "w": w, "y": y, "z": z, "pt": pt, "E": E, "vB": vB, "U": U, "F": F}

    l, r = side(L), side(R)
    c = torch.maximum(_fast(L, Bn, L[6], L[7]), _fast(R, Bn, R[6], R[7]))
    SL, SR = torch.minimum(L[1], R[1]) - c, torch.maximum(L[1], R[1]) + c
    sl, sr = SL - l["u"], SR - r["u"]
    den = sr * r["r"] - sl * l["r"]
    SM = (sr * r["r"] * r["u"] - sl * l["r"] * l["u"] - r["pt"] + l["pt"]) / den
    pts = (sr * r["r"] * l["pt"] - sl * l["r"] * r["pt"] + l["r"] * r["r"] * sr * sl * (r["u"] - l["u"])) / den

    def star(a, s, S):
        rs = a["r"] * s / (S - SM)
        D = a["r"] * s * (S - SM) - Bn * Bn
        weak = D.abs() <= 1e-12 * (a["r"] * s * s + Bn * Bn)
        D = torch.where(weak, 1.0, D)
        f = torch.where(weak, 1.0, (a["r"] * s * s - Bn * Bn) / D)
        g = torch.where(weak, 0.0, Bn * (SM - a["u"]) / D)
        v, w, y, z = a["v"] - a["y"] * g, a["w"] - a["z"] * g, a["y"] * f, a["z"] * f
        vB = SM * Bn + v * y + w * z
        E = (s * a["E"] - a["pt"] * a["u"] + pts * SM + Bn * (a["vB"] - vB)) / (S - SM)
        return {"r": rs, "v": v, "w": w, "y": y, "z": z, "vB": vB, "E": E, "q": torch.sqrt(rs),
                "U": [rs, rs * SM, rs * v, rs * w, E, y, z]}

    ls, rs = star(l, sl, SL), star(r, sr, SR)
    SLs, SRs = SM - Bn.abs() / ls["q"], SM + Bn.abs() / rs["q"]
    sB = torch.copysign(torch.ones_like(Bn), Bn)
    ql, qr = ls["q"], rs["q"]
    qs = ql + qr
    v = (ql * ls["v"] + qr * rs["v"] + (rs["y"] - ls["y"]) * sB) / qs
    w = (ql * ls["w"] + qr * rs["w"] + (rs["z"] - ls["z"]) * sB) / qs
    y = (ql * rs["y"] + qr * ls["y"] + ql * qr * (rs["v"] - ls["v"]) * sB) / qs
    z = (ql * rs["z"] + qr * ls["z"] + ql * qr * (rs["w"] - ls["w"]) * sB) / qs
    vB = SM * Bn + v * y + w * z
    left = SM >= 0
    dE = torch.where(left, -ql * (ls["vB"] - vB) * sB, qr * (rs["vB"] - vB) * sB)
    G = []
    for k in range(7):
        fl, fr = l["F"][k] + SL * (ls["U"][k] - l["U"][k]), r["F"][k] + SR * (rs["U"][k] - r["U"][k])
        rho = torch.where(left, ls["r"], rs["r"])
        us = torch.where(left, ls["U"][k], rs["U"][k])
        uss = (rho, rho * SM, rho * v, rho * w, us + dE, y, z)[k]
        f2 = torch.where(left, fl, fr) + torch.where(left, SLs, SRs) * (uss - us)
        f = torch.where(SLs >= 0, fl, torch.where(SRs <= 0, fr, f2))
        G.append(torch.where(SL >= 0, l["F"][k], torch.where(SR <= 0, r["F"][k], f)))
    return torch.stack([G[0], G[1], G[2], G[3], G[4], psi, G[5], G[6], ch * ch * Bn])


def _mc(a, b):
    m = torch.minimum(0.5 * (a + b).abs(), 2.0 * torch.minimum(a.abs(), b.abs()))
    return torch.where(a * b > 0, torch.copysign(m, a), 0.0)


def _edges(w, recon):
    """Values at the + and - interface from five cells."""
    s0 = _mc(w[2] - w[1], w[3] - w[2])
    if recon == "mc":
        return w[2] + 0.5 * s0, w[2] - 0.5 * s0
    sm, sp = _mc(w[1] - w[0], w[2] - w[1]), _mc(w[3] - w[2], w[4] - w[3])
    dp = 0.5 * (w[2] + w[3]) - (sp - s0) / 6.0 - w[2]
    dm = 0.5 * (w[2] + w[1]) + (sm - s0) / 6.0 - w[2]
    ext = dp * dm > 0
    np_ = torch.where(dp.abs() >= 2.0 * dm.abs(), -2.0 * dm, dp)
    nm_ = torch.where(dm.abs() >= 2.0 * dp.abs(), -2.0 * dp, dm)
    return w[2] + torch.where(ext, 0.0, np_), w[2] + torch.where(ext, 0.0, nm_)


def _predict(W, ch, dtdx, recon):
    """Characteristic normal predictor (Section 3.2) from the five local
    primitive states W: V at the + and - interface, no reference state."""
    V = W[2]
    rho, u, p, Bn, B1, B2 = V[0], V[1], V[4], V[5], V[6], V[7]
    a2 = GAMMA * p / rho
    n2, t2 = Bn * Bn / rho, (B1 * B1 + B2 * B2) / rho
    b2 = n2 + t2
    disc = torch.sqrt((a2 - b2) ** 2 + 4.0 * a2 * t2)
    cf2 = 0.5 * (a2 + b2 + disc)
    cs2 = a2 * n2 / cf2
    cf, cs, ca, a = torch.sqrt(cf2), torch.sqrt(cs2), torch.sqrt(n2), torch.sqrt(a2)
    big = 0.5 * ((a2 - b2).abs() + disc)  # the larger of the two weights (times disc)
    small = torch.where(big > 0, a2 * t2 / big.clamp_min(1e-300), 0.0)
    hot = a2 >= b2
    none = disc <= 0
    d1 = torch.where(none, 1.0, disc)
    af = torch.where(none, 1.0, torch.sqrt(torch.where(hot, big, small) / d1))
    as_ = torch.where(none, 0.0, torch.sqrt(torch.where(hot, small, big) / d1))
    bt = torch.sqrt(B1 * B1 + B2 * B2)
    has = t2 > 1e-24 * a2
    bt = torch.where(has, bt, 1.0)
    e1, e2 = (torch.where(has, B / bt, math.sqrt(0.5)) for B in (B1, B2))
    S = torch.copysign(torch.ones_like(Bn), Bn)
    sq = torch.sqrt(rho)
    # amplitudes w = L V (left vectors scaled by 2 a^2 or 2) and their speeds
    fields = {k: [] for k in ("f+", "f-", "s+", "s-", "a+", "a-", "e", "g+", "g-")}
    for X in W:
        pv, pb = e1 * X[2] + e2 * X[3], e1 * X[6] + e2 * X[7]
        q, r = e1 * X[3] - e2 * X[2], S * (e2 * X[6] - e1 * X[7]) / sq
        xf, yf = af * cf * X[1] - as_ * cs * S * pv, af * X[4] / rho + as_ * a * pb / sq
        xs, ys = as_ * cs * X[1] + af * cf * S * pv, as_ * X[4] / rho - af * a * pb / sq
        for k, v in (("f+", yf + xf), ("f-", yf - xf), ("s+", ys + xs), ("s-", ys - xs), ("a+", q + r), ("a-", q - r),
                     ("e", X[0] - X[4] / a2), ("g+", X[5] + X[8] / ch), ("g-", X[5] - X[8] / ch)):
            fields[k].append(v)
    speed = {"f+": u + cf, "f-": u - cf, "s+": u + cs, "s-": u - cs, "a+": u + ca, "a-": u - ca, "e": u, "g+": ch, "g-": -ch}
    plus, minus, jump = {}, {}, {}
    for k, w in fields.items():
        wp, wm = _edges(w, recon)
        nu = speed[k] * dtdx
        dw, d2 = wp - wm, wp - 2.0 * w[2] + wm
        plus[k] = wp - 0.5 * nu * (dw + d2 * (3.0 - 2.0 * nu))
        minus[k] = wm - 0.5 * nu * (dw - d2 * (3.0 + 2.0 * nu))
        jump[k] = dw
    dB, dps = 0.5 * (jump["g+"] + jump["g-"]), 0.5 * ch * (jump["g+"] - jump["g-"])
    vB = u * Bn + V[2] * B1 + V[3] * B2
    h = 0.5 * dtdx
    out = []
    for w in (plus, minus):
        fs, fd, ss, sd = w["f+"] + w["f-"], w["f+"] - w["f-"], w["s+"] + w["s-"], w["s+"] - w["s-"]
        al, ad = w["a+"] + w["a-"], w["a+"] - w["a-"]
        i2 = 0.5 / a2
        tv = (af * cf * sd - as_ * cs * fd) * S * i2
        tb = (as_ * fs - af * ss) * sq * a * i2
        out.append(torch.stack([
            rho * (af * fs + as_ * ss) * i2 + w["e"],
            (af * cf * fd + as_ * cs * sd) * i2 + h * Bn / rho * dB,
            tv * e1 - 0.5 * e2 * al + h * B1 / rho * dB,
            tv * e2 + 0.5 * e1 * al + h * B2 / rho * dB,
            0.5 * rho * (af * fs + as_ * ss) + h * (GAMMA - 1.0) * (Bn * dps - vB * dB),
            0.5 * (w["g+"] + w["g-"]),
            tb * e1 + 0.5 * S * sq * e2 * ad + h * V[2] * dB,
            tb * e2 - 0.5 * S * sq * e1 * ad + h * V[3] * dB,
            0.5 * ch * (w["g+"] - w["g-"])]))
    return out


def _parabolic(T, v, rho, B, org, lo, hi, ndim, h, case):
    """L_P = sum_d (Pi_+ - Pi_-) / dx_d on the cells [lo, hi) (momentum,
    energy, B) from cell fields (Section 3.1: two-point normal, averaged
    central transverse derivatives, coefficients at the mean state)."""
    out = 0.0
    for d in range(ndim):
        fl, fh = list(lo), list(hi)
        fl[d] -= 1  # faces: right of the cells [lo - 1, hi)

        def at(F, s=0, t=None, k=0):
            m = [0, 0, 0]
            m[d] += s
            if t is not None:
                m[t] += k
            return _at(F, org, [x + y for x, y in zip(fl, m)], [x + y for x, y in zip(fh, m)])

        def grad(F, t):
            if t == d:
                return (at(F, 1) - at(F)) / h
            if t >= ndim:
                return torch.zeros_like(at(F))
            return (at(F, 0, t, 1) - at(F, 0, t, -1) + at(F, 1, t, 1) - at(F, 1, t, -1)) / (4.0 * h)

        E = case["kappa"] * grad(T, d)
        r0, r1 = at(rho), at(rho, 1)
        g = [[grad(v[i], t) for i in range(3)] for t in range(3)]
        div = g[0][0] + g[1][1] + g[2][2]
        mom, mag = [], []
        for i in range(3):
            tau = 0.5 * (r0 + r1) * case["nu"] * (g[d][i] + g[i][d] - (2.0 / 3.0 * div if i == d else 0.0))
            E = E + (r0 * at(v[i]) + r1 * at(v[i], 1)) / (r0 + r1) * tau
            mom.append(tau)
        for i in range(3):
            f = case["eta"] * (grad(B[i], d) - grad(B[d], i))
            E = E + 0.5 * (at(B[i]) + at(B[i], 1)) * f
            mag.append(f)
        P = torch.stack([*mom, E, *mag])
        m = P.shape[-1 - d] - 1
        out = out + (P.narrow(-1 - d, 1, m) - P.narrow(-1 - d, 0, m)) / h
    return out


def _step(U, n, ndim, h, dt, ch, case, faces=False):
    """One CTU step of ghosted blocks U (9, ..., z, y, x): the interior of
    U^(n+1), and with `faces` the n + 1/2 fluxes of each direction."""
    act = [1 if d < ndim else 0 for d in range(3)]
    org = [-NG * a for a in act]
    ring = [-a for a in act], [n[d] + act[d] for d in range(3)]
    zero, top = [0, 0, 0], list(n)
    V = _prim(U)
    recon = case["recon"]
    par = case["kappa"] > 0 or case["nu"] > 0 or case["eta"] > 0

    def local(d, lo, hi, k):
        return _at(V, org, _moved(lo, d, k), _moved(hi, d, k))[PERM[d]]

    def diff(F, d):
        m = F.shape[-1 - d] - 1
        return (F.narrow(-1 - d, 0, m) - F.narrow(-1 - d, 1, m)) / h

    def predict(d, lo, hi):
        return [X[BACK[d]] for X in _predict([local(d, lo, hi, k) for k in range(-2, 3)], ch, dt / h, recon)]

    L1 = []
    for d in range(ndim):
        lo, hi = list(ring[0]), list(ring[1])
        lo[d] -= 1  # left cells of the ring's faces
        if case["corner"]:
            wide = _moved(hi, d, 1)
            P, M = predict(d, lo, wide)
            m = P.shape[-1 - d] - 1
            F = _hlld(P.narrow(-1 - d, 0, m)[PERM[d]], M.narrow(-1 - d, 1, m)[PERM[d]], ch)
        else:
            F = _hlld(local(d, lo, hi, 0), local(d, lo, hi, 1), ch)
        L1.append(diff(F[BACK[d]], d))
    lpn = lph = None
    if par:
        lpn = _parabolic(V[4] / V[0], V[1:4], V[0], V[5:8], org, *ring, ndim, h, case)
        H = _at(U, org, *ring) + 0.5 * dt * sum(L1)
        H[1:8] += 0.5 * dt * lpn
        H = _prim(H)
        lph = _parabolic(H[4] / H[0], H[1:4], H[0], H[5:8], ring[0], zero, top, ndim, h, case)
    total, flux = 0.0, []
    for d in range(ndim):
        lo, hi = _moved(zero, d, -1), _moved(top, d, 1)
        T = 0.0
        for e in range(ndim):
            if e != d:
                T = T + 0.5 * dt * _at(L1[e], ring[0], lo, hi)
        P, M = predict(d, lo, hi)
        states = []
        for X in (P, M):
            C = _cons(X) + T
            if par:
                C[1:8] += 0.5 * dt * _at(lpn, ring[0], lo, hi)
            states.append(_prim(C)[PERM[d]])
        m = P.shape[-1 - d] - 1
        F = _hlld(states[0].narrow(-1 - d, 0, m), states[1].narrow(-1 - d, 1, m), ch)[BACK[d]]
        total = total + diff(F, d)
        if faces:
            flux.append(F)
    if par:
        total[1:8] += lph
    W = _at(U, org, zero, top) + dt * total
    W[8] *= torch.exp(-ALPHA * ch * dt / h)
    return W, flux


# ---- relativistic MHD, ideal gas (Section 2.2)

def _sr_cons(V):
    rho, vx, vy, vz, p, bx, by, bz, psi = V
    v2 = vx * vx + vy * vy + vz * vz
    W = (rho + 4.0 * p) / (1.0 - v2)  # Gamma / (Gamma - 1) = 4
    B2, vB = bx * bx + by * by + bz * bz, vx * bx + vy * by + vz * bz
    D = rho / torch.sqrt(1.0 - v2)
    return [D, (W + B2) * vx - vB * bx, (W + B2) * vy - vB * by, (W + B2) * vz - vB * bz,
            W - p + 0.5 * (B2 + B2 * v2 - vB * vB) - D, bx, by, bz, psi]


def _sr_prim(U):
    """V(U): safeguarded Newton on W = w gamma^2."""
    D, tau = U[0], U[4] + U[0]
    m2 = U[1] * U[1] + U[2] * U[2] + U[3] * U[3]
    B2 = U[5] * U[5] + U[6] * U[6] + U[7] * U[7]
    S = U[1] * U[5] + U[2] * U[6] + U[3] * U[7]
    S2 = S * S

    def at(W):
        X = W + B2
        v2 = (m2 * W * W + S2 * (2.0 * W + B2)) / (W * W * X * X)
        dv = -2.0 / (X * X * X) * (m2 + S2 * (3.0 * W * W + 3.0 * W * B2 + B2 * B2) / (W * W * W))
        g = torch.sqrt((1.0 - v2).clamp_min(0.0))
        p = 0.25 * (W * (1.0 - v2) - D * g)
        dp = 0.25 * ((1.0 - v2) + dv * (0.5 * D / g - W))
        f = W - p + 0.5 * B2 * (1.0 + v2) - 0.5 * S2 / (W * W) - tau
        return v2, p, f, 1.0 - dp + 0.5 * B2 * dv + S2 / (W * W * W)

    lo, hi = torch.zeros_like(tau), 2.0 * tau
    W = tau.clone()
    for _ in range(60):
        v2, p, f, df = at(W)
        low = ~((v2 < 1.0) & (f > 0.0))
        lo, hi = torch.where(low, W, lo), torch.where(low, hi, W)
        N = W - f / df
        last, W = W, torch.where((N > lo) & (N < hi), N, 0.5 * (lo + hi))
        if bool(((W - last).abs() <= 1e-15 * W).all()):
            break
    v2, p, _, _ = at(W)
    v = [(U[k] + S / W * U[k + 4]) / (W + B2) for k in (1, 2, 3)]
    return [D * torch.sqrt(1.0 - v2), *v, p, U[5], U[6], U[7], U[8]]


def _sr_speeds(V):
    v2 = V[1] * V[1] + V[2] * V[2] + V[3] * V[3]
    vB = V[1] * V[5] + V[2] * V[6] + V[3] * V[7]
    w = V[0] + 4.0 * V[4]
    b2 = (V[5] * V[5] + V[6] * V[6] + V[7] * V[7]) * (1.0 - v2) + vB * vB
    cs, ca = GAMMA_SR * V[4] / w, b2 / (w + b2)
    a2 = cs + ca - cs * ca
    q = torch.sqrt((a2 * (1.0 - v2) * (1.0 - v2 * a2 - V[1] * V[1] * (1.0 - a2))).clamp_min(0.0))
    m = V[1] * (1.0 - a2)
    return (m - q) / (1.0 - v2 * a2), (m + q) / (1.0 - v2 * a2)


def _sr_flux(V, U, ch):
    x, y, z, bx, by, bz = V[1], V[2], V[3], V[5], V[6], V[7]
    W = (V[0] + 4.0 * V[4]) / (1.0 - x * x - y * y - z * z)
    ex, ey, ez = z * by - y * bz, x * bz - z * bx, y * bx - x * by
    pt = V[4] + 0.5 * (bx * bx + by * by + bz * bz + ex * ex + ey * ey + ez * ez)
    return [U[0] * x, W * x * x - bx * bx - ex * ex + pt, W * x * y - bx * by - ex * ey, W * x * z - bx * bz - ex * ez,
            U[1] - U[0] * x, V[8], x * by - bx * y, x * bz - bx * z, ch * ch * bx]


def _sr_hll(L, R, ch):
    Bn = 0.5 * (L[5] + R[5]) - 0.5 * (R[8] - L[8]) / ch
    psi = 0.5 * (L[8] + R[8]) - 0.5 * ch * (R[5] - L[5])
    L, R = ([Bn if q == 5 else X[q] for q in range(NV)] for X in (L, R))
    UL, UR = _sr_cons(L), _sr_cons(R)
    FL, FR = _sr_flux(L, UL, ch), _sr_flux(R, UR, ch)
    (a, b), (c, d) = _sr_speeds(L), _sr_speeds(R)
    SL, SR = torch.minimum(a, c), torch.maximum(b, d)
    F = []
    for q in range(NV):
        mid = (SR * FL[q] - SL * FR[q] + SL * SR * (UR[q] - UL[q])) / (SR - SL)
        F.append(torch.where(SL >= 0, FL[q], torch.where(SR <= 0, FR[q], mid)))
    F[5], F[8] = psi, ch * ch * Bn
    return torch.stack(F)


def _sr_rate(U, h):
    V = _sr_prim(U)
    m = 0.0
    for d in range(3):
        a, b = _sr_speeds([V[q] for q in PERM[d]])
        s = torch.maximum(a.abs(), b.abs()) / h
        m = s if d == 0 else torch.maximum(m, s)
    return m.max()


def _sr_step(U, n, h, dt, ch):
    """As _step: MUSCL-Hancock in primitive variables, HLL (Section 3.3)."""
    org, ring = [-NG] * 3, ([-1] * 3, [k + 1 for k in n])
    zero, top = [0, 0, 0], list(n)
    V = torch.stack(_sr_prim(U))

    def local(F, d, lo, hi, k):
        return _at(F, org, _moved(lo, d, k), _moved(hi, d, k))[PERM[d]]

    def diff(F, d):
        m = F.shape[-1 - d] - 1
        return (F.narrow(-1 - d, 0, m) - F.narrow(-1 - d, 1, m)) / h

    L1 = []
    for d in range(3):
        lo, hi = list(ring[0]), list(ring[1])
        lo[d] -= 1
        L1.append(diff(_sr_hll(local(V, d, lo, hi, 0), local(V, d, lo, hi, 1), ch)[BACK[d]], d))
    total = 0.0
    for d in range(3):
        lo, hi = _moved(zero, d, -1), _moved(top, d, 1)
        v0 = local(V, d, lo, hi, 0)
        dV = _mc(v0 - local(V, d, lo, hi, -1), local(V, d, lo, hi, 1) - v0)
        Vp, Vm = v0 + 0.5 * dV, v0 - 0.5 * dV
        Fp, Fm = (torch.stack(_sr_flux(X, _sr_cons(X), ch)) for X in (Vp, Vm))
        half = torch.stack(_sr_prim(local(U, d, lo, hi, 0) - 0.5 * dt / h * (Fp - Fm)))
        T = 0.0
        for e in range(3):
            if e != d:
                T = T + 0.5 * dt * _at(L1[e], ring[0], lo, hi)[PERM[d]]
        P, M = (torch.stack(_sr_prim(torch.stack(_sr_cons(half + s * dV)) + T)) for s in (0.5, -0.5))
        m = P.shape[-1 - d] - 1
        total = total + diff(_sr_hll(P.narrow(-1 - d, 0, m), M.narrow(-1 - d, 1, m), ch)[BACK[d]], d)
    W = _at(U, org, zero, top) + dt * total
    W[8] *= torch.exp(-ALPHA * ch * dt / h)
    return W


PLAIN = {"recon": "ppm", "corner": 0, "kappa": 0.0, "nu": 0.0, "eta": 0.0}


def _level_dt(U):
    return _dt(_rate(_prim(U), 3, LEVEL_H, PLAIN), 0.3, LEVEL_H)


def _wrap(U, ndim):
    """Periodic ghosts of a ghosted block whose interior is set."""
    for d in range(ndim):
        ax = U.dim() - 1 - d
        N = U.shape[ax]
        i = torch.arange(N, device=U.device)
        U = U.index_select(ax, (i - NG) % (N - 2 * NG) + NG)
    return U


def _exact_patch(case, seed):
    n, ndim, h = _dims(case)
    F, dtch = _patch_input(case, seed)
    dt, ch = dtch[0], dtch[1]
    out = _into_ghosted(torch.zeros_like(F), ndim)
    inner, U = _inner(out, ndim), _wrap(_into_ghosted(F, ndim), ndim)
    del F
    M = None
    # in slabs along z (along y in 2-D), each with its four ghost layers
    ax = ndim - 1
    thick = max(8, int(3e6 / max(1, math.prod(n) // n[ax])))
    for a in range(0, n[ax], thick):
        b = min(n[ax], a + thick)
        m = list(n)
        m[ax] = b - a
        slab = U.narrow(3 - ax, a, b - a + 2 * NG)
        if case["kind"] == "jet":
            W = _sr_step(slab, m, h, dt, ch)
            r = _sr_rate(list(W), h)
        else:
            W = _step(slab, m, ndim, h, dt, ch, case)[0]
            r = _rate(_prim(W), ndim, h, case)
        inner.narrow(3 - ax, a, b - a).copy_(W)
        M = r if M is None else torch.maximum(M, r)
    return {"U": out.reshape(NV, -1), "dt": _dt(M, 0.3 if case["kind"] == "jet" else case["cfl"], h)}


def _exact_level(case, seed):
    U = _level_state(case, seed)
    dtch = _level_dt(U)
    out = U.clone()
    _, nreg = _level_windows(case)
    reg = torch.zeros(nreg, dtype=torch.float64, device=U.device)
    cell = roff = 0
    for s, count in _level_groups(case):
        N = s + 2 * NG
        for a in range(0, count, max(1, int(3e6 / N ** 3))):
            k = min(count - a, max(1, int(3e6 / N ** 3)))
            lo = cell + a * N ** 3
            blk = U[:, lo:lo + k * N ** 3].reshape(NV, k, N, N, N)
            W, F = _step(blk, [s] * 3, 3, LEVEL_H, dtch[0], dtch[1], PLAIN, faces=True)
            dst = out[:, lo:lo + k * N ** 3].view(NV, k, N, N, N)
            _inner(dst, 3).copy_(W)
            # registers per patch: (direction, lower and upper plane, variable, face)
            r = reg[roff + a * 6 * NV * s * s:][:k * 6 * NV * s * s].view(k, 3, 2, NV, s, s)
            for d in range(3):
                for side, plane in ((0, 0), (1, s)):
                    r[:, d, side] = (F[d].select(-1 - d, plane) * (dtch[0] * LEVEL_H ** 2)).transpose(0, 1)
        cell += count * N ** 3
        roff += count * 6 * NV * s * s
    return {"U": out, "reg": reg}


def exact(case, seed):
    """The outputs of `run` in float64 by torch alone.  None for tagging (its
    outputs are whole numbers) and for the AMR coarse step: level by level,
    with the ghost shells of some hundred patches filled box by box between
    the substeps, it would take longer than the 20 seconds such a check may."""
    if case["kind"] in ("mhd", "jet"):
        return _exact_patch(case, seed)
    return _exact_level(case, seed) if case["kind"] == "level" else None
