"""The work that a user of the two-body particle-in-cell library has it do, as
cases that can be timed and compared.

Kinds of pass (``case["kind"]``):

  steps    a running simulation advanced by ``steps`` leapfrog steps, then its
           fields read to device tensors: what a production run does between
           two diagnostics.  The field already fills the medium, as it does
           for most of such a run.
  lockin   the same one step at a time, with E_z read after every step: the
           refraction benchmark's lock-in accumulation.
  run      a whole short run of a parameter scan: the context reset, the
           frequencies set, the particles loaded from host arrays, ``steps``
           steps from zero fields under the antenna, the probe, the fields and
           the particles read.
  upload   a run's beginning, end to end: reset, particles loaded from pinned
           host arrays, one step at a time with E_y read asynchronously.
  adjoint  one iteration of an optimisation: probe = PICProbe.apply(omega_b,
           sites, problem), a squared mismatch against a target, backward.

Media (``case["medium"]``):

  neutral   neutral ions, ppc per cell (Sec. 3.1), cold or thermal
  refract   ions of charge +1 and free electrons at the same regular positions
  bragg     a 40 x 40 lattice of neutral ions, one wavelength apart
  crystal   a lattice of +30 ions (period 0.6 wavelengths) in free electrons

Units: c = 1, omega0 = 1, the wavelength is 2 pi.
"""
import math

import numpy as np
import torch

from paper_2208_08038_gb300 import binding as B
from paper_2208_08038_gb300.adjoint import PICProbe, SiteProblem

WAVE = 2.0 * math.pi
M_ION = 197.0 * 1836.15267          # gold atom, electron masses
R_E = 2.8179403262e-15              # classical electron radius [m]
TILE = {1: (16,), 2: (16, 16), 3: (8, 8, 8)}
RES = {1: 64, 2: 32, 3: 16}         # cells per wavelength of the configurations
LAMBDA_M = {"neutral": 12.4e-9, "refract": 56e-9, "bragg": 0.26e-9, "crystal": 0.26e-9}
EVERYTHING = 10_000_000             # particles beyond which no 64-bit result is computed


def _case(name, kind, medium, n, steps, **more):
    n = tuple(n) + (1,) * (3 - len(n))
    d = 3 if n[2] > 1 else (2 if n[1] > 1 else 1)
    c = {"name": name, "kind": kind, "medium": medium, "dims": d, "nx": n[0], "ny": n[1], "nz": n[2], "steps": steps,
         "ppc": 8, "a0": 1e-3, "sigma": 0.0, "margin": 4, "atomic": False, "res": RES[d], "params": 1, "ckpt": 20}
    c.update(more)
    return c


def listed():
    return [
        # the smallest grid and slab a scan uses: latency and launches are all there is
        _case("scan_1d", "run", "refract", (1024,), 500, ppc=2, margin=64, a0=1e-5),
        # the 1D propagation configuration: 2048 cells, a 16-wavelength slab of 16 ions per cell
        _case("medium_1d", "steps", "neutral", (2048,), 50, ppc=16, margin=512),
        # oblique refraction with a field read after every step
        _case("lockin_2d", "lockin", "refract", (192, 160), 16, ppc=1, margin=48, a0=1e-5, res=16),
        # the Bragg crystal: a large grid with few ions, open on both axes
        _case("bragg_2d", "steps", "bragg", (2048, 2048), 10),
        # the partially ionised crystal: free electrons carry the work, a strong field
        _case("crystal_2d", "steps", "crystal", (2048, 1024), 10, ppc=4, margin=512, a0=0.3, sigma=4.4e-3),
        # 3D medium, small: half a million ions, less than one tile per block
        _case("medium_3d_small", "steps", "neutral", (64, 32, 32), 10, sigma=1e-3, margin=0),
        # 3D medium, middle
        _case("medium_3d", "steps", "neutral", (256, 128, 128), 4, sigma=1e-3),
        # the FP32-atomic deposit, which a user picks for speed over bit-exact reruns
        _case("medium_3d_atomic", "steps", "neutral", (128, 64, 64), 5, sigma=1e-3, margin=16, atomic=True),
        # the 3D configuration itself: 264 million ions
        _case("medium_3d_full", "steps", "neutral", (512, 256, 256), 2, sigma=1e-3),
        # the beginning of a 3D run end to end, ahead of the field in most tiles
        _case("upload_3d", "upload", "neutral", (128, 64, 64), 12, sigma=1e-3),
        # gradients with respect to a few frequencies and sites on the 1D grid
        _case("adjoint_1d", "adjoint", "neutral", (2048,), 300, ppc=2, margin=64, params=8),
        # the adjoint configuration: 1024 x 1024 cells, 1024 frequencies, 4096 sites, 400 steps
        _case("adjoint_2d", "adjoint", "neutral", (1024, 1024), 400, ppc=8, params=1024),
    ]


def draw(rng):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    def cells(lo, hi, tile):
        return tile * max(1, round(log(lo, hi) / tile))

    what = rng.choice(("steps1", "run", "lockin", "bragg", "crystal", "steps2", "steps3", "steps3", "steps3", "upload",
                       "adjoint1", "adjoint2"))
    a0 = log(1e-3, 1e-2)
    if what == "steps1":
        nx = cells(512, 65536, 16)
        return _case("", "steps", "neutral", (nx,), rng.randint(10, 100), ppc=rng.randint(1, 24), margin=nx // rng.randint(3, 8),
                     a0=a0, atomic=rng.random() < 0.25)
    if what == "run":
        return _case("", "run", "refract", (cells(512, 4096, 16),), rng.randint(200, 600), ppc=rng.randint(1, 4), margin=64,
                     a0=1e-5)
    if what == "lockin":
        return _case("", "lockin", "refract", (cells(128, 512, 16), cells(64, 512, 16)), rng.randint(4, 24), ppc=1, margin=48,
                     a0=1e-5, res=16)
    if what == "bragg":
        return _case("", "steps", "bragg", (cells(512, 3072, 16), cells(512, 3072, 16)), rng.randint(2, 12), a0=a0)
    if what == "crystal":
        nx = cells(768, 3072, 16)
        return _case("", "steps", "crystal", (nx, cells(128, 1536, 16)), rng.randint(2, 10), ppc=rng.randint(1, 6),
                     margin=nx // 4, a0=rng.uniform(0.1, 0.4), sigma=4.4e-3)
    if what == "steps2":
        nx = cells(96, 1536, 16)
        return _case("", "steps", "neutral", (nx, cells(64, 1024, 16)), rng.randint(2, 20), ppc=rng.randint(1, 10),
                     margin=nx // 8, a0=a0, atomic=rng.random() < 0.25)
    if what == "steps3":
        nx = cells(32, 320, 8)
        return _case("", "steps", "neutral", (nx, cells(24, 144, 8), cells(24, 144, 8)), rng.randint(1, 8),
                     ppc=rng.randint(1, 12), sigma=1e-3, margin=0 if nx < 96 else nx // 6, a0=a0, atomic=rng.random() < 0.3)
    if what == "upload":
        return _case("", "upload", "neutral", (cells(48, 160, 8), cells(32, 80, 8), cells(32, 80, 8)), rng.randint(4, 12),
                     ppc=rng.randint(1, 8), sigma=1e-3, a0=a0)
    if what == "adjoint1":
        nx = cells(1024, 4096, 16)
        return _case("", "adjoint", "neutral", (nx,), rng.randint(250, 400), ppc=rng.randint(1, 8), margin=64,
                     params=rng.randint(2, 32), ckpt=rng.randint(5, 40))
    ny = cells(32, 768, 16)
    return _case("", "adjoint", "neutral", (cells(256, 768, 16), ny), rng.randint(300, 400), ppc=rng.randint(1, 8), params=ny,
                 ckpt=rng.randint(5, 25))


# ---------------------------------------------------------------------------
# the problem of a case: grid, species, laser, initial fields; FP64 arrays on the device

def _problem(case, seed):
    d, kind, medium = case["dims"], case["kind"], case["medium"]
    n = (case["nx"], case["ny"], case["nz"])
    dx = WAVE / case["res"]
    dev = "cuda"
    g = torch.Generator(device=dev)
    g.manual_seed(1009 * int(seed) + 7)

    def uniform(*shape):
        return torch.rand(*shape, generator=g, device=dev, dtype=torch.float64)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device=dev, dtype=torch.float64)

    def grid(axes):  # cell corners, x fastest
        m = torch.meshgrid(*[torch.as_tensor(a, dtype=torch.float64, device=dev) for a in reversed(axes)], indexing="ij")
        return torch.stack([x.reshape(-1) for x in reversed(m)], 1)

    margin = case["margin"]
    # the 3D box without a margin is periodic everywhere (a piece of the bulk, without the antenna)
    open_x = 0 if d == 3 and margin == 0 else 1
    p = {"d": d, "n": n, "dx": dx, "dt": 0.95 * dx / math.sqrt(d), "bc": (open_x, 1 if medium == "bragg" else 0, 0), "species": []}
    two = {"kind": "two", "mc": M_ION, "lambda_m": LAMBDA_M[medium], "pidx": None}
    lo, hi = margin, n[0] - margin
    comp, theta, waist, xa = 1, 0.0, 0.0, 2 if d == 3 else 8
    if medium == "neutral":
        density = {1: 0.01, 2: 0.01, 3: 0.02}[d]
        ppc = case["ppc"]
        omega = np.array([3.0])
        if kind == "adjoint":  # the slab of the adjoint configuration, its ions grouped on lattice sites
            density, wide = (0.05, 16) if d == 1 else (density, 16)
            comp, lo = 2, (lo if d == 1 else 64)
            hi = lo + 64
            sx = (hi - lo) // wide
            sites = grid([np.arange(sx) * wide + lo + 0.5 * wide] + ([np.arange(n[1]) + 0.5] if d == 2 else [])) * dx
            ns, per = len(sites), ppc * wide
            off = (uniform(ns * per, d) - 0.5) * torch.tensor([wide, 1.0][:d], device=dev, dtype=torch.float64) * dx
            site = torch.arange(ns, device=dev).repeat_interleave(per)
            # FP32 parameters, as an optimiser holds them
            sites = sites.float().double()
            omega = (2.5 + uniform(case["params"])).float().double().cpu().numpy()
            if d == 2:
                two["pidx"] = (site // sx) % case["params"]
            else:
                two["pidx"] = site * case["params"] // ns
            p.update(sites=sites, off=off, site=site, probe=[128 + 64 + n[0] * j for j in range(n[1])] if d == 2 else [hi + 64])
            x = sites[site] + off
            u = torch.zeros(len(x), 3, device=dev, dtype=torch.float64)
        else:
            total = ppc * (hi - lo) * n[1] * n[2]
            if total > EVERYTHING:
                x = u = None  # generated by the library on the device
                p["fill"] = ((lo, 0, 0)[:d], (hi, n[1], n[2])[:d], ppc, int(seed), case["sigma"])
            else:
                cell = grid([np.arange(lo, hi), np.arange(n[1]), np.arange(n[2])][:d])
                x = (cell.repeat_interleave(ppc, 0) + uniform(total, d)) * dx
                u = case["sigma"] * normal(total, 3) if case["sigma"] > 0 else torch.zeros(total, 3, device=dev, dtype=torch.float64)
            waist = 6 * WAVE if d == 3 else 0.0
        p["species"].append({**two, "Zb": 1.0, "qc": 0.0, "w": density / ppc, "omega": omega, "x": x, "u": u})
    elif medium == "refract":
        ppc = case["ppc"]
        density = {1: 8.14e-3, 2: 0.166}[d]
        Zb = {1: 78.0, 2: 20.0}[d]
        hi = lo + n[0] // 4 if d == 1 else n[0]
        axes = [(np.arange(ppc * lo, ppc * hi) + 0.5) / ppc] + ([np.arange(n[1]) + 0.5] if d == 2 else [])
        x = grid(axes) * dx
        u = torch.zeros(len(x), 3, device=dev, dtype=torch.float64)
        omega = float((2.0 if d == 2 else 1.5) + 0.5 * uniform(1).item())
        p["species"].append({**two, "Zb": Zb, "qc": 1.0, "w": density / ppc, "omega": np.array([omega]), "x": x, "u": u,
                             "lambda_m": 12.4e-9 if d == 1 else 56e-9})
        p["species"].append({"kind": "free", "q": -1.0, "m": 1.0, "w": density / ppc, "x": x.clone(), "u": u.clone()})
        if d == 2:
            comp, theta, waist = 2, math.radians(30.0), 2 * WAVE
    elif medium == "bragg":
        ns = [min(40, (m - 64) // case["res"]) for m in n[:2]]
        mid = [0.5 * m * dx for m in n[:2]]
        s = grid([np.arange(k) + 0.5 for k in ns]) * WAVE
        s = s + torch.tensor([mid[a] - 0.5 * ns[a] * WAVE for a in range(2)], device=dev, dtype=torch.float64)
        x = s.repeat_interleave(4, 0)
        x = x + 0.01 * WAVE * normal(len(x), 2)
        p["species"].append({**two, "Zb": 1.0, "qc": 0.0, "w": 0.01 * case["res"] ** 2 / 4, "omega": np.array([4.0]), "x": x,
                             "u": torch.zeros(len(x), 3, device=dev, dtype=torch.float64)})
        theta, waist = math.radians(30.0), 8 * WAVE
    else:
        period = 0.6 * WAVE
        nsx, nsy = int((hi - lo) * dx / period), int(n[1] * dx / period)
        s = grid([lo * dx + (np.arange(nsx) + 0.5) * period, (np.arange(nsy) + 0.5) * period])
        x = s.repeat_interleave(4, 0)
        p["species"].append({**two, "Zb": 49.0, "qc": 30.0, "w": 0.1 / 30 * (period / dx) ** 2 / 4, "omega": np.array([4.0]),
                             "x": x, "u": torch.zeros(len(x), 3, device=dev, dtype=torch.float64)})
        cell = grid([np.arange(lo, hi), np.arange(n[1])]).repeat_interleave(case["ppc"], 0)
        p["species"].append({"kind": "free", "q": -1.0, "m": 1.0, "w": 0.1 / case["ppc"], "x": (cell + uniform(len(cell), 2)) * dx,
                             "u": case["sigma"] * normal(len(cell), 3)})
    yc, zc = 0.5 * n[1] * dx, 0.5 * n[2] * dx
    phase = 0.3 * int(seed) % WAVE
    p["laser"] = {"comp": comp, "a0": case["a0"], "theta": theta, "waist": waist, "fwhm": 0.0, "t0": 0.0, "ramp": 2 * WAVE,
                  "phase": phase, "ia": xa, "yc": yc - (0.5 * n[0] - xa) * dx * math.tan(theta), "zc": zc}
    if kind == "run":
        p["laser"].update(fwhm=2 * WAVE, t0=3 * WAVE)
        p["probe"] = [lo - 16]  # in front of the slab: the reflection
    elif kind == "upload":
        p["laser"].update(fwhm=10 * WAVE, t0=15 * WAVE)
    p["fields"] = None
    if kind in ("steps", "lockin"):
        # a pulse of 10 wavelengths in the middle of the box, travelling along the laser's direction
        c, s = math.cos(theta), math.sin(theta)

        def wave(shift):  # shift: half cells of the component's Yee location
            ax = [(torch.arange(n[a], device=dev, dtype=torch.float64) + (0.5 if shift[a] and a < d else 0.0)) * dx for a in range(3)]
            X, Y, Z = ax[0][None, None, :] - 0.5 * n[0] * dx, ax[1][None, :, None] - yc, ax[2][:, None, None] - zc
            along, across = c * X + s * Y, c * Y - s * X
            w = case["a0"] * torch.exp(-2 * math.log(2.0) * (along / (10 * WAVE)) ** 2) * torch.sin(along + phase)
            if waist > 0:
                w = w * torch.exp(-(across ** 2 + Z ** 2) / waist ** 2)
            return w.expand(n[2], n[1], n[0])

        zero = torch.zeros(n[2], n[1], n[0], device=dev, dtype=torch.float64)
        if comp == 1:
            f = [-s * wave((1, 0, 0)) if s else zero, c * wave((0, 1, 0)), zero, zero, zero, wave((1, 1, 0))]
        else:
            f = [zero, zero, wave((0, 0, 1)), s * wave((0, 1, 1)) if s else zero, -c * wave((1, 0, 1)), zero]
        p["fields"] = [x.float() for x in f]
    return p


def prepare(case, seed):
    p = _problem(case, seed)
    d, n = p["d"], p["n"]
    kind = case["kind"]
    ctx = B.Context(d, n[:d], (p["dx"],) * d, p["dt"], p["bc"][:d], tile=TILE[d],
                    deposit_mode=B.BP_DEPOSIT_ATOMIC if case["atomic"] else B.BP_DEPOSIT_SORTED)
    L = p["laser"]
    if p["bc"][0]:
        ctx.add_laser(L["comp"], L["a0"], 1.0, L["theta"], L["waist"], L["fwhm"], L["t0"], L["ramp"], L["phase"], L["ia"],
                      L["yc"], L["zc"])
    state = {"kind": kind, "ctx": ctx, "steps": case["steps"], "load": []}
    for s in p["species"]:
        if s["kind"] == "two":
            sid = ctx.add_two_body(s["Zb"], s["qc"], s["mc"], s["w"], s["lambda_m"], s["omega"])
        else:
            sid = ctx.add_free(s["q"], s["m"], s["w"])
        if "fill" in p:
            ctx.set_medium(sid, *p["fill"])
            continue
        x, u = (t.cpu() for t in (s["x"], s["u"]))
        if kind == "upload":
            x, u = x.pin_memory(), u.pin_memory()
        pidx = s.get("pidx")
        state["load"].append((sid, x.numpy(), u.numpy(), None if pidx is None else pidx.to(torch.int32).cpu().numpy(), s.get("omega")))
        if kind in ("steps", "lockin"):
            ctx.load_particles(*state["load"][-1][:4])
    if p["fields"] is not None:
        for k, f in enumerate(p["fields"]):
            ctx.write_field(k, f.cpu().numpy())
    if "probe" in p:
        state["probe"] = ctx.add_probe(L["comp"], p["probe"], case["steps"])
    if kind == "adjoint":
        sid, _, _, pidx, omega = state["load"][0]
        state["problem"] = SiteProblem(ctx, sid, state["probe"], p["site"].cpu().numpy(), p["off"].cpu().numpy(), pidx,
                                       case["steps"], case["ckpt"])
        state["omega"], state["sites"] = torch.from_numpy(omega).float(), p["sites"].float().cpu()
        state["target"] = _target(case, p, seed)
    elif kind == "lockin":
        state["frames"] = torch.empty(case["steps"], n[2], n[1], n[0], device="cuda")
    elif kind == "upload":
        state["frame"] = torch.empty(n[2], n[1], n[0], pin_memory=True)
    state["fields"] = torch.empty(9, n[2], n[1], n[0], device="cuda")
    return state


def _target(case, p, seed):
    """The recorded wave that the adjoint's loss compares with: the launched
    wave's amplitude with a phase of the seed's own at every probe point."""
    phase = np.random.default_rng(int(seed)).uniform(0.2, 1.0, len(p["probe"]))
    t = p["dt"] * np.arange(1, case["steps"] + 1)
    return torch.from_numpy(0.5 * case["a0"] * np.sin(t[:, None] + phase[None, :]))


def _read(state):
    ctx, f = state["ctx"], state["fields"]
    for k in range(9):
        ctx.read_field_device(k, f[k].data_ptr())
    return {"E": f[0:3], "B": f[3:6], "J": f[6:9]}


def run(state):
    ctx, kind = state["ctx"], state["kind"]
    if kind == "steps":
        ctx.step(state["steps"])
        return _read(state)
    if kind == "lockin":
        for k in range(state["steps"]):
            ctx.step(1)
            ctx.read_field_device(B.EZ, state["frames"][k].data_ptr())
        return {"frames": state["frames"], **_read(state)}
    if kind == "run":
        ctx.reset()
        for sid, x, u, pidx, omega in state["load"]:
            if omega is not None:
                ctx.set_omega(sid, omega)
            ctx.load_particles(sid, x, u, pidx)
        ctx.step(state["steps"])
        out = {"probe": ctx.read_probe(state["probe"]), **_read(state)}
        for sid, x, _, _, omega in state["load"]:  # the state itself is FP32
            x1, x2, u1, u2 = (a.astype(np.float32) for a in ctx.read_particles(sid, len(x)))
            out["free" if omega is None else "ions"] = [x1, u1] if omega is None else [x1, x2, u1, u2]
        return out
    if kind == "upload":
        ctx.reset()
        for sid, x, u, pidx, _ in state["load"]:
            ctx.load_particles(sid, x, u, pidx)
        for _ in range(state["steps"]):
            ctx.step(1)
            ctx.read_field_async(B.EY, state["frame"].numpy())
        ctx.sync()
        return {"frame": state["frame"], **_read(state)}
    omega, sites = state["omega"].clone().requires_grad_(), state["sites"].clone().requires_grad_()
    probe = PICProbe.apply(omega, sites, state["problem"])
    loss = ((probe - state["target"]) ** 2).sum()
    loss.backward()
    return {"probe": probe.detach().float(), "omega": omega.grad, "sites": sites.grad}  # the record itself is FP32


def _counts(case):
    """(two-body ions, free particles) of a case."""
    nx, ny, nz, lo = case["nx"], case["ny"], case["nz"], case["margin"]
    if case["kind"] == "adjoint":
        return 64 * ny * case["ppc"], 0
    if case["medium"] == "neutral":
        return case["ppc"] * (nx - 2 * lo) * ny * nz, 0
    if case["medium"] == "refract":
        k = case["ppc"] * (nx // 4) if case["dims"] == 1 else (nx - lo) * ny
        return k, k
    if case["medium"] == "bragg":
        return 4 * math.prod(min(40, (m - 64) // case["res"]) for m in (nx, ny)), 0
    period = 0.6 * case["res"]
    return 4 * int((nx - 2 * lo) / period) * int(ny / period), case["ppc"] * (nx - 2 * lo) * ny


def work(case):
    """Bytes: in every step each particle's state (cell, offsets, momenta and,
    for an ion, the displacement and the second body's momenta) and E and B
    are read and written once, 4 bytes a value; an uploaded position and
    momentum is read once; a field that is read out is written once.  The
    adjoint adds the checkpoint's copy, the recomputed step and a reverse step
    that reads the state and carries 12 adjoints per ion and 6 per cell.
    Flops: the gather of six components from 3^d nodes at each body, the Boris
    rotations, the force and the deposit of three components over 3^d nodes."""
    d, steps = case["dims"], case["steps"]
    ions, free = _counts(case)
    cells = case["nx"] * case["ny"] * case["nz"]
    state = ions * 4 * (1 + d + 9) + free * 4 * (1 + d + 3)
    body = 6 * 2 * 3 ** d + 3 * 3 * 3 ** d + 140
    step_b, step_f = 2 * state + 48 * cells, (2 * ions + free) * body + 36 * cells
    if case["kind"] == "adjoint":
        reverse = state + 2 * 48 * ions + 24 * cells + 48 * cells
        ck = -(-steps // case["ckpt"]) * 2 * (state + 24 * cells)
        return {"bytes": steps * (2 * step_b + reverse) + ck, "flops": steps * (2 * step_f + 2 * step_f)}
    out = 36 * cells + (4 * cells * steps if case["kind"] in ("lockin", "upload") else 0)
    load = 8 * (ions + free) * (d + 3) if case["kind"] in ("run", "upload") else 0
    return {"bytes": steps * step_b + out + load, "flops": steps * step_f}


# ---------------------------------------------------------------------------
# the same computation in 64 bits, in plain torch

def _shape(u):
    a = u.abs()
    return torch.where(a <= 0.5, 0.75 - u * u, torch.where(a < 1.5, 0.5 * (1.5 - a) ** 2, torch.zeros_like(u)))


class _Sim:
    """The leapfrog step of Sec. 2 on the Yee grid with quadratic shapes, in
    FP64: staggered gather, Boris with the modified Coulomb field, Esirkepov
    deposit, Mur faces.  Every update is out of place, so autograd follows it."""

    CHUNK = 1 << 20

    def __init__(self, p):
        self.d, self.n, self.dx, self.dt, self.bc = p["d"], p["n"], p["dx"], p["dt"], p["bc"]
        self.laser, self.step_no = p["laser"], 0
        shape = (self.n[2], self.n[1], self.n[0])
        kw = dict(device="cuda", dtype=torch.float64)
        f = p["fields"]
        self.F = [torch.zeros(shape, **kw) if f is None else f[k].double() for k in range(6)]
        self.J = [torch.zeros(shape, **kw)] * 3
        ax = [torch.arange(m, device="cuda") for m in self.n]
        self.C = [ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]]
        self.shape = shape
        self.species = []
        for s in p["species"]:
            q = dict(s)
            q["x"] = s["x"]
            q["r"] = torch.zeros(len(s["x"]), 3, **kw)
            q["alive"] = torch.ones(len(s["x"]), **kw)
            if s["kind"] == "two":
                q["q2"], q["m2"] = -s["Zb"], s["Zb"]
                q["q1"], q["m1"] = s["qc"] + s["Zb"], s["mc"] - s["Zb"]
                q["kappa"] = R_E * 2 * math.pi / s["lambda_m"]
                if s["qc"] == 0:
                    q["u1"], q["u2"] = s["u"], s["u"]
                else:
                    q["u1"] = (q["m1"] + q["m2"]) * s["u"] / (q["m1"] - q["m2"] * q["q1"] / q["q2"])
                    q["u2"] = -q["q1"] * q["u1"] / q["q2"]
                self.set_omega(q, torch.as_tensor(s["omega"], **kw))
            else:
                q["q1"], q["m1"], q["u1"] = s["q"], s["m"], s["u"]
            self.species.append(q)
        self.masks = [self._masks(c) for c in range(3)]
        self.outer = [self._edge({a for a in range(3) if a != c}) for c in range(3)]

    def set_omega(self, q, omega):
        mr = q["m1"] * q["m2"] / (q["m1"] + q["m2"])
        ac = (abs(q["q1"] * q["q2"]) * q["kappa"] / (mr * omega * omega)) ** (1.0 / 3.0)
        q["ac"] = ac[q["pidx"]] if q["pidx"] is not None else ac[0]

    def _edge(self, half):
        """Cells off the last node of an open axis on which the component sits half a cell in."""
        m = torch.zeros(self.shape, dtype=torch.bool, device="cuda")
        for a in range(self.d):
            if self.bc[a] and a in half:
                m = m | (self.C[a] == self.n[a] - 1)
        return m

    def _masks(self, c):
        """E component c: the nodes of the interior update, and per pass, open axis and side the Mur nodes."""
        outer = self._edge({c})
        count = torch.zeros(self.shape, dtype=torch.int32, device="cuda")
        first = torch.full(self.shape, -1, dtype=torch.int32, device="cuda")
        for a in range(self.d):
            if self.bc[a] and a != c:
                on = ((self.C[a] == 0) | (self.C[a] == self.n[a] - 1)).expand(self.shape)
                first = torch.where(on & (first < 0), torch.full_like(first, a), first)
                count = count + on.int()
        mur = []
        for k in range(1, sum(self.bc[: self.d]) + 1):
            for a in range(self.d):
                if self.bc[a] and a != c:
                    for side in (0, 1):
                        m = (count == k) & (first == a) & (self.C[a] == (0 if side == 0 else self.n[a] - 1)) & ~outer
                        if bool(m.any()):
                            mur.append((k, a, side, m))
        return (count == 0) & ~outer, mur

    def _diff(self, f, a, forward):
        """The difference along axis a over dx; zero along an axis the grid does not have."""
        if a >= self.d:
            return torch.zeros_like(f)
        r = torch.roll(f, -1 if forward else 1, 2 - a)
        return ((r - f) if forward else (f - r)) / self.dx

    def _curl(self, f, forward):
        return [self._diff(f[(c + 2) % 3], (c + 1) % 3, forward) - self._diff(f[(c + 1) % 3], (c + 2) % 3, forward) for c in range(3)]

    def _half_b(self):
        c = self._curl(self.F[:3], True)
        for k in range(3):
            self.F[3 + k] = torch.where(self.outer[k], self.F[3 + k], self.F[3 + k] - 0.5 * self.dt * c[k])

    def _index(self, nodes):
        """Flat indices of nodes (one list of integer tensors per axis, to be combined), and whether they are on the grid."""
        idx, ok, stride = 0, True, 1
        for a in range(self.d):
            m = nodes[a]
            if self.bc[a]:
                ok = ok & (m >= 0) & (m < self.n[a])
                m = m.clamp(0, self.n[a] - 1)
            else:
                m = torch.remainder(m, self.n[a])
            idx = idx + m * stride
            stride *= self.n[a]
        return idx, ok

    def _spread(self, per_axis):
        """Per-axis tensors [N, k] as factors of a [N, k, ..] stencil."""
        return [t.reshape([len(t)] + [t.shape[1] if b == a else 1 for b in range(self.d)]) for a, t in enumerate(per_axis)]

    def _gather(self, x):
        X = x / self.dx
        out = []
        for k in range(6):
            half = {k} if k < 3 else {a for a in range(3) if a != k - 3}
            nodes, w = [], []
            for a in range(self.d):
                s = X[:, a] - (0.5 if a in half else 0.0)
                near = torch.floor(s.detach() + 0.5)
                m = near[:, None] + torch.arange(-1, 2, device="cuda")
                nodes.append(m.long())
                w.append(_shape(s[:, None] - m))
            idx, ok = self._index(self._spread(nodes))
            weight = math.prod(self._spread(w))
            v = self.F[k].reshape(-1)[idx] * ok
            out.append((v * weight).reshape(len(x), -1).sum(1))
        return torch.stack(out[:3], 1), torch.stack(out[3:], 1)

    @staticmethod
    def _boris(h, E, Bf, u):
        um = u + h * E
        t = h * Bf / torch.sqrt(1 + (um * um).sum(1, keepdim=True))
        s = 2 * t / (1 + (t * t).sum(1, keepdim=True))
        up = um + torch.linalg.cross(um + torch.linalg.cross(um, t), s)
        return up + h * E

    def _deposit(self, J, qw, x0, dx, v):
        """The current of bodies of charge times weight qw [N] moved from x0 by dx."""
        X0, X1 = x0 / self.dx, (x0 + dx) / self.dx
        nodes, S0, DS = [], [], []
        for a in range(self.d):
            m = torch.floor(X0[:, a].detach() + 0.5)[:, None] + torch.arange(-2, 3, device="cuda")
            s0 = _shape(X0[:, a, None] - m)
            nodes.append(m.long())
            S0.append(s0)
            DS.append(_shape(X1[:, a, None] - m) - s0)
        idx, ok = self._index(self._spread(nodes))
        for c in range(3):
            other = [a for a in range(self.d) if a != c]
            s, ds = self._spread(S0), self._spread(DS)
            if len(other) == 2:
                a, b = other
                fac = s[a] * s[b] + 0.5 * (ds[a] * s[b] + s[a] * ds[b]) + ds[a] * ds[b] / 3
            elif len(other) == 1:
                fac = s[other[0]] + 0.5 * ds[other[0]]
            else:
                fac = torch.ones_like(s[0])
            lead = qw.reshape([-1] + [1] * self.d)
            if c < self.d:
                val = -lead * self.dx / self.dt * torch.cumsum(ds[c], 1 + c) * fac
            else:
                val = lead * v[:, c].reshape(lead.shape) * fac
            val = (val * ok).expand(idx.shape)
            J[c] = J[c].index_add(0, idx.reshape(-1), val.reshape(-1))

    def _antenna(self, J):
        L, t = self.laser, (self.step_no + 0.5) * self.dt
        ny, nz = self.n[1], self.n[2]
        kw = dict(device="cuda", dtype=torch.float64)
        y = (torch.arange(ny, **kw) + (0.5 if L["comp"] == 1 else 0.0)) * self.dx if self.d >= 2 else torch.zeros(1, **kw)
        z = (torch.arange(nz, **kw) + (0.5 if L["comp"] == 2 else 0.0)) * self.dx if self.d >= 3 else torch.zeros(1, **kw)
        ty, tz = (y - L["yc"])[None, :], (z - L["zc"])[:, None]
        tau = t - ty * math.sin(L["theta"]) + 0 * tz
        if L["fwhm"] > 0:
            env = torch.exp(-2 * math.log(2.0) * ((tau - L["t0"]) / L["fwhm"]) ** 2)
        else:
            env = torch.sin(0.5 * math.pi * (tau / L["ramp"]).clamp(0, 1)) ** 2
        if L["waist"] > 0:
            env = env * torch.exp(-((ty * math.cos(L["theta"])) ** 2 + tz ** 2) / L["waist"] ** 2)
        f = L["a0"] * env * torch.sin(tau + L["phase"])
        sheet = torch.zeros(self.shape, **kw)
        sheet[:, :, L["ia"]] = -2 / self.dx * (math.cos(L["theta"]) if L["comp"] == 2 else 1.0) * f
        J[L["comp"]] = J[L["comp"]] + sheet

    def step(self):
        self._half_b()
        cells = math.prod(self.n)
        J = [torch.zeros(cells, device="cuda", dtype=torch.float64) for _ in range(3)]
        d, dt = self.d, self.dt
        for s in self.species:
            parts = []
            for i in range(0, len(s["x"]), self.CHUNK):
                cut = slice(i, i + self.CHUNK)
                x, r, u1 = s["x"][cut], s["r"][cut], s["u1"][cut]
                qw = s["w"] * s["alive"][cut]
                E1, B1 = self._gather(x)
                if s["kind"] == "two":
                    u2 = s["u2"][cut]
                    x2 = x - r[:, :d]
                    E2, B2 = self._gather(x2)
                    ac = s["ac"][cut] if s["ac"].ndim else s["ac"]
                    force = s["kappa"] * ((r * r).sum(1) + ac * ac)[:, None] ** -1.5 * r
                    u1 = self._boris(s["q1"] * dt / (2 * s["m1"]), E1 + s["q2"] * force, B1, u1)
                    u2 = self._boris(s["q2"] * dt / (2 * s["m2"]), E2 - s["q1"] * force, B2, u2)
                    v1 = u1 / torch.sqrt(1 + (u1 * u1).sum(1, keepdim=True))
                    v2 = u2 / torch.sqrt(1 + (u2 * u2).sum(1, keepdim=True))
                    self._deposit(J, s["q2"] * qw, x2, dt * v2[:, :d], v2)
                    r = r + dt * (v1 - v2)
                else:
                    u1 = self._boris(s["q1"] * dt / (2 * s["m1"]), E1, B1, u1)
                    v1 = u1 / torch.sqrt(1 + (u1 * u1).sum(1, keepdim=True))
                    u2 = u1
                self._deposit(J, s["q1"] * qw, x, dt * v1[:, :d], v1)
                x = x + dt * v1[:, :d]
                parts.append((x, r, u1, u2))
            s["x"], s["r"], s["u1"], s["u2"] = (torch.cat(t) for t in zip(*parts))
            if s["kind"] == "free":  # removed once its cell leaves [2, n - 2) on an open axis
                c = torch.floor(s["x"].detach() / self.dx)
                for a in range(d):
                    if self.bc[a]:
                        s["alive"] = s["alive"] * ((c[:, a] >= 2) & (c[:, a] < self.n[a] - 2))
        J = [j.reshape(self.shape) for j in J]
        if self.bc[0]:
            self._antenna(J)
        self.J = J
        self._half_b()
        old = self.F[:3]
        curl = self._curl(self.F[3:], False)
        new = [torch.where(self.masks[c][0], old[c] + dt * (curl[c] - J[c]), old[c]) for c in range(3)]
        for k in range(1, sum(self.bc[:d]) + 1):
            for c in range(3):
                for q, a, side, m in self.masks[c][1]:
                    if q == k:
                        to = 1 if side else -1
                        km = (dt - self.dx) / (dt + self.dx)
                        v = torch.roll(old[c], to, 2 - a) + km * (torch.roll(new[c], to, 2 - a) - old[c])
                        new[c] = torch.where(m, v, new[c])
        self.F[:3] = new
        self.step_no += 1

    def fields(self):
        return {"E": torch.stack(self.F[:3]), "B": torch.stack(self.F[3:]), "J": torch.stack(self.J)}


def exact(case, seed):
    ions, free = _counts(case)
    kind, nodes = case["kind"], 5 ** case["dims"]
    if kind == "adjoint":
        # autograd keeps every step
        if (ions * nodes * 40 + 30 * case["nx"] * case["ny"]) * 8 * case["steps"] > 60e9:
            return None
    elif (ions + free) > EVERYTHING or (2 * ions + free) * nodes * case["steps"] > 1.5e10:
        return None
    p = _problem(case, seed)
    sim = _Sim(p)
    if kind == "adjoint":
        s = sim.species[0]
        omega = torch.as_tensor(s["omega"], device="cuda").clone().requires_grad_()
        sites = p["sites"].clone().requires_grad_()
        sim.set_omega(s, omega)
        s["x"] = sites[p["site"]] + p["off"]
        at = torch.as_tensor(p["probe"], device="cuda")
        rows = []
        for _ in range(case["steps"]):
            sim.step()
            rows.append(sim.F[p["laser"]["comp"]].reshape(-1)[at])
        probe = torch.stack(rows)
        loss = ((probe - _target(case, p, seed).cuda()) ** 2).sum()
        loss.backward()
        return {"probe": probe.detach().cpu(), "omega": omega.grad.cpu(), "sites": sites.grad.cpu()}
    with torch.no_grad():
        rows, frames = [], []
        for _ in range(case["steps"]):
            sim.step()
            if kind == "run":
                rows.append(sim.F[p["laser"]["comp"]].reshape(-1)[p["probe"]])
            if kind == "lockin":
                frames.append(sim.F[2])
        out = sim.fields()
        if kind == "run":
            out["probe"] = torch.stack(rows).cpu()
            for s in sim.species:
                x1 = torch.zeros(len(s["x"]), 3, dtype=torch.float64, device="cuda")
                x1[:, :1] = s["x"]
                two = s["kind"] == "two"
                x2 = x1 - s["r"]
                out["ions" if two else "free"] = [t.cpu() for t in ([x1, x2, s["u1"], s["u2"]] if two else [x1, s["u1"]])]
        if kind == "lockin":
            out["frames"] = torch.stack(frames)
        if kind == "upload":
            out["frame"] = sim.F[1].cpu()
        return out
