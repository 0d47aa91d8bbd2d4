"""The work a user of this package has it do, as timed cases.

Every case goes through the package's public binding (`pic.Context`, `pic.Species*`,
`adjoint.ProbeEnergy`).  Most are whole runs from initial conditions: FP64 positions and Yee fields
in hand, deposit rho^0, advance a number of steps in one call, read the advanced fields, J, rho, the
momenta and the positions of the tracked particles (in the order of their ids: the library re-orders
the particle arrays).  The others are the reverse step, the probe-energy gradient, the
field solve and the transforms, which programs also call by themselves.

`exact` restates each of them with plain torch operations in 64 bits (torch.fft transforms, one
gather or index_add per stencil node, PSATD coefficients by Gauss-Legendre quadrature of the
analytic solution, autograd for the reverse mode), without this package.
"""
import math

import numpy as np
import torch

from paper_2106_12919_gb300 import adjoint, pic

_VARIANT = {"standard": pic.STANDARD, "galilean": pic.GALILEAN, "averaged": pic.AVERAGED}
_CYCLE = {"hybrid": pic.PIC_CYCLE_HYBRID, "fdtd": pic.PIC_CYCLE_HYBRID_FDTD}


def _case(name, kind, family, form, shape, ppc, steps, drop=0, order=None, pusher="boris", filter=0, tile="8x8x8"):
    d = {"kind": kind, "family": family, "form": form, "nx": shape[0], "ny": shape[1], "nz": shape[2], "ppc": ppc,
         "steps": steps, "drop": drop, "order": order or _FAMILY[family]["order"], "pusher": pusher, "filter": filter,
         "tile": tile}
    return dict(d, name=name) if name else d


# method and spacings of each family of runs: the configurations of workloads.py (thermal plasma, laser
# wakefield, drifting pair plasma, beam-driven wakefield, seed wave) and the FDTD form of the laser one
_FAMILY = {
    "thermal": dict(dx=(1.0, 1.0, 1.0), variant="standard", center=(8, 8, 8), spectral=(0, 0, 0), order=1,
                    cycle="hybrid", gamma=0.0),
    "laser": dict(dx=(0.2, 0.2, 0.04), variant="standard", center=(8, 8, 16), spectral=(0, 0, 0), order=3,
                  cycle="hybrid", gamma=0.0),
    "drift": dict(dx=(1.0, 1.0, 1.0), variant="galilean", center=(8, 8, 8), spectral=(16, 16, 16), order=2,
                  cycle="hybrid", gamma=130.0),
    "beam": dict(dx=(0.1, 0.1, 0.02), variant="averaged", center=(8, 8, 16), spectral=(16, 16, 16), order=3,
                 cycle="hybrid", gamma=1000.0),
    "laser_fdtd": dict(dx=(0.2, 0.2, 0.04), variant="standard", center=(8, 8, 16), spectral=(4, 4, 16), order=3,
                       cycle="fdtd", gamma=0.0),
    "seed": dict(dx=(1.0, 1.0, 1.0), variant="standard", center=(8, 8, 8), spectral=(0, 0, 0), order=1,
                 cycle="hybrid", gamma=0.0),
}


def listed():
    return [
        # one step of a small plasma, as in an interactive or coupled loop: launches and latency
        _case("thermal_f32_32_one_step", "run", "thermal", "fp32", (32, 32, 32), 8, 1),
        # the thermal-plasma configuration, 32^3 and 8 per cell, 10 steps, a ragged particle count
        _case("thermal_f64_32", "run", "thermal", "fp64", (32, 32, 32), 8, 10, drop=37),
        # the drifting electron-positron plasma of the Galilean stability runs, two species
        _case("drift_f32_64x64x256", "run", "drift", "fp32", (64, 64, 256), 2, 20, drop=1001),
        # the laser-wakefield box at its configured size
        _case("laser_f32_128x128x512", "run", "laser", "fp32", (128, 128, 512), 2, 10),
        # the same physics in the FP64 form at the size used for convergence checks
        _case("laser_f64_64x64x256", "run", "laser", "fp64", (64, 64, 256), 2, 4, drop=513),
        # the paper's production settings: Vay's pusher and the bilinear filter
        _case("laser_f32_vay_64x64x512", "run", "laser", "fp32", (64, 64, 512), 3, 10, drop=77, pusher="vay", filter=1),
        # the beam-driven wakefield box at its configured size (68.1M particles), tiles as the benchmark takes them
        _case("beam_f32_256x256x1024", "run", "beam", "fp32", (256, 256, 1024), 1, 6, tile="8x16x8"),
        # the averaged Galilean form in FP64
        _case("beam_f64_64x64x256", "run", "beam", "fp64", (64, 64, 256), 1, 4),
        # the hybrid scheme around the finite-difference solver
        _case("fdtd_f32_128x128x256", "run", "laser_fdtd", "fp32", (128, 128, 256), 2, 6),
        # one reverse step of the differentiable probe problem (64^3, 4 per cell, CIC)
        _case("adjoint_64", "adjoint", "seed", "fp64", (64, 64, 64), 4, 1),
        # the probe-energy loss and its gradient through autograd, forward and backward
        _case("gradient_32", "gradient", "seed", "fp64", (32, 32, 32), 4, 8, order=3),
        # the FP64 field solve by itself (transforms, update, transforms)
        _case("solve_f64_128x128x256", "solve", "beam", "fp64", (128, 128, 256), 0, 1),
    ]


def draw(rng):
    def grid(lo, hi):
        """powers of two per axis, 16..1024 along z, with lo <= log2 cells <= hi"""
        while True:
            e = [rng.randint(4, 8), rng.randint(4, 8), rng.randint(4, 10)]
            if lo <= sum(e) <= hi:
                return tuple(1 << v for v in e)

    def ragged(shape):
        return rng.randint(1, max(2, shape[0] * shape[1] * shape[2] // 16))

    kind = rng.choice(["f32", "f32", "f32", "f32", "f64", "f64", "fdtd", "adjoint", "gradient", "solve", "transform"])
    if kind == "f32":
        shape = grid(15, 25)
        family = rng.choice(["thermal", "laser", "drift", "beam"])
        big = shape[0] * shape[1] * shape[2] > 1 << 23
        return _case(None, "run", family, "fp32", shape, 1 if big else rng.randint(1, 6),
                     rng.choice([1, 2, 3]) if big else rng.randint(1, 12), ragged(shape),
                     order=rng.choice([None, 1, 2, 3]), pusher=rng.choice(["boris", "boris", "vay"]),
                     filter=rng.choice([0, 0, 1, 2]), tile=rng.choice(["8x8x8", "8x8x8", "8x16x8", "16x8x8", "4x8x8"]))
    if kind == "f64":
        shape = grid(13, 20)
        return _case(None, "run", rng.choice(["thermal", "laser", "drift", "beam"]), "fp64", shape, rng.randint(1, 5),
                     rng.randint(1, 6), ragged(shape), order=rng.choice([None, 1, 2, 3]),
                     pusher=rng.choice(["boris", "boris", "vay"]), filter=rng.choice([0, 0, 1]))
    if kind == "fdtd":
        shape = grid(15, 22)
        return _case(None, "run", "laser_fdtd", rng.choice(["fp32", "fp32", "fp64"]), shape, rng.randint(1, 3),
                     rng.randint(1, 6), ragged(shape), order=rng.choice([1, 2, 3]))
    if kind == "adjoint":
        shape = grid(13, 19)
        return _case(None, "adjoint", "seed", "fp64", shape, rng.randint(1, 5), 1, ragged(shape), order=rng.randint(1, 3))
    if kind == "gradient":
        shape = grid(12, 16)
        return _case(None, "gradient", "seed", "fp64", shape, rng.randint(1, 4), rng.randint(2, 8), ragged(shape),
                     order=rng.randint(1, 3))
    if kind == "solve":
        return _case(None, "solve", rng.choice(["laser", "drift", "beam"]), "fp64", grid(13, 23), 0, 1)
    return _case(None, "transform", "laser", rng.choice(["fp32", "fp64"]), grid(13, 24), 0, 1)


# ---------------------------------------------------------------------------------------------------
# what a program has in hand
# ---------------------------------------------------------------------------------------------------
def _shape(case):
    return case["nx"], case["ny"], case["nz"]


def _params(case):
    f = _FAMILY[case["family"]]
    shape = _shape(case)
    center = tuple(min(o, n) for o, n in zip(f["center"], shape))
    spectral = tuple(min(o, n) for o, n in zip(f["spectral"], shape))
    dt = f["dx"][2]
    if f["cycle"] == "fdtd":  # 0.9 of the Courant limit of these orders
        s = sum((2.0 * sum(abs(w) for w in _fd_weights(spectral[a] // 2)) / f["dx"][a]) ** 2 for a in range(3))
        dt = 0.9 * 2.0 / math.sqrt(s)
    beta = math.sqrt(1.0 - 1.0 / f["gamma"] ** 2) if f["gamma"] else 0.0
    return dict(shape=shape, dx=f["dx"], dt=dt, order=case["order"], center=center, variant=f["variant"],
                v_gal=(0.0, 0.0, beta), spectral=spectral, cycle=f["cycle"])


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _stratified(g, shape, ppc, drop, dx):
    """ppc particles uniform in every cell, then the last `drop` of a random choice left out"""
    n = shape[0] * shape[1] * shape[2]
    idx = torch.arange(n, device="cuda").repeat_interleave(ppc)
    if drop:
        keep = torch.ones(idx.numel(), dtype=torch.bool, device="cuda")
        keep[torch.randperm(idx.numel(), device="cuda", generator=g)[:drop]] = False
        idx = idx[keep]
    iz = idx % shape[2]
    r = idx // shape[2]
    cell = [r // shape[1], r % shape[1], iz]
    return [((cell[a] + torch.rand(idx.numel(), dtype=torch.float64, device="cuda", generator=g)) * dx[a])
            for a in range(3)]


def _normal(g, n, s=1.0):
    return s * torch.randn(n, dtype=torch.float64, device="cuda", generator=g)


def _state0(case, seed):
    """Yee E, B (lists of FP64 (Nx, Ny, Nz) arrays) and the species [(x, y, z, ux, uy, uz, w, q, m)] at t = 0"""
    p = _params(case)
    shape, dx, family = p["shape"], p["dx"], case["family"]
    g = _gen(seed)
    zero = lambda: torch.zeros(shape, dtype=torch.float64, device="cuda")  # noqa: E731
    E, B = [zero() for _ in range(3)], [zero() for _ in range(3)]
    dV = dx[0] * dx[1] * dx[2]
    L = [shape[a] * dx[a] for a in range(3)]

    def at(a, off):
        v = (torch.arange(shape[a], dtype=torch.float64, device="cuda") + off) * dx[a]
        return v.reshape([-1 if b == a else 1 for b in range(3)])

    x = _stratified(g, shape, case["ppc"], case["drop"], dx)
    n = x[0].numel()
    w = torch.full((n,), dV / case["ppc"], dtype=torch.float64, device="cuda")
    none = lambda: torch.zeros(n, dtype=torch.float64, device="cuda")  # noqa: E731
    if family == "thermal":
        sp = [(*x, *[_normal(g, n, 0.01) for _ in range(3)], w, -1.0, 1.0)]
    elif family in ("laser", "laser_fdtd"):
        w = w * torch.clamp(x[2] / (50 * dx[2]), max=1.0)
        k0 = 2 * math.pi / (30 * dx[2])
        w0, ell, zl = 20 * dx[0], 60 * dx[2], min(150, shape[2] // 2) * dx[2]

        def pulse(ox, oy, oz):
            r2 = (at(0, ox) - L[0] / 2) ** 2 + (at(1, oy) - L[1] / 2) ** 2
            z = at(2, oz) - zl
            return 2.0 * k0 * torch.exp(-r2 / w0 ** 2) * torch.exp(-(z / ell) ** 2) * torch.cos(k0 * z)

        E[1], B[0] = pulse(0.0, 0.5, 0.0), -pulse(0.0, 0.5, 0.5)
        sp = [(*x, none(), none(), none(), w, -1.0, 1.0)]
    elif family == "drift":
        u0 = math.sqrt(_FAMILY[family]["gamma"] ** 2 - 1.0)
        ue, up = [[_normal(g, n, 1e-3) for _ in range(3)] for _ in range(2)]
        sp = [(*x, ue[0], ue[1], ue[2] + u0, w, -1.0, 1.0),
              (*_stratified(g, shape, case["ppc"], case["drop"], dx), up[0], up[1], up[2] + u0, w.clone(), 1.0, 1.0)]
    elif family == "beam":
        nb = max(64, shape[0] * shape[1] * shape[2] // 67)
        sr, sz = 4 * dx[0], 10 * dx[2]
        c = (L[0] / 2, L[1] / 2, 0.75 * L[2])
        xb = [torch.remainder(c[a] + (sz if a == 2 else sr) * _normal(g, nb), L[a]) for a in range(3)]
        zb = torch.zeros(nb, dtype=torch.float64, device="cuda")
        wb = torch.full_like(zb, 10.0 * (2 * math.pi) ** 1.5 * sr * sr * sz / nb)
        ub = torch.full_like(zb, math.sqrt(_FAMILY[family]["gamma"] ** 2 - 1.0))
        sp = [(*x, none(), none(), none(), w, -1.0, 1.0), (*xb, zb, zb.clone(), ub, wb, -1.0, 1.0)]
    else:  # seed wave
        z = at(2, 0.0) - L[2] / 2
        E[0] = (1e-2 * torch.exp(-(z / 8.0) ** 2) * torch.cos(2 * math.pi * at(2, 0.0) / 16.0)).expand(shape).contiguous()
        sp = [(*x, *[_normal(g, n, 0.05) for _ in range(3)], w, -1.0, 1.0)]
    return p, E, B, sp


def _context(case, p, **more):
    return pic.Context(p["shape"], p["dx"], p["dt"], p["order"], p["center"], _VARIANT[p["variant"]], p["v_gal"],
                       p["spectral"], tile=tuple(int(t) for t in case["tile"].split("x")),
                       precision=pic.PIC_FP32 if case["form"] == "fp32" else pic.PIC_FP64,
                       filter_passes=case["filter"], cycle=_CYCLE[p["cycle"]],
                       pusher=pic.PIC_PUSHER_VAY if case["pusher"] == "vay" else pic.PIC_PUSHER_BORIS, **more)


def _waves(case, seed, count):
    """smooth random periodic fields of order one with a spectrum (as fields and deposits have), plus noise"""
    shape, g, out = _shape(case), _gen(seed), []
    for _ in range(count):
        f = 0.1 * torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)
        for _ in range(4):
            t = 0.0
            for a in range(3):
                k = int(torch.randint(1, max(2, shape[a] // 8), (1,), device="cuda", generator=g))
                v = torch.arange(shape[a], dtype=torch.float64, device="cuda") * (2 * math.pi * k / shape[a])
                t = t + v.reshape([-1 if b == a else 1 for b in range(3)])
            f = f + torch.cos(t + 6.28 * torch.rand(1, dtype=torch.float64, device="cuda", generator=g))
        out.append(f)
    return out


def _adjoints(case, seed, n):
    """incoming adjoints of a reverse step: of E, B, rho (grid) and of the positions and momenta"""
    return _waves(case, seed + 7, 7), [_normal(_gen(seed + 8 + a), n, 1e-2) for a in range(6)]


def _probe(shape):
    return tuple(max(0, s // 2 - 8) for s in shape), tuple(min(s, s // 2 + 8) for s in shape)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "transform":
        p = _params(case)
        dt = torch.float32 if case["form"] == "fp32" else torch.float64
        return {"case": case, "ctx": _context(case, p), "F": [f.reshape(-1).to(dt) for f in _waves(case, seed, 6)]}
    if kind == "solve":
        p = _params(case)
        return {"case": case, "p": p, "ctx": _context(case, p), "F": [f.reshape(-1) for f in _waves(case, seed, 11)]}
    p, E, B, sp = _state0(case, seed)
    dt = torch.float32 if case["form"] == "fp32" else torch.float64
    E, B = [f.reshape(-1).to(dt) for f in E], [f.reshape(-1).to(dt) for f in B]
    if kind == "gradient":
        ctx = _context(case, p, sort_interval=0)
        run_ = adjoint.Rollout(ctx, [pic.Species(*sp[0])], case["steps"], *_probe(p["shape"]), checkpoint=4)
        return {"case": case, "E": torch.stack(E), "B": torch.stack(B), "u": sp[0][3:6], "run": run_}
    if kind == "adjoint":
        ctx = _context(case, p, sort_interval=0)
        f, q = _adjoints(case, seed, sp[0][0].numel())
        return {"case": case, "ctx": ctx, "E": E, "B": B, "sp": [pic.Species(*sp[0])],
                "fb": [a.reshape(-1) for a in f], "pb": q}
    ids = [torch.arange(s[0].numel(), device="cuda") for s in sp]
    return {"case": case, "p": p, "ctx": _context(case, p), "E": E, "B": B, "sp": sp, "id": ids}


# ---------------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------------
def _by_id(id, v):
    out = torch.empty_like(v)
    out[id] = v
    return out


def _tracks(p, x0, id, x, dtype):
    """x^n of the particles in id order, followed across the periodic boundary from x^0"""
    out = []
    for a in range(3):
        L = p["shape"][a] * p["dx"][a]
        x1 = _by_id(id, x[a])
        d = x1 - x0[a]
        out.append(torch.where(d > 0.5 * L, x1 - L, torch.where(d < -0.5 * L, x1 + L, x1)).to(dtype))
    return out


def _run(s):
    case, p, ctx = s["case"], s["p"], s["ctx"]
    f32 = case["form"] == "fp32"
    E, B = [a.clone() for a in s["E"]], [a.clone() for a in s["B"]]
    J, rho = [torch.empty_like(E[0]) for _ in range(3)], torch.empty_like(E[0])
    if f32:
        sp = [pic.Species32.from_positions(ctx, *v, id=i.clone()) for v, i in zip(s["sp"], s["id"])]
        ctx.deposit_rho32(sp, rho)
        ctx.step32(E, B, J, rho, sp, case["steps"])
    else:
        sp = [pic.Species(*[a.clone() for a in v[:7]], v[7], v[8], id=i.clone()) for v, i in zip(s["sp"], s["id"])]
        ctx.deposit_rho(sp, rho)
        ctx.step(E, B, J, rho, sp, case["steps"])
    out = {"E": E, "B": B, "J": J, "rho": rho}
    for q, v in enumerate(sp):
        d = ctx.species32_to_species(v) if f32 else v
        out["u%d" % q] = [_by_id(v.id, u) for u in (v.ux, v.uy, v.uz)]
        out["x%d" % q] = _tracks(p, s["sp"][q], d.id, (d.x, d.y, d.z), E[0].dtype)
    return out


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "run":
        return _run(s)
    if kind == "transform":
        ctx = s["ctx"]
        spec = [torch.empty(2 * ctx.nmode, dtype=s["F"][0].dtype, device="cuda") for _ in s["F"]]
        back = [torch.empty_like(f) for f in s["F"]]
        (ctx.fft_forward32 if case["form"] == "fp32" else ctx.fft_forward)(s["F"], spec)
        work_ = [v.clone() for v in spec]  # the inverse overwrites its spectra
        (ctx.fft_inverse32 if case["form"] == "fp32" else ctx.fft_inverse)(work_, back)
        return {"spec": spec, "back": back}
    if kind == "solve":
        F, ctx = s["F"], s["ctx"]
        E, B = [a.clone() for a in F[0:3]], [a.clone() for a in F[3:6]]
        avg = s["p"]["variant"] == "averaged"
        A = [torch.empty_like(E[0]) for _ in range(6)] if avg else []
        ctx.maxwell_step(E, B, F[6:9], F[9], F[10], A[0:3] if avg else None, A[3:6] if avg else None)
        return {"E": E, "B": B, "avg": A}
    if kind == "adjoint":
        fb = [a.clone() for a in s["fb"]]
        pb = dict(zip(("x", "y", "z", "ux", "uy", "uz"), [a.clone() for a in s["pb"]]))
        s["ctx"].adjoint_step(s["E"], s["B"], s["sp"], fb[0:3], fb[3:6], fb[6], [pb])
        return {"E": fb[0:3], "B": fb[3:6], "rho": fb[6], "p": pb}
    E, B = s["E"].clone().requires_grad_(), s["B"].clone().requires_grad_()
    u = [a.clone().requires_grad_() for a in s["u"]]
    loss = adjoint.ProbeEnergy.apply(E, B, *u, s["run"])
    loss.backward()
    return {"loss": loss.detach(), "E": E.grad, "B": B.grad, "u": [a.grad for a in u]}


# ---------------------------------------------------------------------------------------------------
# what one pass cannot do without
# ---------------------------------------------------------------------------------------------------
def _particles(case):
    n = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] in ("transform", "solve"):
        return 0
    one = n * case["ppc"] - case["drop"]
    return 2 * one if case["family"] == "drift" else one + (max(64, n // 67) if case["family"] == "beam" else 0)


def work(case):
    n, np_ = case["nx"] * case["ny"] * case["nz"], _particles(case)
    b = 4 if case["form"] == "fp32" else 8
    nodes = (case["order"] + 1) ** 3
    fft = 2.5 * n * math.log2(n)
    if case["kind"] == "transform":
        return {"bytes": b * n * (6 + 6 + 6), "flops": 12 * fft}
    if case["kind"] == "solve":
        return {"bytes": b * n * (11 + 12), "flops": (11 + 12) * fft + 150 * n}
    if case["kind"] == "adjoint":
        return {"bytes": b * (n * 20 + np_ * 19), "flops": 35 * fft + np_ * (nodes * 90 + 400)}
    per_step = {"bytes": b * (n * 16 + np_ * 14), "flops": 10 * fft + 150 * n + np_ * (nodes * 22 + 250)}
    if case["kind"] == "gradient":  # forward, recomputed forward and reverse of every step
        per_step = {"bytes": 3 * per_step["bytes"], "flops": 2 * per_step["flops"] + 35 * fft + np_ * (nodes * 90 + 400)}
    # in: FP64 positions, momenta, weights, ids and the fields; out: fields, J, rho, momenta, positions
    ends = n * b * 16 + np_ * (64 + 6 * b)
    return {"bytes": case["steps"] * per_step["bytes"] + ends, "flops": case["steps"] * per_step["flops"]}


# ---------------------------------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ---------------------------------------------------------------------------------------------------
def _alpha_s(m, n):
    """Fornberg weights of the staggered first derivative (and, over 2n - 1, of its difference form)"""
    d = 1.0
    for i in range(1, m + 1):
        d *= (2 * i - 1) / 2
    return (1 if n % 2 else -1) * d * d * 4 / ((2 * n - 1) * math.factorial(m - n) * math.factorial(m + n - 1))


def _alpha_c(m, n):
    return (1 if n % 2 else -1) * 2 * math.factorial(m) ** 2 / (math.factorial(m - n) * math.factorial(m + n))


def _fd_weights(m):
    return [_alpha_s(m, n) / (2 * n - 1) for n in range(1, max(1, m) + 1)]


def _axis(N, dx, spectral, center):
    """per Fourier index: [k]_s, [k]_c, centering symbol, half-cell shift, bilinear filter symbol"""
    j = np.rint(np.fft.fftfreq(N) * N).astype(np.int64)
    sinp = lambda q, d: np.sin(np.pi * (np.mod(q, 2 * d) / d))  # noqa: E731
    cosp = lambda q, d: np.cos(np.pi * (np.mod(q, 2 * d) / d))  # noqa: E731
    if spectral == 0:
        ks = kc = 2 * np.pi * j / (N * dx)
    else:
        m = spectral // 2
        ks = sum(_alpha_s(m, n) * sinp(j * (2 * n - 1), N) / ((n - 0.5) * dx) for n in range(1, m + 1))
        kc = sum(_alpha_c(m, n) * sinp(2 * j * n, N) / (n * dx) for n in range(1, m + 1))
    zeta = sum(_alpha_s(center // 2, n) * cosp(j * (2 * n - 1), N) for n in range(1, center // 2 + 1))
    half = cosp(j, N) - 1j * sinp(j, N)
    return [torch.from_numpy(np.asarray(v)).cuda() for v in (ks, kc, zeta, half, cosp(j, N) ** 2)]


_STAG = ((1, 0, 0), (0, 1, 0), (0, 0, 1), (0, 1, 1), (1, 0, 1), (1, 1, 0))  # E^x .. B^z


class _Exact:
    """The hybrid cycle in plain torch: FP64, differentiable."""

    def __init__(self, p, filter_passes=0, vay=False):
        self.p, self.shape, self.dx, self.dt, self.vay = p, p["shape"], p["dx"], p["dt"], vay
        self.vg = p["v_gal"] if p["variant"] != "standard" else (0.0, 0.0, 0.0)
        self.passes = filter_passes
        if p["cycle"] == "fdtd":
            return
        nzh = self.shape[2] // 2 + 1
        ax = [_axis(self.shape[a], self.dx[a], p["spectral"][a], p["center"][a]) for a in range(3)]
        ax[2] = [v[:nzh] for v in ax[2]]
        self.k, kc, self.zeta, self.half, self.flt = ([ax[a][i].reshape([-1 if b == a else 1 for b in range(3)])
                                                      for a in range(3)] for i in range(5))
        # the coefficients depend on k_x, k_y through their squares only (v_gal along z)
        q = [self.k[0][: self.shape[0] // 2 + 1], self.k[1][:, : self.shape[1] // 2 + 1], self.k[2]]
        phi = torch.sqrt(q[0] ** 2 + q[1] ** 2 + q[2] ** 2) * self.dt
        a = (self.vg[2] * kc[2] * self.dt).expand(phi.shape)
        co = self._coefficients(phi, a, p["variant"] == "averaged")
        ix = torch.arange(self.shape[0], device="cuda")
        iy = torch.arange(self.shape[1], device="cuda")
        self.fold = (torch.minimum(ix, self.shape[0] - ix), torch.minimum(iy, self.shape[1] - iy))
        self.co = co

    def _coefficients(self, phi, a, averaged):
        dt = self.dt
        x, w = np.polynomial.legendre.leggauss(20)
        x, w = (x + 1) / 2, w / 2
        sinc = lambda v: torch.sinc(v / math.pi)  # noqa: E731
        cis = lambda v: torch.polar(torch.ones_like(v), v)  # noqa: E731
        sa = sinc(a / 2)
        K1 = K2 = K3 = 0
        for s, ws in zip(x, w):
            g = ws * s * sinc(phi * s)
            K1 = K1 + g * cis(a * s)
            K2 = K2 + g * (1 - s) * sinc(a * (1 - s) / 2) / sa * cis(a * s / 2)
            K3 = K3 - g * s * sinc(a * s / 2) / sa * cis(a * (1 + s) / 2)
        th2 = cis(a)
        co = {"TC": th2 * torch.cos(phi), "TS": th2 * (dt * sinc(phi)), "X1": K1 * dt ** 2, "X2": K2 * dt ** 2,
              "TX3": K3 * dt ** 2, "X4": dt * (1j * a * K1 - th2 * sinc(phi))}
        if averaged:
            F = lambda b: cis(b) * sinc(b / 2)  # noqa: E731
            P2 = Y1 = Q = 0
            for s, ws in zip(x + 0.5, w):
                P2 = P2 + ws * s * sinc(phi * s) * cis(a * s)
                for r, wr in zip(x, w):
                    u, wu = s * r, ws * s * wr
                    d = s - u
                    Y1 = Y1 + wu * u * sinc(phi * u) * cis(a * u)
                    Q = Q + wu * d * sinc(phi * d) * u * sinc(a * u / 2) / sa * cis(a * (d + (u - 1) / 2))
            co.update({"P1": 0.5 * (F(a + phi) + F(a - phi)), "P2": -dt * P2, "Y1": dt ** 2 * Y1, "Y2": -1j * dt ** 2 * Q,
                       "Y3": -1j * dt ** 2 * (Y1 - Q), "Y4": dt * (1j * a * Y1 - P2)})
        return co

    def c(self, name):
        return self.co[name][self.fold[0]][:, self.fold[1]]

    def fwd(self, f):
        return torch.fft.fftn(torch.fft.rfft(f.reshape(self.shape), dim=2), dim=(0, 1))

    def inv(self, F):
        return torch.fft.irfft(torch.fft.ifftn(F, dim=(0, 1)), n=self.shape[2], dim=2).reshape(-1)

    def phase(self, F, stag, back=False):
        for a in range(3):
            if stag[a]:
                F = F * (self.half[a].conj() if back else self.half[a])
        return F

    def nodal(self, EB):
        out = []
        for c in range(6):
            G = EB[c]
            for a in range(3):
                if _STAG[c][a]:
                    G = G * self.zeta[a]
            out.append(self.inv(G))
        return out

    def solve(self, EB, J, rn, rp):
        k = self.k
        cross = lambda v: [k[1] * v[2] - k[2] * v[1], k[2] * v[0] - k[0] * v[2], k[0] * v[1] - k[1] * v[0]]  # noqa: E731
        E, B = EB[:3], EB[3:]
        kE, kB, kJ = cross(E), cross(B), cross(J)
        TC, TS, X1, X4 = (self.c(v) for v in ("TC", "TS", "X1", "X4"))
        r = 1j * (self.c("TX3") * rn - self.c("X2") * rp)
        new = [TC * E[a] + 1j * TS * kB[a] + X4 * J[a] + r * k[a] for a in range(3)]
        new += [TC * B[a] - 1j * TS * kE[a] + 1j * X1 * kJ[a] for a in range(3)]
        if self.p["variant"] != "averaged":
            return new, new
        P1, P2, Y1, Y4 = (self.c(v) for v in ("P1", "P2", "Y1", "Y4"))
        r = self.c("Y3") * rn + self.c("Y2") * rp
        avg = [P1 * E[a] - 1j * P2 * kB[a] + Y4 * J[a] + r * k[a] for a in range(3)]
        avg += [P1 * B[a] + 1j * P2 * kE[a] + 1j * Y1 * kJ[a] for a in range(3)]
        return new, avg

    def smooth(self, F):
        for a in range(3):
            F = F * self.flt[a] ** self.passes
        return F

    # particles
    def weights(self, x, a):
        t, P = x / self.dx[a], self.p["order"]
        base = torch.floor(t.detach() + 0.5) if P == 2 else torch.floor(t.detach())
        d = t - base
        if P == 1:
            w, lo = [1 - d, d], base
        elif P == 2:
            w, lo = [0.5 * (0.5 - d) ** 2, 0.75 - d ** 2, 0.5 * (0.5 + d) ** 2], base - 1
        else:
            w = [(1 - d) ** 3 / 6, (4 - 6 * d ** 2 + 3 * d ** 3) / 6, (1 + 3 * d + 3 * d ** 2 - 3 * d ** 3) / 6, d ** 3 / 6]
            lo = base - 1
        step = (self.shape[1] * self.shape[2], self.shape[2], 1)[a]
        i = lo.to(torch.int64)
        return [(torch.remainder(i + n, self.shape[a]) * step, v) for n, v in enumerate(w)]

    def nodes(self, x):
        wx, wy, wz = (self.weights(x[a], a) for a in range(3))
        for ix, sx in wx:
            for iy, sy in wy:
                ixy, sxy = ix + iy, sx * sy
                for iz, sz in wz:
                    yield ixy + iz, sxy * sz

    def gather(self, F, x):
        out = [0.0] * len(F)
        for i, s in self.nodes(x):
            out = [o + s * f[i] for o, f in zip(out, F)]
        return out

    def deposit(self, x, values, into=None):
        n = self.shape[0] * self.shape[1] * self.shape[2]
        into = into or [torch.zeros(n, dtype=torch.float64, device="cuda") for _ in values]
        for i, s in self.nodes(x):
            for o, v in zip(into, values):
                o.index_add_(0, i, s * v)
        return into

    def push(self, f, u, k):
        dot = lambda a, b: a[0] * b[0] + a[1] * b[1] + a[2] * b[2]  # noqa: E731
        cross = lambda a, b: [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]  # noqa: E731
        E, B = f[:3], f[3:]
        if self.vay:
            g0 = torch.sqrt(1 + dot(u, u))
            v = [c / g0 for c in u]
            vb = cross(v, B)
            up = [u[c] + 2 * k * E[c] + k * vb[c] for c in range(3)]
            t = [k * b for b in B]
            t2, ut = dot(t, t), dot(up, t)
            b = t2 + ut ** 2
            s = 1 + dot(up, up) - t2
            R = torch.sqrt(s * s + 4 * b)
            g = torch.sqrt(torch.where(s >= 0, 0.5 * (s + R), 2 * b / (R - s).clamp_min(1e-300)))
            t = [c / g for c in t]
            ut, ct = dot(up, t), cross(up, t)
            return [(up[c] + ut * t[c] + ct[c]) / (1 + dot(t, t)) for c in range(3)]
        um = [u[c] + k * E[c] for c in range(3)]
        gm = torch.sqrt(1 + dot(um, um))
        t = [k * B[c] / gm for c in range(3)]
        s = [2 * c / (1 + dot(t, t)) for c in t]
        ct = cross(um, t)
        up = [um[c] + ct[c] for c in range(3)]
        cs = cross(up, s)
        return [um[c] + cs[c] + k * E[c] for c in range(3)]

    def particles(self, F, sp):
        """sp: [(x[3] unwrapped, u[3], w, q, m)] -> advanced species, nodal J, rho"""
        dV = self.dx[0] * self.dx[1] * self.dx[2]
        J = rho = None
        new = []
        for x, u, w, q, m in sp:
            f = self.gather(F, x)
            u = self.push(f, u, q * self.dt / (2 * m))
            g = torch.sqrt(1 + u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
            v = [c / g for c in u]
            qw = w * (q / dV)
            mid = [x[a] + 0.5 * self.dt * (v[a] - self.vg[a]) for a in range(3)]
            x = [x[a] + self.dt * (v[a] - self.vg[a]) for a in range(3)]
            J = self.deposit(mid, [qw * c for c in v], J)
            rho = self.deposit(x, [qw], rho)
            new.append((x, u, w, q, m))
        return new, J, rho[0]

    def rho0(self, sp):
        dV = self.dx[0] * self.dx[1] * self.dx[2]
        rho = None
        for x, _, w, q, _ in sp:
            rho = self.deposit(x, [w * (q / dV)], rho)
        return rho[0]

    def spectra(self, E, B):
        return [self.phase(self.fwd(f), _STAG[c]) for c, f in enumerate(list(E) + list(B))]

    def advance(self, E, B, rho, sp, steps):
        """Yee E, B, nodal rho^0 -> the same after the steps, with the last J (Yee)"""
        if self.p["cycle"] == "fdtd":
            return self.advance_fdtd(E, B, sp, steps)
        EB, rn = self.spectra(E, B), self.fwd(rho)
        F = self.nodal(EB)
        for s in range(steps):
            sp, J, rho = self.particles(F, sp)
            Jh = [self.smooth(self.fwd(J[a]) * self.zeta[a]) for a in range(3)]
            rp = self.fwd(rho)
            EB, G = self.solve(EB, Jh, self.smooth(rn), self.smooth(rp))
            rn = rp
            if s < steps - 1:
                F = self.nodal(G)
        out = [self.inv(self.phase(EB[c], _STAG[c], True)) for c in range(6)]
        J = [self.inv(self.phase(Jh[a], _STAG[a], True)) for a in range(3)]
        return out[:3], out[3:], J, rho, sp

    # the finite-difference cycle
    def center(self, f, stag, to_nodes):
        f = f.reshape(self.shape)
        for a in range(3):
            if stag[a]:
                m, o = self.p["center"][a] // 2, 0
                for n in range(1, m + 1):
                    d = 1 if to_nodes else 0
                    o = o + 0.5 * _alpha_s(m, n) * (torch.roll(f, -(n - d), a) + torch.roll(f, n - 1 + d, a))
                f = o
        return f.reshape(-1)

    def diff(self, f, a, half):
        o, d = 0, 0 if half else 1
        for n, w in enumerate(_fd_weights(self.p["spectral"][a] // 2), 1):
            o = o + w / self.dx[a] * (torch.roll(f, -(n - d), a) - torch.roll(f, n - 1 + d, a))
        return o

    def curl(self, f, half):
        return [self.diff(f[2], 1, half) - self.diff(f[1], 2, half), self.diff(f[0], 2, half) - self.diff(f[2], 0, half),
                self.diff(f[1], 0, half) - self.diff(f[0], 1, half)]

    def advance_fdtd(self, E, B, sp, steps):
        E, B = [f.reshape(self.shape) for f in E], [f.reshape(self.shape) for f in B]
        for _ in range(steps):
            F = [self.center(f, _STAG[c], True) for c, f in enumerate(E + B)]
            sp, J, rho = self.particles(F, sp)
            J = [self.center(J[a], _STAG[a], False) for a in range(3)]
            B = [b - 0.5 * self.dt * c for b, c in zip(B, self.curl(E, True))]
            E = [e + self.dt * (c - j.reshape(self.shape)) for e, c, j in zip(E, self.curl(B, False), J)]
            B = [b - 0.5 * self.dt * c for b, c in zip(B, self.curl(E, True))]
        return [f.reshape(-1) for f in E], [f.reshape(-1) for f in B], J, rho, sp


def exact(case, seed):
    kind = case["kind"]
    if kind == "transform":
        F = _waves(case, seed, 6)
        if case["form"] == "fp32":
            F = [f.float().double() for f in F]
        n = case["nx"] * case["ny"] * case["nz"]
        spec = [torch.view_as_real(torch.fft.fftn(torch.fft.rfft(f, dim=2), dim=(0, 1))).reshape(-1) for f in F]
        return {"spec": spec, "back": [f.reshape(-1) * n for f in F]}
    if kind == "solve":
        p = _params(case)
        x, F = _Exact(p), _waves(case, seed, 11)
        EB = x.spectra(F[0:3], F[3:6])
        J = [x.phase(x.fwd(F[6 + a]), _STAG[a]) for a in range(3)]
        EB, G = x.solve(EB, J, x.fwd(F[9]), x.fwd(F[10]))
        out, avg = [[x.inv(x.phase(H[c], _STAG[c], True)) for c in range(6)] for H in (EB, G)]
        return {"E": out[:3], "B": out[3:], "avg": avg if p["variant"] == "averaged" else []}
    p, E, B, sp = _state0(case, seed)
    if case["form"] == "fp32":  # the fields a program has in hand are FP32
        E, B = [f.float().double() for f in E], [f.float().double() for f in B]
    E, B = [f.reshape(-1) for f in E], [f.reshape(-1) for f in B]
    x = _Exact(p, case["filter"], case["pusher"] == "vay")
    sp = [(list(v[0:3]), list(v[3:6]), v[6], v[7], v[8]) for v in sp]
    if kind == "run":
        if case["steps"] * (_particles(case) * (case["order"] + 1) ** 3) > 3e10:
            return None
        with torch.no_grad():
            E1, B1, J, rho, new = x.advance(E, B, x.rho0(sp), sp, case["steps"])
        out = {"E": E1, "B": B1, "J": J, "rho": rho}
        for q, v in enumerate(new):
            out["u%d" % q] = v[1]
            out["x%d" % q] = v[0]
        return out
    if kind == "adjoint":
        f, q = _adjoints(case, seed, sp[0][0][0].numel())
        leaves = [t.detach().requires_grad_() for t in E + B + [x.rho0(sp)] + sp[0][0] + sp[0][1]]
        E1, B1, _, rho, new = x.advance(leaves[0:3], leaves[3:6], leaves[6],
                                        [(leaves[7:10], leaves[10:13], *sp[0][2:])], 1)
        g = torch.autograd.grad(E1 + B1 + [rho] + new[0][0] + new[0][1], leaves, [a.reshape(-1) for a in f] + q)
        return {"E": g[0:3], "B": g[3:6], "rho": g[6], "p": dict(zip(("x", "y", "z", "ux", "uy", "uz"), g[7:13]))}
    if case["steps"] * _particles(case) * (case["order"] + 1) ** 3 > 2e8:  # the graph would not fit
        return None
    leaves = [t.detach().requires_grad_() for t in E + B + sp[0][1]]
    E1, B1, _, _, _ = x.advance(leaves[0:3], leaves[3:6], x.rho0(sp), [(sp[0][0], leaves[6:9], *sp[0][2:])],
                                case["steps"])
    (lo, hi), dV = _probe(p["shape"]), p["dx"][0] * p["dx"][1] * p["dx"][2]
    loss = 0.0
    for c in E1 + B1:
        loss = loss + 0.5 * dV * (c.reshape(p["shape"])[lo[0]:hi[0], lo[1]:hi[1], lo[2]:hi[2]] ** 2).sum()
    g = torch.autograd.grad(loss, leaves)
    return {"loss": loss.detach(), "E": torch.stack(g[0:3]), "B": torch.stack(g[3:6]), "u": list(g[6:9])}
