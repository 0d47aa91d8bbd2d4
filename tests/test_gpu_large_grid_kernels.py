"""The kernels that only large grids or particular arrays reach, against the oracle: centering stencils
and finite differences from register windows (every order they are built for, the first order beyond,
arrays off the 16-byte boundary), the two sides of the k-space update's split, tiles with more particles
than the sort holds in shared memory, more tiles than its one-launch scan takes, and the widening of
FP32 values that are not normal numbers, the windowed deposit of rho, and the FP64 tiled push's chunks."""
import numpy as np
import pytest

from helpers import TOL, context_for, field_rel_err, species_to_dev, to_dev, to_host
from oracle import fdtd, grid, particles, step
from test_gpu_fp32 import _oracle_run, as_oracle_species, ctx32, dev32, momentum_errors, species32

pytestmark = pytest.mark.gpu

WINDOW = (64, 128, 128)      # 2^20 cells: the smallest grid whose centering takes the window kernels
BELOW = (64, 64, 128)        # one launch for all components


def _params(shape, **kw):
    p = dict(shape=shape, dx=(0.5, 0.7, 0.3), dt=0.1, shape_order=2, centering_order=(4, 4, 8), variant=0,
             v_gal=(0.0, 0.0, 0.0), spectral_order=(0, 0, 0), c=1.0, eps0=1.0)
    p.update(kw)
    return p


def _off(a, dtype, skip):
    """Device copy of a that starts skip elements past an aligned address."""
    import torch
    buf = torch.empty(a.size + skip, dtype=dtype, device="cuda")
    buf[skip:] = torch.from_numpy(np.ascontiguousarray(a).reshape(-1)).to(dtype).cuda()
    return buf[skip:]


@pytest.mark.parametrize("shape,corder,skip", [
    (WINDOW, (2, 6, 16), 0), (WINDOW, (4, 16, 14), 0), (WINDOW, (6, 12, 12), 0), (WINDOW, (8, 4, 10), 0),
    (WINDOW, (10, 2, 8), 0), (WINDOW, (12, 10, 6), 0), (WINDOW, (14, 8, 4), 0), (WINDOW, (16, 14, 2), 0),
    (WINDOW, (18, 4, 32), 0), (WINDOW, (4, 8, 16), 1), (BELOW, (2, 32, 16), 0), (BELOW, (8, 4, 6), 1),
    ((8, 1024, 128), (8, 16, 16), 0), ((1024, 64, 16), (16, 16, 16), 0)])
def test_centering_windows(shape, corder, skip):
    """Tolerance: a pass sums 2 m <= 32 terms whose weights sum to less than 1.95 in magnitude, so it adds at
    most (m + 1) 2^-53 1.95 max|f| with max|f| < 6; two passes, on both sides: 4 17 1.2e-16 1.95 6 1.95 = 1.9e-13."""
    import torch
    ctx = context_for(_params(shape, centering_order=corder))
    rng = np.random.default_rng(3)
    F = [rng.normal(size=shape) for _ in range(6)]
    out = [_off(np.zeros(ctx.ncell), torch.float64, skip) for _ in range(6)]
    ctx.center_to_nodal([_off(f, torch.float64, skip) for f in F], out)
    names = grid.E_NAMES + grid.B_NAMES
    for c in range(6):
        ref = grid.center_to_nodal(F[c], names[c], corder)
        np.testing.assert_allclose(to_host(out[c]).reshape(shape), ref, rtol=0, atol=1.9e-13)
    ctx.center_to_yee([_off(f, torch.float64, skip) for f in F[:3]], out[:3])
    for c in range(3):
        ref = grid.center_to_yee(F[c], grid.J_NAMES[c], corder)
        np.testing.assert_allclose(to_host(out[c]).reshape(shape), ref, rtol=0, atol=1.9e-13)


@pytest.mark.parametrize("shape,m", [((8, 8, 16), m) for m in range(1, 9)] + [((16, 32, 32), m) for m in range(1, 10)])
def test_finite_differences(shape, m):
    """One FDTD field step at every z order of the vector kernel and the first beyond, TOL as elsewhere."""
    dx = (0.5, 0.7, 0.3)
    orders = tuple(min(o, n) for o, n in zip((2 * (m % 8) + 2, 2 * ((m + 1) % 9) + 2, 2 * m), shape))
    p = _params(shape, dx=dx, spectral_order=orders, dt=0.8 * fdtd.courant_limit(orders, dx, 1.3), c=1.3, eps0=0.7)
    ctx = context_for(p, cycle=3)
    rng = np.random.default_rng(m)
    E, B, J = [[rng.normal(size=shape) for _ in range(3)] for _ in range(3)]
    dE, dB = [to_dev(a) for a in E], [to_dev(a) for a in B]
    ctx.maxwell_step(dE, dB, [to_dev(a) for a in J], None, None)
    rE, rB = fdtd.yee_update(E, B, J, p["dt"], orders, dx, 1.3, 0.7)
    assert field_rel_err([to_host(a).reshape(shape) for a in dE], rE) < TOL
    assert field_rel_err([to_host(a).reshape(shape) for a in dB], rB) < TOL


@pytest.mark.parametrize("cycle,corder,orders,skip", [
    (0, (2, 4, 16), (0, 0, 0), 0), (0, (6, 8, 10), (16, 8, 16), 0), (0, (18, 4, 4), (0, 0, 0), 2),
    (1, (4, 4, 4), (8, 8, 8), 0), (2, (4, 4, 4), (8, 8, 8), 0),
    (3, (4, 4, 16), (4, 4, 16), 0), (3, (2, 12, 14), (2, 8, 12), 0), (3, (8, 8, 8), (4, 4, 8), 2)])
def test_step32_on_a_large_grid(cycle, corder, orders, skip):
    """One FP32 call of one step: the fields it gathers, the J it returns (both centered in real space) and
    the new E and B, for every cycle.  FP32 rounding (2^-24) through at most 20 additions of terms of one
    size, and through transforms of 20 stages: 1e-5, the bound of the FP32 form."""
    import torch
    shape, dx = WINDOW, (0.5, 0.7, 0.3)
    dt = 0.8 * fdtd.courant_limit(tuple(o or 2 for o in orders), dx, 1.0) if cycle == 3 else 0.2
    p = _params(shape, centering_order=corder, spectral_order=orders, dt=dt)
    ctx = ctx32(p, cycle=cycle)
    rng = np.random.default_rng(cycle)
    n = 6000
    sp = [{k: rng.uniform(0, shape[a] * dx[a], n) for a, k in enumerate("xyz")}]
    sp[0].update({k: rng.normal(0, 0.3, n) for k in ("ux", "uy", "uz")}, w=rng.uniform(0.5, 1.5, n), q=-1.0, m=1.0)
    E, B = [[rng.normal(size=shape).astype(np.float32).astype(np.float64) for _ in range(3)] for _ in range(2)]
    d = species32(ctx, sp)
    op = step.Params(**p, cycle=cycle)
    st = _oracle_run(op, E, B, as_oracle_species(ctx, d), 1)
    dE, dB, J = [[_off(a, torch.float32, skip) for a in f] for f in (E, B, [np.zeros(shape)] * 3)]
    rho = torch.empty(ctx.ncell, dtype=torch.float32, device="cuda")
    ctx.deposit_rho32(d, rho)
    ctx.step32(dE, dB, J, rho, d, 1)
    ctx.sync()
    for got, ref in ((dE, st["E"]), (dB, st["B"]), (J, st["J"]), ([rho], [st["rho"]])):
        assert field_rel_err([to_host(a).astype(np.float64).reshape(shape) for a in got], ref) < 1e-5
    assert max(momentum_errors(as_oracle_species(ctx, d), st["species"])) < 1e-5


@pytest.mark.parametrize("shape", [(64, 64, 128), (64, 64, 256)])  # both sides of the split by grid size
@pytest.mark.parametrize("variant,v", [(0, (0.0, 0.0, 0.0)), (1, (0.0, 0.0, 0.99)), (2, (0.2, 0.1, -0.3))])
def test_update_split(shape, variant, v):
    import torch
    p = _params(shape, variant=variant, v_gal=v, spectral_order=(8, 16, 0), dt=0.25)
    ctx = context_for(p)
    rng = np.random.default_rng(17)
    E, B, J = [[rng.normal(size=shape) for _ in range(3)] for _ in range(3)]
    rn, rp = rng.normal(size=shape), rng.normal(size=shape)
    Eo, Bo, avg, _ = step.maxwell_update(step.Params(**p), E, B, J, rn, rp)
    Ed, Bd = [to_dev(a) for a in E], [to_dev(a) for a in B]
    av = [torch.empty(ctx.ncell, dtype=torch.float64, device="cuda") for _ in range(6)]
    ctx.maxwell_step(Ed, Bd, [to_dev(a) for a in J], to_dev(rn), to_dev(rp), av[:3] if variant == 2 else None,
                     av[3:] if variant == 2 else None)
    got = [(Ed, Eo), (Bd, Bo)] + ([(av[:3], avg[0]), (av[3:], avg[1])] if variant == 2 else [])
    for g, r in got:
        assert field_rel_err([to_host(a).reshape(shape) for a in g], r) < TOL


@pytest.mark.parametrize("shape,tile,n,crowd", [((16, 16, 32), (8, 8, 8), 1, 0), ((16, 16, 32), (8, 8, 8), 4095, 4095),
                                                ((16, 16, 32), (8, 8, 8), 9000, 4097),
                                                ((16, 16, 32), (8, 8, 8), 30000, 20000),
                                                ((16, 32, 32), (8, 16, 8), 30000, 20000),
                                                ((128, 128, 128), (2, 2, 2), 40000, 5000)])
def test_step32_sorts(shape, tile, n, crowd):
    """Two FP32 steps that sort before each, crowd of the particles in one tile: nothing lost or mixed up, and
    J, rho and the momenta as the oracle's within the FP32 form's 1e-5."""
    import torch
    p = _params(shape, shape_order=3)
    ctx = ctx32(p, tile=tile, sort_interval=1)
    rng = np.random.default_rng(n)
    sp = [{k: rng.uniform(0, shape[a] * p["dx"][a], n) for a, k in enumerate("xyz")}]
    for a, k in enumerate("xyz"):
        sp[0][k][:crowd] = rng.uniform(tile[a], 2 * tile[a], crowd) % shape[a] * p["dx"][a]
    sp[0].update({k: rng.normal(0, 0.5, n) for k in ("ux", "uy", "uz")}, w=rng.uniform(0.5, 1.5, n), q=-1e-3, m=1.0)
    d = species32(ctx, sp)
    w0 = to_host(d[0].w).copy()
    Z = [np.zeros(shape)] * 3
    st = _oracle_run(step.Params(**p), Z, Z, as_oracle_species(ctx, d), 2)
    E, B, J = [[dev32(a) for a in Z] for _ in range(3)]
    rho = torch.empty(ctx.ncell, dtype=torch.float32, device="cuda")
    ctx.deposit_rho32(d, rho)
    ctx.step32(E, B, J, rho, d, 2)
    ctx.sync()
    ids = to_host(d[0].id)
    np.testing.assert_array_equal(np.sort(ids), np.arange(n))
    np.testing.assert_array_equal(to_host(d[0].w), w0[ids])
    for got, ref in ((J, st["J"]), ([rho], [st["rho"]])):
        assert field_rel_err([to_host(a).astype(np.float64).reshape(shape) for a in got], ref) < 1e-5
    assert max(momentum_errors(as_oracle_species(ctx, d), st["species"])) < 1e-5


def test_widening_of_special_values():
    import torch
    from paper_2106_12919_gb300 import pic
    ctx = ctx32(_params((8, 8, 16)))
    tiny, big = np.float32(1e-45), np.finfo(np.float32).max
    v = np.array([0.0, -0.0, tiny, -tiny, 1e-39, -1.1754942e-38, 1.17549435e-38, big, -big, np.inf, -np.inf, np.nan,
                  1.0, -1.5, 2.0 ** -126, 3.0e-44], dtype=np.float32)
    z = torch.zeros(v.size, dtype=torch.float32, device="cuda")
    s32 = pic.Species32(torch.zeros(v.size, dtype=torch.int32, device="cuda"), z, z, z, dev32(v), dev32(-v),
                        dev32(v[::-1]), dev32(v), -1.0, 1.0)
    s = ctx.species32_to_species(s32)
    ctx.sync()
    for got, want in zip((s.ux, s.uy, s.uz, s.w), (v, -v, v[::-1], v)):
        got, want = to_host(got), want.astype(np.float64)
        np.testing.assert_array_equal(np.isnan(got), np.isnan(want))
        ok = ~np.isnan(want)
        np.testing.assert_array_equal(got[ok].view(np.int64), want[ok].view(np.int64))


def test_splitting_of_special_values():
    """FP64 -> FP32 on the bit patterns: ties, results that are subnormal, overflow or are not finite, offsets
    down to 2^-1074, positions outside the box; and back (offsets below 2^-20 included), bit for bit."""
    import torch
    from paper_2106_12919_gb300 import pic
    shape, dx = (8, 16, 1024), (1.0, 0.25, 0.04)
    ctx = ctx32(_params(shape, dx=dx))
    rng = np.random.default_rng(9)
    k = np.arange(4000)
    pos = [np.where(k % 4 == 0, (k % shape[a]) + 2.0 ** -(k % 70), np.where(
        k % 4 == 1, np.nextafter((k % shape[a]) + 1.0, 0.0), np.where(
            k % 4 == 2, 2.0 ** -(k * 0.27), (k % shape[a]) + (2 * (k % 512) + 1) * 2.0 ** -25))) * dx[a] for a in range(3)]
    pos = [np.clip(v, 0.0, np.nextafter(shape[a] * dx[a], 0.0)) for a, v in enumerate(pos)]
    u = rng.normal(size=k.size) * 10.0 ** rng.uniform(-46, 39, k.size)
    u[:500] = (1.0 + k[:500] * 2.0 ** -24) * 2.0 ** (k[:500] % 250 - 125.0)
    u[500:512] = [0.0, -0.0, np.inf, -np.inf, np.nan, 1e300, -1e300, 1e-300, 2.0 ** -150, 3.4028235677973366e38, 1e-45, 5e-324]
    dev = [to_dev(v) for v in (*pos, u, -u, u[::-1], u)]
    s = pic.Species32.from_positions(ctx, *dev, -1.0, 1.0)
    ctx.sync()
    ref = [particles.cell_offset_split(v, dx[a], shape[a]) for a, v in enumerate(pos)]
    np.testing.assert_array_equal(to_host(s.cell), particles.linear_cell(ref[0][0], ref[1][0], ref[2][0], shape))
    with np.errstate(all="ignore"):
        want32 = [v.astype(np.float32) for v in (u, -u, u[::-1], u)]
    for got, want in zip((s.fx, s.fy, s.fz, s.ux, s.uy, s.uz, s.w), [r[1] for r in ref] + want32):
        got = to_host(got)
        ok = ~np.isnan(want)
        np.testing.assert_array_equal(np.isnan(got), ~ok)
        np.testing.assert_array_equal(got[ok].view(np.uint32), want[ok].view(np.uint32))
    b = ctx.species32_to_species(s)
    ctx.sync()
    for a, got in enumerate((b.x, b.y, b.z)):
        np.testing.assert_array_equal(to_host(got), particles.cell_offset_join(ref[a][0], ref[a][1], dx[a]))
    # outside the box: the cell wraps, the offset is that of the position
    far = [np.array([-0.3, -17.6, 1e9 + 0.5, 3e12, -0.0]) * dx[a] for a in range(3)]
    z = to_dev(np.zeros(5))
    s = pic.Species32.from_positions(ctx, *[to_dev(v) for v in far], z, z, z, z, -1.0, 1.0)
    ctx.sync()
    for a, got in enumerate((s.fx, s.fy, s.fz)):
        t = far[a] * (1.0 / dx[a])
        f = (t - np.floor(t)).astype(np.float32)
        np.testing.assert_array_equal(to_host(got), np.where(f == 1.0, np.float32(0.0), f))


@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("kind", ["sorted", "random", "faces", "peak", "spread", "ramp", "inf"])
def test_deposit_rho32_windows(order, kind):
    """rho of enough particles for the windowed deposit: chunks it sums itself, and the ones it leaves to the
    per-particle path (random order, a full cell among empty ones, amounts orders apart, an infinite one).
    FP32 weights (four roundings) and sums: 2e-6, the bound of the FP32 deposit."""
    import torch
    from paper_2106_12919_gb300 import pic
    shape, n = (32, 64, 128), 700001
    p = _params(shape, shape_order=order)
    ctx = ctx32(p)
    rng = np.random.default_rng(order)
    cell = rng.integers(0, ctx.ncell, n)
    if kind != "random":
        cell = np.sort(cell)
    if kind == "peak":
        cell[:1500] = 77
    f = [rng.random(n, dtype=np.float32) for _ in range(3)]
    if kind == "faces":
        for a in range(3):
            f[a][a::5] = (0.0, -0.0, 0.5)[a]
            f[a][a + 1::7] = np.nextafter(np.float32(1), np.float32(0))
    w = rng.uniform(0.5, 1.5, n).astype(np.float32)
    if kind == "spread":
        w *= (10.0 ** rng.uniform(-6, 0, n)).astype(np.float32)
    if kind == "ramp":
        w = ((cell % shape[2]) / shape[2]).astype(np.float32)
    if kind == "inf":
        w[n // 2] = np.inf
    u = torch.zeros(n, dtype=torch.float32, device="cuda")
    s = pic.Species32(torch.from_numpy(cell.astype(np.int32)).cuda(), *[dev32(v) for v in f], u, u, u, dev32(w), -1.0, 1.0)
    rho = torch.empty(ctx.ncell, dtype=torch.float32, device="cuda")
    ctx.deposit_rho32([s], rho)
    ctx.sync()
    got = to_host(rho).astype(np.float64).reshape(shape)
    ix, iy, iz = cell // (shape[1] * shape[2]), cell // shape[2] % shape[1], cell % shape[2]
    sp = {k: (i + g.astype(np.float64)) * p["dx"][a] for a, (k, i, g) in enumerate(zip("xyz", (ix, iy, iz), f))}
    sp.update(w=w.astype(np.float64), q=-1.0, m=1.0)
    if kind == "inf":  # the nodes around that particle, and no others
        assert 1 <= np.count_nonzero(~np.isfinite(got)) <= (order + 1) ** 3
        sp["w"][n // 2] = 0.0
        ok = np.isfinite(got)
        got[~ok] = 0.0
        ref = particles.deposit_rho(sp, shape, p["dx"], order) * ok
    else:
        ref = particles.deposit_rho(sp, shape, p["dx"], order)
    assert field_rel_err([got], [ref]) < 2e-6


@pytest.mark.parametrize("n", [255, 256, 257, 513, 400000, 1300001])
def test_tiled64_chunk_sizes(n):
    """FP64 tiled push with chunks from 256 to 2048 particles (a rule on the count), a quarter of them in one tile."""
    import torch
    shape, dx = (8, 16, 32), (0.5, 1.0, 0.25)
    p = _params(shape, dx=dx)
    ctx = context_for(p, sort_interval=0)
    rng = np.random.default_rng(n)
    s = {k: rng.uniform(0, shape[a] * dx[a], n) for a, k in enumerate("xyz")}
    for a, k in enumerate("xyz"):
        s[k][:n - n // 4 if n < 1000 else n // 4] *= (1.0, 0.5, 0.25)[a]
    s.update({k: rng.normal(0, 0.3, n) for k in ("ux", "uy", "uz")}, w=rng.uniform(0.5, 1.5, n), q=-1.0, m=1.0)
    F = [rng.normal(size=shape) for _ in range(6)]
    ref, Jref, rho_ref = particles.push_and_deposit(s, F[:3], F[3:], shape, dx, p["dt"], 2, p["v_gal"])
    (d,) = species_to_dev([s])
    Jd = [torch.empty(ctx.ncell, dtype=torch.float64, device="cuda") for _ in range(3)]
    rd = torch.empty(ctx.ncell, dtype=torch.float64, device="cuda")
    ctx.push_deposit([to_dev(f) for f in F[:3]], [to_dev(f) for f in F[3:]], [d], Jd, rd)
    ctx.sync()
    assert field_rel_err([to_host(a).reshape(shape) for a in Jd], Jref) < TOL
    assert field_rel_err([to_host(rd).reshape(shape)], [rho_ref]) < TOL
    order = np.argsort(to_host(d.id))
    for k in ("ux", "uy", "uz"):
        assert np.max(np.abs(to_host(getattr(d, k))[order] - ref[k])) < 1e-12 * np.max(np.abs(ref[k]))


@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("kind", ["below", "first", "sorted", "faces", "spread", "outside", "inf"])
def test_deposit_rho_tiled64(order, kind):
    """FP64 rho by itself, on both sides of the count from which it is summed per tile, against the oracle."""
    import torch
    shape, dx = (16, 16, 32), (0.5, 1.0, 0.25)
    ctx = context_for(_params(shape, dx=dx, shape_order=order))
    rng = np.random.default_rng(order)
    n = 2 ** 18 - 1 if kind == "below" else 2 ** 18 if kind == "first" else 300007
    s = {k: rng.uniform(0, shape[a] * dx[a], n) for a, k in enumerate("xyz")}
    s.update({k: np.zeros(n) for k in ("ux", "uy", "uz")}, w=rng.uniform(0.5, 1.5, n), q=-1.0, m=1.0)
    if kind == "sorted":
        s["x"].sort()
    elif kind == "faces":
        for a, k in enumerate("xyz"):
            s[k][a::3] = rng.integers(0, shape[a], s[k][a::3].size) * dx[a]
            s[k][:50], s[k][50:100] = np.nextafter(shape[a] * dx[a], 0.0), 0.5 * dx[a]
    elif kind == "spread":
        s["w"] *= 10.0 ** rng.uniform(-8, 0, n)
    elif kind == "outside":
        for a, k in enumerate("xyz"):
            s[k][:500] += shape[a] * dx[a] * rng.integers(-1, 2, 500)
    elif kind == "inf":
        s["w"][n // 2] = np.inf
    (d,) = species_to_dev([s])
    rho = torch.empty(ctx.ncell, dtype=torch.float64, device="cuda")
    ctx.deposit_rho([d], rho)
    ctx.sync()
    got = to_host(rho).reshape(shape)
    ok = np.isfinite(got)
    assert np.count_nonzero(~ok) <= ((order + 1) ** 3 if kind == "inf" else 0) and (kind == "inf") == (not ok.all())
    if kind == "inf":
        s["w"][n // 2] = 0.0
    ref = particles.deposit_rho(s, shape, dx, order)
    assert field_rel_err([np.where(ok, got, 0.0)], [ref * ok]) < TOL
