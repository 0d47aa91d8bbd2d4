"""Precision of the deposits node by node: where the density falls off by orders of magnitude, and with amounts
that do, every node keeps the relative precision of its format, whatever its neighbours hold."""
import numpy as np
import pytest

from helpers import context_for, species_from_dev, species_to_dev, to_dev, to_host
from oracle import particles

pytestmark = pytest.mark.gpu

DX = (0.5, 1.0, 0.25)  # powers of two: x / dx is exact


def _params(shape, order):
    return dict(shape=shape, dx=DX, dt=0.05, shape_order=order, centering_order=(4, 4, 4), variant=0,
                v_gal=(0.0, 0.0, 0.0), spectral_order=(0, 0, 0), c=1.0, eps0=1.0)


@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("kind", ["even", "holes", "amounts"])
def test_rho32(order, kind):
    """A node that sums c contributions of one sign, each of at most 8 roundings, is off by at most
    (c + 8) 2^-24 of itself."""
    import torch
    from paper_2106_12919_gb300 import pic
    shape, n = (32, 32, 64), 700001
    ctx = context_for(_params(shape, order), precision=pic.PIC_FP32)
    rng = np.random.default_rng(order)
    cell = np.sort(rng.integers(0, ctx.ncell, n))
    if kind == "holes":
        cell = np.sort(np.where(rng.random(n) < 0.98, cell // 64 * 64 + cell % 16, cell))
    f = [rng.random(n, dtype=np.float32) for _ in range(3)]
    w = rng.uniform(0.5, 1.5, n).astype(np.float32)
    if kind == "amounts":
        w *= np.where(rng.random(n) < 0.05, 1.0, 1 / 15.0).astype(np.float32)
    dev = lambda a: torch.from_numpy(a).cuda()
    u = torch.zeros(n, dtype=torch.float32, device="cuda")
    s = pic.Species32(dev(cell.astype(np.int32)), *map(dev, f), u, u, u, dev(w), 1.0, 1.0)
    rho = torch.empty(ctx.ncell, dtype=torch.float32, device="cuda")
    ctx.deposit_rho32([s], rho)
    ctx.sync()
    ijk = cell // (shape[1] * shape[2]), cell // shape[2] % shape[1], cell % shape[2]
    sp = {k: (ijk[a] + f[a].astype(np.float64)) * DX[a] for a, k in enumerate("xyz")}
    ref = particles.deposit_rho(dict(sp, w=w.astype(np.float64), q=1.0, m=1.0), shape, DX, order)
    # the number of contributions of every node
    base = [particles.shape_weights(sp[k], 1.0 / DX[a], order)[0] for a, k in enumerate("xyz")]
    count = np.zeros(shape)
    for o in np.ndindex(*[order + 1] * 3):
        np.add.at(count, tuple((base[a] + o[a]) % shape[a] for a in range(3)), 1)
    err = np.abs(to_host(rho).astype(np.float64).reshape(shape) - ref)
    assert np.all(err <= (count + 8) * 2.0 ** -24 * ref)


def _weights(t, order):
    """First node, weights and magnitudes of their derivatives at t = x / dx, in long double."""
    LD = np.longdouble
    b = np.floor(t + LD(0.5)) if order == 2 else np.floor(t)
    d = t - b
    if order == 2:
        a, c = LD(0.5) - d, LD(0.5) + d
        w, g = [a * a / 2, LD(0.75) - d * d, c * c / 2], [a, 2 * np.abs(d), c]
    else:
        e = 1 - d
        w = [e ** 3 / 6, (4 - 6 * d * d + 3 * d ** 3) / 6, (4 - 6 * e * e + 3 * e ** 3) / 6, d ** 3 / 6]
        g = [e * e / 2, d * (2 - d * LD(1.5)), e * (2 - e * LD(1.5)), d * d / 2]
    return b.astype(np.int64) - 1, w, g


def _nodes(pos, shape, order):
    """Per node of the particles' blocks: its index, its weight and the weight's change per cell of error."""
    lo, w, g = zip(*[_weights(pos[a].astype(np.longdouble) / np.longdouble(DX[a]), order) for a in range(3)])
    for i, j, k in np.ndindex(*[order + 1] * 3):
        ix = tuple((lo[a] + n) % shape[a] for a, n in enumerate((i, j, k)))
        yield ix, w[0][i] * w[1][j] * w[2][k], (g[0][i] * w[1][j] * w[2][k] + w[0][i] * g[1][j] * w[2][k]
                                               + w[0][i] * w[1][j] * g[2][k]).astype(np.float64)


def _deposit_bound(got, pos, amount, shape, order, ulp):
    """|got - exact|, and its bound: c contributions of amounts and weights of a few roundings each, summed in
    FP64, (8 c + 64) 2^-53 of sum |contribution|; and positions known to ulp cells."""
    ref, mag, amb, count = np.zeros(shape, np.longdouble), np.zeros(shape), np.zeros(shape), np.zeros(shape)
    for ix, w, g in _nodes(pos, shape, order):
        np.add.at(ref, ix, w * amount)
        np.add.at(mag, ix, np.abs(w * amount).astype(np.float64))
        np.add.at(amb, ix, g * np.abs(amount).astype(np.float64) * ulp)
        np.add.at(count, ix, 1)
    return np.abs((got.astype(np.longdouble) - ref).astype(np.float64)), (8 * count + 64) * 2.0 ** -53 * mag + amb


@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("kind", ["even", "fields", "amounts", "bunch", "sparse"])
def test_fp64_push(order, kind):
    """FP64 push and deposits: fields and amounts that fall by 10^10 over the 8 cells of a tile, a bunch with
    its tails.  A gathered component is off by at most 128 2^-53 of A = sum w |F| (64 terms, their weights of a few
    roundings each)."""
    import torch
    shape, n = (16, 16, 32), 4000 if kind == "sparse" else 24000
    ctx = context_for(_params(shape, order), sort_interval=0)
    rng = np.random.default_rng(order)
    L = [shape[a] * DX[a] for a in range(3)]
    x = [rng.uniform(0, L[a], n) for a in range(3)]
    if kind == "bunch":
        x = [np.mod(L[a] / 2 + rng.normal(0, 1.2 * DX[a], n), L[a]) for a in range(3)]
    fall = lambda z: 10.0 ** (-10 * (z % 8) / 8)
    w = rng.uniform(0.5, 1.5, n) * (fall(x[2] / DX[2]) if kind == "amounts" else 1.0)
    F = [rng.normal(size=shape) * (fall(np.arange(shape[2])) if kind in ("fields", "amounts") else 1.0) for _ in range(3)]
    s = dict(x=x[0], y=x[1], z=x[2], ux=np.zeros(n), uy=np.zeros(n), uz=np.zeros(n), w=w, q=-1.0, m=1.0)
    (d,) = species_to_dev([s])
    E, Z = [to_dev(f) for f in F], to_dev(np.zeros(shape))
    J, rho = [torch.empty(ctx.ncell, dtype=torch.float64, device="cuda") for _ in range(3)], torch.empty_like(Z)
    ctx.push_deposit(E, [Z, Z, Z], [d], J, rho)
    ctx.sync()
    new = species_from_dev([d])[0]
    u = [new[k] for k in ("ux", "uy", "uz")]
    f, A = [np.zeros(n, np.longdouble) for _ in F], [np.zeros(n) for _ in F]
    for ix, weight, _ in _nodes(x, shape, order):
        for c in range(3):
            v = weight * F[c][ix]
            f[c] += v
            A[c] += np.abs(v).astype(np.float64)
    dt = 0.05
    for c in range(3):  # u = 2 (q dt / 2 m) E
        assert np.all(np.abs((u[c].astype(np.longdouble) + f[c] * np.longdouble(dt)).astype(np.float64))
                      <= 128 * 2.0 ** -53 * dt * A[c])
    v = [a / np.sqrt(1 + sum(b.astype(np.longdouble) ** 2 for b in u)) for a in u]
    mid = [np.mod(x[a] + 0.5 * (dt * v[a].astype(np.float64)), L[a]) for a in range(3)]
    qw = -w.astype(np.longdouble) / np.longdouble(DX[0] * DX[1] * DX[2])
    for c in range(3):
        err, bound = _deposit_bound(to_host(J[c]).reshape(shape), mid, qw * v[c], shape, order,
                                    max(np.spacing(L[a]) / DX[a] for a in range(3)))
        assert np.all(err <= bound)
    err, bound = _deposit_bound(to_host(rho).reshape(shape), [new[k] for k in "xyz"], qw, shape, order, 0.0)
    assert np.all(err <= bound)


@pytest.mark.parametrize("kind", ["even", "amounts", "bunch"])
def test_fp64_rho(kind):
    """rho by itself: the bound of the push's rho."""
    import torch
    shape, n = (8, 16, 16), 2 ** 18 + 1
    ctx = context_for(_params(shape, 3))
    rng = np.random.default_rng(3)
    L = [shape[a] * DX[a] for a in range(3)]
    x = [rng.uniform(0, L[a], n) for a in range(3)]
    if kind == "bunch":
        x = [np.mod(L[a] / 2 + rng.normal(0, DX[a], n), L[a]) for a in range(3)]
    w = rng.uniform(0.5, 1.5, n) * (10.0 ** (-10 * (x[2] / DX[2] % 8) / 8) if kind == "amounts" else 1.0)
    z = np.zeros(n)
    (d,) = species_to_dev([dict(x=x[0], y=x[1], z=x[2], ux=z, uy=z, uz=z, w=w, q=-1.0, m=1.0)])
    rho = torch.empty(ctx.ncell, dtype=torch.float64, device="cuda")
    ctx.deposit_rho([d], rho)
    ctx.sync()
    qw = -w.astype(np.longdouble) / np.longdouble(DX[0] * DX[1] * DX[2])
    err, bound = _deposit_bound(to_host(rho).reshape(shape), x, qw, shape, 3, 0.0)
    assert np.all(err <= bound)
