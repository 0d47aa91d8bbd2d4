"""Precision of the deposits node by node: where the density falls off by orders of magnitude, and with amounts
that do, every node keeps the relative precision of its format, whatever its neighbours hold."""
import numpy as np
import pytest

from helpers import context_for, to_host
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
