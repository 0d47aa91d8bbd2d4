"""FP32 contexts with tiles of more than 4096 cells: pic_bin32 sorts them over the whole grid, pic_step32 runs
without tiles."""
import numpy as np
import pytest

from helpers import field_rel_err, to_host
from oracle import step
from test_gpu_fp32 import _oracle_run, as_oracle_species, ctx32, dev32, species32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("tile", [(16, 16, 32), (32, 32, 64)])
def test_large_tiles(order, tile):
    import torch
    shape, dx = (32, 32, 64), (0.5, 0.7, 0.3)
    p = dict(shape=shape, dx=dx, dt=0.1, shape_order=order, centering_order=(4, 4, 8), variant=0,
             v_gal=(0.0, 0.0, 0.0), spectral_order=(0, 0, 0), c=1.0, eps0=1.0)
    ctx = ctx32(p, tile=tile)
    rng = np.random.default_rng(order)
    for n in (1, 3000, 500, 9000):
        s = {k: rng.uniform(0, shape[a] * dx[a], n) for a, k in enumerate("xyz")}
        s.update({k: rng.normal(0, 0.3, n) for k in ("ux", "uy", "uz")}, w=rng.uniform(0.5, 1.5, n), q=-1e-3, m=1.0)
        (d,) = species32(ctx, [s])
        cell = to_host(d.cell).astype(np.int64)
        c = cell // (shape[1] * shape[2]), cell // shape[2] % shape[1], cell % shape[2]
        nt = [shape[a] // tile[a] for a in range(3)]
        tid = (c[0] // tile[0] * nt[1] + c[1] // tile[1]) * nt[2] + c[2] // tile[2]
        key = tid * np.prod(tile) + (c[1] % tile[1] * tile[0] + c[0] % tile[0]) * tile[2] + c[2] % tile[2]
        off = torch.empty(ctx.num_tiles() + 1, dtype=torch.int64, device="cuda")
        for _ in range(2):  # the second leaves it as it is
            ctx.bin32(d, off)
            ctx.sync()
            np.testing.assert_array_equal(to_host(off), np.concatenate([[0], np.cumsum(np.bincount(tid, minlength=nt[0] * nt[1] * nt[2]))]))
            ids = to_host(d.id)
            np.testing.assert_array_equal(np.sort(ids), np.arange(n))
            np.testing.assert_array_equal(to_host(d.cell), cell[ids])
            assert np.all(np.diff(key[ids]) >= 0)
        # a step: J and rho within the FP32 form's 1e-5 of the oracle's
        Z = [np.zeros(shape)] * 3
        st = _oracle_run(step.Params(**p), Z, Z, as_oracle_species(ctx, [d]), 1)
        E, B, J = [[dev32(a) for a in Z] for _ in range(3)]
        rho = torch.empty(ctx.ncell, dtype=torch.float32, device="cuda")
        ctx.deposit_rho32([d], rho)
        ctx.step32(E, B, J, rho, [d], 1)
        ctx.sync()
        for got, ref in ((J, st["J"]), ([rho], [st["rho"]])):
            assert field_rel_err([to_host(a).astype(np.float64).reshape(shape) for a in got], ref) < 1e-5
