"""Scratch that a context keeps between calls and enlarges: calls with more species or particles than the
ones before, each against the oracle."""
import numpy as np
import pytest

from helpers import field_rel_err, to_host
from oracle import step
from test_gpu_fp32 import _oracle_run, as_oracle_species, ctx32, dev32, species32

pytestmark = pytest.mark.gpu


def _params(shape, **kw):
    p = dict(shape=shape, dx=(0.5, 0.7, 0.3), dt=0.1, shape_order=2, centering_order=(4, 4, 8), variant=0,
             v_gal=(0.0, 0.0, 0.0), spectral_order=(0, 0, 0), c=1.0, eps0=1.0)
    p.update(kw)
    return p


def _species(rng, p, n):
    s = {k: rng.uniform(0, p["shape"][a] * p["dx"][a], n) for a, k in enumerate("xyz")}
    s.update({k: rng.normal(0, 0.3, n) for k in ("ux", "uy", "uz")}, w=rng.uniform(0.5, 1.5, n), q=-1e-3, m=1.0)
    return s


@pytest.mark.parametrize("shape,tile,counts", [((16, 16, 32), (8, 8, 8), (1, 3, 2, 8, 9)),
                                               ((128, 128, 128), (2, 2, 2), (1, 3))])  # 16 and 2^18 tiles
def test_step32_with_more_species(shape, tile, counts):
    """FP32 calls of different numbers of species on one context (its counts are kept, and cleared by every
    binning; of 9 species one is not binned); J and rho within the FP32 form's 1e-5."""
    import torch
    p = _params(shape)
    ctx = ctx32(p, tile=tile)
    rng = np.random.default_rng(4)
    Z = [np.zeros(shape)] * 3
    for nsp in counts:
        d = species32(ctx, [_species(rng, p, int(n)) for n in rng.integers(1, 3000, nsp)])
        st = _oracle_run(step.Params(**p), Z, Z, as_oracle_species(ctx, d), 1)
        E, B, J = [[dev32(a) for a in Z] for _ in range(3)]
        rho = torch.empty(ctx.ncell, dtype=torch.float32, device="cuda")
        ctx.deposit_rho32(d, rho)
        ctx.step32(E, B, J, rho, d, 1)
        ctx.sync()
        for got, ref in ((J, st["J"]), ([rho], [st["rho"]])):
            assert field_rel_err([to_host(a).astype(np.float64).reshape(shape) for a in got], ref) < 1e-5
