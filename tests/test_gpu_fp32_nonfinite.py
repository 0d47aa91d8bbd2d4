"""FP32 tiled push with a few non-finite particles: they deposit nothing, and the J and rho of all others
are the oracle's."""
import numpy as np
import pytest

from helpers import field_rel_err, to_host
from oracle import step
from test_gpu_fp32 import _oracle_run, as_oracle_species, ctx32, dev32, species32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("vz", [0.0, 0.9])  # 0.9: the tiles follow the plasma, J over one z node more
def test_nonfinite_particles_deposit_nothing(order, vz):
    """Two calls of one step (the second starts with the NaN momenta of the first).  J and rho within the FP32
    form's 1e-5 of a run without those particles."""
    import torch
    shape, dx, n = (16, 16, 32), (0.5, 0.7, 0.3), 6000
    p = dict(shape=shape, dx=dx, dt=0.3, shape_order=order, centering_order=(4, 4, 8), variant=1 if vz else 0,
             v_gal=(0.0, 0.0, vz), spectral_order=(0, 0, 0), c=1.0, eps0=1.0)
    ctx = ctx32(p)
    rng = np.random.default_rng(order)
    s = {k: rng.uniform(0, shape[a] * dx[a], n) for a, k in enumerate("xyz")}
    s.update({k: rng.normal(0, 0.02, n) for k in ("ux", "uy", "uz")}, w=rng.uniform(0.5, 1.5, n), q=-1e-3, m=1.0)
    s["ux"][5], s["uy"][17], s["uz"][18], s["w"][23] = np.nan, np.inf, -np.inf, np.inf
    d = species32(ctx, [s])
    bad = [5, 17, 18, 23]
    ok = as_oracle_species(ctx, d)
    for k in ("x", "y", "z", "ux", "uy", "uz", "w"):
        ok[0][k] = np.delete(ok[0][k], bad)
    Z = [np.zeros(shape)] * 3
    st = _oracle_run(step.Params(**p), Z, Z, ok, 2)
    E, B, J = [[dev32(a) for a in Z] for _ in range(3)]
    rho = torch.empty(ctx.ncell, dtype=torch.float32, device="cuda")
    ctx.deposit_rho32(species32(ctx, [{k: np.delete(v, bad) if isinstance(v, np.ndarray) else v for k, v in s.items()}]),
                      rho)
    for _ in range(2):
        ctx.step32(E, B, J, rho, d, 1)
    ctx.sync()
    for got, ref in ((J, st["J"]), ([rho], [st["rho"]])):
        assert field_rel_err([to_host(a).astype(np.float64).reshape(shape) for a in got], ref) < 1e-5
