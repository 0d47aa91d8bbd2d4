"""Tiled FP64 push (integer node sums) against the oracle at the edges of its range: chunks of a tile
at and around their limits, positions on cell faces and at the ends of the box, moves past the deposit
window, amounts spread over orders of magnitude, positions outside the box, a grid one tile wide, and
non-finite fields."""
import numpy as np
import pytest

from helpers import TOL, context_for, field_rel_err, species_from_dev, species_to_dev, to_dev, to_host
from oracle import particles

pytestmark = pytest.mark.gpu

SHAPE, DX, DT = (8, 16, 32), (0.5, 1.0, 0.25), 0.2
L = [SHAPE[a] * DX[a] for a in range(3)]


def _species(rng, n, lo=(0.0, 0.0, 0.0), hi=L, u=0.3):
    return {"x": rng.uniform(lo[0], hi[0], n), "y": rng.uniform(lo[1], hi[1], n), "z": rng.uniform(lo[2], hi[2], n),
            "ux": rng.normal(0, u, n), "uy": rng.normal(0, u, n), "uz": rng.normal(0, u, n),
            "w": rng.uniform(0.5, 1.5, n), "q": -1.0, "m": 1.0}


def _case(kind, rng):
    if kind.startswith("tile"):  # all particles in tile (0, 1, 2), a few spread ones beside them
        n = int(kind[4:])
        s = _species(rng, n, (0.0, 8 * DX[1], 16 * DX[2]), (8 * DX[0], 16 * DX[1], 24 * DX[2]))
        more = _species(rng, 40)
        return {k: (np.concatenate([s[k], more[k]]) if isinstance(s[k], np.ndarray) else s[k]) for k in s}, DT
    s = _species(rng, 3000)
    if kind == "faces":
        for a, k in enumerate("xyz"):
            s[k][:1000] = rng.integers(0, SHAPE[a], 1000) * DX[a]
            s[k][1000:1500] = (rng.integers(0, SHAPE[a], 500) + 0.5) * DX[a]
            s[k][1500:1600] = np.nextafter(L[a], 0.0)
            s[k][1600:1700] = 0.0
            s[k][1700:1800] = 1e-300
    elif kind == "fast":
        return s, 6.0 * DT
    elif kind == "uneven":
        fast = rng.random(3000) < 0.01
        for k in ("ux", "uy", "uz"):
            s[k] = s[k] * np.where(fast, 10.0, 1e-5)
        s["w"] = s["w"] * 10.0 ** rng.uniform(-6, 0, 3000)
    elif kind == "outside":
        for a, k in enumerate("xyz"):
            s[k][:200] += L[a] * rng.integers(-1, 2, 200)
    return s, DT


@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("kind", ["tile15", "tile16", "tile2048", "tile2049", "tile4097", "faces", "fast", "uneven",
                                  "outside", "nan"])
def test_push_deposit(order, kind):
    import torch
    rng = np.random.default_rng(order)
    s, dt = _case(kind, rng)
    p = dict(shape=SHAPE, dx=DX, dt=dt, shape_order=order, centering_order=(4, 4, 4), variant=1,
             v_gal=(0.0, 0.1, 0.4), spectral_order=(0, 0, 0), c=1.0, eps0=1.0)
    ctx = context_for(p, sort_interval=0)
    F = [rng.normal(size=SHAPE) for _ in range(6)]
    if kind == "nan":
        F[1][3, 5, 20] = np.nan
        F[4][7, 15, 31] = np.inf
    with np.errstate(all="ignore"):
        ref, Jref, rho_ref = particles.push_and_deposit(s, F[:3], F[3:], SHAPE, DX, dt, order, p["v_gal"])
    dsp = species_to_dev([s])
    Jd = [torch.empty(ctx.ncell, dtype=torch.float64, device="cuda") for _ in range(3)]
    rd = torch.empty(ctx.ncell, dtype=torch.float64, device="cuda")
    ctx.push_deposit([to_dev(f) for f in F[:3]], [to_dev(f) for f in F[3:]], dsp, Jd, rd)
    ctx.sync()
    got = species_from_dev(dsp)[0]
    if kind == "nan":  # the particles that do not see the non-finite nodes, and only those, are unharmed
        for k in ("ux", "uy", "uz"):
            ok = np.isfinite(ref[k])
            assert 0 < np.count_nonzero(~ok) < ok.size
            np.testing.assert_array_equal(np.isfinite(got[k]), ok)
            assert np.max(np.abs(got[k][ok] - ref[k][ok])) < 1e-12 * np.max(np.abs(ref[k][ok]))
        return
    assert field_rel_err([to_host(a).reshape(SHAPE) for a in Jd], Jref) < TOL
    assert field_rel_err([to_host(rd).reshape(SHAPE)], [rho_ref]) < TOL
    for a, k in enumerate("xyz"):
        assert np.max(np.abs(got[k] - ref[k])) < 1e-12 * L[a]
    for k in ("ux", "uy", "uz"):
        assert np.max(np.abs(got[k] - ref[k])) < 1e-12 * np.max(np.abs(ref[k]))
