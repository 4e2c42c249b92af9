"""FP64 gather deposit in fixed point against the FP64 oracle's grids.

A contribution is off by a few units of 2^-61 of the field's largest value (weights of 62
bits, three products), so a node that takes k of them is off by less than 8 k 2^-61 of it;
the oracle's own FP64 sums by about k 2^-53 of the largest partial sum. The bound below,
1e-14 of the largest node per 100 particles of the fullest node's reach, covers both.
"""
import numpy as np
import pytest

from oracle import estimator as est
from paper_2005_06170_gb300 import catalogs

pytestmark = pytest.mark.gpu


def _grids(pk, pos, vel, mass, L, ng, order):
    import torch
    ctx = pk.Context(0)
    p = pk.params(L, ng, 4, order=order, precision=pk.F64)
    dev = [torch.from_numpy(a).cuda() if a is not None else None for a in (pos, vel, mass)]
    grids = torch.empty((4, ng, ng, ng + 2), dtype=torch.float64, device="cuda")
    mom = torch.zeros(16, dtype=torch.float64, device="cuda")
    scratch = torch.empty(ctx.scratch_bytes_tuned(p, len(pos)), dtype=torch.uint8, device="cuda")
    ctx.assign(pk.catalog_from_tensors(*dev), p, grids, mom, scratch)
    ctx.sync()
    out = grids[..., :ng].cpu().numpy()
    ctx.close()
    return out


# 24^3: 8^3 tiles; 32^3 and 48^3: 8 x 8 x 16; 16^3: the reach of order 5 spans 13 x 13 x 21
# cells and wraps onto itself (FP64 atomics); 30000 in one cell: carries and a reduced scale
@pytest.mark.parametrize("order", [2, 3, 4, 5])
@pytest.mark.parametrize("ng,n,kind", [(24, 3000, "uniform"), (32, 40000, "uniform"), (48, 1, "uniform"),
                                       (48, 9000, "edges"), (32, 30000, "one cell"), (16, 2000, "uniform")])
def test_fixed_point_grids_match_oracle(gpu_lib, order, ng, n, kind):
    L = 100.0
    cat = catalogs.poisson(n, L, seed=5 + ng, dtype=np.float64, unit_mass=False)
    pos, vel, mass = cat["pos"], cat["vel"], cat["mass"]
    if kind == "edges":  # offsets of 0, 1/2 and just below 1, and values over twelve decades
        u = np.random.Generator(np.random.PCG64(9)).choice([0.0, 0.5, 1.0 - 2.0 ** -53, 2.0 ** -60], size=(n, 3))
        pos = np.mod((np.floor(pos * ng / L) + u) * (L / ng), L)
        mass = mass * 10.0 ** np.random.Generator(np.random.PCG64(8)).uniform(-6, 6, n)
    if kind == "one cell":
        pos = (np.array([7.0, 15.0, 31.0 % ng]) + pos / L) * (L / ng)
    got = _grids(gpu_lib, np.ascontiguousarray(pos), vel, mass, L, ng, order)
    ref = est.assign(pos, vel, mass, L=L, ng=ng, order=order)
    crowd = n if kind == "one cell" else max(1.0, 64.0 * n / ng ** 3)
    for f in range(4):
        scale = max(np.abs(ref[f]).max(), np.abs(mass).max() * (np.abs(vel).max() if f else 1.0))
        assert np.max(np.abs(got[f] - ref[f])) <= 1e-14 * (1.0 + crowd / 100.0) * scale


def test_nonfinite_values_reach_the_grid(gpu_lib):
    """A NaN velocity makes its field's nodes NaN and leaves the other fields alone, as FP64
    sums do (the fixed-point path steps aside)."""
    cat = catalogs.poisson(500, 50.0, seed=3, dtype=np.float64)
    vel = cat["vel"].copy()
    vel[7, 1] = np.nan
    got = _grids(gpu_lib, cat["pos"], vel, None, 50.0, 32, 4)
    ref = est.assign(cat["pos"], np.where(np.isnan(vel), 0.0, vel), None, L=50.0, ng=32, order=4)
    assert np.isnan(got[2]).any() and np.isfinite(got[[0, 1, 3]]).all()
    for f in (0, 1, 3):
        assert np.max(np.abs(got[f] - ref[f])) <= 1e-13 * np.abs(ref[f]).max()
