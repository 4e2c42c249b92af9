"""Crowded lists of sparse catalogues (keys of several cells). The runs of a tile hold particles
below and above its reach, and a bank group of more than 128 particles exceeds the ranks its
list is ordered by: the particles out of reach must stay out of the adds all the same. In the
checked build an add outside the reach's padding raises PKMOM_EDATA. Listed grids equal those
deposited node by node bit for bit, and the oracle's within the rounding the scale rule gives
(a tile of n particles rounds to steps of at most 2 w3 n max|q| / 2^30, half a step at random
per contribution, so six standard deviations of a node are below 3 sqrt(n) steps; 1e-6 of the
largest node and value for the FP32 weights and products)."""
import numpy as np
import pytest

from oracle import estimator as est

pytestmark = pytest.mark.gpu
W3 = {1: 1.0, 2: 1.0, 3: 0.421875, 4: 0.2962963, 5: 0.2148770}


def _cells(cells, L, ng, seed):
    """One particle at a random place of each cell, with velocities."""
    rng = np.random.Generator(np.random.PCG64(seed))
    cells = np.asarray(cells, dtype=np.float64)
    pos = np.mod((cells + rng.uniform(0.02, 0.98, cells.shape)) * (L / ng), L).astype(np.float32)
    return pos, rng.normal(0.0, 100.0, cells.shape).astype(np.float32)


def _crowd(cell, count, z_strays):
    """count particles in a cell and four in its row at each stray z."""
    out = [cell] * count
    for z in z_strays:
        out += [(cell[0], cell[1], z)] * 4
    return out


def _grids(pk, pos, vel, L, ng, order, tuning, checked):
    import torch
    ctx = pk.Context(0, checked=checked)
    ctx.set_tuning(*tuning)
    p = pk.params(L, ng, 4, order=order)
    grids = torch.empty((4, ng, ng, ng + 2), dtype=torch.float32, device="cuda")
    mom = torch.zeros(16, dtype=torch.float64, device="cuda")
    scratch = torch.empty(ctx.scratch_bytes_tuned(p, len(pos)), dtype=torch.uint8, device="cuda")
    ctx.assign(pk.catalog_from_tensors(torch.from_numpy(pos).cuda(), torch.from_numpy(vel).cuda()), p, grids, mom,
               scratch)
    ctx.sync()
    ctx.close()
    return grids[..., :ng].cpu().numpy()


# 48^3, 16^3 tiles, lists of 256: 130 to 200 particles in a cell of two tiles, strays in the
# cells of their runs of four beyond the reach (12 to 15 below the corner at 16, 32 to 35 above;
# 44 to 47 and 16 to 19 around the box's corner). 64^3, 16 x 16 x 32 tiles, lists of 4096: bank
# groups beyond 128 without a crowded cell.
@pytest.mark.parametrize("order,ng,tuning,kind", [(o, 48, (-1, -1), k) for o in (1, 2, 3, 4, 5) for k in (130, 200)] +
                         [(o, 64, (1, 4096), 0) for o in (1, 2, 3, 4, 5)])
def test_particles_out_of_reach_stay_out(gpu_lib, order, ng, tuning, kind):
    L = 96.0
    if kind:
        cells = _crowd((20, 21, 20), kind, (12, 13, 14, 15, 32, 33, 34, 35))
        cells += _crowd((3, 2, 1), kind, (44, 45, 46, 47, 16, 17, 18, 19))
    else:
        rng = np.random.Generator(np.random.PCG64(2))
        cells = np.concatenate([rng.integers((18, 18, 34), (30, 30, 62), (3850, 3)),
                                rng.integers((18, 18, 28), (30, 30, 32), (200, 3))])
    pos, vel = _cells(cells, L, ng, seed=order + ng)
    n = len(pos)
    listed = [_grids(gpu_lib, pos, vel, L, ng, order, tuning, checked) for checked in (False, True)]
    by_node = _grids(gpu_lib, pos, vel, L, ng, order, (tuning[0], 0), False)
    assert np.array_equal(listed[0], by_node) and np.array_equal(listed[1], by_node)
    ref = est.assign(pos, vel, None, L=L, ng=ng, order=order)
    q = [1.0] + [np.abs(vel[:, a]).max() for a in range(3)]
    for f in range(4):
        tol = 3.0 * np.sqrt(n) * 2.0 * W3[order] * n * q[f] / 2.0 ** 30 + 1e-6 * (np.abs(ref[f]).max() + q[f])
        assert np.max(np.abs(listed[0][f] - ref[f])) <= tol, f
