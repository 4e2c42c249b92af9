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
# 4 to 1 below and 16 to 19 above the box's corner); cubic order has such keys from 192^3 on. 64^3, 16 x 16 x 32 tiles, lists of 4096: bank
# groups beyond 128 without a crowded cell.
@pytest.mark.parametrize("order,ng,tuning,kind", [(o, 48, (-1, -1), k) for o in (1, 2, 3, 4, 5) for k in (130, 200)] +
                         [(4, 192, (-1, -1), 200)] + [(o, 64, (1, 4096), 0) for o in (1, 2, 3, 4, 5)] +
                         [(4, 192, (1, 4096), 0)])
def test_particles_out_of_reach_stay_out(gpu_lib, order, ng, tuning, kind):
    L = 96.0
    if kind:
        cells = _crowd((20, 21, 20), kind, (12, 13, 14, 15, 32, 33, 34, 35))
        cells += _crowd((3, 2, 1), kind, (ng - 4, ng - 3, ng - 2, ng - 1, 16, 17, 18, 19))
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


@pytest.mark.parametrize("at", [0.0, 7.5])
def test_dense_tiles_of_runs(gpu_lib, at):
    """Cubic order, keys of four cells, a clump on a tile's corner (the box's) and inside a tile:
    dense tiles find a cell's particles, some with more than 256, in its run. A lost or misplaced
    particle changes a node by 0.01 to 1 of its value."""
    L, ng, n = 192.0, 192, 60000
    rng = np.random.Generator(np.random.PCG64(8))
    pos = np.mod(rng.normal(at, 1.4, (n, 3)), L).astype(np.float32)
    pos[pos >= np.float32(L)] = 0
    vel = rng.normal(0.0, 100.0, (n, 3)).astype(np.float32)
    got = [_grids(gpu_lib, pos, vel, L, ng, 4, (-1, -1), checked) for checked in (False, True)]
    ref = est.assign(pos, vel, None, L=L, ng=ng, order=4)
    q = [1.0] + [np.abs(vel[:, a]).max() for a in range(3)]
    for f in range(4):
        tol = 3.0 * np.sqrt(n) * 2.0 * W3[4] * n * q[f] / 2.0 ** 30 + 1e-6 * (np.abs(ref[f]).max() + q[f])
        for g in got:
            assert np.max(np.abs(g[f] - ref[f])) <= tol, f


@pytest.mark.parametrize("kind", ["row", "clump", "edge"])
def test_crowded_small_tiles_at_order_five(gpu_lib, kind):
    """8^3 tiles at order 5: crowded tiles are deposited a particle per warp straight from their
    ranges (one row far above the others; many particles a cell; a clump on the box's corner,
    whose ranges wrap), the others from lists."""
    L, ng, n = 80.0, 40, 6000
    rng = np.random.Generator(np.random.PCG64(5))
    cells = rng.integers(0, ng, (n, 3))
    m = n // 2
    if kind == "row":
        cells[:m, :2] = 21, 13
    if kind == "clump":
        cells[:] = rng.integers(16, 19, (n, 3))
    if kind == "edge":
        cells[:m] = rng.integers(-2, 2, (m, 3)) % ng
    pos, vel = _cells(cells, L, ng, seed=7)
    got = [_grids(gpu_lib, pos, vel, L, ng, 5, (-1, -1), checked) for checked in (False, True)]
    by_node = _grids(gpu_lib, pos, vel, L, ng, 5, (-1, 0), False)
    assert np.array_equal(got[0], by_node) and np.array_equal(got[1], by_node)
    ref = est.assign(pos, vel, None, L=L, ng=ng, order=5)
    q = [1.0] + [np.abs(vel[:, a]).max() for a in range(3)]
    for f in range(4):
        tol = 3.0 * np.sqrt(n) * 2.0 * W3[5] * n * q[f] / 2.0 ** 30 + 1e-6 * (np.abs(ref[f]).max() + q[f])
        assert np.max(np.abs(got[0][f] - ref[f])) <= tol, f
