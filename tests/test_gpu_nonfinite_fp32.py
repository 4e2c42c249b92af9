"""FP32 catalogues with NaN or infinite velocities. They are accepted (positions alone are
checked), and what they reach is not defined, but nothing else may change: the other fields
and, for NaN, which leaves a field's scale alone, the nodes of the field away from them equal
bit for bit those of the same catalogue with zeros in their place. The gather tiles add every
node of a stencil with weight zero outside the tile, beside the list of the particles."""
import numpy as np
import pytest

from paper_2005_06170_gb300 import catalogs

pytestmark = pytest.mark.gpu


def _grids(pk, ctx, pos, vel, L, ng, order):
    import torch
    p = pk.params(L, ng, 4, order=order)
    grids = torch.empty((4, ng, ng, ng + 2), dtype=torch.float32, device="cuda")
    mom = torch.zeros(16, dtype=torch.float64, device="cuda")
    scratch = torch.empty(ctx.scratch_bytes_tuned(p, len(pos)), dtype=torch.uint8, device="cuda")
    ctx.assign(pk.catalog_from_tensors(torch.from_numpy(pos).cuda(), torch.from_numpy(vel).cuda()), p, grids, mom,
               scratch)
    ctx.sync()
    return grids[..., :ng].cpu().numpy()


def _far(pos, L, ng, bad):
    """Nodes more than three cells from every bad particle on some axis."""
    node = np.arange(ng)
    near = np.zeros((ng, ng, ng), bool)
    for u in pos[bad].astype(np.float64) * ng / L:
        d = [np.abs((node - x + ng / 2) % ng - ng / 2) <= 3.0 for x in u]
        near |= d[0][:, None, None] & d[1][None, :, None] & d[2][None, None, :]
    return ~near


# 48^3: 16^3 tiles, keys of four cells; 40^3: 8^3 tiles, sparse and at two particles a cell
# (lists in several parts); "crowd": half of the particles in a cell (one particle a warp)
@pytest.mark.parametrize("order", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("ng,n,kind", [(48, 3000, ""), (40, 3000, ""), (40, 128000, ""), (48, 1200, "crowd"),
                                       (40, 1200, "crowd")])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_nonfinite_velocities_stay_in_place(gpu_lib, order, ng, n, kind, value):
    L = 100.0
    cat = catalogs.poisson(n, L, seed=ng + n, dtype=np.float32)
    pos, vel = cat["pos"], cat["vel"]
    if kind:
        pos[: n // 2] = (np.float32(20.0) + pos[: n // 2] / np.float32(L)) * np.float32(L / ng)
    bad = np.arange(0, n, max(1, n // 40))
    zeros, broken = vel.copy(), vel.copy()
    zeros[bad[:, None], [0, 2]], broken[bad[:, None], [0, 2]] = 0.0, value
    ctx = gpu_lib.Context(0)
    want, got = (_grids(gpu_lib, ctx, pos, v, L, ng, order) for v in (zeros, broken))
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[2], want[2])
    if np.isnan(value):
        far = _far(pos, L, ng, bad)
        assert far.any() and np.array_equal(got[1][far], want[1][far]) and np.array_equal(got[3][far], want[3][far])
    assert np.array_equal(_grids(gpu_lib, ctx, pos, zeros, L, ng, order), want)  # and the context goes on
    ctx.close()
