"""FP32 moments whose warp sums leave FP32's range: m^2 v^2 of 1e37 a particle (masses in solar
masses), where 32 lanes' sums pass 3.4e38. Against FP64 sums of the same FP32 values: products
of three or four factors round three times, the compensated sums once more in effect: 4 2^-24
of the sum of magnitudes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [32, 33, 4096, 100003, 3000000])
@pytest.mark.parametrize("layout", ["aligned", "unaligned"])
@pytest.mark.parametrize("m0,v0", [(1e15, 3e3), (None, 3e18)])
def test_large_moments_stay_finite(gpu_lib, n, layout, m0, v0):
    import torch
    rng = np.random.Generator(np.random.PCG64(n))
    L, ng = 100.0, 32
    pos = rng.uniform(0.0, L, (n, 3)).astype(np.float32)
    pos[pos >= np.float32(L)] = 0
    vel = (v0 * rng.choice([-1.0, 1.0], (n, 3)) * rng.uniform(0.8, 1.0, (n, 3))).astype(np.float32)
    mass = None if m0 is None else (m0 * rng.uniform(0.8, 1.0, n)).astype(np.float32)
    dev = [torch.from_numpy(a).cuda() for a in (pos, vel)]
    if layout == "unaligned":  # one value off 16 bytes: the kernel for arbitrary arrays
        dev[1] = torch.cat([dev[1].new_zeros(1), dev[1].reshape(-1)])[1:].view(n, 3)
    dm = None if mass is None else torch.from_numpy(mass).cuda()
    ctx = gpu_lib.Context(0)
    p = gpu_lib.params(L, ng, 8)
    grids = torch.empty((4, ng, ng, ng + 2), dtype=torch.float32, device="cuda")
    mom = torch.zeros(16, dtype=torch.float64, device="cuda")
    scratch = torch.empty(ctx.scratch_bytes(p, n), dtype=torch.uint8, device="cuda")
    ctx.assign(gpu_lib.catalog_from_tensors(*dev, dm), p, grids, mom, scratch)
    ctx.sync()
    got = mom.cpu().numpy()
    ctx.close()
    m = np.ones(n) if mass is None else mass.astype(np.float64)
    v = vel.astype(np.float64)
    terms = [m, m * m] + [m * v[:, a] for a in range(3)] + [m * m * v[:, a] for a in range(3)]
    terms += [m * m * v[:, a] * v[:, b] for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]
    for k, t in enumerate(terms):
        assert abs(got[k] - t.sum()) <= 4.0 * 2.0 ** -24 * np.abs(t).sum(), k
    assert got[14] == n
