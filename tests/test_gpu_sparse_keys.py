"""Sparse FP32 catalogues sort by runs of two or four cells: a tile passes over the particles
of the runs that stick out of its reach, finds the scale of its reach where its row bound
passes 256, and a dense tile picks a cell's particles out of its run. Grids listed and node
by node are the same bit for bit (tiles without cells of more than 256 particles), and
those of the oracle within the rounding the scale rule
gives: a tile of at most n particles rounds each contribution to a step of at most
2 w3 n max|q| / 2^30 (w3: the largest product of three weights), half a step at random per
contribution and at most n of them in a node, so six standard deviations are below
3 sqrt(n) steps; and 1e-6 of the largest node for the FP32 weights and products. A lost or
misplaced particle changes a node by 0.01 to 1 of its value."""
import numpy as np
import pytest

from oracle import estimator as est
from paper_2005_06170_gb300 import catalogs

pytestmark = pytest.mark.gpu


def _cat(kind, n, L, ng):
    rng = np.random.Generator(np.random.PCG64(ng + n))
    cat = catalogs.poisson(n, L, seed=n + ng, dtype=np.float32)
    if kind == "rows":  # a third of the particles in one column of cells: row bounds beyond 256
        cat["pos"][: n // 3, :2] = (L / ng) * (np.float32(5.0) + rng.random((n // 3, 2), dtype=np.float32))
    if kind == "blob":  # nine tenths in a blob of three cells: dense tiles, crowded runs
        m = 9 * n // 10
        cat["pos"][:m] = np.mod(rng.normal(0.0, 1.5 * L / ng, (m, 3)), L).astype(np.float32)
        cat["pos"][cat["pos"] >= np.float32(L)] = 0
    return cat


@pytest.mark.parametrize("order", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("kind,ng,n", [("uniform", 32, 1500), ("uniform", 24, 700), ("uniform", 48, 20000),
                                       ("rows", 48, 9000), ("rows", 40, 4000), ("blob", 96, 40000), ("blob", 72, 20000),
                                       ("uniform", 16, 200)])
def test_sparse_key_grids_match_oracle(gpu_lib, order, kind, ng, n):
    import torch
    L = 100.0
    cat = _cat(kind, n, L, ng)
    ctx = gpu_lib.Context(0)
    p = gpu_lib.params(L, ng, 4, order=order)
    pos, vel = torch.from_numpy(cat["pos"]).cuda(), torch.from_numpy(cat["vel"]).cuda()
    out = []
    for cap in (-1, 0):  # listed, and node by node
        ctx.set_tuning(-1, cap)
        grids = torch.empty((4, ng, ng, ng + 2), dtype=torch.float32, device="cuda")
        mom = torch.zeros(16, dtype=torch.float64, device="cuda")
        scratch = torch.empty(ctx.scratch_bytes_tuned(p, n), dtype=torch.uint8, device="cuda")
        ctx.assign(gpu_lib.catalog_from_tensors(pos, vel), p, grids, mom, scratch)
        ctx.sync()
        out.append(grids[..., :ng].clone())
    ctx.set_tuning(-1, -1)
    ctx.close()
    if kind != "blob":  # dense cubic tiles round the sums of 256 particles of a cell, in sort order
        assert torch.equal(out[0], out[1])
    ref = est.assign(cat["pos"], cat["vel"], None, L=L, ng=ng, order=order)
    w3 = {1: 1.0, 2: 1.0, 3: 0.421875, 4: 0.2962963, 5: 0.2148770}[order]
    q = [np.ones(n)] + [np.abs(cat["vel"][:, a].astype(np.float64)) for a in range(3)]
    for f in range(4):
        step = 2.0 * w3 * n * q[f].max() / 2.0 ** 30
        tol = 3.0 * np.sqrt(n) * step + 1e-6 * np.abs(ref[f]).max() + 1e-6 * q[f].max()
        assert np.max(np.abs(out[0][f].double().cpu().numpy() - ref[f])) <= tol, f
