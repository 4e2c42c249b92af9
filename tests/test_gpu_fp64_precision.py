"""FP64 grids keep FP64's precision of every particle. The fixed-point deposit is off by less
than 6 2^-61 of the scale of a pass per contribution, and a pass takes particles down to
2^-9 of its scale: at most 1.5 2^-50 of a particle's own mass (first grid) or largest momentum
component (the others), below the 15 roundings of 2^-53 of FP64 products (three weights of
four, three products). Light and slow particles have passes of their own, and crowds lose
no bits.

Grid units (L = ng) make the offsets in the cells exact, so that references differ by the
roundings alone."""
from math import comb, factorial

import numpy as np
import pytest

from oracle import estimator as est

pytestmark = pytest.mark.gpu


def _grids(pk, pos, vel, mass, ng, order, checked=False):
    import torch
    ctx = pk.Context(0, checked=checked)
    p = pk.params(float(ng), ng, 4, order=order, precision=pk.F64)
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() if a is not None else None for a in (pos, vel, mass)]
    grids = torch.empty((4, ng, ng, ng + 2), dtype=torch.float64, device="cuda")
    mom = torch.zeros(16, dtype=torch.float64, device="cuda")
    scratch = torch.empty(ctx.scratch_bytes_tuned(p, len(pos)), dtype=torch.uint8, device="cuda")
    ctx.assign(pk.catalog_from_tensors(*dev), p, grids, mom, scratch)
    ctx.sync()
    out = grids[..., :ng].cpu().numpy()
    ctx.close()
    return out


def _weights(u, order):
    """First nodes and B-spline weights of one axis in long double: truncated powers from the
    nearer end of the support, so that small weights keep their relative precision."""
    first = np.floor(u + (0.5 if order % 2 else 0.0)) - (order - 1) // 2
    w = []
    for k in range(order):
        x = np.abs(u.astype(np.longdouble) - (first + k))
        s = np.zeros(len(u), np.longdouble)
        for j in range(order):
            s += (-1) ** j * comb(order, j) * np.maximum(np.longdouble(order) / 2 - x - j, 0) ** (order - 1)
        w.append(s / factorial(order - 1))
    return first.astype(int), w


def _deposit(pos, q, ng, order, reach=False):
    """Grid of one field in long double; reach: every weight one (the sum over the particles
    that reach a node)."""
    axes = [_weights(pos[:, a], order) for a in range(3)]
    grid = np.zeros((ng, ng, ng), np.longdouble)
    for k in np.ndindex(order, order, order):
        node = tuple((axes[a][0] + k[a]) % ng for a in range(3))
        np.add.at(grid, node, q if reach else q * axes[0][1][k[0]] * axes[1][1][k[1]] * axes[2][1][k[2]])
    return grid


def _reaching(pos, nodes, ng):
    """Particles within three nodes of the marked ones on every axis."""
    for axis in range(3):
        nodes = np.any([np.roll(nodes, d, axis) for d in range(-3, 4)], axis=0)
    return nodes[tuple(np.floor(pos).astype(int).T % ng)]


# 24^3: 8^3 tiles, 32^3: 8 x 8 x 16; few light particles a tile and many, without masses too;
# a mass, or the speed, 2^9 to 2^40 below the largest
@pytest.mark.parametrize("order", [2, 3, 4, 5])
@pytest.mark.parametrize("ng,n,share", [(24, 3000, 0.1), (32, 4000, 0.1), (32, 60000, 0.5), (24, 40000, 1e-4)])
@pytest.mark.parametrize("what,orders", [("mass", 9), ("mass", 25), ("speed", 9), ("speed", 40), ("slow, no mass", 20),
                                         ("both", 30)])
def test_light_and_slow_particles_keep_their_digits(gpu_lib, order, ng, n, share, what, orders):
    rng = np.random.Generator(np.random.PCG64(ng + order + orders))
    pos = rng.uniform(0.0, ng, (n, 3))
    pos[pos >= ng] = 0.0
    vel = rng.choice([-1.0, 1.0], (n, 3)) * rng.uniform(100.0, 200.0, (n, 3))
    mass = None if "no mass" in what else rng.uniform(0.75, 0.99, n)
    low = rng.random(n) < share
    low[:2] = True, False
    low[(pos < ng / 4).all(axis=1)] = True  # a corner of its own, where only they are
    if what in ("mass", "both"):  # both: every level between, in mass and in speed
        mass[low] *= 2.0 ** -(orders if what == "mass" else rng.integers(9, orders, low.sum()))
    if what == "both":
        vel[low] *= 2.0 ** -rng.integers(9, orders, low.sum())[:, None].astype(float)
    elif what != "mass":
        vel[low] *= 2.0 ** -orders
    got = _grids(gpu_lib, pos, vel, mass, ng, order)
    ref = est.assign(pos, vel, mass, L=float(ng), ng=ng, order=order)
    own = est.assign(pos, np.abs(vel), mass, L=float(ng), ng=ng, order=order)  # sums of magnitudes
    normal = est.assign(pos[~low], np.abs(vel[~low]), None if mass is None else mass[~low], L=float(ng), ng=ng,
                        order=order)
    q = [np.ones(n) if mass is None else mass]
    q += [q[0] * vel[:, a] for a in range(3)]
    for f in range(4):
        only = (normal[f] == 0.0) & (own[f] > 0.0)
        assert only.any()
        near = low & _reaching(pos, only, ng)
        value = q[f][near].astype(np.longdouble)
        size = np.abs(q[0] if f == 0 else np.max(np.abs(q[1:]), axis=0))[near].astype(np.longdouble)
        error = np.abs(got[f] - _deposit(pos[near], value, ng, order))[only]
        # the contributions, and four roundings of the node (its passes and the result)
        bound = 1.5 * 2.0 ** -50 * _deposit(pos[near], size, ng, order, reach=True) + 2.0 ** -51 * own[f]
        assert np.all(error <= bound[only]), float(np.max(error / bound[only]))
        top = (1.0 if mass is None else mass.max()) * (200.0 if f else 1.0)
        assert np.max(np.abs(got[f] - ref[f])) <= 1e-14 * (1.0 + 64.0 * n / ng ** 3 / 100.0) * max(own[f].max(), top)


@pytest.mark.parametrize("order,copies", [(2, 1), (2, 1000), (3, 1000), (4, 10), (4, 1000), (5, 100)])
def test_crowded_nodes_are_exact(gpu_lib, order, copies):
    """2000 particles of one cell, many times each: high sums of 64 bits, no scale of the crowd."""
    ng, n = 32, 2000
    rng = np.random.Generator(np.random.PCG64(order + copies))
    pos = np.array([8.0, 15.0, 31.0]) + rng.uniform(0.0, 0.999, (n, 3))
    vel = rng.choice([-1.0, 1.0], (n, 3)) * rng.uniform(100.0, 200.0, (n, 3))
    mass = rng.uniform(0.5, 1.0, n)
    got = _grids(gpu_lib, np.tile(pos, (copies, 1)), np.tile(vel, (copies, 1)), np.tile(mass, copies), ng, order)
    q = [mass.astype(np.longdouble)] + [mass * vel[:, a] for a in range(3)]
    axes = [_weights(pos[:, a], order) for a in range(3)]
    first = [a[0].min() for a in axes]
    for f in range(4):
        value = q[f].astype(np.longdouble)
        top = 2.0 ** np.ceil(np.log2(float(np.abs(value).max())))
        ref = {}
        for k in np.ndindex(order, order, order):
            c = value * axes[0][1][k[0]] * axes[1][1][k[1]] * axes[2][1][k[2]]
            for at in {tuple(x) for x in np.stack([axes[a][0] + k[a] for a in range(3)], 1)}:
                here = np.all([axes[a][0] + k[a] == at[a] for a in range(3)], axis=0)
                node = tuple(x % ng for x in at)
                ref[node] = ref.get(node, np.longdouble(0)) + copies * c[here].sum()
        for node, r in ref.items():
            # 6 units of 2^-61 a contribution, the node's own rounding, the reference's of 2^-63
            tol = 6.0 * 2.0 ** -61 * top * n * copies + (2.0 ** -53 + 64 * 2.0 ** -63) * abs(float(r)) + \
                2.0 ** -59 * copies * float(np.abs(value).sum())
            assert abs(float(got[f][node] - r)) <= tol, (f, node)
    assert first[0] >= 0


def test_checked_build_with_light_particles(gpu_lib):
    rng = np.random.Generator(np.random.PCG64(4))
    ng, n = 32, 30000
    pos, vel = rng.uniform(0.0, ng, (n, 3)), rng.normal(0.0, 100.0, (n, 3))
    pos[: n // 2] = 5.0 + pos[: n // 2] / ng
    vel[::40] *= 1e-6
    a, b = (_grids(gpu_lib, pos, vel, None, ng, 4, checked) for checked in (False, True))
    assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(a))
