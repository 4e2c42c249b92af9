"""pkmom_estimate_host copies velocities and masses beside the histogram and the scan, which
need positions alone: catalogues that alternate on one context, in either layout, pinned or
not, give the spectra of the device estimate. The same kernels run on the same bytes: the
only difference allowed is the FP64 rounding of the deposit's order-dependent sums."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ng,fp64,mass,pinned,soa", [
    (1, 32, False, False, True, False),
    (1001, 32, True, True, False, False),
    (300_000, 64, True, True, True, True),
    (2_000_003, 128, False, True, True, True),
    (2_000_003, 128, False, False, False, False),
    (4_000_000, 160, False, False, True, False),
])
def test_host_estimates_equal_device_estimates(gpu_lib, n, ng, fp64, mass, pinned, soa):
    import torch
    pk = gpu_lib
    dt = np.float64 if fp64 else np.float32
    p = pk.params(250.0, ng, 16, precision=pk.F64 if fp64 else pk.F32)
    ctx, stream = pk.Context(0), torch.cuda.Stream()
    rng = np.random.default_rng(n + ng)
    cats, refs = [], []

    def catalog(pos, vel, m, address):
        c = pk.Catalog(n=n, stride=1, dtype=p.precision, mass=address(m) if mass else None)
        for f, r in zip(("x", "y", "z", "vx", "vy", "vz"), [*pos, *vel]):
            setattr(c, f, address(r))
        return c

    for _ in range(3):
        a = [torch.from_numpy((rng.random((n, 3)) * 250).astype(dt)), torch.from_numpy(rng.normal(0, 90, (n, 3)).astype(dt))]
        a.append(torch.from_numpy(rng.uniform(0.5, 2, n).astype(dt)) if mass else None)
        if soa:
            a[:2] = [t.T.contiguous() for t in a[:2]]
        d = [None if t is None else t.cuda() for t in a]
        if soa:
            ref = torch.empty((pk.NROWS, p.nbins), dtype=torch.float64, device="cuda")
            c = catalog(*d, lambda t: t.data_ptr())
            assert ctx._L.pkmom_estimate(ctx._h, ctypes.byref(c), ctypes.byref(p), ref.data_ptr(), None) == 0
        else:
            ref = ctx.estimate(d[0], d[1], p, mass=d[2])
        ctx.sync()
        refs.append(ref.cpu().numpy())
        cats.append([t.pin_memory() if pinned and t is not None else t for t in a])
    for k in (0, 1, 2, 0, 2, 1):
        pos, vel, m = (None if t is None else t.numpy() for t in cats[k])
        if soa:
            out = np.empty((pk.NROWS, p.nbins))
            c = catalog(pos, vel, m, lambda t: t.ctypes.data)
            assert ctx._L.pkmom_estimate_host(ctx._h, ctypes.byref(c), ctypes.byref(p), out.ctypes.data,
                                              stream.cuda_stream) == 0
        else:
            out = ctx.estimate_host(pos, vel, p, mass=m, stream=stream)
        np.testing.assert_allclose(out, refs[k], rtol=1e-12, atol=1e-12 * np.nanmax(np.abs(refs[k])), equal_nan=True)
    ctx.close()
