"""The queued (|k|, mu) binning at the edges of its range: one bin, an odd number (the middle
bin is its own mirror), the most bins it takes and one more (which the per-bin kernel takes),
bins along an axis (modes exactly on bin edges, whose mirror images fall elsewhere), single
and empty shells. Counts exact; spectra within the tolerances of test_gpu_mu."""
import numpy as np
import pytest

from oracle import mu as omu
from paper_2005_06170_gb300 import catalogs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("ng,nb,nmu,direction", [(24, 5, 1, (0.3, -0.5, 0.81)), (32, 7, 3, (1.0, 0.0, 0.0)),
                                                 (40, 30, 8, (0.0, 0.0, 1.0)), (32, 1, 9, (0.0, -1.0, 0.0)),
                                                 (48, 6, 16, (1.0, 1.0, 0.0)), (24, 5, 17, (0.0, 0.0, 1.0))])
def test_queued_mu_binning_matches_oracle(gpu_lib, dtype, ng, nb, nmu, direction):
    import torch
    pk = gpu_lib
    L = 100.0
    c = catalogs.poisson(6000, L, seed=ng + nmu, dtype=dtype, bulk=(90.0, -40.0, 20.0))
    p = pk.params(L, ng, nb, precision=pk.F32 if dtype == np.float32 else pk.F64, theta_scale=0.02)
    ctx = pk.Context(0)
    out = ctx.estimate_mu(torch.from_numpy(c["pos"]).cuda(), torch.from_numpy(c["vel"]).cuda(), p, nmu,
                          direction=direction)
    again = ctx.estimate_mu(torch.from_numpy(c["pos"]).cuda(), torch.from_numpy(c["vel"]).cuda(), p, nmu,
                            direction=direction)
    ctx.sync()
    g, g2 = pk.as_mu_dict(out, nb, nmu), pk.as_mu_dict(again, nb, nmu)
    ctx.close()
    o = omu.spectra_mu(c["pos"], c["vel"], None, L=L, ng=ng, nbins=nb, nmu=nmu, direction=direction, theta_scale=0.02)
    n = o["n_modes"]
    np.testing.assert_array_equal(g["n_modes"], n)
    ok = n > 0
    rtol = 1e-4 if dtype == np.float32 else 1e-9
    np.testing.assert_allclose(g["mu"][ok], o["mu_mean"][ok], atol=1e-6)
    sn_dt = np.sqrt(o["SN_dd"] * o["SN_tt"])
    scale = {"P_dd": o["SN_dd"], "P_tt": o["SN_tt"], "P_tt_b": o["SN_tt"], "Re_dt": sn_dt, "Im_dt": sn_dt,
             "Re_dt_b": sn_dt, "Im_dt_b": sn_dt, "P_pp": np.abs(o["P_pp"]) + o["SN_dd"] * 3 * 300.0 ** 2,
             "P_pp_b": np.abs(o["P_pp_b"]) + o["SN_dd"] * 3 * 300.0 ** 2}
    for key, sn in scale.items():
        floor = np.maximum(np.abs(o[key][ok]), np.abs(sn[ok]) / np.sqrt(n[ok]))
        assert np.max(np.abs(g[key][ok] - o[key][ok]) / floor) <= rtol, key
        np.testing.assert_allclose(g2[key][ok], g[key][ok], rtol=1e-12, atol=1e-12 * np.abs(g[key][ok]).max())
