"""Adjoint and interpolation of more channels than one slab of the lanes-over-
channels form holds, with a partial last slab, and at the edges of its widths.
Against the brute-force oracle (the bounds of the other adjoint tests)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [63, 64, 65, 100, 128, 129, 260])
@pytest.mark.parametrize("n", [5, 400])
def test_many_channels(n, C):
    import torch
    from paper_1604_06667_gb300 import Gridder
    rng = np.random.Generator(np.random.PCG64(n + C))
    nt, r = 500, 0.2
    lon, lat = 10.0 + rng.uniform(-1, 1, n), -30.0 + rng.uniform(-1, 1, n)
    lon_t, lat_t = 10.0 + rng.uniform(-1, 1, nt), -30.0 + rng.uniform(-1, 1, nt)
    om = rng.uniform(0.2, 2.0, n).astype(np.float32)
    g = Gridder(lon_t, lat_t, n_channels=C)
    g.set_kernel("gauss1d", (r / 3.0,), r, nside=512)
    W = torch.empty(nt, device="cuda")
    g.grid_oneshot(lon, lat, torch.ones((n, C)), weights=torch.from_numpy(om), out_weights=W)
    y = rng.normal(size=(nt, C)).astype(np.float32)
    k = oracle.gauss1d(r / 3.0, r)
    x = g.degrid(torch.from_numpy(y).cuda(), map_weights=W).cpu().numpy()
    args = (lon_t, lat_t, lon, lat)
    ref = oracle.degrid_bruteforce(*args, y.astype(np.float64), k, om.astype(np.float64))
    mag = oracle.degrid_bruteforce(*args, np.abs(y).astype(np.float64), k, om.astype(np.float64))
    assert np.all(np.abs(x - ref) <= 2e-5 * mag + 1e-30)
    v = torch.empty(n, device="cuda")
    z = g.interp(torch.from_numpy(y).cuda(), out_weights=v).cpu().numpy()
    g.close()
    v = v.cpu().numpy()
    zr, vr = oracle.interp_bruteforce(*args, y.astype(np.float64), k)
    za, _ = oracle.interp_bruteforce(*args, np.abs(y).astype(np.float64), k)
    on = vr > 0
    assert np.array_equal(on, v > 0) and np.all(np.isnan(z[~on]))
    assert np.all(np.abs(v[on] - vr[on]) <= 1e-5 * vr[on])
    assert np.all(np.abs(z[on] - zr[on]) <= 1e-5 * za[on])
