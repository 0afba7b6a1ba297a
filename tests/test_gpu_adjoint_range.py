"""The adjoint with sample weights whose sums are far from one: map / W or its
products with the kernel leave FP32's range although the result does not.
Against the brute-force oracle (the bound of the other adjoint tests)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [1, 4, 20, 100])
@pytest.mark.parametrize("om,y", [(1e-34, 1e6), (1e-30, 1e7), (1e33, 1e-8), (1e34, 1e3), (1e-3, 1e-3)])
def test_extreme_sample_weights(om, y, C):
    import torch
    from paper_1604_06667_gb300 import Gridder
    rng = np.random.Generator(np.random.PCG64(C))
    n, nt, r = 2000, 300, 0.15
    lon, lat = 50.0 + rng.uniform(-1, 1, n), 20.0 + rng.uniform(-1, 1, n)
    lon_t, lat_t = 50.0 + rng.uniform(-1, 1, nt), 20.0 + rng.uniform(-1, 1, nt)
    w = (om * rng.uniform(0.5, 2.0, n)).astype(np.float32)
    m = (y * rng.normal(size=(nt, C))).astype(np.float32)
    k = oracle.gauss1d(r / 3.0, r)
    g = Gridder(lon_t, lat_t, n_channels=C)
    g.set_kernel("gauss1d", (r / 3.0,), r, nside=1024)
    W = oracle.grid_bruteforce(lon_t, lat_t, lon, lat, np.ones((n, 1)), k, w.astype(np.float64)).wsum
    g.grid_oneshot(lon, lat, torch.ones((n, C)), weights=torch.from_numpy(w))
    x = g.degrid(torch.from_numpy(m).cuda(), map_weights=torch.from_numpy(W.astype(np.float32)).cuda())
    x = x.cpu().numpy()
    g.close()
    args = (lon_t, lat_t, lon, lat)
    ref = oracle.degrid_bruteforce(*args, m.astype(np.float64), k, w.astype(np.float64))
    mag = oracle.degrid_bruteforce(*args, np.abs(m).astype(np.float64), k, w.astype(np.float64))
    assert np.all(np.isfinite(x))
    assert np.all(np.abs(x - ref) <= 2e-5 * mag)
