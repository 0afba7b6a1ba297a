"""Adds whose samples crowd on a few target tiles: full tiles are shared among
blocks, the others are not, in one call; accumulated over three scans, with
non-finite values in one of them.  Against the brute-force oracle (1e-5 of S,
the FP32 form's bound)."""
import numpy as np
import pytest

import oracle
from _parity import FP32_TOL, compare_maps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [9, 37, 64, 130])
@pytest.mark.parametrize("n", [400, 9000])
def test_scans_on_part_of_the_map(n, C):
    import torch
    from paper_1604_06667_gb300 import Gridder
    rng = np.random.Generator(np.random.PCG64(n + C))
    x = np.linspace(-1.0, 1.0, 40)
    lon_t, lat_t = (a.ravel() for a in np.meshgrid(200.0 + x, x))
    g = Gridder(lon_t, lat_t, n_channels=C)
    g.set_kernel("gauss1d", (0.05,), 0.15, hpx_maxres=0.07)
    parts = []
    for k in range(3):
        lon = 200.0 + rng.uniform(-1.0, 1.0, n)
        lat = -0.9 + 0.8 * k + rng.uniform(0.0, 0.2, n)      # a strip of the map
        lon[-50:], lat[-50:] = 200.0 + rng.uniform(-1, 1, 50), rng.uniform(-1, 1, 50)
        data = 2.0 + rng.standard_normal((n, C)).astype(np.float32)
        om = rng.uniform(0.2, 2.0, n).astype(np.float32)
        if k == 1:                                           # taken out by their weight
            om[::11] = 0.0
            data[::11] = np.nan
        g.grid(lon, lat, torch.from_numpy(data), weights=torch.from_numpy(om))
        parts.append((lon, lat, np.nan_to_num(data).astype(np.float64), om.astype(np.float64)))
    w = torch.empty(lon_t.size, device="cuda")
    out = g.get_datacube(out_weights=w)
    lon, lat, data, om = (np.concatenate([p[i] for p in parts]) for i in range(4))
    ref = oracle.grid_bruteforce(lon_t, lat_t, lon, lat, data, oracle.gauss1d(0.05, 0.15), om)
    compare_maps(out.cpu().numpy(), w.cpu().numpy(), ref, FP32_TOL)
