"""Tiles of targets where the axes of their cuts change: fields on the equator,
at middle latitude, where meridians converge and around a pole, wide fields and
the whole sky, just below and above the number of targets that one block
finishes in shared memory.  Against the brute-force oracle (1e-5 of S, the FP32
form's bound)."""
import numpy as np
import pytest

import oracle
from _parity import FP32_TOL, compare_maps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nt", [33, 4096, 4097, 9001])
@pytest.mark.parametrize("lon0,lat0,side", [(0.0, 0.0, 4.0), (120.0, 30.0, 4.0), (300.0, -75.0, 4.0),
                                            (77.0, 90.0, 3.0), (200.0, 40.0, 60.0), (0.0, 0.0, 360.0)])
def test_cuts_along_own_axes(lon0, lat0, side, nt):
    import torch
    from paper_1604_06667_gb300 import Gridder
    rng = np.random.Generator(np.random.PCG64(nt + int(side) + int(abs(lat0))))

    def draw(n):
        if side == 360.0:
            return rng.uniform(0.0, 360.0, n), np.degrees(np.arcsin(rng.uniform(-1.0, 1.0, n)))
        if lat0 == 90.0:
            return rng.uniform(0.0, 360.0, n), 90.0 - side * np.sqrt(rng.uniform(0.0, 1.0, n))
        lat = lat0 + side * rng.uniform(-0.5, 0.5, n)
        return lon0 + side * rng.uniform(-0.5, 0.5, n) / np.cos(np.radians(lat0)), lat

    r = 0.1 * min(side, 90.0)
    lon, lat = draw(4000)
    lon_t, lat_t = draw(nt)
    data = 2.0 + rng.standard_normal((4000, 1)).astype(np.float32)
    g = Gridder(lon_t, lat_t)
    g.set_kernel("gauss1d", (r / 3,), r, hpx_maxres=r / 2)
    w = torch.empty(nt, device="cuda")
    out = g.grid_oneshot(lon, lat, torch.from_numpy(data), out_weights=w)
    ref = oracle.grid_bruteforce(lon_t, lat_t, lon, lat, data.astype(np.float64), oracle.gauss1d(r / 3, r),
                                 np.ones(4000))
    assert g.info()["n_pairs"] == ref.npairs
    compare_maps(out.cpu().numpy().reshape(nt, 1), w.cpu().numpy(), ref, FP32_TOL)
