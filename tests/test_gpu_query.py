"""The candidate query (pixel intervals of the tiles' discs, FP32 with a
margin) may propose too many samples but never miss one: exact pair counts and
maps against the brute-force oracle next to the poles, across the longitude
seam, at the smallest and largest nside, and for discs that hold a pole or
cover most of the sphere."""
import numpy as np
import pytest

import oracle
from _parity import FP32_TOL, compare_maps

pytestmark = pytest.mark.gpu


def _cap(rng, n, lat0, lon0, radius):
    """n directions uniform in a cap."""
    c = 1.0 - rng.random(n) * (1.0 - np.cos(np.radians(radius)))
    t, a = np.arccos(c), rng.uniform(0.0, 2.0 * np.pi, n)
    v = np.stack([np.sin(t) * np.cos(a), np.sin(t) * np.sin(a), np.cos(t)])
    b, l = np.radians(90.0 - lat0), np.radians(lon0)
    x = np.cos(b) * v[0] + np.sin(b) * v[2]
    z = -np.sin(b) * v[0] + np.cos(b) * v[2]
    lon = np.degrees(np.arctan2(np.sin(l) * x + np.cos(l) * v[1], np.cos(l) * x - np.sin(l) * v[1]))
    return lon, np.degrees(np.arctan2(z, np.hypot(x, v[1])))


@pytest.mark.parametrize("lat0,lon0,radius,support,nside", [
    (90.0, 0.0, 1.0, 0.1, 2048),       # the pole inside the field
    (-89.95, 40.0, 0.2, 0.03, 8192),   # discs that just hold or just miss it
    (89.0, 180.0, 1.0, 0.5, 512),      # the seam next to a pole
    (0.0, 180.0, 2.0, 0.2, 4096),
    (41.81, 359.9, 0.5, 0.05, 8192),   # the cap / belt boundary
    (-20.0, 10.0, 0.02, 0.002, 8192),  # margins as large as the tiles' pixels
    (30.0, 100.0, 60.0, 25.0, 3),
    (-70.0, 200.0, 90.0, 80.0, 1),
    (50.0, 20.0, 180.0, 100.0, 16),    # the whole sphere, more than a hemisphere in reach
])
def test_no_candidate_is_missed(lat0, lon0, radius, support, nside):
    import torch
    from paper_1604_06667_gb300 import Gridder
    rng = np.random.Generator(np.random.PCG64(nside * 1000 + int(10 * (lat0 + 90))))
    lon_t, lat_t = _cap(rng, 333, lat0, lon0, radius)
    lon, lat = _cap(rng, 3000, lat0, lon0, radius)
    data = 1.0 + rng.random((lon.size, 2)).astype(np.float32)
    g = Gridder(lon_t, lat_t, n_channels=2)
    g.set_kernel("gauss1d", (support / 3.0,), support, nside=nside)
    g.grid(lon, lat, torch.from_numpy(data))
    w = torch.empty(lon_t.size, device="cuda")
    out = g.get_datacube(out_weights=w).cpu().numpy()
    pairs = g.info()["n_pairs"]
    g.close()
    ref = oracle.grid_bruteforce(lon_t, lat_t, lon, lat, data.astype(np.float64),
                                 oracle.gauss1d(support / 3.0, support))
    assert pairs == ref.npairs
    compare_maps(out, w.cpu().numpy(), ref, FP32_TOL)
