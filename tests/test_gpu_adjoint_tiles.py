"""The tiled adjoint and interpolation gather (circular kernels) at the edges of
its tiles: sample counts around 64 and 8, channel counts on both sides of every
width, coverage with gaps, both poles and the longitude seam, many rings per
tile, supports above the series' range, dead samples, and non-finite map values,
which stay within the support.  Against the brute-force oracle (the bounds of
the other adjoint tests)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _fields(name, rng, n):
    """Sample and target positions."""
    if name == "gaps":          # two patches far apart
        lon = np.where(rng.random(n) < 0.5, 10.0, 40.0) + rng.uniform(-0.6, 0.6, n)
        lat = 20.0 + rng.uniform(-0.6, 0.6, n)
        lon_t = np.where(rng.random(500) < 0.5, 10.0, 40.0) + rng.uniform(-0.6, 0.6, 500)
        return lon, lat, lon_t, 20.0 + rng.uniform(-0.6, 0.6, 500), 0.1, 1024
    if name == "pole":
        lon, lon_t = rng.uniform(0.0, 360.0, n), rng.uniform(0.0, 360.0, 500)
        return lon, 90.0 - rng.uniform(0.0, 1.5, n), lon_t, 90.0 - rng.uniform(0.0, 1.5, 500), 0.2, 512
    if name == "seam":
        lon = (360.0 + rng.uniform(-0.7, 0.7, n)) % 360.0
        lon_t = rng.uniform(-0.7, 0.7, 500)
        return lon, -88.0 + rng.uniform(-0.7, 0.7, n), lon_t, -88.0 + rng.uniform(-0.7, 0.7, 500), 0.1, 2048
    if name == "rings":         # more rings per tile than one batch of intervals
        return (rng.uniform(0.0, 3.0, n), rng.uniform(-1.5, 1.5, n), rng.uniform(0.0, 3.0, 500),
                rng.uniform(-1.5, 1.5, 500), 1.0, 8192)
    return (rng.uniform(0.0, 30.0, n), rng.uniform(-15.0, 15.0, n), rng.uniform(0.0, 30.0, 500),
            rng.uniform(-15.0, 15.0, 500), 9.0, 32)       # "wide": d from the arc sine


@pytest.mark.parametrize("field", ["gaps", "pole", "seam", "rings", "wide"])
@pytest.mark.parametrize("n,C", [(1, 1), (7, 3), (63, 1), (64, 8), (65, 2), (700, 9), (3000, 4), (1500, 20)])
def test_adjoint_and_interpolation(field, n, C):
    import torch
    from paper_1604_06667_gb300 import Gridder
    rng = np.random.Generator(np.random.PCG64(1000 * len(field) + n + C))
    lon, lat, lon_t, lat_t, r, nside = _fields(field, rng, n)
    om = rng.uniform(0.2, 2.0, n).astype(np.float32)
    om[n // 2] = 0.0
    g = Gridder(lon_t, lat_t, n_channels=C)
    g.set_kernel("gauss1d", (r / 3.0,), r, nside=nside)
    g.grid_oneshot(lon, lat, torch.ones((n, C)), weights=torch.from_numpy(om))
    y = rng.normal(size=(lon_t.size, C)).astype(np.float32)
    k = oracle.gauss1d(r / 3.0, r)
    # the operator's weight map from the oracle: the gather alone is tested here
    W = oracle.grid_bruteforce(lon_t, lat_t, lon, lat, np.ones((n, 1)), k, om.astype(np.float64)).wsum
    W = torch.from_numpy(W.astype(np.float32)).cuda()
    x = g.degrid(torch.from_numpy(y).cuda(), map_weights=W).cpu().numpy()
    args = (lon_t, lat_t, lon, lat)
    ref = oracle.degrid_bruteforce(*args, y.astype(np.float64), k, om.astype(np.float64))
    mag = oracle.degrid_bruteforce(*args, np.abs(y).astype(np.float64), k, om.astype(np.float64))
    assert np.all(np.abs(x - ref) <= 2e-5 * mag + 1e-30)
    v = torch.empty(n, device="cuda")
    z = g.interp(torch.from_numpy(y).cuda(), out_weights=v).cpu().numpy()
    v = v.cpu().numpy()
    zr, vr = oracle.interp_bruteforce(*args, y.astype(np.float64), k)
    za, _ = oracle.interp_bruteforce(*args, np.abs(y).astype(np.float64), k)
    on = vr > 0
    assert np.array_equal(on, v > 0) and np.all(np.isnan(z[~on]))
    assert np.all(np.abs(v[on] - vr[on]) <= 1e-5 * vr[on])
    assert np.all(np.abs(z[on] - zr[on]) <= 1e-5 * za[on])
    # a NaN and an infinity in the map reach exactly the samples within their support
    bad = y.copy()
    bad[3, 0], bad[100, C - 1] = np.nan, np.inf
    zb = g.interp(torch.from_numpy(bad).cuda()).cpu().numpy()
    g.close()
    zo, _ = oracle.interp_bruteforce(*args, np.where(np.isfinite(bad), 0.0, 1.0), k)
    hit = np.nan_to_num(zo) > 0
    assert np.array_equal(~np.isfinite(zb[on]), hit[on])
    fine = on[:, None] & ~hit
    assert np.all(np.abs(zb - zr)[fine] <= 1e-5 * za[fine])
