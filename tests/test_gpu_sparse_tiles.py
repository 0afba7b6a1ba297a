"""Maps of many targets and few samples, at most 8 channels: tiles with no
candidate, one, up to 64 (a lane per target), up to 128 (groups on one stage)
and more, tiles of more sample ranges than are kept, every kernel and width,
samples of weight zero with non-finite values, a NaN that reaches exactly the
targets within its support, adds, and other layouts.  Against the brute-force
oracle (1e-5 of S, the FP32 form's bound)."""
import numpy as np
import pytest

import oracle
from _parity import FP32_TOL, compare_maps

pytestmark = pytest.mark.gpu

KERNELS = {
    "gauss1d": (("gauss1d", (0.05,), 0.15), lambda: oracle.gauss1d(0.05, 0.15), 1024),
    "rings": (("gauss1d", (0.2,), 0.6), lambda: oracle.gauss1d(0.2, 0.6), 8192),
    "gauss2d": (("gauss2d", (0.06, 0.03, 25.0), 0.15), lambda: oracle.gauss2d(0.06, 0.03, 25.0, 0.15), 1024),
    "wide": (("gauss1d", (4.0,), 9.0), lambda: oracle.gauss1d(4.0, 9.0), 32),
}


def _samples(rng, n, crowd):
    """n samples over a 4-degree field, a crowd of them within 0.02 degrees."""
    lon, lat = 200.0 + rng.uniform(-2.0, 2.0, n), rng.uniform(-2.0, 2.0, n)
    lon[:crowd] = 200.3 + rng.uniform(-0.01, 0.01, crowd)
    lat[:crowd] = 0.4 + rng.uniform(-0.01, 0.01, crowd)
    return lon, lat


@pytest.mark.parametrize("kernel", sorted(KERNELS))
@pytest.mark.parametrize("C", [1, 2, 3, 8])
@pytest.mark.parametrize("n,crowd", [(1, 0), (40, 3), (900, 61), (1500, 129), (2500, 700)])
def test_few_samples_per_tile(n, crowd, C, kernel):
    import torch
    from paper_1604_06667_gb300 import Gridder
    rng = np.random.Generator(np.random.PCG64(n + C))
    (kt, kp, r), ok, nside = KERNELS[kernel]
    x = np.linspace(-2.0, 2.0, 143)
    lon_t, lat_t = (a.ravel() for a in np.meshgrid(200.0 + x, x))
    lon, lat = _samples(rng, n, crowd)
    data = 2.0 + rng.standard_normal((n, C)).astype(np.float32)
    om = rng.uniform(0.2, 2.0, n).astype(np.float32)
    if n > 1:
        om[::9] = 0.0
        data[::9] = np.nan                              # these do not take part
    g = Gridder(lon_t, lat_t, n_channels=C)
    g.set_kernel(kt, kp, r, nside=nside)
    w = torch.empty(lon_t.size, device="cuda")
    out = g.grid_oneshot(lon, lat, torch.from_numpy(data), weights=torch.from_numpy(om), out_weights=w)
    ref = oracle.grid_bruteforce(lon_t, lat_t, lon, lat, np.nan_to_num(data).astype(np.float64), ok(),
                                 om.astype(np.float64))
    assert g.info()["n_pairs"] == ref.npairs
    compare_maps(out.cpu().numpy(), w.cpu().numpy(), ref, FP32_TOL)
    # the same twice, added up, by the kept index and in the other layout
    d2 = torch.from_numpy(np.nan_to_num(data)).cuda()
    g.reset()
    g.grid(lon, lat, d2, weights=torch.from_numpy(om))
    g.grid(None, None, d2)
    out2 = g.get_datacube(out_weights=w, channel_major=True).cpu().numpy().T
    g.close()
    ref.wsum = 2.0 * ref.wsum
    compare_maps(out2, w.cpu().numpy(), ref, FP32_TOL)


@pytest.mark.parametrize("C", [1, 5])
def test_nan_reaches_its_support_only(C):
    import torch
    from paper_1604_06667_gb300 import Gridder
    rng = np.random.Generator(np.random.PCG64(3))
    x = np.linspace(-2.0, 2.0, 143)
    lon_t, lat_t = (a.ravel() for a in np.meshgrid(200.0 + x, x))
    lon, lat = _samples(rng, 1200, 200)
    data = 2.0 + rng.standard_normal((1200, C)).astype(np.float32)
    data[5, 0], data[700, C - 1] = np.nan, np.inf       # in the crowd and outside
    g = Gridder(lon_t, lat_t, n_channels=C)
    g.set_kernel("gauss1d", (0.05,), 0.15, nside=1024)
    out = g.grid_oneshot(lon, lat, torch.from_numpy(data)).cpu().numpy()
    g.close()
    k = oracle.gauss1d(0.05, 0.15)
    hit = oracle.grid_bruteforce(lon_t, lat_t, lon, lat, np.where(np.isfinite(data), 0.0, 1.0), k)
    ref = oracle.grid_bruteforce(lon_t, lat_t, lon, lat, np.where(np.isfinite(data), data, 0.0).astype(np.float64), k)
    on = ref.wsum > 0
    reached = hit.out[on] > 0
    assert np.array_equal(~np.isfinite(out[on]), reached)
    fine = ~reached
    assert np.all((np.abs(out[on] - ref.out[on]) <= FP32_TOL * ref.sabs[on])[fine])
