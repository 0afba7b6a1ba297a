"""The sort of the samples by RING index at the edges of its forms: parts of one
cluster (from one key to a full cluster of each size), then tiles with
look-back.  Exact: sorted by pixel, ties in the order of the input."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside", [4, 64, 4096])
@pytest.mark.parametrize("n", [1, 31, 257, 8191, 32767, 32769, 49152, 49153, 131073])
def test_order_of_samples(n, nside):
    import torch
    from paper_1604_06667_gb300 import Gridder
    rng = np.random.Generator(np.random.PCG64(n + nside))
    lon = rng.uniform(0.0, 360.0, n)
    lat = np.degrees(np.arcsin(rng.uniform(-1.0, 1.0, n)))
    lon[n // 2:], lat[n // 2:] = 77.0, 12.0          # one pixel holds half of them
    g = Gridder(np.array([77.0]), np.array([12.0]))
    g.set_kernel("gauss1d", (0.05,), 0.1, nside=nside)
    pix = oracle.ang2pix(nside, lon, lat)
    for data in (np.ones(n, np.float32), np.zeros(n, np.float32)):   # the second run reuses the scratch
        g.reset()
        g.grid(lon, lat, torch.from_numpy(data[:, None]))
        got, perm, _ = g.export_index(n)
        order = np.argsort(pix, kind="stable")
        assert np.array_equal(perm.cpu().numpy(), order)
        assert np.array_equal(got.cpu().numpy(), pix[order])
