"""Replays of a captured sort on other coordinates in the same buffers, with one
digit pass (nside 4: 8-bit keys) and several, above the size that one cluster
sorts.  Against the brute-force oracle (1e-5 of S, the FP32 form's bound)."""
import numpy as np
import pytest

import oracle
from _parity import compare_maps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside", [4, 64])
def test_replay_on_new_coordinates(nside):
    import torch
    from paper_1604_06667_gb300 import Batch, Gridder
    n, nt, r = 60_000, 200, 6.0
    rng = np.random.Generator(np.random.PCG64(nside))

    def sky(k):
        return rng.uniform(0.0, 360.0, k), np.degrees(np.arcsin(rng.uniform(-1.0, 1.0, k)))

    lon_t, lat_t = sky(nt)
    data = 2.0 + rng.standard_normal((n, 1)).astype(np.float32)
    g = Gridder(lon_t, lat_t)
    g.set_kernel("gauss1d", (r / 3.0,), r, nside=nside)
    lon, lat = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
    out, w = torch.empty((nt, 1), device="cuda"), torch.empty(nt, device="cuda")
    # a narrow field first: its digit counts are far from those of the sky
    fields = [(rng.uniform(10.0, 14.0, n), rng.uniform(-3.0, 3.0, n)), sky(n), sky(n)]
    lon.copy_(torch.from_numpy(fields[0][0]))
    lat.copy_(torch.from_numpy(fields[0][1]))
    b = Batch([(g, lon, lat, torch.from_numpy(data).cuda(), out, w)]).capture()
    for x, y in fields:
        lon.copy_(torch.from_numpy(x))
        lat.copy_(torch.from_numpy(y))
        torch.cuda.synchronize()
        b.run()
        b.sync()
        ref = oracle.grid_bruteforce(lon_t, lat_t, x, y, data.astype(np.float64),
                                     oracle.gauss1d(r / 3.0, r))
        compare_maps(out.cpu().numpy(), w.cpu().numpy(), ref)
    b.close()
    g.close()
