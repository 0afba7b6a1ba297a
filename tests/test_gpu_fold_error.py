"""Rounding of the FP32 form on maps of few tiles: its chains of additions are no
longer than those of the register-blocked form, which shares a tile's candidates
among several blocks there.  The RMS errors of the two forms on the same inputs,
against the brute-force oracle: chains of equal length give a ratio of 1; the RMS
over more than 10,000 values is good to a few per cent, so 1.15 is allowed (one
chain per tile: 1.3 to 2.8)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,side,n", [(16, 200, 60_000), (21, 113, 62_000), (37, 110, 60_000), (66, 52, 15_000),
                                      (130, 48, 12_000), (300, 24, 8_000)])
def test_error_against_shared_candidates(C, side, n):
    import torch
    from paper_1604_06667_gb300 import Gridder
    rng = np.random.Generator(np.random.PCG64(C + side))
    size, r = 2.0, 0.15
    x = (np.arange(side) + 0.5) / side * size - 0.5 * size
    lon_t, lat_t = (a.ravel() for a in np.meshgrid(60.0 + x, x))
    lon, lat = 60.0 + size * (rng.random(n) - 0.5), size * (rng.random(n) - 0.5)
    data = 3.0 + rng.standard_normal((n, C)).astype(np.float32)
    pick = rng.choice(lon_t.size, min(lon_t.size, 1500), replace=False)
    ref = oracle.grid_bruteforce(lon_t[pick], lat_t[pick], lon, lat, data.astype(np.float64), oracle.gauss1d(r / 3, r))
    g = Gridder(lon_t, lat_t, n_channels=C)
    g.set_kernel("gauss1d", (r / 3,), r, hpx_maxres=r / 6)
    rms = []
    for shape in (-1, next(i for i, c in enumerate((4, 8, 16, 32, 64, 128, 256)) if C <= c or c == 256)):
        g.set_f32_shape(shape)
        out = g.grid_oneshot(lon, lat, torch.from_numpy(data)).double().cpu().numpy()[pick]
        on = ref.wsum > 0
        rms.append(np.sqrt(np.mean(((out[on] - ref.out[on]) / ref.sabs[on]) ** 2)))
    g.close()
    assert rms[0] <= 1.15 * rms[1], rms
