"""d/dsigma at the channel counts where its sums change form (lanes over
candidates up to 8 channels, over channels above, several slabs) and where a
block of the epilogue holds many targets or part of one.  Against the
brute-force oracle, with the bounds of the adjoint tests: dR and the scalar to
1e-4 (FP32 weights and sums, FP64 epilogue)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [1, 2, 8, 9, 37, 300])
def test_width_derivative_forms(C):
    import torch
    from paper_1604_06667_gb300 import Gridder
    rng = np.random.Generator(np.random.PCG64(900 + C))
    n, nt = 5000, 333
    lon, lat = 80.0 + rng.uniform(-1, 1, n), 35.0 + rng.uniform(-1, 1, n)
    lon_t, lat_t = 80.0 + rng.uniform(-1.5, 1.5, nt), 35.0 + rng.uniform(-1.5, 1.5, nt)
    data = 2.0 + rng.standard_normal((n, C)).astype(np.float32)
    om = rng.uniform(0.2, 2.0, n).astype(np.float32)
    gr = rng.standard_normal((nt, C)).astype(np.float32)
    g = Gridder(lon_t, lat_t, n_channels=C)
    g.set_kernel("gauss1d", (0.06,), 0.18, hpx_maxres=0.09)
    d = torch.from_numpy(data)
    g.grid_oneshot(lon, lat, d, weights=torch.from_numpy(om))
    dR, ds = g.dsigma(d, grad_out=torch.from_numpy(gr))
    dR = dR.double().cpu().numpy()
    ref = oracle.dsigma_bruteforce(lon_t, lat_t, lon, lat, data.astype(np.float64),
                                   oracle.gauss1d(0.06, 0.18), om.astype(np.float64))
    on = np.isfinite(ref[:, 0])
    assert 0 < on.sum() < nt                     # some targets see no sample
    assert np.array_equal(on, np.isfinite(dR[:, 0]))
    assert np.max(np.abs(dR[on] - ref[on])) <= 1e-4 * np.abs(ref[on]).max()
    terms = gr.astype(np.float64)[on] * ref[on]
    assert abs(float(ds) - terms.sum()) <= 1e-4 * np.abs(terms).sum()
