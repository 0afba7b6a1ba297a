"""The FP32 gridder's forms at the edges of their ranges: channel counts on
both sides of every width, one to several steps and shares of candidates,
every kernel type, BF16 and FP32 rows of any alignment, weights with zeros on
non-finite samples, adds that accumulate and adds that reuse the index.  Against the
brute-force oracle (1e-5 of S, the FP32 form's bound)."""
import numpy as np
import pytest

import oracle
from _parity import FP32_TOL, compare_maps

pytestmark = pytest.mark.gpu

KERNELS = {
    "gauss1d": (("gauss1d", (0.05,), 0.15), lambda: oracle.gauss1d(0.05, 0.15)),
    "gauss2d": (("gauss2d", (0.06, 0.03, 25.0), 0.15), lambda: oracle.gauss2d(0.06, 0.03, 25.0, 0.15)),
    "tsinc": (("tsinc", (0.05, 0.2), 0.15), lambda: oracle.tapered_sinc(0.05, 0.2, 0.15)),
    # support above the series' range: d from the arc sine
    "wide": (("gauss1d", (4.0,), 9.0), lambda: oracle.gauss1d(4.0, 9.0)),
    "wide2d": (("gauss2d", (4.0, 2.0, -40.0), 9.0), lambda: oracle.gauss2d(4.0, 2.0, -40.0, 9.0)),
}


def _inputs(n, nt, C, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    lon = 200.0 + rng.uniform(-1.0, 1.0, n)
    lat = 40.0 + rng.uniform(-0.8, 0.8, n)
    lon_t = 200.0 + rng.uniform(-1.05, 1.05, nt)
    lat_t = 40.0 + rng.uniform(-0.85, 0.85, nt)
    data = 2.0 + rng.standard_normal((n, C)).astype(np.float32)
    om = rng.uniform(0.2, 2.0, n).astype(np.float32)
    return lon, lat, lon_t, lat_t, data, om


@pytest.mark.parametrize("kernel", sorted(KERNELS))
@pytest.mark.parametrize("C", [1, 2, 3, 5, 8, 9, 32, 37, 64, 100, 257])
def test_channel_counts_and_kernels(C, kernel):
    import torch
    from paper_1604_06667_gb300 import Gridder
    (kt, kp, r), ok = KERNELS[kernel]
    n = 4000 if kernel.startswith("wide") else 9000
    lon, lat, lon_t, lat_t, data, om = _inputs(n, 450, C, 17 * C + len(kernel))
    om[::7] = 0.0
    data[::7] = np.nan                      # weight zero: these samples do not take part
    g = Gridder(lon_t, lat_t, n_channels=C)
    g.set_kernel(kt, kp, r, nside=64 if kernel.startswith("wide") else 1024)
    w = torch.empty(lon_t.size, device="cuda")
    out = g.grid_oneshot(lon, lat, torch.from_numpy(data), weights=torch.from_numpy(om), out_weights=w)
    pairs = g.info()["n_pairs"]
    ref = oracle.grid_bruteforce(lon_t, lat_t, lon, lat, np.nan_to_num(data).astype(np.float64), ok(),
                                 om.astype(np.float64))
    assert pairs == ref.npairs
    if kernel == "tsinc":                   # signed weights: N and W against sum |w|
        on = ref.wsum > 0.2 * np.nanmax(ref.wsum)
        got = out.cpu().numpy()[on]
        assert np.max(np.abs(got - ref.out[on]) / ref.sabs[on]) < 4 * FP32_TOL
    else:
        compare_maps(out.cpu().numpy(), w.cpu().numpy(), ref, FP32_TOL)
    # the same samples again by the kept index, on other values, accumulated twice
    d2 = np.flip(np.nan_to_num(data), axis=0).copy()
    g.set_kernel(kt, kp, r, nside=64 if kernel.startswith("wide") else 1024)
    g.grid(lon, lat, torch.from_numpy(d2), weights=torch.from_numpy(om))
    g.grid(None, None, torch.from_numpy(d2).cuda())
    out2 = g.get_datacube(out_weights=w, channel_major=True).cpu().numpy().T
    g.close()
    ref2 = oracle.grid_bruteforce(lon_t, lat_t, lon, lat, d2.astype(np.float64), ok(), om.astype(np.float64))
    if kernel != "tsinc":
        ref2.wsum = 2.0 * ref2.wsum
        compare_maps(out2, w.cpu().numpy(), ref2, FP32_TOL)


@pytest.mark.parametrize("n,nt", [(1, 1), (3, 70), (255, 64), (257, 129), (40000, 40), (300000, 10)])
@pytest.mark.parametrize("C,dtype", [(1, "f32"), (1, "bf16"), (4, "f32"), (7, "bf16"), (33, "f32"),
                                     (45, "bf16"), (130, "f32")])
def test_sizes_shares_and_alignment(n, nt, C, dtype):
    """From one sample and target to many candidate shares per tile, rows that
    start on a 4-byte (FP32) or 2-byte (BF16) boundary only."""
    import torch
    from paper_1604_06667_gb300 import Gridder, _capi
    if n * C > 3_000_000:
        n = 3_000_000 // C
    (kt, kp, r), ok = KERNELS["gauss1d"]
    lon, lat, lon_t, lat_t, data, _ = _inputs(n, nt, C, n + nt + C)
    buf = torch.empty(n * C + 1, dtype=torch.float32 if dtype == "f32" else torch.bfloat16, device="cuda")
    buf[1:] = torch.from_numpy(data.ravel()).cuda()
    d = buf[1:].reshape(n, C)
    g = Gridder(lon_t, lat_t, n_channels=C)
    g.set_kernel(kt, kp, r, nside=1024)
    g.set_path(_capi.CG_PATH_FP32)
    w = torch.empty(nt, device="cuda")
    out = g.grid_oneshot(lon, lat, d, out_weights=w)
    pairs = g.info()["n_pairs"]
    g.close()
    ref = oracle.grid_bruteforce(lon_t, lat_t, lon, lat, d.float().cpu().numpy().astype(np.float64), ok())
    assert pairs == ref.npairs
    compare_maps(out.cpu().numpy(), w.cpu().numpy(), ref, FP32_TOL)
