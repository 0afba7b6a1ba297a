"""The bounded waits inside the FP32 gridder for more than 8 channels: the hook
keeps one warp of every block from staging, so the other warps' waits run out
with their own copies in flight.  The batch reports CG_ETIMEOUT, and the same
handles then grid correctly, twice.  One case per way that rows reach shared
memory (gathered, copied element by element, converted from BF16) and one of
several channel slabs.  Against the brute-force oracle (1e-5 of S)."""
import numpy as np
import pytest

import oracle
import workloads
from _parity import compare_maps, kernel_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,dtype", [(16, "f32"), (32, "f32"), (37, "f32"), (44, "bf16"), (128, "f32"), (300, "f32")])
def test_waits_run_out_and_handle_recovers(C, dtype):
    import torch
    from paper_1604_06667_gb300 import Batch, Gridder, _capi
    wl = workloads.random_field(700 + C, 9000, 20, C, 140.0, 40.0, 1.0, 2.5 / 60.0)
    d = torch.from_numpy(wl.data).cuda()
    if dtype == "bf16":
        d = d.to(torch.bfloat16)
    g = Gridder(wl.lon_t, wl.lat_t, n_channels=C)
    g.set_kernel("gauss1d", (wl.kernel["sigma"],), wl.support, wl.hpx_maxres)
    g.set_path(_capi.CG_PATH_FP32)
    out, w = torch.empty((wl.n_targets, C), device="cuda"), torch.empty(wl.n_targets, device="cuda")
    b = Batch([(g, wl.lon_s, wl.lat_s, d, out, w)]).set_fused(True).debug_hold(True, 2_000_000).capture()
    b.run()
    with pytest.raises(_capi.CygridError) as ei:
        b.sync()
    assert ei.value.status == _capi.CG_ETIMEOUT
    b.debug_hold(False).capture()
    ref = oracle.grid_bruteforce(wl.lon_t, wl.lat_t, wl.lon_s, wl.lat_s,
                                 d.float().cpu().numpy().astype(np.float64), kernel_of(wl))
    for _ in range(2):
        b.run()
        b.sync()
        compare_maps(out.cpu().numpy(), w.cpu().numpy(), ref)
    b.close()
    g.close()
