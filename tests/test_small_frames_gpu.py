"""Frames of few subapertures project inside the spot kernel, larger ones or those of many layers in a
launch of their own: on both sides of the rule's limits the slopes match the oracle, and a handle
measured through a batch (always a launch of its own) gives the same bits (GPU)."""
import dataclasses

import numpy as np
import pytest

from paper_1408_0698_gb300 import inputs, native
from _gpu import check_against_oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,N,nd,n_sub,layers,screen", [
    (8, 16, 8, 20, 1, 256), (8, 16, 8, 20, 3, 300), (8, 16, 8, 20, 4, 256), (3, 8, 4, 36, 6, 128), (3, 8, 4, 40, 6, 128),
    (9, 21, 7, 5, 2, 513), (11, 22, 11, 9, 1, 256), (16, 32, 16, 3, 1, 256), (5, 15, 5, 4, 6, 256)])
@pytest.mark.parametrize("lgs", [False, True])
def test_frames_around_the_limits(n, N, nd, n_sub, layers, screen, lgs):
    cfg = inputs.config1(inputs.PREC_FP32)
    cfg.geometries = [inputs.Geometry(n_sub, n, N, nd, 0.5, inputs.PREC_FP32)]
    dx = 8.0 / (n_sub * n)
    ar = np.arange(layers, dtype=np.float64)
    cfg.layers = inputs.Layers(alt_m=2000.0 * ar, wind_vx_mps=3.0 + ar, wind_vy_mps=-5.0 * ar, x0_m=0.3 * ar, y0_m=-0.2 * ar,
                               weights=np.full(layers, 1.0 / layers), screen_size=screen,
                               screen_dx_m=1.13 * dx if screen * 1.13 * dx > 10 else 12.0 / screen)
    if lgs:
        cfg.stars = [dataclasses.replace(inputs.config2().stars[0], geometry_index=0)]
    scr = inputs.make_screens(cfg.layers, 11)
    w = native.Wfs(cfg, seed=5, noise=False)
    d = torch.as_tensor(scr).cuda()
    out, again = (torch.zeros((max(w.total, 1), 2), device="cuda") for _ in range(2))
    native.wfs_measure(w.h, d.data_ptr(), 0.37, out.data_ptr(), 0)
    b = native.wfs_batch_create([w.h])
    native.wfs_batch_measure(b, [d.data_ptr()], [0.37], [again.data_ptr()], 0)
    torch.cuda.synchronize()
    native.wfs_sync_status(w.h)
    native.wfs_batch_destroy(b)
    assert torch.equal(out, again)
    check_against_oracle(cfg, scr, 0.37, out.cpu().numpy(), w.layouts)
    w.close()
