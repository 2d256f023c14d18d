"""The projection's blocks at their edges (GPU, against the FP64 oracle with the open-loop bars): block
widths of one column to a full block and a remainder, one to three row parts per subaperture, screens
whose rows have no 16-byte alignment, screens hardly larger than the footprint (boxes across both
periodic edges), many layers, and more (sensor, layer) pairs than a block of threads keeps."""
import dataclasses

import numpy as np
import pytest

from paper_1408_0698_gb300 import inputs, native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from _gpu import run_library  # noqa: E402
from test_parity_gpu import _check_wfs, _small_cfg  # noqa: E402


@pytest.mark.parametrize("n_sub,n,N,nd", [(65, 1, 2, 1), (13, 5, 10, 5), (7, 11, 22, 11), (6, 12, 24, 12), (9, 22, 44, 4),
                                          (4, 32, 64, 32)])
@pytest.mark.parametrize("S", ["odd", "mod4", "tight", "pow2"])
def test_blocks(n_sub, n, N, nd, S):
    lgs = N >= 2 * n - 1 and n > 1
    cfg = _small_cfg(n_sub, n, N, nd, lgs)
    P = n_sub * n
    size = {"odd": P + 21, "mod4": (P + 26) // 4 * 4 + 2, "tight": (P // 2 + 8) // 4 * 4, "pow2": cfg.layers.screen_size}[S]
    if S == "odd":
        size |= 1
    cfg = dataclasses.replace(cfg, layers=dataclasses.replace(cfg.layers, screen_size=size))
    scr = inputs.make_screens(cfg.layers, 4)
    for t in (0.0, 0.317):
        gpu, w = run_library(cfg, scr, t)
        _check_wfs(cfg, scr, t, gpu)
        w.close()


def test_many_layers_and_sensors():
    cfg = _small_cfg(6, 6, 12, 6, False)
    alts = np.linspace(0.0, 9e3, 32)
    cfg.layers = inputs._layers(alts, np.ones(32), 0.1, 20.0, 64, 4.0 / 36)
    cfg.stars = [dataclasses.replace(cfg.stars[0], theta_x_rad=k * 2e-6) for k in range(20)]  # 640 pairs
    scr = inputs.make_screens(cfg.layers, 4)
    gpu, w = run_library(cfg, scr, 0.05)
    _check_wfs(cfg, scr, 0.05, gpu)
    w.close()
