"""The FP32 warp-per-subaperture spot kernel (N <= 32, 3 <= n <= 16) where its folded transforms can
go wrong: odd and even sizes, the smallest and largest of its range, a single detector pixel, and
odd pixel counts whose generator pairs straddle two subapertures (GPU, against the FP64 oracle with
the open-loop bars)."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1408_0698_gb300 import inputs, native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from _gpu import run_library  # noqa: E402
from test_parity_gpu import _check_wfs, _small_cfg  # noqa: E402

GEOMETRIES = [  # n, N, nd
    (3, 5, 5), (3, 32, 1), (4, 7, 7), (4, 31, 31), (5, 9, 3), (6, 11, 11), (6, 32, 32), (7, 13, 13), (8, 15, 5),
    (9, 32, 8), (10, 19, 19), (11, 21, 7), (12, 24, 12), (13, 25, 25), (14, 28, 4), (15, 29, 29), (16, 31, 31), (16, 32, 2),
]


@pytest.mark.parametrize("n,N,nd", GEOMETRIES)
@pytest.mark.parametrize("lgs,per_slice", [(False, False), (True, False), (True, True)])
def test_row_geometries(n, N, nd, lgs, per_slice):
    cfg = _small_cfg(5, n, N, nd, lgs)
    if per_slice:
        cfg = dataclasses.replace(cfg, stars=[dataclasses.replace(s, per_slice=True) for s in cfg.stars])
    scr = inputs.make_screens(cfg.layers, 6)
    gpu, w = run_library(cfg, scr, 0.004)
    _check_wfs(cfg, scr, 0.004, gpu)
    w.close()


@pytest.mark.parametrize("n,N,nd", [(4, 14, 7), (6, 25, 5), (8, 32, 16), (10, 32, 16), (16, 32, 32)])
@pytest.mark.parametrize("photons", [30.0, 4000.0])
def test_row_noise_counts(n, N, nd, photons):
    """Counts from the stored means by the oracle's generator: equal except where a draw sits on a
    rounding boundary (the bar of the noise stage: 99.99 % of the pixels; read noise to 1e-4)."""
    cfg = _small_cfg(6, n, N, nd, False, photons=photons)
    scr = inputs.make_screens(cfg.layers, 8)
    gpu, w = run_library(cfg, scr, 0.007, seed=31, noise=True)
    E, C = gpu[0]["E"].reshape(-1), gpu[0]["C"].reshape(-1)
    ref = oracle.noise_image(E, cfg.stars[0].read_noise_e, 31, 0, 0.007, 0)[0]
    assert np.sum(np.abs(C - ref) > 1e-4) <= max(1, 1e-4 * C.size)
    c = (nd - 1) / 2
    C = C.reshape(-1, nd, nd).astype(np.float64)
    tot = C.sum(axis=(1, 2))
    x = np.arange(nd) - c
    want = np.stack([(C * x).sum(axis=(1, 2)), (C * x[:, None]).sum(axis=(1, 2))], axis=1) / np.where(tot > 0, tot, 1)[:, None]
    ok = tot > 20.0
    np.testing.assert_allclose(gpu[0]["slopes"][ok], want[ok], atol=1e-4 * nd)
    w.close()


@pytest.mark.parametrize("lgs,noise", [(True, True), (False, True), (True, False)])
def test_static_entry_equals_the_handle_on_32_points(lgs, noise):
    cfg = _small_cfg(9, 10, 32, 16, lgs)
    scr = torch.as_tensor(inputs.make_screens(cfg.layers, 3)).cuda()
    w = native.Wfs(cfg, seed=5, noise=noise)
    tel, stars, geoms, lay, keep = native.marshal(cfg)
    out = [torch.full((w.total, 2), float("nan"), device="cuda") for _ in range(2)]
    stream = torch.cuda.current_stream().cuda_stream
    native.wfs_measure(w.h, scr.data_ptr(), 0.01, out[0].data_ptr(), stream)
    native.wfs_measure_one_static(tel, geoms[0], stars[0], lay, scr.data_ptr(), 0.01, 5, 0, noise, out[1].data_ptr(),
                                  w.total, stream)
    torch.cuda.synchronize()
    assert np.array_equal(out[0].cpu().numpy(), out[1].cpu().numpy())
    w.close()
