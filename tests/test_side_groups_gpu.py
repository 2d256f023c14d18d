"""Sensors of a geometry that is not the handle's largest (GPU): such a group runs on a side stream, and its
slopes and stages are those of the same stars measured by a handle of their own, bit for bit, and the
oracle's."""
import dataclasses

import numpy as np
import pytest

from paper_1408_0698_gb300 import inputs, native

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
from _gpu import run_library  # noqa: E402
from test_parity_gpu import _check_wfs  # noqa: E402


def _cfg(side, precision, big, uplink=0.0):
    """Config 2's layers on its telescope: a geometry of `big` and two LGS of a smaller geometry `side`
    = (n_sub, n, N, nd), of 3 and 5 sodium slices."""
    base = inputs.config2()
    n_sub, n, N, nd = side
    geoms = [big[0], inputs.Geometry(n_sub, n, N, nd, 0.5, precision)]
    lgs = [s for s in base.stars if s.is_lgs][:2]
    stars = list(big[1])
    for k, s in enumerate(lgs):
        h, w = inputs.sodium_slices(90e3, n_slices=3 + 2 * k)
        stars.append(dataclasses.replace(s, geometry_index=1, na_alt_m=h, na_weight=w, per_slice=True,
                                         spot_fwhm_rad=0.9 * inputs.ARCSEC, uplink_diameter_m=uplink, uplink_samples=12))
    return dataclasses.replace(base, geometries=geoms, stars=stars)


def _alone(cfg):
    stars = [dataclasses.replace(s, geometry_index=0) for s in cfg.stars if s.geometry_index == 1]
    return dataclasses.replace(cfg, geometries=[cfg.geometries[1]], stars=stars)


NGS_BIG = (inputs.Geometry(40, 6, 24, 12, 0.5, inputs.PREC_FP32),
           [dataclasses.replace(inputs.config1().stars[0], geometry_index=0)])
LGS_BIG = (inputs.Geometry(36, 8, 32, 16, 0.5, inputs.PREC_BF16X3),
           [dataclasses.replace(inputs.config2().stars[0], geometry_index=0, per_slice=True)])


@pytest.mark.parametrize("side,precision", [
    ((24, 10, 32, 16), inputs.PREC_BF16X3), ((12, 10, 32, 16), inputs.PREC_FP16S), ((9, 8, 32, 16), inputs.PREC_BF16X3),
    ((12, 10, 32, 16), inputs.PREC_FP32), ((9, 6, 24, 12), inputs.PREC_BF16X3), ((5, 10, 40, 20), inputs.PREC_FP32)])
@pytest.mark.parametrize("big,uplink", [(NGS_BIG, 0.0), (LGS_BIG, 0.4)])
def test_per_slice_side_group(side, precision, big, uplink):
    cfg = _cfg(side, precision, big, uplink)
    scr = inputs.make_screens(cfg.layers, 31)
    together, w = run_library(cfg, scr, 0.013)
    plain, _ = run_library(cfg, scr, 0.013, stages=False, handle=w)
    alone, v = run_library(_alone(cfg), scr, 0.013)
    assert len(alone) == 2 and w.layouts[0].n_valid > sum(L.n_valid for L in w.layouts[1:])
    for a, b, c in zip(together[1:], alone, plain[1:]):
        for key in ("slopes", "opd", "I", "E", "C"):
            np.testing.assert_array_equal(a[key], b[key], err_msg=key)
        np.testing.assert_array_equal(c["slopes"], b["slopes"])
    sel = [np.arange(k, L.n_valid, 1 + L.n_valid // 40, dtype=np.int32) for k, L in enumerate(w.layouts)]
    _check_wfs(cfg, scr, 0.013, together, sel=sel)
    w.close()
    v.close()


@pytest.mark.parametrize("n_sub,n,N,nd,precision,lgs,layers", [
    (20, 8, 16, 8, inputs.PREC_BF16X3, False, 1), (36, 6, 24, 12, inputs.PREC_FP16S, False, 3),
    (36, 6, 24, 12, inputs.PREC_BF16X3, True, 10), (10, 10, 32, 16, inputs.PREC_FP32, True, 3),
    (7, 16, 32, 32, inputs.PREC_FP32, False, 2), (3, 9, 21, 7, inputs.PREC_FP32, True, 10)])
def test_fp32_side_group_has_its_projection(n_sub, n, N, nd, precision, lgs, layers):
    """A side group of the warp-per-subaperture kernel, below and above the largest group's limits for
    projecting in the spot kernel: a projection launch of its own, the same bits as alone."""
    base = inputs.config2(inputs.PREC_BF16X3)
    ar = np.arange(layers, dtype=np.float64)
    lay = dataclasses.replace(base.layers, alt_m=1000.0 * ar, wind_vx_mps=3.0 + ar, wind_vy_mps=-5.0 * ar, x0_m=0.3 * ar,
                              y0_m=-0.2 * ar, weights=np.full(layers, 1.0 / layers))
    star = dataclasses.replace(base.stars[0 if lgs else 3], geometry_index=1)
    cfg = dataclasses.replace(base, layers=lay, geometries=base.geometries + [inputs.Geometry(n_sub, n, N, nd, 0.5, precision)],
                              stars=base.stars + [star])
    scr = torch.as_tensor(inputs.make_screens(lay, 3)).cuda()
    w, v = native.Wfs(cfg, seed=2), native.Wfs(_alone(cfg), seed=2)
    a, b = (torch.zeros((x.total, 2), device="cuda") for x in (w, v))
    native.wfs_measure(w.h, scr.data_ptr(), 0.021, a.data_ptr(), 0)
    native.wfs_measure(v.h, scr.data_ptr(), 0.021, b.data_ptr(), 0)
    native.wfs_timing_enable(w.h, True)
    native.wfs_measure(w.h, scr.data_ptr(), 0.021, a.data_ptr(), 0)
    torch.cuda.synchronize()
    assert native.wfs_timing_read(w.h)["project"][0] == 2
    assert torch.equal(a[-v.total:], b) and bool(torch.any(b != 0))
    w.close()
    v.close()
