"""The LGS per-slice model with layers or mirrors above the lowest slices, as a low beacon has them (GPU): such
a slice sees the layer through a negative cone, projected like any other against the oracle; slices whose
footprint on a layer would not fit the screen are refused."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1408_0698_gb300 import inputs, native

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
from _gpu import run_library, slope_rms  # noqa: E402
from test_parity_gpu import SLOPE_RMS, _check_wfs  # noqa: E402


def _cfg(n, N, nd, precision, alts, slices):
    base = inputs.config2()
    ar = np.arange(len(alts), dtype=np.float64)
    lay = dataclasses.replace(base.layers, alt_m=np.asarray(alts), wind_vx_mps=3.0 + ar, wind_vy_mps=-5.0 * ar,
                              x0_m=0.3 * ar, y0_m=-0.2 * ar, weights=np.full(len(alts), 1.0 / len(alts)),
                              screen_dx_m=1.03 * 8.0 / (14 * n))
    star = dataclasses.replace(base.stars[0], geometry_index=0, range_m=10e3, per_slice=True,
                               na_alt_m=np.asarray(slices), na_weight=np.full(len(slices), 1.0 / len(slices)))
    return dataclasses.replace(base, geometries=[inputs.Geometry(14, n, N, nd, 0.5, precision)], stars=[star], layers=lay)


SIZES = [(6, 24, 12, inputs.PREC_FP32), (10, 32, 16, inputs.PREC_FP32), (10, 32, 16, inputs.PREC_BF16X3),
         (10, 40, 20, inputs.PREC_FP32)]


@pytest.mark.parametrize("n,N,nd,precision", SIZES)
def test_layer_above_a_slice(n, N, nd, precision):
    cfg = _cfg(n, N, nd, precision, [0.0, 4e3, 9.2e3], [8.8e3, 9.2e3, 10e3])
    scr = inputs.make_screens(cfg.layers, 12)
    for t in (0.0, 0.23):
        gpu, w = run_library(cfg, scr, t)
        _check_wfs(cfg, scr, t, gpu)
        w.close()


@pytest.mark.parametrize("n,N,nd,precision", SIZES)
def test_mirror_above_a_slice(n, N, nd, precision):
    cfg = _cfg(n, N, nd, precision, [0.0, 4e3], [8.8e3, 10e3])
    scr = inputs.make_screens(cfg.layers, 13)
    dms = [inputs.Dm(15, 8.0 / 14, 0.0, 5), inputs.Dm(13, 0.8, 9.3e3, 4)]
    m2a = [inputs.modal_base(d, 3 + i, amplitude_m=2e-8) for i, d in enumerate(dms)]
    w = native.Wfs(cfg)
    Ms = [torch.as_tensor(M).cuda() for M in m2a]
    cm = inputs.random_control_matrix(9, 2 * w.total, seed=5, scale=0.5)
    gain = np.full(9, 0.4)
    cm_d, g_d = torch.as_tensor(cm).cuda(), torch.as_tensor(gain.astype(np.float32)).cuda()
    lp = native.wfs_loop_create(w.h, [native.wfs_dm(d.n_act, d.pitch_m, d.alt_m, d.coupling, d.support, d.n_modes,
                                                    M.data_ptr()) for d, M in zip(dms, Ms)], cm_d.data_ptr(), g_d.data_ptr())
    c0 = np.random.default_rng(8).standard_normal(9).astype(np.float32)
    c_d = torch.as_tensor(c0).cuda()
    st = torch.cuda.current_stream().cuda_stream
    native.wfs_loop_set_coeffs(lp, w.h, c_d.data_ptr(), st)
    s = torch.zeros((w.total, 2), device="cuda")
    native.wfs_loop_step(lp, w.h, torch.as_tensor(scr).cuda().data_ptr(), 0.01, s.data_ptr(), st)
    torch.cuda.synchronize()
    native.wfs_sync_status(w.h)
    s_ref, _ = oracle.loop_step(cfg, scr, 0.01, dms, m2a, cm, gain, c0.astype(np.float64))
    assert slope_rms(s.cpu().numpy(), s_ref) < SLOPE_RMS
    native.wfs_loop_destroy(lp)
    w.close()


def test_footprints_larger_than_the_screen_are_refused():
    # nothing is launched: the cone of a slice at 30 m on a layer at 9.2 km is -306
    with pytest.raises(native.WfsError, match="WFS_EINVAL"):
        native.Wfs(_cfg(6, 24, 12, inputs.PREC_FP32, [0.0, 9.2e3], [30.0, 10e3]))
