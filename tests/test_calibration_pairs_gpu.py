"""Push-pull pairs from one wavefront (32-point tensor-core geometries): the interaction matrix of the
tensor-core kernel against that of the FP32 kernel, which measures every mode and its negative as two
instances (GPU)."""
import ctypes
import dataclasses

import numpy as np
import pytest

from paper_1408_0698_gb300 import inputs, native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _im(precision, n, lgs, n_modes, amplitude):
    D, n_sub = 8.0, 14
    cfg = inputs.config1(precision)
    cfg.geometries = [inputs.Geometry(n_sub, n, 32, 16, 0.5, precision)]
    cfg.layers = dataclasses.replace(cfg.layers, screen_dx_m=D / (n_sub * n))
    if lgs:
        cfg.stars = [inputs.config2().stars[0]]
    w = native.Wfs(cfg, seed=3, noise=True)  # a calibration takes no noise
    dm = inputs.Dm(n_sub + 1, D / n_sub, 0.0, n_modes)
    m2a = torch.as_tensor(inputs.modal_base(dm, 5, amplitude_m=3e-8)).cuda()
    cm, gain = torch.zeros((1, 1), device="cuda"), torch.zeros(n_modes, device="cuda")
    lp = native.wfs_loop_create(w.h, [native.wfs_dm(dm.n_act, dm.pitch_m, 0.0, dm.coupling, dm.support, n_modes,
                                                    ctypes.c_void_p(m2a.data_ptr()))], cm.data_ptr(), gain.data_ptr())
    im = torch.full((n_modes + 1, 2 * w.total), float("nan"), device="cuda")
    native.wfs_loop_calibrate(lp, w.h, 0, amplitude, im.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    native.wfs_sync_status(w.h)
    native.wfs_loop_destroy(lp)
    w.close()
    im = im.cpu().numpy()
    assert np.all(np.isnan(im[n_modes:]))
    return im[:n_modes].astype(np.float64)


@pytest.mark.parametrize("n", [8, 10])
@pytest.mark.parametrize("lgs", [False, True])
@pytest.mark.parametrize("precision,n_modes,amplitude", [(inputs.PREC_BF16X3, 70, 1.0), (inputs.PREC_FP16S, 64, -0.7),
                                                         (inputs.PREC_BF16X3, 1, 2.0)])
def test_pairs_match_two_instances(n, lgs, precision, n_modes, amplitude):
    # a slope of either precision is within 1e-4 px RMS of the exact one by a wide margin (its bar is
    # 1e-3), and a row is a difference of two over twice the amplitude
    a, b = _im(precision, n, lgs, n_modes, amplitude), _im(inputs.PREC_FP32, n, lgs, n_modes, amplitude)
    tol = 1e-4 / abs(amplitude)
    assert np.sqrt(np.mean(b ** 2)) > 100 * tol  # the modes move the spots
    assert np.sqrt(np.mean((a - b) ** 2)) < tol
    assert np.max(np.abs(a - b)) < 5 * tol
