"""The error of a push-pull pair measured from one wavefront (32-point tensor-core geometries), against the
FP64 oracle's interaction matrix: no larger than that of the same modes pushed and pulled in two
measurements, whose roundings are independent and average out (GPU)."""
import ctypes
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1408_0698_gb300 import inputs, native

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [8, 10])
@pytest.mark.parametrize("lgs", [False, True])
# the operands' split, the same in both forms, is most of the error in BF16X3 and little of it in FP16S: a
# hundredth is left there for what the FP32 roundings can differ by
@pytest.mark.parametrize("precision,most", [(inputs.PREC_FP16S, 1.0), (inputs.PREC_BF16X3, 1.01)])
def test_pair_error(n, lgs, precision, most):
    D, n_sub, n_modes, amplitude = 8.0, 20, 37, 1.0
    cfg = inputs.config1(precision)
    cfg.geometries = [inputs.Geometry(n_sub, n, 32, 16, 0.5, precision)]
    cfg.layers = dataclasses.replace(cfg.layers, screen_dx_m=D / (n_sub * n))
    if lgs:
        cfg.stars = [inputs.config2().stars[0]]
    dm = inputs.Dm(n_sub + 1, D / n_sub, 0.0, n_modes)
    m2a_host = inputs.modal_base(dm, 5, amplitude_m=3e-8)
    ref = oracle.interaction_matrix(cfg, 0, [dm], [m2a_host], amplitude)
    w = native.Wfs(cfg, seed=3, noise=False)
    m2a = torch.as_tensor(m2a_host).cuda()
    cm, gain = torch.zeros((n_modes, 2 * w.total), device="cuda"), torch.zeros(n_modes, device="cuda")
    lp = native.wfs_loop_create(w.h, [native.wfs_dm(dm.n_act, dm.pitch_m, 0.0, dm.coupling, dm.support, n_modes,
                                                    ctypes.c_void_p(m2a.data_ptr()))], cm.data_ptr(), gain.data_ptr())
    st = torch.cuda.current_stream().cuda_stream
    im = torch.zeros((n_modes, 2 * w.total), device="cuda")
    native.wfs_loop_calibrate(lp, w.h, 0, amplitude, im.data_ptr(), st)
    # a mode in the beam, then its negative (a coefficient takes its shape out of the beam)
    flat = torch.zeros((cfg.layers.n_layers, cfg.layers.screen_size, cfg.layers.screen_size), device="cuda")
    s = torch.zeros((2, n_modes, w.total, 2), device="cuda")
    for k in range(n_modes):
        for i, sign in enumerate((-1.0, 1.0)):
            c = torch.zeros(n_modes, device="cuda")
            c[k] = sign * amplitude
            native.wfs_loop_set_coeffs(lp, w.h, c.data_ptr(), st)
            native.wfs_loop_step(lp, w.h, flat.data_ptr(), 0.0, s[i, k].data_ptr(), st)
    torch.cuda.synchronize()
    native.wfs_sync_status(w.h)
    native.wfs_loop_destroy(lp)
    two = ((s[0] - s[1]) / (2 * amplitude)).reshape(n_modes, -1).cpu().numpy()
    ref = np.asarray(ref, np.float64).reshape(n_modes, -1)
    err = [np.sqrt(np.mean((x.astype(np.float64) - ref) ** 2)) for x in (im.cpu().numpy(), two)]
    assert err[1] < 1e-5 / amplitude  # the two measurements are the oracle's modes
    assert err[0] <= most * err[1], err[0] / err[1]
    w.close()
