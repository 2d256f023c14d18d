"""Calibration layers, several modes per tile with the weights of every support unrolled: interaction
matrices of mirrors from one actuator per screen pixel (a tile's actuators are staged in parts) to
coarse ones, with mode counts around the pairs and the tile's eight modes, against the oracle (GPU)."""
import numpy as np
import pytest

from paper_1408_0698_gb300 import inputs, native
import oracle
from test_loop_gpu import _Loop, _calibrate, _small_cfg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("support,n_act,pitch,n_modes", [
    (1, 85, 0.05, 3), (2, 40, 0.11, 8), (3, 81, 0.05, 9), (4, 30, 0.16, 1), (5, 12, 0.4, 17),
    (6, 60, 0.07, 2), (7, 9, 0.5, 5), (8, 85, 0.05, 10), (8, 2, 3.0, 1)])
def test_layers_of_many_modes_match_oracle(support, n_act, pitch, n_modes):
    cfg, amp = _small_cfg(), 0.5
    dm = inputs.Dm(n_act, pitch, 0.0, n_modes, coupling=0.3, support=support)
    M = inputs.modal_base(dm, 60 + support, amplitude_m=2e-8)
    L = _Loop(cfg, [dm], [M], np.zeros((n_modes, 2)), np.zeros(n_modes))
    im = _calibrate(L, 0, amp, native.wfs_num_valid(L.w.h, 0))
    ref = oracle.interaction_matrix(cfg, 0, [dm], [M], amp)
    L.close()
    # FP32 slopes are within 1e-4 px of the exact ones by a wide margin (their bar is 1e-3 RMS); a row
    # is a difference of two over twice the amplitude.  A wrong or missing weight of the smallest
    # influence that matters moves a layer by percents.
    tol = 1e-4 / amp
    assert np.sqrt(np.mean(ref ** 2)) > 10 * tol
    assert np.max(np.abs(im - ref)) < tol
