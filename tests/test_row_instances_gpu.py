"""The FP32 warp-per-subaperture kernel takes another instance (registers, CTAs per SM) by the number of
subapertures of a launch: the same star measured in launches on every side of those limits gives the
same bits, with and without noise and in the LGS per-slice model, and the oracle's slopes (GPU)."""
import dataclasses

import numpy as np
import pytest

from paper_1408_0698_gb300 import inputs, native

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
from _gpu import check_against_oracle, run_library  # noqa: E402


def _cfg(n, N, nd, stars, per_slice):
    """Stars of 40 x 40 (1,264 subapertures each) on config 2's layers: 1, 2 and 3 of them fit the SMs at
    two CTAs of eight warps, at three, and not at once."""
    base = inputs.config2()
    dx = 8.0 / (40 * n)
    lay = dataclasses.replace(base.layers, screen_dx_m=1.04 * dx)
    all_stars = [dataclasses.replace(s, per_slice=per_slice) if s.is_lgs else s for s in base.stars]
    return dataclasses.replace(base, geometries=[inputs.Geometry(40, n, N, nd, 0.5, inputs.PREC_FP32)], layers=lay,
                               stars=[all_stars[i] for i in stars])


@pytest.mark.parametrize("n,N,nd", [(10, 32, 16), (8, 32, 16), (6, 24, 12), (9, 21, 7), (12, 24, 24)])
@pytest.mark.parametrize("per_slice", [False, True])
@pytest.mark.parametrize("first", [0, 3])  # an LGS, the NGS
def test_same_bits_in_launches_of_any_size(n, N, nd, per_slice, first):
    others = [i for i in (0, 1, 2, 3) if i != first]
    got = []
    for k in (1, 2, 3):
        cfg = _cfg(n, N, nd, [first] + others[: k - 1], per_slice)
        scr = inputs.make_screens(cfg.layers, 17)
        runs = []
        for noise in (False, True):
            r, w = run_library(cfg, scr, 0.019, seed=4, noise=noise)
            runs.append(r[0])
            if not noise:
                assert w.total == k * w.layouts[0].n_valid and 1216 < w.layouts[0].n_valid <= 1280
                check_against_oracle(cfg, scr, 0.019, np.concatenate([x["slopes"] for x in r]), w.layouts)
            w.close()
        got.append(runs)
    for runs in got[1:]:
        for a, b in zip(runs, got[0]):
            for key in ("slopes", "opd", "I", "E", "C"):
                np.testing.assert_array_equal(a[key], b[key], err_msg=key)
