"""The copies of a projection box (GPU): screens at every offset from a 16-byte boundary give the OPD and the
slopes of aligned ones bit for bit, for boxes inside the screen and across its periodic edges, from one
column to the widest, and on screens narrower than a box."""
import dataclasses

import pytest

from paper_1408_0698_gb300 import inputs, native

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
from test_parity_gpu import _small_cfg  # noqa: E402


@pytest.mark.parametrize("n_sub,n,N,nd", [(1, 3, 6, 3), (13, 5, 10, 5), (8, 8, 16, 8), (7, 11, 22, 11), (4, 32, 64, 32)])
@pytest.mark.parametrize("S", ["tight", "wide"])
def test_offsets_give_the_same_bits(n_sub, n, N, nd, S):
    cfg = _small_cfg(n_sub, n, N, nd, True)
    P = n_sub * n
    size = (P // 2 + 8) // 4 * 4 if S == "tight" else (2 * P + 16) // 4 * 4
    cfg = dataclasses.replace(cfg, layers=dataclasses.replace(cfg.layers, screen_size=size))
    scr = torch.as_tensor(inputs.make_screens(cfg.layers, 4)).cuda().reshape(-1)
    w = native.Wfs(cfg, seed=1)
    n_opd = sum(L.n_valid * L.n * L.n for L in w.layouts)
    buf = torch.empty(scr.numel() + 4, device="cuda")
    for t in (0.0, 0.317, 5.2, 77.7):
        got = []
        for off in range(4):
            buf[off:off + scr.numel()] = scr
            opd, out = torch.full((n_opd,), float("nan"), device="cuda"), torch.full((w.total, 2), float("nan"), device="cuda")
            native.wfs_measure_stages(w.h, buf.data_ptr() + 4 * off, t, out.data_ptr(), opd.data_ptr())
            torch.cuda.synchronize()
            native.wfs_sync_status(w.h)
            got.append((opd, out))
        assert bool(torch.isfinite(got[0][0]).all())
        for opd, out in got[1:]:
            assert torch.equal(opd, got[0][0]) and torch.equal(out, got[0][1])
    w.close()
