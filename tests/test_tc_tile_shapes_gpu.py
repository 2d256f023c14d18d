"""The tensor-core kernel with six warpgroups per CTA (large launches, or the tuner's choice) measures
every class bit for bit as the handles alone do with two (GPU)."""
import numpy as np
import pytest

from paper_1408_0698_gb300 import inputs, native
from test_batch_gpu import _alone, _instances, _setup

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", [inputs.PREC_BF16X3, inputs.PREC_FP16S])
@pytest.mark.parametrize("count,cap,noise", [(1, 0, True), (16, 152, False), (16, 3, True)])
def test_six_warpgroups_give_the_same_results(prec, count, cap, noise, tmp_path, monkeypatch):
    path = tmp_path / "tune.txt"
    monkeypatch.setenv("GBWFS_TUNE_CACHE", str(path))
    insts = [c for c in _instances(3 * count + 6, 4400, prec) if c.geometries[0].precision == prec
             and c.geometries[0].n_fft == 32][:count]
    assert insts
    hs, scr, outs = _setup(insts, noise)
    ts = [0.002 + 1e-4 * i for i in range(len(hs))]
    b = native.wfs_batch_create([w.h for w in hs])
    native.wfs_batch_tune(b, [s.data_ptr() for s in scr], ts, [o.data_ptr() for o in outs], 0)
    native.wfs_batch_destroy(b)
    forced = [f"{ln.split()[0]} {cap} 24" for ln in path.read_text().split("\n") if ln.strip()]
    path.write_text("\n".join(forced) + "\n")
    b = native.wfs_batch_create([w.h for w in hs])
    assert all(c["cta_warps"] == 24 for c in native.wfs_batch_info(b))
    for o in outs:
        o.zero_()
    native.wfs_batch_measure(b, [s.data_ptr() for s in scr], ts, [o.data_ptr() for o in outs], 0)
    torch.cuda.synchronize()
    for i, (o, r) in enumerate(zip(outs, _alone(hs, scr, ts))):
        assert np.array_equal(o.cpu().numpy(), r), i
    native.wfs_batch_destroy(b)
    for w in hs:
        w.close()
