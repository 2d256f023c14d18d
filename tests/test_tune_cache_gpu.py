"""Launch shapes saved for a kernel that is gone are not taken for the one that has its number (GPU)."""
import pytest

from paper_1408_0698_gb300 import inputs, native

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_shapes_of_a_deleted_kernel_are_not_taken(tmp_path, monkeypatch):
    path = tmp_path / "tune.txt"
    name = torch.cuda.get_device_name(0).replace(" ", "_")
    path.write_text("".join(f"kind1_n10_N32_nd16_sub{1 << k}_{name} 304 4\n" for k in range(20)))
    monkeypatch.setenv("GBWFS_TUNE_CACHE", str(path))
    cfg = inputs.config1(inputs.PREC_FP32)
    cfg.geometries = [inputs.Geometry(12, 10, 32, 16, 0.5, inputs.PREC_FP32)]
    w = native.Wfs(cfg, seed=1)
    b = native.wfs_batch_create([w.h])
    info = native.wfs_batch_info(b)
    assert [(c["kind"], c["grid_cap"], c["cta_warps"]) for c in info] == [(1, 0, 0)]
    scr = torch.as_tensor(inputs.make_screens(cfg.layers, 1)).cuda()
    out = torch.empty((w.total, 2), device="cuda")
    native.wfs_batch_tune(b, [scr.data_ptr()], [0.0], [out.data_ptr()], 0)
    tuned = [(c["grid_cap"], c["cta_warps"]) for c in native.wfs_batch_info(b)]
    native.wfs_batch_destroy(b)
    b = native.wfs_batch_create([w.h])
    assert [(c["grid_cap"], c["cta_warps"]) for c in native.wfs_batch_info(b)] == tuned != [(0, 0)]
    native.wfs_batch_destroy(b)
    w.close()
