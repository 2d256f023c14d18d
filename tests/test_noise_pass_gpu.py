"""The noise stage's pair kernel at the edges of its range, and the choice between the noise pass
and the centroid in the spot kernel (32-point geometries; GPU)."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_1408_0698_gb300 import inputs, native

pytestmark = pytest.mark.gpu


def _noise(e, pixel0, offset=0, ron=2.5):
    buf_e = torch.zeros(e.numel() + offset, device="cuda")
    buf_c = torch.full((e.numel() + offset,), float("nan"), device="cuda")
    buf_e[offset:] = e
    native.wfs_noise_apply(buf_e[offset:].data_ptr(), e.numel(), ron, 77, 3, 0.125, pixel0,
                           buf_c[offset:].data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert torch.isnan(buf_c[:offset]).all()
    return buf_c[offset:].cpu().numpy()


@pytest.mark.parametrize("first,count,offset", [(0, 1, 0), (1, 1, 0), (1, 2, 1), (0, 3, 1), (5, 62, 0), (7, 511, 3),
                                                (64, 513, 1), (0xFFFFFFFD - 1000, 1000, 0)])
def test_noise_range_is_a_slice_of_the_whole(first, count, offset):
    # a pixel's noise depends on its index alone, whatever range, alignment or neighbour it is drawn with
    base = max(0, first - 3) & ~1
    e = torch.as_tensor(inputs.random_expected_image(first - base + count + 5, 11)).cuda()
    whole = _noise(e, base)
    part = _noise(e[first - base: first - base + count], first, offset)
    np.testing.assert_array_equal(part, whole[first - base: first - base + count])


def test_noise_of_means_without_a_draw_and_large_means():
    e = torch.tensor([0.0, -1.0, float("nan"), 15.999999, 16.0, 1e-30, 400.0, 3e-8], device="cuda")
    c = _noise(e, 0, ron=0.0)
    assert np.all(c[[0, 1, 2, 5]] == 0.0) and np.all(c >= 0.0) and np.all(c == np.rint(c)) and c[6] > 200


def _elt_small(n, lgs, precision):
    cfg = inputs.config1(precision)
    cfg.geometries = [inputs.Geometry(12, n, 32, 16, 0.5, precision)]
    cfg.layers = dataclasses.replace(cfg.layers, screen_dx_m=8.0 / (12 * n))
    if lgs:
        cfg.stars = [inputs.config2().stars[0]]
    return cfg


@pytest.mark.parametrize("n,lgs,precision", [(10, True, inputs.PREC_BF16X3), (8, False, inputs.PREC_FP16S),
                                             (10, True, inputs.PREC_FP32), (8, True, inputs.PREC_FP32)])
def test_batch_follows_the_noise_switch(n, lgs, precision):
    """A class of a batch takes the noise pass while one of its instances has noise on; its noise-free
    instances give the same slopes either way, those of the handle alone."""
    cfg = _elt_small(n, lgs, precision)
    scr = torch.as_tensor(inputs.make_screens(cfg.layers, 5)).cuda()
    ws = [native.Wfs(cfg, seed=9 + i, noise=False) for i in range(2)]
    sp = torch.cuda.current_stream().cuda_stream

    def alone():
        out = []
        for w in ws:
            s = torch.full((w.total, 2), float("nan"), device="cuda")
            native.wfs_measure(w.h, scr.data_ptr(), 0.01, s.data_ptr(), sp)
            out.append(s)
        torch.cuda.synchronize()
        return [s.cpu().numpy() for s in out]

    b = native.wfs_batch_create([w.h for w in ws])

    def batched(subset):
        out = [torch.full((w.total, 2), float("nan"), device="cuda") for w in ws]
        args = ([scr.data_ptr()] * 2, [0.01] * 2, [s.data_ptr() for s in out], sp)
        if subset:
            native.wfs_batch_measure_subset(b, 0, [0, 1], *args)
        else:
            native.wfs_batch_measure(b, *args)
        torch.cuda.synchronize()
        return [s.cpu().numpy() for s in out]

    quiet = alone()
    for noise in ((0, 0), (0, 1), (0, 0), (1, 1)):
        for w, k in zip(ws, noise):
            native.wfs_set_noise(w.h, k)
        ref = alone()
        for subset in (False, True):
            for got, want in zip(batched(subset), ref):
                np.testing.assert_array_equal(got, want)
        for i in range(2):
            assert np.array_equal(ref[i], quiet[i]) == (not noise[i])
    native.wfs_batch_destroy(b)
    for w in ws:
        w.close()
