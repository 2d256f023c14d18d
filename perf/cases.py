"""The measured workloads of the Shack-Hartmann library: what a Monte-Carlo simulation, a
calibration or a loop has the library do, through its public entry points.

Kinds of case:

* ``frame``: one open-loop frame of every guide star of a handle (``wfs_measure``; with
  ``stages``, ``wfs_measure_stages`` and its four intermediate outputs);
* ``batch``: frames of many uneven one-star instances in one call (``wfs_batch_measure``);
* ``loop``: one closed-loop step (``wfs_loop_step``) and the read-back of the coefficients;
* ``calibrate``: the push-pull interaction matrix of one star over the modes of a mirror
  (``wfs_loop_calibrate``);
* ``noise``: the detector-noise stage alone on given expected images (``wfs_noise_apply``).

Detector noise is on where a simulation of that kind runs with it and the result can be held
against another build's: a Poisson draw decided on a rounding boundary of its mean moves a slope
by a whole photon, so the larger geometries beside the headline frame are measured noise-free
(as error budgets and calibrations are), where a 64-bit reference exists too, and the noise
stage has a case of its own.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1408_0698_gb300 import inputs, native

PRECISIONS = {"fp32": inputs.PREC_FP32, "bf16x3": inputs.PREC_BF16X3, "fp16s": inputs.PREC_FP16S}
#: The tensor-core geometries (n_pix, n_fft, n_det) of the configurations.
TC_GEOMETRIES = [(8, 16, 8), (6, 24, 12), (8, 32, 16), (10, 32, 16)]


def _frame(name, **kw):
    """A frame case: a telescope, one geometry for the full-pupil sensors, optional 2 x 2 NGS."""
    c = {"kind": "frame", "diameter": 8.0, "obstruction": 0.0, "n_sub": 20, "n_pix": 8, "n_fft": 16,
         "n_det": 8, "precision": "fp32", "lgs": 0, "ngs": 1, "ngs_2x2": 0, "ring_arcsec": 60.0,
         "layers": 1, "top_m": 0.0, "screen": 256, "slices": 8, "uplink_m": 0.0, "per_slice": False,
         "noise": False, "stages": False}
    c.update(kw)
    if name:
        c["name"] = name
    return c


_ELT = dict(diameter=39.0, obstruction=0.28, n_sub=80, n_pix=10, n_fft=32, n_det=16, lgs=6, ngs=0, ngs_2x2=3,
            ring_arcsec=45.0, layers=10, top_m=20e3, screen=2048)
_MCAO = dict(n_sub=40, n_pix=6, n_fft=24, n_det=12, lgs=3, ngs=1, layers=3, top_m=10e3, screen=512)


def listed():
    return [
        # the smallest call in use: one 20 x 20 NGS on an 8 m telescope, noise on (latency, launches)
        _frame("ngs_8m_fp32", noise=True),
        # an 8 m MCAO frame, 3 LGS + 1 NGS 40 x 40, on the tensor-core kernel of its geometry
        _frame("mcao_8m_bf16x3", precision="bf16x3", **_MCAO),
        # the same in plain FP32 with every intermediate stage written (checking, visualisation)
        _frame("mcao_8m_fp32_stages", stages=True, **_MCAO),
        # a sensor outside the configured sizes: odd pixels, odd DFT, an odd number of subapertures
        _frame("odd_4m_fp32", diameter=4.2, obstruction=0.3, n_sub=37, n_pix=9, n_fft=21, n_det=7, lgs=2, ngs=1,
               layers=5, top_m=14e3, screen=768, slices=5),
        # the headline: the ELT frame, 6 LGS 80 x 80 + 3 NGS 2 x 2, 10 layers, noise on
        _frame("elt_bf16x3", precision="bf16x3", noise=True, **_ELT),
        # the ELT frame noise-free in plain FP32 (reference precision)
        _frame("elt_fp32", **_ELT),
        # the ELT frame in the more accurate split with the laser uplink tip-tilt on
        _frame("elt_fp16s_uplink", precision="fp16s", uplink_m=0.4, **_ELT),
        # the ELT frame with one wavefront and one DFT per sodium slice
        _frame("elt_slices_bf16x3", precision="bf16x3", per_slice=True, **_ELT),
        # a parameter sweep's step: 64 uneven one-star instances in one call
        {"name": "batch_64_bf16x3", "kind": "batch", "instances": 64, "precision": "bf16x3", "draw": 4000},
        # one closed-loop step of the ELT frame with its three mirrors (8200 modes)
        dict(_frame("loop_elt_bf16x3", precision="bf16x3", **_ELT), kind="loop", mirrors=3, mode_share=1.0),
        # the ground mirror's interaction matrix: 5000 modes, push-pull, one 80 x 80 LGS
        {"name": "calibrate_m4_bf16x3", "kind": "calibrate", "n_sub": 80, "n_pix": 10, "precision": "bf16x3",
         "n_act": 81, "modes": 5000},
        # the noise stage on the ELT frame's detector pixels (6 x 4632 subapertures of 16 x 16)
        {"name": "noise_7m_pixels", "kind": "noise", "pixels": 6 * 4632 * 256, "mean": 500.0 / 256},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["frame", "batch", "loop", "calibrate", "noise"], [12, 2, 2, 2, 2])[0]
    if kind == "noise":
        return {"kind": kind, "pixels": _log(rng, 20_001, 7_113_728), "mean": round(math.exp(rng.uniform(-2.0, 3.5)), 3)}
    if kind == "batch":
        return {"kind": kind, "instances": _log(rng, 3, 64), "precision": rng.choice(list(PRECISIONS)),
                "draw": rng.randrange(1 << 20)}
    if kind == "calibrate":
        n_sub = rng.randint(20, 80)
        return {"kind": kind, "n_sub": n_sub, "n_pix": rng.choice([8, 10]), "precision": rng.choice(list(PRECISIONS)),
                "n_act": n_sub + 1, "modes": _log(rng, 5, 300)}
    if kind == "frame" and rng.random() < 0.4:  # the plain FP32 geometries, odd sizes among them
        n = rng.randint(3, 16)
        b = rng.randint(1, 3)
        nd = rng.randint(-(-(2 * n - 1) // b), max(-(-(2 * n - 1) // b), 40 // b))
        geom, precision = (n, b * nd, nd), "fp32"
    else:
        geom, precision = rng.choice(TC_GEOMETRIES), rng.choice(list(PRECISIONS))
    n, N, nd = geom
    elt = rng.random() < 0.4
    D = round(rng.uniform(25.0, 40.0) if elt else rng.uniform(3.0, 12.0), 2)
    n_sub = rng.randint(41, 80) if elt else _log(rng, 7, 40)
    if kind == "loop":
        n_sub = max(n_sub, 20)
    lgs = rng.randint(0, 6)
    ngs = rng.randint(0 if lgs else 1, 2)
    per_slice = kind == "frame" and lgs > 0 and rng.random() < 0.25
    layers = rng.randint(1, 10)
    c = _frame(None, kind=kind, diameter=D, obstruction=rng.choice([0.0, 0.14, 0.28]), n_sub=n_sub, n_pix=n, n_fft=N,
               n_det=nd, precision=precision, lgs=lgs, ngs=ngs, ngs_2x2=rng.randint(0, 3) if elt else 0,
               ring_arcsec=round(rng.uniform(10.0, 60.0), 1), layers=layers,
               top_m=round(rng.uniform(5e3, 20e3)) if layers > 1 else 0.0,
               screen=-(-max(128, int(1.5 * n_sub * n + 64)) // 128) * 128, slices=rng.randint(3, 8),
               uplink_m=rng.choice([0.0, 0.0, 0.3, 0.5]) if lgs else 0.0, per_slice=per_slice,
               stages=kind == "frame" and not elt and rng.random() < 0.2)
    c["noise"] = kind == "frame" and ((N == 32 and nd == 16 and not per_slice and precision != "fp32")
                                      or (n_sub <= 20 and lgs == 0 and ngs == 1)) and rng.random() < 0.5
    if kind == "loop":
        c.update(mirrors=rng.randint(1, 3), mode_share=round(rng.uniform(0.1, 1.0), 2))
    return c


# ----------------------------------------------------------------------- descriptions

def _layer_set(alts, weights, S, dx):
    alts, w = np.asarray(alts, dtype=np.float64), np.asarray(weights, dtype=np.float64)
    d = np.radians(36.0 * np.arange(len(alts)))
    return inputs.Layers(alt_m=alts, wind_vx_mps=10.0 * np.cos(d), wind_vy_mps=10.0 * np.sin(d), x0_m=np.zeros(len(alts)),
                         y0_m=np.zeros(len(alts)), screen_size=int(S), screen_dx_m=dx, r0_m=0.157, L0_m=25.0,
                         weights=w / w.sum())


def _lgs(r, az, slices, geometry=0, **kw):
    h, w = inputs.sodium_slices(90e3, n_slices=slices)
    return inputs.GuideStar(is_lgs=True, theta_x_rad=r * math.cos(az), theta_y_rad=r * math.sin(az), range_m=90e3,
                            wavelength_m=inputs.LAMBDA_NA, geometry_index=geometry, launch_x_m=5.0 * math.cos(az),
                            launch_y_m=5.0 * math.sin(az), spot_fwhm_rad=inputs.ARCSEC, na_alt_m=h, na_weight=w, **kw)


def _ngs(r, az, wavelength=700e-9, geometry=0, photons=500.0):
    return inputs.GuideStar(is_lgs=False, theta_x_rad=r * math.cos(az), theta_y_rad=r * math.sin(az), range_m=math.inf,
                            wavelength_m=wavelength, geometry_index=geometry, photons_per_subap=photons)


def _config(c):
    """The frame's description (inputs.Config) of a frame or loop case."""
    ring = c["ring_arcsec"] * inputs.ARCSEC
    geoms = [inputs.Geometry(c["n_sub"], c["n_pix"], c["n_fft"], c["n_det"], 0.5, PRECISIONS[c["precision"]])]
    stars = [_lgs(ring, 2 * math.pi * k / c["lgs"], c["slices"], uplink_diameter_m=c["uplink_m"], uplink_samples=24,
                  per_slice=c["per_slice"]) for k in range(c["lgs"])]
    stars += [_ngs(0.0 if k == 0 else ring, k * 2.1) for k in range(c["ngs"])]
    if c["ngs_2x2"]:
        geoms.append(inputs.Geometry(2, 32, 64, 32, 0.5, inputs.PREC_FP32))
        stars += [_ngs(60.0 * inputs.ARCSEC, 2 * math.pi * k / c["ngs_2x2"], 1650e-9, 1, 5000.0) for k in range(c["ngs_2x2"])]
    weights = ([0.5, 0.1, 0.08, 0.07, 0.06, 0.05, 0.045, 0.035, 0.03, 0.03])[: c["layers"]]
    lay = _layer_set(np.linspace(0.0, c["top_m"], c["layers"]), weights, c["screen"], c["diameter"] / (c["n_sub"] * c["n_pix"]))
    return inputs.Config("frame", inputs.Telescope(c["diameter"], c["obstruction"]), geoms, stars, lay, seed=0)


def _instances(c):
    """The batch's one-star descriptions."""
    return inputs.config4_instances(c["instances"], seed=c["draw"], precision=PRECISIONS[c["precision"]])


def _calibration(c):
    """One LGS on the pupil of the calibrated mirror, and the mirror (one actuator per corner)."""
    D = 39.0 * c["n_sub"] / 80
    lay = _layer_set([0.0], [1.0], 128 * -(-c["n_sub"] * c["n_pix"] // 50), D / (c["n_sub"] * c["n_pix"]))
    geom = inputs.Geometry(c["n_sub"], c["n_pix"], 32, 16, 0.5, PRECISIONS[c["precision"]])
    cfg = inputs.Config("calibration", inputs.Telescope(D, 0.28), [geom], [_lgs(45.0 * inputs.ARCSEC, 0.0, 8)], lay, seed=0)
    return cfg, inputs.Dm(c["n_act"], D / c["n_sub"], 0.0, c["modes"])


def _mirrors(c):
    """The loop's mirrors: the ELT's three, scaled to the pupil and to a share of their modes."""
    scale = c["diameter"] / 39.0
    out = []
    for d in inputs.elt_dms()[: c["mirrors"]]:
        n = max(5, int(round((c["n_sub"] + 1) if d.alt_m == 0.0 else d.n_act * max(0.4, scale))))
        pitch = c["diameter"] / c["n_sub"] if d.alt_m == 0.0 else d.pitch_m
        out.append(inputs.Dm(n, pitch, d.alt_m, max(4, min(n * n, int(d.n_modes * c["mode_share"] * n * n / d.n_act ** 2)))))
    return out


# ----------------------------------------------------------------------- inputs

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _screens(lay, g):
    """[L][S][S] FP32 von Karman OPD screens (metres) of a layer set, made on the GPU."""
    S, dx = lay.screen_size, lay.screen_dx_m
    k = torch.fft.fftfreq(S, d=dx, dtype=torch.float64, device="cuda")
    k2 = k[:, None] ** 2 + k[None, :] ** 2 + lay.L0_m ** -2
    out = torch.empty((lay.n_layers, S, S), device="cuda")
    for l in range(lay.n_layers):
        r0 = lay.r0_m * float(lay.weights[l]) ** -0.6
        amp = (0.023 * r0 ** (-5.0 / 3.0) * k2 ** (-11.0 / 6.0)).sqrt() / (S * dx)
        amp[0, 0] = 0.0
        noise = torch.complex(torch.randn((S, S), generator=g, device="cuda"), torch.randn((S, S), generator=g, device="cuda"))
        out[l] = torch.fft.fft2(noise * amp.float()).real * (inputs.R0_WAVELENGTH / (2 * math.pi))
    return out


def _time(seed):
    return (seed * 7 % 500 + 1) * 1e-3  # a step of a run of half a second at 1 kHz


def _stream():
    return torch.cuda.current_stream().cuda_stream


class State:
    """What a user's program holds: the handle (and loop or batch) and its device buffers."""

    def __init__(self, **kw):
        self.loop = self.batch = None
        self.handles = []
        self.__dict__.update(kw)

    def __del__(self):
        try:
            if self.loop:
                native.wfs_loop_destroy(self.loop)
            if self.batch:
                native.wfs_batch_destroy(self.batch)
            for w in self.handles:
                w.close()
        except Exception:
            pass


def _modal_base(dm, g):
    return torch.randn((dm.n_act * dm.n_act, dm.n_modes), generator=g, device="cuda") * 1e-8


def _loop(w, dms, m2a, cm, gain):
    structs = [native.wfs_dm(d.n_act, d.pitch_m, d.alt_m, d.coupling, d.support, d.n_modes, ctypes.c_void_p(m.data_ptr()))
               for d, m in zip(dms, m2a)]
    return native.wfs_loop_create(w.h, structs, cm.data_ptr(), gain.data_ptr())


def _loop_inputs(c, g, n_slopes):
    dms = _mirrors(c)
    n = sum(d.n_modes for d in dms)
    m2a = [_modal_base(d, g) for d in dms]
    cm = (torch.rand((n, n_slopes), generator=g, device="cuda") - 0.5) * (2e-3 / math.sqrt(n_slopes))
    gain = 0.3 + 0.2 * torch.rand(n, generator=g, device="cuda")
    return dms, m2a, cm, gain


def _expected(c, g):
    """Expected photon counts of detector pixels: most faint, some bright, as in a spot."""
    e = torch.rand(c["pixels"], generator=g, device="cuda") ** 6 * (7.0 * c["mean"])
    e[torch.rand(c["pixels"], generator=g, device="cuda") < 0.02] = 0.0
    return e


def prepare(case, seed):
    c, g = case, _generator(seed)
    if c["kind"] == "noise":
        return State(case=c, seed=seed, expected=_expected(c, g), counts=torch.empty(c["pixels"], device="cuda"))
    if c["kind"] == "batch":
        cfgs = _instances(c)
        ws = [native.Wfs(f, seed=seed + i, noise=False) for i, f in enumerate(cfgs)]
        scr = [_screens(f.layers, g) for f in cfgs]
        out = [torch.empty((w.total, 2), device="cuda") for w in ws]
        ts = [_time(seed + i) for i in range(len(ws))]
        return State(case=c, handles=ws, batch=native.wfs_batch_create([w.h for w in ws]), screens=scr, slopes=out, ts=ts)
    if c["kind"] == "calibrate":
        cfg, dm = _calibration(c)
        w = native.Wfs(cfg, seed=seed, noise=False)
        m2a = _modal_base(dm, g)
        cm, gain = torch.zeros((1, 1), device="cuda"), torch.zeros(dm.n_modes, device="cuda")  # not read by a calibration
        return State(case=c, handles=[w], loop=_loop(w, [dm], [m2a], cm, gain), keep=(m2a, cm, gain),
                     im=torch.empty((dm.n_modes, 2 * w.total), device="cuda"))
    cfg = _config(c)
    w = native.Wfs(cfg, seed=seed, noise=c["noise"])
    s = State(case=c, handles=[w], screens=_screens(cfg.layers, g), t=_time(seed), slopes=torch.empty((w.total, 2), device="cuda"))
    if c["kind"] == "loop":
        dms, m2a, cm, gain = _loop_inputs(c, g, 2 * w.total)
        s.keep, s.coeffs = (m2a, cm, gain), torch.empty(cm.shape[0], device="cuda")
        s.loop = _loop(w, dms, m2a, cm, gain)
    if c["stages"]:
        size = {k: 0 for k in ("opd", "intensity", "expected", "counts")}
        for L in w.layouts:
            for k, n in (("opd", L.n), ("intensity", L.n_fft), ("expected", L.n_det), ("counts", L.n_det)):
                size[k] += L.n_valid * n * n
        s.out = {k: torch.empty(n, device="cuda") for k, n in size.items()}
    return s


def run(s):
    kind = s.case["kind"]
    if kind == "noise":
        native.wfs_noise_apply(s.expected.data_ptr(), s.expected.numel(), 3.0, s.seed, 1, _time(s.seed), 0,
                               s.counts.data_ptr(), _stream())
        return s.counts
    if kind == "batch":
        native.wfs_batch_measure(s.batch, [x.data_ptr() for x in s.screens], s.ts, [x.data_ptr() for x in s.slopes], _stream())
        return s.slopes
    w = s.handles[0]
    if kind == "calibrate":
        native.wfs_loop_calibrate(s.loop, w.h, 0, 1.0, s.im.data_ptr(), _stream())
        return s.im
    if kind == "loop":
        native.wfs_loop_step(s.loop, w.h, s.screens.data_ptr(), s.t, s.slopes.data_ptr(), _stream())
        native.wfs_loop_get_coeffs(s.loop, w.h, s.coeffs.data_ptr(), _stream())
        return {"slopes": s.slopes, "coeffs": s.coeffs}
    if s.case["stages"]:
        native.wfs_measure_stages(w.h, s.screens.data_ptr(), s.t, s.slopes.data_ptr(), s.out["opd"].data_ptr(),
                                  s.out["intensity"].data_ptr(), s.out["expected"].data_ptr(), s.out["counts"].data_ptr(), _stream())
        return dict(s.out, slopes=s.slopes)
    native.wfs_measure(w.h, s.screens.data_ptr(), s.t, s.slopes.data_ptr(), _stream())
    return s.slopes


# ----------------------------------------------------------------------- work

def _valid(tel, geom):
    """(lit pixels [n_valid][n][n], ids [n_valid]) of a geometry's valid subapertures."""
    P = geom.n_sub * geom.n_pix_sub
    x = (np.arange(P) - (P - 1) / 2.0) * (tel.diameter_m / P)
    r2 = x[:, None] ** 2 + x[None, :] ** 2
    lit = (r2 <= (tel.diameter_m / 2) ** 2) & (r2 >= (tel.obstruction * tel.diameter_m / 2) ** 2)
    lit = lit.reshape(geom.n_sub, geom.n_pix_sub, geom.n_sub, geom.n_pix_sub).transpose(0, 2, 1, 3)
    lit = lit.reshape(-1, geom.n_pix_sub, geom.n_pix_sub)
    ids = np.flatnonzero(lit.mean(axis=(1, 2)) >= geom.valid_fill)
    return lit[ids], ids


def _frame_work(cfg, stages=False):
    """Screen pixels under the stars' footprints once per layer, the slopes, and the projection,
    transform, elongation and centroid operations with each transform as an FFT over its rows."""
    L, D = cfg.layers, cfg.telescope.diameter_m
    S, ds, step = L.screen_size, L.screen_dx_m, 8
    grid = (np.arange(0, S, step) - S / 2) * ds
    pixels = 0
    for h in L.alt_m:
        seen = np.zeros((len(grid), len(grid)), dtype=bool)
        for st in cfg.stars:
            r = D / 2 * (1 - h / st.range_m if st.is_lgs else 1.0)
            r2 = (grid[:, None] - st.theta_y_rad * h) ** 2 + (grid[None, :] - st.theta_x_rad * h) ** 2
            seen |= (r2 <= r * r) & (r2 >= (cfg.telescope.obstruction * r) ** 2)
        pixels += int(seen.sum()) * step * step
    work = {"bytes": 4.0 * pixels, "flops": 0.0}
    for st in cfg.stars:
        geom = cfg.geometries[st.geometry_index]
        n, N, nd = geom.n_pix_sub, geom.n_fft, geom.n_det
        nv = len(_valid(cfg.telescope, geom)[1])
        ns = len(st.na_alt_m) if st.is_lgs and st.per_slice else 1
        fft = 5.0 * N * math.log2(N) * (n + N)
        per = ns * (8.0 * n * n * L.n_layers + fft + 3 * N * N) + 6 * nd * nd + (fft + 6.0 * N * n if st.is_lgs else N * N)
        work["bytes"] += nv * (8.0 + (4.0 * (n * n + N * N + 2 * nd * nd) if stages else 0.0))
        work["flops"] += nv * per
    return work


def work(case):
    c = case
    if c["kind"] == "noise":
        return {"bytes": 8.0 * c["pixels"], "flops": 60.0 * c["pixels"]}  # one generator block per pixel pair
    if c["kind"] == "batch":
        each = [_frame_work(f) for f in _instances(c)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    if c["kind"] == "calibrate":
        cfg, dm = _calibration(c)
        w = _frame_work(cfg)
        nv = len(_valid(cfg.telescope, cfg.geometries[0])[1])
        return {"bytes": 4.0 * dm.n_modes * (dm.n_act ** 2 + 2 * nv), "flops": 2.0 * dm.n_modes * w["flops"]}
    cfg = _config(c)
    w = _frame_work(cfg, c["stages"])
    if c["kind"] == "loop":
        ns = 2 * sum(len(_valid(cfg.telescope, cfg.geometries[s.geometry_index])[1]) for s in cfg.stars)
        dms = _mirrors(c)
        n = sum(d.n_modes for d in dms)
        cells = float(n) * ns + sum(float(d.n_modes) * d.n_act ** 2 for d in dms)
        w = {"bytes": w["bytes"] + 4.0 * cells + 8.0 * n, "flops": w["flops"] + 2.0 * cells}
    return w


# ----------------------------------------------------------------------- 64-bit reference

def _f64(a):
    return torch.as_tensor(np.asarray(a, dtype=np.float64), device="cuda")


def _bilinear(screen, u, v):
    """Periodic bilinear samples of a screen at column u, row v (pixels)."""
    S = screen.shape[0]
    iu, iv = u.floor(), v.floor()
    f, g = u - iu, v - iv
    i0, j0 = iu.long() % S, iv.long() % S
    i1, j1 = (i0 + 1) % S, (j0 + 1) % S
    at = lambda j, i: screen[j, i].double()  # noqa: E731
    return (1 - g) * ((1 - f) * at(j0, i0) + f * at(j0, i1)) + g * ((1 - f) * at(j1, i0) + f * at(j1, i1))


def _uplink_tilt(L, screens, st, t):
    """(x, y) angle by which the launch beam's spot moves on the sodium layer."""
    n, D, H = st.uplink_samples, st.uplink_diameter_m, st.range_m
    o = (torch.arange(n, dtype=torch.float64, device="cuda") - (n - 1) / 2) * (D / n)
    ox, oy = o[None, :].expand(n, n), o[:, None].expand(n, n)
    inside = (ox * ox + oy * oy <= D * D / 4).double()
    tx = ty = 0.0
    for l in range(L.n_layers):
        h = float(L.alt_m[l])
        x = st.launch_x_m * (1 - h / H) + st.theta_x_rad * h + ox - (L.x0_m[l] + L.wind_vx_mps[l] * t)
        y = st.launch_y_m * (1 - h / H) + st.theta_y_rad * h + oy - (L.y0_m[l] + L.wind_vy_mps[l] * t)
        val = _bilinear(screens[l], L.screen_size / 2 + x / L.screen_dx_m, L.screen_size / 2 + y / L.screen_dx_m) * inside
        tx += float((ox * val).sum() / (ox * ox * inside).sum()) * (H - h) / H
        ty += float((oy * val).sum() / (oy * oy * inside).sum()) * (H - h) / H
    return tx, ty


def _gaussian(N, shift, sigma):
    """[...][N] periodic Gaussian profiles about the shifts (minimum image)."""
    d = torch.arange(N, dtype=torch.float64, device="cuda") - shift[..., None]
    d = d - N * torch.floor(d / N + 0.5)
    return torch.exp(-d * d / (2 * sigma * sigma))


def _measure64(cfg, st, screens, t, stages=False, chunk=2048):
    """One star's noise-free frame in 64 bits: slopes [n_valid][2], and with stages the OPD, the
    intensity and the expected image of each subaperture."""
    geom, L, D = cfg.geometries[st.geometry_index], cfg.layers, cfg.telescope.diameter_m
    n, N, nd, ns = geom.n_pix_sub, geom.n_fft, geom.n_det, geom.n_sub
    lit, ids = _valid(cfg.telescope, geom)
    P, S, ds = ns * n, L.screen_size, L.screen_dx_m
    dx = D / P
    pos = (torch.arange(P, dtype=torch.float64, device="cuda") - (P - 1) / 2) * dx
    up = _uplink_tilt(L, screens, st, t) if st.is_lgs and st.uplink_diameter_m > 0 else (0.0, 0.0)
    slices = [(st.range_m, 1.0)]
    if st.is_lgs and st.per_slice:
        slices = [(float(h), float(w) / float(np.sum(st.na_weight))) for h, w in zip(st.na_alt_m, st.na_weight)]
    F = (_f64(np.arange(N)) - (N - 1) / 2)[:, None] * (_f64(np.arange(n)) - (n - 1) / 2)[None, :]
    F = torch.polar(torch.ones_like(F), -2 * math.pi * torch.remainder(F, N) / N)
    sy, sx = torch.as_tensor(ids // ns, device="cuda"), torch.as_tensor(ids % ns, device="cuda")
    lit = torch.as_tensor(lit, device="cuda").double()
    got = {"slopes": [], "opd": [], "intensity": [], "expected": []}
    c = (nd - 1) / 2
    axis = torch.arange(nd, dtype=torch.float64, device="cuda") - c
    for b in range(0, len(ids), chunk):
        ys = pos.reshape(ns, n)[sy[b:b + chunk]][:, :, None]
        xs = pos.reshape(ns, n)[sx[b:b + chunk]][:, None, :]
        inten = 0.0
        for k, (h_s, w_s) in enumerate(slices):
            opd = (up[0] * xs + up[1] * ys).expand(-1, n, n).clone()
            for l in range(L.n_layers):
                h = float(L.alt_m[l])
                cone = 1.0 - h / h_s if st.is_lgs else 1.0
                u = S / 2 + (cone * xs + st.theta_x_rad * h - (L.x0_m[l] + L.wind_vx_mps[l] * t)) / ds
                v = S / 2 + (cone * ys + st.theta_y_rad * h - (L.y0_m[l] + L.wind_vy_mps[l] * t)) / ds
                opd += _bilinear(screens[l], u.expand(-1, n, n), v.expand(-1, n, n))
            if stages and k == 0:
                got["opd"].append(opd.reshape(-1))
            if st.is_lgs and st.per_slice:
                opd = opd + 0.5 * ((xs - st.launch_x_m) ** 2 + (ys - st.launch_y_m) ** 2) * (1 / st.range_m - 1 / h_s)
            X = torch.polar(lit[b:b + chunk], 2 * math.pi / st.wavelength_m * (opd - opd[:, :1, :1]))
            Y = F @ X @ F.T
            inten = inten + w_s * (Y.real ** 2 + Y.imag ** 2)
        if stages:
            got["intensity"].append(inten.reshape(-1))
        if st.is_lgs:
            pix = st.wavelength_m / (N * dx)
            sigma = st.spot_fwhm_rad / (2 * math.sqrt(2 * math.log(2))) / pix
            alts, weights = ([st.range_m], [1.0]) if st.per_slice else (st.na_alt_m, st.na_weight)
            curv = _f64(1 / st.range_m - 1 / np.asarray(alts))
            K = _f64(weights)[None, :, None] * _gaussian(N, (ys.mean(dim=1) - st.launch_y_m) * curv / pix, sigma)
            K = K.transpose(1, 2) @ _gaussian(N, (xs.mean(dim=2) - st.launch_x_m) * curv / pix, sigma)
            K = K / K.sum(dim=(1, 2), keepdim=True)
            inten = torch.fft.irfft2(torch.fft.rfft2(inten) * torch.fft.rfft2(K), s=(N, N))
        B = inten.reshape(-1, nd, N // nd, nd, N // nd).sum(dim=(2, 4))
        fill = lit[b:b + chunk].mean(dim=(1, 2))
        tot = B.sum(dim=(1, 2))
        E = B * (st.photons_per_subap * fill / tot)[:, None, None]
        got["slopes"].append(torch.stack(((B * axis).sum(dim=(1, 2)) / tot, (B * axis[:, None]).sum(dim=(1, 2)) / tot), dim=1))
        if stages:
            got["expected"].append(E.reshape(-1))
    return {k: torch.cat(v) if v else torch.zeros((0, 2) if k == "slopes" else 0, dtype=torch.float64, device="cuda")
            for k, v in got.items()}


def _influence(dm, S, ds):
    """[S][n_act] influence of each actuator of an axis at the screen grid's points."""
    u = ((torch.arange(S, dtype=torch.float64, device="cuda") - S / 2) * ds / dm.pitch_m)[:, None]
    u = u - (torch.arange(dm.n_act, dtype=torch.float64, device="cuda") - (dm.n_act - 1) / 2)[None, :]
    edge = dm.coupling ** (dm.support ** 2)
    return (dm.coupling ** (u * u) - edge).clamp(min=0) / (1 - edge)


def exact(case, seed):
    c, g = case, _generator(seed)
    if c["kind"] == "noise":
        return None  # photon counts of a seeded generator
    if c["kind"] == "batch":
        out = []
        for i, cfg in enumerate(_instances(c)):
            out.append(_measure64(cfg, cfg.stars[0], _screens(cfg.layers, g), _time(seed + i))["slopes"])
        return out
    if c["kind"] == "calibrate":
        if c["modes"] > 400:
            return None  # ten times the time of the others
        cfg, dm = _calibration(c)
        m2a = _modal_base(dm, g)
        L = cfg.layers
        W = _influence(dm, L.screen_size, L.screen_dx_m)
        rows = []
        for m in range(dm.n_modes):
            shape = W @ m2a[:, m].double().reshape(dm.n_act, dm.n_act) @ W.T
            s = [_measure64(cfg, cfg.stars[0], shape[None] * a, 0.0, chunk=8192)["slopes"].reshape(-1) for a in (1.0, -1.0)]
            rows.append((s[0] - s[1]) / 2)
        return torch.stack(rows)
    cfg = _config(c)
    if c["noise"] and not c["stages"]:
        return None
    screens = _screens(cfg.layers, g)
    each = [_measure64(cfg, st, screens, _time(seed), c["stages"]) for st in cfg.stars]
    slopes = torch.cat([e["slopes"] for e in each])
    if c["kind"] == "loop":
        _, _, cm, gain = _loop_inputs(c, g, slopes.numel())
        s = slopes.reshape(-1)
        return {"slopes": slopes, "coeffs": gain.double() * torch.cat([x.double() @ s for x in cm.split(512)])}
    if c["stages"]:
        out = {k: torch.cat([e[k] for e in each]) for k in ("opd", "intensity", "expected")}
        return dict(out, counts=None if c["noise"] else out["expected"], slopes=None if c["noise"] else slopes)
    return slopes
