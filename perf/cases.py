"""What a user of the imaging library has it do: the calls whose speed matters, with their sizes.

Every case runs through the public Python entry points (`epic.Plan`, `epic.Batch`, `epic.moff_image`,
`epic.fengine`) on synthetic voltages of the array layouts of `synth.py`: `prepare` makes the layout,
the voltages and the plan a program keeps, `run` is one call (for the calibration one training step),
`exact` is the same result in 64 bits from plain torch and numpy.

The float64 accumulators of the imaging calls are the caller's own buffers; their values are returned
as the images, which are the accumulators divided by the number of samples.
"""
import math

import numpy as np
import torch

from paper_1510_08318_gb300 import epic, synth

DEV = "cuda"

# ------------------------------------------------------------------------------ the cases
_IMAGE = {"kind": "image", "xform": "fft", "gains": False, "autocorr": False}


def listed():
    return [
        # one all-sky snapshot of a small test array (16 antennas, one channel, 64 samples), with the
        # auto-correlation term: the smallest call, as in the quick-look display of a station
        dict(_IMAGE, name="tiny_snapshot", array="tiny", n_ant=16, n_pad=64, n_chan=1, n_pol=1, n_time=64,
             vdtype="c64", autocorr=True),
        # a short block of a 256-antenna station's stream (16 channels, 250 samples, calibrated, with the
        # auto-correlation term) in the default FP32 transform: what a live imager runs per block
        dict(_IMAGE, name="lwa_block_fft", array="lwa", n_ant=256, n_pad=128, n_chan=16, n_pol=2, n_time=250,
             vdtype="ci4", gains=True, autocorr=True),
        # a full integration of the same station (128 channels, 1024 samples, 4+4-bit) with the
        # tensor-core transform: the largest imaging call, throughput counts
        dict(_IMAGE, name="lwa_full_dftgemm", array="lwa", n_ant=256, n_pad=128, n_chan=128, n_pol=2, n_time=1024,
             vdtype="ci4", xform="dftgemm"),
        # full-polarisation images (XX, YY, XY) of a part of the band, calibrated
        dict(name="lwa_xpol_dftgemm", kind="xpol", array="lwa", n_ant=256, n_pad=128, n_chan=32, n_pol=2, n_time=256,
             vdtype="ci4", xform="dftgemm", gains=True),
        # the dense hexagonal array of 331 dishes: one node's share of the band at 256 x 256, FP16 voltages
        dict(_IMAGE, name="hera_f16", array="hera", n_ant=331, n_pad=256, n_chan=128, n_pol=1, n_time=256,
             vdtype="f16"),
        # a wide array on the finest grid, two-pass transform, an odd number of samples
        dict(_IMAGE, name="wide_512", array="disk", n_ant=400, n_pad=512, n_chan=8, n_pol=1, n_time=101,
             vdtype="f16", xform="fft_twopass"),
        # one gain-calibration step: image, loss against the model image, gradient of the gains
        dict(name="calibration_step", kind="calib", array="disk", n_ant=1024, n_pad=256, n_chan=32, n_pol=1,
             n_time=64, vdtype="c64"),
        # a dozen heterogeneous sub-arrays of every grid size imaged by one batch call
        dict(name="batch_subarrays", kind="batch", structure=4, n_sub=12, n_time=128, max_ant=1024, max_chan=32),
        # the correlator: visibilities of every antenna pair over the full integration
        dict(name="correlate_lwa", kind="correlate", array="lwa", n_ant=256, n_pad=128, n_chan=128, n_pol=2,
             n_time=1024, vdtype="ci4", gains=True),
        # imaging of one integration's visibilities
        dict(name="fx_image_lwa", kind="fx_image", array="lwa", n_ant=256, n_pad=128, n_chan=64, n_pol=2),
        # the channeliser ahead of the imager: 4+4-bit samples to 128-channel FP16 spectra
        dict(name="fengine_c128", kind="fengine", n_ant=256, n_pol=2, n_chan=128, n_time=1024, vdtype="ci4",
             out="f16"),
        # the gridded fields of every sample written out for a transform done elsewhere
        dict(name="grid_lwa", kind="grid", array="lwa", n_ant=256, n_pad=128, n_chan=16, n_pol=2, n_time=1024,
             vdtype="ci4", gains=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _fit(c, limit):
    """Shorten a case until its padded pixels over all samples are at most `limit`."""
    per = c["n_chan"] * c["n_pol"] * c["n_pad"] ** 2
    c["n_time"] = max(1, min(c["n_time"], limit // per))
    return c


def draw(rng):
    kind = rng.choice(["image", "image", "image", "image", "xpol", "calib", "batch", "correlate", "fx_image",
                       "fengine", "grid"])
    lwa = dict(array="lwa", n_ant=_log_int(rng, 48, 512), n_pad=128, n_chan=_log_int(rng, 1, 64),
               n_pol=rng.choice([1, 2]), n_time=_log_int(rng, 16, 1024), vdtype=rng.choice(["ci4", "ci4", "f16"]))
    gains = rng.choice([False, True])
    if kind == "image":
        array = rng.choice(["tiny", "lwa", "lwa", "hera", "disk", "disk"])
        c = dict(_IMAGE, gains=gains, autocorr=rng.choice([False, True]))
        if array == "tiny":
            c.update(array="tiny", n_ant=_log_int(rng, 8, 64), n_pad=64, n_chan=_log_int(rng, 1, 8), n_pol=1,
                     n_time=_log_int(rng, 16, 512), vdtype="c64")
        elif array == "lwa":
            c.update(lwa, xform=rng.choice(["fft", "dftgemm"]))
        elif array == "hera":
            side = rng.randint(5, 11)
            c.update(array="hera", n_ant=3 * side * (side - 1) + 1, n_pad=256, n_chan=_log_int(rng, 2, 64), n_pol=1,
                     n_time=_log_int(rng, 16, 256), vdtype="f16")
        else:
            n_pad = rng.choice([256, 512])
            c.update(array="disk", n_ant=_log_int(rng, 64, 1024), n_pad=n_pad, n_chan=_log_int(rng, 1, 16), n_pol=1,
                     n_time=_log_int(rng, 16, 256), vdtype=rng.choice(["f16", "c64"]),
                     xform="fft" if n_pad == 256 else "fft_twopass")
        return _fit(c, 1 << 30)
    if kind == "xpol":
        c = dict(kind="xpol", xform=rng.choice(["fft", "dftgemm"]), gains=gains, **lwa)
        c.update(n_pol=2, n_chan=min(c["n_chan"], 24))
        return _fit(c, 1 << 28)
    if kind == "calib":
        return _fit(dict(kind="calib", array="disk", n_ant=_log_int(rng, 128, 1024), n_pad=256,
                         n_chan=_log_int(rng, 2, 32), n_pol=1, n_time=_log_int(rng, 8, 96), vdtype="c64"), 1 << 27)
    if kind == "batch":
        return dict(kind="batch", structure=rng.randint(10, 10 ** 6), n_sub=rng.randint(3, 9),
                    n_time=rng.randint(16, 96), max_ant=512, max_chan=24)
    if kind == "correlate":
        return dict(kind="correlate", gains=gains, **lwa)
    if kind == "fx_image":
        return dict(kind="fx_image", array="lwa", n_ant=_log_int(rng, 48, 256), n_pad=128,
                    n_chan=_log_int(rng, 1, 64), n_pol=rng.choice([1, 2]))
    if kind == "fengine":
        return dict(kind="fengine", n_ant=_log_int(rng, 48, 300), n_pol=rng.choice([1, 2]),
                    n_chan=rng.choice([32, 64, 128, 256, 512]), n_time=_log_int(rng, 16, 256),
                    vdtype=rng.choice(["ci4", "ci4", "f16"]), out="f16")
    c = dict(kind="grid", gains=gains, **lwa)
    c.update(n_chan=min(c["n_chan"], 16))
    return _fit(c, 1 << 28)


# ------------------------------------------------------------------------------ array layouts
def _array(case, seed):
    """pos, footprints (kern_ptr, kern_dxdy, kern_w), dx, origin, n_grid, channel frequencies."""
    rng = np.random.default_rng([seed, 11])
    A, NG, C = case["n_ant"], case["n_pad"] // 2, case["n_chan"]
    if case["array"] == "tiny":          # 2 m squares in a 20 m box, half-wavelength grid at 60 MHz
        freqs = 60e6 + 25e3 * np.arange(C)
        dx = synth.C_LIGHT / 60e6 / 2
        pos, reach = synth.layout_rect(rng, A, 20.0, 20.0), 1.0
        kern = [synth.kernel_square(2.0, dx / 4)] * A
    elif case["array"] == "lwa":         # Gaussian apertures in a 100 m x 110 m ellipse, 30-80 MHz
        freqs = np.linspace(30e6, 80e6, 128)[:C]
        dx = synth.C_LIGHT / 80e6 / 2
        pos, reach = synth.layout_ellipse(rng, A, 100.0, 110.0), 4.5
        kern = [synth.kernel_gaussian(1.5, dx / 4)] * A
    elif case["array"] == "hera":        # 14 m dishes in a hexagon, 2.5 m grid, 100-200 MHz
        freqs = np.linspace(100e6, 200e6, 1024)[:C]
        side = int(round((3 + math.sqrt(12 * A - 3)) / 6))
        dx = 2.5
        pos, reach = synth.layout_hex(side, 14.0), 7.0
        kern = [synth.kernel_disk(14.0, dx / 4)] * A
    else:                                # Gaussian apertures in a 300 m disk filling the grid, 50-80 MHz
        freqs = np.linspace(50e6, 80e6, 32)[:C]
        dx = (300.0 + 9.0) / NG
        pos, reach = synth.layout_disk(rng, A, 300.0), 4.5
        kern = [synth.kernel_gaussian(1.5, dx / 4)] * A
    return pos, synth.pack_kernels(kern), dx, synth.centred_origin(pos, reach, dx, NG), NG, freqs


def _sub_cases(case):
    """The sub-arrays of a batch: antenna and channel counts log-uniform, every grid size in turn."""
    rng = np.random.default_rng(case["structure"])
    subs = []
    for s in range(case["n_sub"]):
        n_pad = (128, 512, 64, 256, 32)[s % 5]
        subs.append(dict(
            n_pad=n_pad, n_pol=1, n_time=case["n_time"], vdtype="f16",
            n_ant=int(round(math.exp(rng.uniform(math.log(32), math.log(case["max_ant"]))))),
            n_chan=int(round(math.exp(rng.uniform(math.log(4), math.log(case["max_chan"]))))),
            diam=float(rng.uniform(60.0, 300.0)), kernels=int(rng.integers(1 << 30))))
    return subs


def _sub_array(sub, seed):
    """Squares, Gaussians and disks of 1-14 m mixed antenna by antenna in a disk."""
    rng, krng = np.random.default_rng([seed, 12]), np.random.default_rng(sub["kernels"])
    A, NG = sub["n_ant"], sub["n_pad"] // 2
    dx = (sub["diam"] + 21.0) / (NG - 1)
    pos = synth.layout_disk(rng, A, sub["diam"])
    kern = []
    for size, kind in zip(krng.uniform(1.0, 14.0, A), krng.integers(0, 3, A)):
        step = max(dx / 2, size / 64)
        kern.append(synth.kernel_square(size, step) if kind == 0 else
                    synth.kernel_gaussian(size / 4, step) if kind == 1 else synth.kernel_disk(size, step))
    packed = synth.pack_kernels(kern)
    reach = float(np.abs(packed[1]).max())
    return pos, packed, dx, synth.centred_origin(pos, reach, dx, NG), NG, np.linspace(50e6, 200e6, sub["n_chan"])


# ------------------------------------------------------------------------------ inputs
def _sky(array, seed):
    rng = np.random.default_rng([seed, 13])
    if array == "lwa":                   # power-law source counts over the visible hemisphere
        sky = synth.sky_powerlaw_hemisphere(rng, 200, 1.0, 100.0)
        return sky, math.sqrt(sky.flux.sum() / 0.1)
    return synth.sky_box(rng, 3 if array == "tiny" else 50, 0.7, 1.0, 10.0), 1.0


def _voltages(sky, noise, pos, freqs, n_time, n_pol, seed, gains=None):
    """[T, C, P, A] complex64: point sources with fresh phases every sample, and receiver noise."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    A = len(pos)
    out = torch.empty((n_time, len(freqs), n_pol, A), dtype=torch.complex64, device=DEV)
    geo = torch.from_numpy(np.outer(sky.l, pos[:, 0]) + np.outer(sky.m, pos[:, 1])).to(DEV)
    amp = torch.from_numpy(np.sqrt(sky.flux)).to(DEV, torch.float32)
    for c, f in enumerate(freqs):
        turn = torch.remainder(geo * (f / synth.C_LIGHT), 1.0) * (-2 * math.pi)
        steer = torch.polar(torch.ones_like(turn), turn).to(torch.complex64)
        ph = torch.rand((n_time * n_pol, len(amp)), generator=gen, device=DEV) * (2 * math.pi)
        v = (torch.polar(amp.expand_as(ph).contiguous(), ph) @ steer).view(n_time, n_pol, A)
        if noise:
            v += noise * torch.randn((n_time, n_pol, A), dtype=torch.complex64, generator=gen, device=DEV)
        out[:, c] = v if gains is None else v * gains
    return out


def _encode(v, vdtype):
    """The library's voltage formats: complex64, FP16 pairs, or signed 4+4-bit at an rms of two levels."""
    if vdtype == "c64":
        return v
    x = torch.view_as_real(v)
    if vdtype == "f16":
        return x.to(torch.float16)
    n = (x * (2.0 / x.square().mean().sqrt())).round().clamp(-7, 7).to(torch.int16)
    return ((n[..., 0] & 15) * 16 + (n[..., 1] & 15)).to(torch.uint8)


def _decode64(volt, vdtype):
    if vdtype == "c64":
        return volt.to(torch.complex128)
    if vdtype == "f16":
        return torch.view_as_complex(volt.to(torch.float64))
    b = volt.to(torch.int16)
    hi, lo = b >> 4, b & 15
    return torch.complex((hi - 16 * (hi > 7)).to(torch.float64), (lo - 16 * (lo > 7)).to(torch.float64))


def _gains(shape, seed):
    g = synth.random_gains(np.random.default_rng([seed, 14]), shape)
    return torch.from_numpy(g).to(DEV)


def _plan(arr, c, n_pol=None):
    pos, (ptr, dxdy, w), dx, origin, NG, freqs = arr
    return epic.Plan(pos, ptr, dxdy, w, dx, origin, NG, c["n_pad"], len(freqs), c["n_pol"], c["vdtype"], 0)


def _inputs(case, seed):
    """Layout, encoded voltages and gains of an imaging or correlator case."""
    arr = _array(case, seed)
    sky, noise = _sky(case["array"], seed)
    v = _voltages(sky, noise, arr[0], arr[5], case["n_time"], case["n_pol"], seed)
    g = _gains((case["n_chan"], case["n_pol"], case["n_ant"]), seed) if case.get("gains") else None
    return arr, _encode(v, case["vdtype"]), g


def _calib_inputs(case, seed):
    """Voltages corrupted by per-antenna gains, the model image of the sources, the starting gains."""
    arr = _array(case, seed)
    sky, noise = _sky(case["array"], seed)
    true = _gains((case["n_ant"],), seed)
    volt = _voltages(sky, noise, arr[0], arr[5], case["n_time"], 1, seed, gains=true)
    clean = _voltages(sky, 0.0, arr[0], arr[5], case["n_time"], 1, seed + 1)
    model = _images64(_map64(arr), clean.to(torch.complex128), case["n_pad"]).to(torch.float32)
    start = (1.0 / true) * _gains((case["n_chan"], 1, case["n_ant"]), seed + 2).abs()
    return arr, volt, model, start.to(torch.complex64).contiguous()


def _vis_inputs(case, seed):
    """Visibilities [C, P, A, A] of a 64-sample integration of the array's voltages."""
    arr = _array(case, seed)
    sky, noise = _sky(case["array"], seed)
    v = _voltages(sky, noise, arr[0], arr[5], 64, case["n_pol"], seed).permute(1, 2, 3, 0).contiguous()
    return arr, (v @ v.conj().transpose(-1, -2) / 64).contiguous()


def _feng_inputs(case, seed):
    """Time samples [T C, P, A]: receiver noise and one carrier common to all antennas."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    n = case["n_time"] * case["n_chan"]
    x = torch.randn((n, case["n_pol"], case["n_ant"]), dtype=torch.complex64, generator=gen, device=DEV)
    ph = torch.remainder(torch.arange(n, device=DEV, dtype=torch.float64) * 0.1337, 1.0) * (2 * math.pi)
    x += torch.polar(torch.full_like(ph, 0.5), ph).to(torch.complex64)[:, None, None]
    return _encode(x, case["vdtype"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fengine":
        return {"case": case, "raw": _feng_inputs(case, seed)}
    if kind == "batch":
        plans, volts = [], []
        for i, sub in enumerate(_sub_cases(case)):
            arr = _sub_array(sub, seed + i)
            sky = synth.sky_box(np.random.default_rng([seed + i, 13]), 20, 0.7, 1.0, 10.0)
            plans.append(_plan(arr, sub))
            volts.append(_encode(_voltages(sky, 1.0, arr[0], arr[5], sub["n_time"], 1, seed + i), "f16"))
        batch = epic.Batch(plans)
        acc, img = batch.alloc()
        batch.autotune(volts, acc)
        return {"case": case, "plans": plans, "batch": batch, "volts": volts, "acc": acc, "img": img}
    if kind == "calib":
        arr, volt, model, start = _calib_inputs(case, seed)
        return {"case": case, "plan": _plan(arr, case), "volt": volt, "model": model,
                "gains": start.requires_grad_(True)}
    if kind == "fx_image":
        arr, vis = _vis_inputs(case, seed)
        return {"case": case, "plan": _plan(arr, dict(case, vdtype="ci4")), "vis": vis}
    arr, volt, gains = _inputs(case, seed)
    plan = _plan(arr, case)
    if case.get("xform", "fft") != "fft":
        plan.set_transform(case["xform"])
    s = {"case": case, "plan": plan, "volt": volt, "gains": gains}
    C, P, NP = case["n_chan"], case["n_pol"], case["n_pad"]
    if kind == "image":
        s["accum"] = torch.zeros((C, P, NP, NP), dtype=torch.float64, device=DEV)
        s["power"] = torch.zeros((C, P, case["n_ant"]), dtype=torch.float64, device=DEV) if case["autocorr"] else None
    elif kind == "xpol":
        s["accum4"] = torch.zeros((C, 4, NP, NP), dtype=torch.float64, device=DEV)
    return s


# ------------------------------------------------------------------------------ one pass
def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "image":
        out = s["plan"].image(s["volt"], s["gains"], accum=s["accum"], power=s["power"],
                              want_autocorr=case["autocorr"])
        return {"image": out["image"], "autocorr": out["autocorr"]}
    if kind == "xpol":
        out = s["plan"].image_xpol(s["volt"], s["gains"], accum4=s["accum4"])
        return {"image": out["image"], "cross": out["cross"]}
    if kind == "calib":
        g = s["gains"]
        g.grad = None
        image = epic.moff_image(g, s["volt"], s["plan"])
        loss = (image - s["model"]).square().sum()
        loss.backward()
        return {"image": image.detach(), "grad": g.grad}
    if kind == "batch":
        s["batch"].image(s["volts"], s["acc"], s["img"])
        return s["img"]
    if kind == "correlate":
        return s["plan"].correlate(s["volt"], s["gains"])
    if kind == "fx_image":
        return s["plan"].fx_image(s["vis"])
    if kind == "fengine":
        return epic.fengine(s["raw"], case["n_chan"], case["vdtype"], case["out"])
    return s["plan"].grid(s["volt"], s["gains"])


# ------------------------------------------------------------------------------ the least work
_VOLT_BYTES = {"c64": 8, "f16": 4, "ci4": 1}
_FOOT = {"tiny": 2.0, "lwa": 20.0, "hera": 30.0, "disk": 14.0}   # mapping entries per antenna, roughly


def _image_work(c, n_images, n_planes, out_bytes):
    """Bytes and flops of imaging n_images padded grids into n_planes: voltages in, accumulators out;
    pruned radix-2 count of the 2-D transform, the gridding and |F|^2."""
    n, a = c["n_pad"], c["n_ant"]
    lines = n + n // 2
    foot = _FOOT.get(c.get("array"), 30.0)
    flops = n_images * (5.0 * n * math.log2(n) * lines + 4.0 * foot * a + 4.0 * n * n)
    volts = c["n_time"] * c["n_chan"] * c["n_pol"] * a
    return {"bytes": volts * _VOLT_BYTES[c["vdtype"]] + n_planes * n * n * out_bytes, "flops": flops}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [work(dict(s, kind="image", autocorr=False)) for s in _sub_cases(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    C, P, A = case["n_chan"], case["n_pol"], case["n_ant"]
    if kind == "fengine":
        n = case["n_time"] * C * P * A
        return {"bytes": n * (_VOLT_BYTES[case["vdtype"]] + _VOLT_BYTES[case["out"]]), "flops": 5.0 * n * math.log2(C)}
    NP = case["n_pad"]
    if kind == "fx_image":
        # the lag cells that an antenna pair reaches: one multiply-add each per plane
        return {"bytes": C * P * (8.0 * A * A + 4.0 * NP * NP),
                "flops": C * P * (A * A / 2 * 81 * 8.0 + 5.0 * NP * NP * 2 * math.log2(NP))}
    T = case["n_time"]
    volt = T * C * P * A * _VOLT_BYTES[case["vdtype"]]
    if kind == "correlate":
        return {"bytes": volt + 8.0 * C * P * A * A, "flops": C * P * 8.0 * T * A * (A + 1) / 2}
    if kind == "grid":
        return {"bytes": volt + 8.0 * T * C * P * (NP // 2) ** 2, "flops": 4.0 * _FOOT[case["array"]] * A * T * C * P}
    if kind == "xpol":
        return _image_work(case, 2 * C * T, C, 4 * 8 + 2 * 4 + 8)
    w = _image_work(case, C * P * T, C * P, 8 + 4 + (4 if case.get("autocorr") else 0))
    if kind == "calib":                  # the image and its adjoint
        w = {"bytes": 2 * w["bytes"], "flops": 3 * w["flops"]}
    return w


# ------------------------------------------------------------------------------ 64-bit results
def _map64(arr):
    """The antenna-to-grid mapping as a dense real matrix [cells, A]: every footprint sample's weight is
    added to its nearest cell."""
    pos, (ptr, dxdy, w), dx, origin, NG, _ = arr
    ant = np.repeat(np.arange(len(pos)), np.diff(ptr))
    cell = np.floor((pos[ant] + dxdy - origin) / dx + 0.5).astype(np.int64)
    m = np.zeros((NG * NG, len(pos)))
    np.add.at(m, (cell[:, 1] * NG + cell[:, 0], ant), w.real)
    return torch.from_numpy(m).to(DEV)


def _fields64(m, v):
    """Gridded fields [n, NG, NG] of calibrated voltages v [n, A]."""
    ng = int(math.isqrt(m.shape[0]))
    return torch.complex(v.real @ m.T, v.imag @ m.T).view(-1, ng, ng)


def _transform64(e, n_pad):
    """sum_g E(g) exp(+2 pi i g.k / N_p), k = 0 at the centre."""
    return torch.fft.fftshift(torch.fft.ifft2(e, s=(n_pad, n_pad), norm="forward"), dim=(-2, -1))


def _chunks(n, n_pad):
    step = max(1, (1 << 30) // (16 * n_pad * n_pad))
    return [(i, min(n, i + step)) for i in range(0, n, step)]


def _images64(m, v, n_pad):
    """Time-averaged |F|^2 [C, P, N_p, N_p] of calibrated voltages v [T, C, P, A]."""
    T, C, P, A = v.shape
    out = torch.zeros((C, P, n_pad, n_pad), dtype=torch.float64, device=DEV)
    for c in range(C):
        for p in range(P):
            for i, j in _chunks(T, n_pad):
                f = _transform64(_fields64(m, v[i:j, c, p]), n_pad)
                out[c, p] += (f.real.square() + f.imag.square()).sum(0) / T
    return out


def _apply64(volt, case, gains):
    v = _decode64(volt, case["vdtype"])
    return v if gains is None else v * gains.to(torch.complex128)


def exact(case, seed):
    kind = case["kind"]
    if kind == "fengine":
        x = _decode64(_feng_inputs(case, seed), case["vdtype"])
        x = x.view(case["n_time"], case["n_chan"], case["n_pol"], case["n_ant"])
        return torch.view_as_real(torch.fft.fft(x, dim=1))
    if kind == "batch":
        out = []
        for i, sub in enumerate(_sub_cases(case)):
            arr = _sub_array(sub, seed + i)
            sky = synth.sky_box(np.random.default_rng([seed + i, 13]), 20, 0.7, 1.0, 10.0)
            v = _encode(_voltages(sky, 1.0, arr[0], arr[5], sub["n_time"], 1, seed + i), "f16")
            out.append(_images64(_map64(arr), _decode64(v, "f16"), sub["n_pad"]))
        return out
    if kind == "calib":
        arr, volt, model, start = _calib_inputs(case, seed)
        m, T, NP = _map64(arr), case["n_time"], case["n_pad"]
        images, grads = [], []
        for c in range(case["n_chan"]):
            g = start[c, 0].to(torch.complex128).requires_grad_(True)
            f = _transform64(_fields64(m, volt[:, c, 0].to(torch.complex128) * g), NP)
            image = (f.real.square() + f.imag.square()).sum(0) / T
            (image - model[c, 0].to(torch.float64)).square().sum().backward()
            images.append(image.detach())
            grads.append(g.grad)
        return {"image": torch.stack(images)[:, None], "grad": torch.stack(grads)[:, None]}
    if kind == "fx_image":
        arr, vis = _vis_inputs(case, seed)
        NP, A = case["n_pad"], case["n_ant"]
        k = _transform64(_map64(arr).T.reshape(A, NP // 2, NP // 2).to(torch.complex128), NP).reshape(A, -1)
        out = torch.empty((case["n_chan"], case["n_pol"], NP, NP), dtype=torch.float64, device=DEV)
        for c in range(case["n_chan"]):
            for p in range(case["n_pol"]):
                y = vis[c, p].to(torch.complex128) @ k.conj()
                out[c, p] = (k * y).sum(0).real.view(NP, NP)
        return out
    arr, volt, gains = _inputs(case, seed)
    v = _apply64(volt, case, gains)
    T, C, P, A = v.shape
    if kind == "correlate":
        out = torch.empty((C, P, A, A), dtype=torch.complex128, device=DEV)
        for c in range(C):
            x = v[:, c].permute(1, 2, 0)
            out[c] = x @ x.conj().transpose(-1, -2) / T
        return out
    m, NP = _map64(arr), case["n_pad"]
    if kind == "grid":
        return _fields64(m, v.reshape(-1, A)).view(T, C, P, NP // 2, NP // 2)
    if kind == "xpol":
        image = _images64(m, v, NP)
        cross = torch.zeros((C, NP, NP), dtype=torch.complex128, device=DEV)
        for c in range(C):
            for i, j in _chunks(T, NP):
                f = [_transform64(_fields64(m, v[i:j, c, p]), NP) for p in (0, 1)]
                cross[c] += (f[0] * f[1].conj()).sum(0) / T
        return {"image": image, "cross": cross}
    out = {"image": _images64(m, v, NP), "autocorr": None}
    if case["autocorr"]:
        k = _transform64(m.T.reshape(A, NP // 2, NP // 2).to(torch.complex128), NP)
        beam = (k.real.square() + k.imag.square()).view(A, -1)
        power = (v.real.square() + v.imag.square()).mean(0)
        out["autocorr"] = (power @ beam).view(C, P, NP, NP)
    return out
