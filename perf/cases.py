"""What is timed: the calls a user of this library makes, over the range of sizes they come in.

Every case goes through the C ABI's Python binding (``paper_2605_28451_gb300.bfpfft``)
or, for autofocus, through the ``torch.autograd`` wrapper.  Kinds:

* ``fft``       a forward transform of a batch, then the 1/N-shifted inverse of the result (a
                forward-inverse pair is the unit the benchmark counts);
* ``uneven``    one batch of mixed lengths by one plan, forward;
* ``sar``       range compression of a raw echo and, for ``stage = "image"``, the azimuth
                compression that makes the image;
* ``rda``       the image with range-cell-migration correction and range-dependent filters;
* ``spectral``  forward, multiply by a filter (one for all lines or one per line), inverse;
* ``autofocus`` image entropy and its gradient by the phase correction, one optimiser step's work.

Inputs follow the seeded recipes of ``paper_2605_28451_gb300.synth`` (unit Gaussian lines, the
point-target scene, the phase-error model), drawn on the GPU so that they are quick to make.
``exact`` repeats each chain in complex128 with torch.fft and nothing of this library.
"""

import math

import torch

from paper_2605_28451_gb300 import autofocus as GA
from paper_2605_28451_gb300 import bfpfft as B
from paper_2605_28451_gb300 import synth

DEV = "cuda:0"
STORAGE = {"f32": B.F32, "f16": B.F16_BFP, "e4m3": B.E4M3_BFP, "e5m2": B.E5M2_BFP}
POINT_BYTES = {"f32": 8, "f16": 4, "e4m3": 2, "e5m2": 2}
FP8 = {"e4m3": torch.float8_e4m3fn, "e5m2": torch.float8_e5m2}
ARITH = {"f32": B.ARITH_F32, "tc": B.ARITH_F16_MUL_F32_ACC}
APERTURE = synth.AZIMUTH_APERTURE


def listed():
    return [
        # the smallest call: a handful of short lines, as one radar pulse's channels; launches and host time count
        {"name": "fft_f16_256x8", "kind": "fft", "n": 256, "batch": 8, "storage": "f16", "arith": "f32"},
        # the paper's Table II workload: N = 4096, batch 256
        {"name": "fft_f16_4096x256", "kind": "fft", "n": 4096, "batch": 256, "storage": "f16", "arith": "f32"},
        # an ordinary batch of short lines with a count that fits no tile
        {"name": "fft_f16_1024x30011", "kind": "fft", "n": 1024, "batch": 30011, "storage": "f16", "arith": "f32"},
        # the benchmark's headline: FP16 operands, FP32 accumulation on the tensor cores
        {"name": "fft_tc_4096x65536", "kind": "fft", "n": 4096, "batch": 65536, "storage": "f16", "arith": "tc"},
        # FP8 storage (Section VII)
        {"name": "fft_e4m3_4096x16384", "kind": "fft", "n": 4096, "batch": 16384, "storage": "e4m3", "arith": "f32"},
        # the FP32 comparison path on long range lines
        {"name": "fft_f32_16384x1001", "kind": "fft", "n": 16384, "batch": 1001, "storage": "f32", "arith": "f32"},
        # the longest lines, odd count
        {"name": "fft_f16_65536x601", "kind": "fft", "n": 65536, "batch": 601, "storage": "f16", "arith": "f32"},
        # the mixed-length batch: 20,000 transforms of 256 .. 65536 points, one plan as created
        {"name": "uneven_f16_20000", "kind": "uneven", "count": 20000, "storage": "f16"},
        # the benchmark's SAR image: complex64 echo to FP16 image
        {"name": "sar_image_4096x4096", "kind": "sar", "stage": "image", "n_az": 4096, "n_rg": 4096, "raw": "f32",
         "out": "f16", "arith": "f32"},
        # the same scene size with range-cell-migration correction
        {"name": "rda_4096x4096", "kind": "rda", "n_az": 4096, "n_rg": 4096, "out": "f16"},
        # a spectral layer: per-channel weights, modes truncated, odd number of lines
        {"name": "spectral_f16_1024x20001", "kind": "spectral", "n": 1024, "lines": 20001, "per_line": True,
         "x": "f16", "out": "f16", "arith": "f32"},
        # one autofocus gradient step on a 4096 x 4096 scene
        {"name": "autofocus_f16_4096x4096", "kind": "autofocus", "n_az": 4096, "n_rg": 4096, "rc": "f16", "arith": "f32"},
    ]


def _log_uniform(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["fft", "fft", "fft", "uneven", "sar", "sar", "rda", "spectral", "autofocus"])
    if kind == "fft":
        storage = rng.choice(["f16", "f16", "f16", "f32", "e4m3", "e5m2"])
        arith = "tc" if storage != "f32" and rng.random() < 0.25 else "f32"
        n = 4096 if arith == "tc" else 1 << rng.randint(4, 16)
        batch = _log_uniform(rng, 1, max(1, (1 << 26) // n))
        return {"kind": kind, "n": n, "batch": batch, "storage": storage, "arith": arith}
    if kind == "uneven":
        return {"kind": kind, "count": _log_uniform(rng, 20, 8000), "storage": rng.choice(["f16", "f16", "f32", "e4m3"])}
    if kind == "sar":
        stage = rng.choice(["range", "image"])
        arith = rng.choice(["f32", "f32", "tc"])
        n_rg = 4096 if arith == "tc" else 1 << rng.randint(9, 13)
        if stage == "range":
            n_az = _log_uniform(rng, 17, (1 << 24) // n_rg)
        else:
            n_az = 4096 if arith == "tc" else 1 << rng.randint(9, min(13, 24 - n_rg.bit_length() + 1))
        out = "f16" if arith == "tc" else rng.choice(["f16", "f16", "f32"])
        return {"kind": kind, "stage": stage, "n_az": n_az, "n_rg": n_rg, "raw": rng.choice(["f32", "f16"]),
                "out": out, "arith": arith}
    if kind == "rda":
        n_az = 1 << rng.randint(11, 13)
        n_rg = 1 << rng.randint(10, 24 - n_az.bit_length() + 1)
        return {"kind": kind, "n_az": n_az, "n_rg": min(n_rg, 8192), "out": rng.choice(["f16", "f32"])}
    if kind == "spectral":
        arith = rng.choice(["f32", "f32", "f32", "tc"])
        n = 4096 if arith == "tc" else 1 << rng.randint(8, 14)
        per_line = rng.random() < 0.5
        lines = _log_uniform(rng, 3, (1 << 24) // n)
        return {"kind": kind, "n": n, "lines": lines, "per_line": per_line, "x": rng.choice(["f16", "f32"]),
                "out": "f16" if arith == "tc" else rng.choice(["f16", "f32"]), "arith": arith}
    arith = rng.choice(["f32", "f32", "tc"])
    n_az = 4096 if arith == "tc" else 1 << rng.randint(10, 13)
    return {"kind": kind, "n_az": n_az, "n_rg": _log_uniform(rng, 101, (1 << 24) // n_az),
            "rc": rng.choice(["f16", "f16", "f32"]), "arith": arith}


# ---- inputs ------------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _to_storage(z, storage):
    """complex64 [...] -> the storage layout: complex64, or [..., 2] in the 16- or 8-bit type."""
    if storage == "f32":
        return z.contiguous()
    v = torch.view_as_real(z)
    return v.to(torch.float16 if storage == "f16" else FP8[storage]).contiguous()


def _lines(shape, seed, storage):
    """re, im ~ N(0, 1) in the storage type (Table II's workload)."""
    if storage == "f32":
        return torch.view_as_complex(torch.randn(tuple(shape) + (2,), device=DEV, generator=_gen(seed)))
    x = torch.randn(tuple(shape) + (2,), device=DEV, generator=_gen(seed), dtype=torch.float16)
    return x if storage == "f16" else x.to(FP8[storage])


def _values(x):
    """Stored points as complex128."""
    if x.is_complex():
        return x.to(torch.complex128)
    return torch.view_as_complex(x.to(torch.float64))


def _like(z, storage):
    """An exact complex128 result in the layout run() returns it in."""
    return z if storage == "f32" else torch.view_as_real(z)


def _empty(shape, storage):
    if storage == "f32":
        return torch.empty(shape, dtype=torch.complex64, device=DEV)
    return torch.empty(tuple(shape) + (2,), dtype=torch.float16 if storage == "f16" else FP8[storage], device=DEV)


def _c64(a):
    return torch.from_numpy(a.astype("complex64")).to(DEV)


def _targets(n_az, n_rg, seed):
    """Target cells (eta, r) and amplitudes 10^(-k/7); any scene size of the declared ranges."""
    g = torch.Generator().manual_seed(seed)
    u = torch.rand((synth.N_TARGETS, 2), generator=g, dtype=torch.float64)
    return [(int(n_az * (0.1 + 0.8 * float(a))), int(n_rg * (0.1 + 0.8 * float(b))), 10.0 ** (-k / 7.0))
            for k, (a, b) in enumerate(u)]


def _noise(shape, std, seed):
    v = torch.randn(tuple(shape) + (2,), device=DEV, generator=_gen(seed))
    return torch.view_as_complex(v.mul_(std))


def _aperture(n_az):
    """An even azimuth chirp length that fits the scene."""
    return min(APERTURE, max(2, n_az // 2 * 2))


def _echo(n_az, n_rg, seed, migrating):
    """Raw point-target echo (Section VI): every target's azimuth chirp times its range pulse, with
    the hyperbolic range history when the cells migrate, plus noise 20 dB below the unit target."""
    raw = _noise((n_az, n_rg), math.sqrt(synth.NOISE_VARIANCE / 2), seed + 1)
    m, k, fs = synth.range_chirp_params()
    geo = synth.radar_geometry(APERTURE)
    ap = _aperture(n_az)
    ka = synth.AZIMUTH_DOPPLER_FRACTION / APERTURE
    rr = torch.arange(n_rg, device=DEV, dtype=torch.float64)
    for eta, r, a in _targets(n_az, n_rg, seed):
        e0, e1 = max(eta - ap // 2, 0), min(eta + ap // 2, n_az)
        t = torch.arange(e0, e1, device=DEV, dtype=torch.float64) - eta
        if migrating:
            rk = float(synth.slant_range_m(r, n_rg, geo))
            re = torch.sqrt(rk * rk + (geo.speed_mps * t / geo.prf_hz) ** 2)
            d, ph = (re - rk) / geo.range_cell_m, -4 * math.pi * (re - rk) / geo.wavelength_m
        else:
            d, ph = torch.zeros_like(t), -math.pi * ka * t * t
        tau = (rr[None, :] - r - d[:, None]) / fs
        inside = (tau >= -m / fs / 2) & (tau < m / fs / 2)
        phase = math.pi * k * tau * tau + ph[:, None]
        raw[e0:e1] += (torch.polar(inside.to(phase.dtype) * a, phase)).to(torch.complex64)
    return raw


def _references(n_az, n_rg):
    """Time-domain reference lines of the matched filters, complex64."""
    pulse = synth.range_chirp()
    cut = max(0, (pulse.shape[0] - n_rg + 1) // 2)
    ref_r = synth.centred_reference(pulse[cut:pulse.shape[0] - cut], n_rg)
    ref_a = synth.centred_reference(synth.azimuth_chirp(_aperture(n_az)), n_az) if n_az else None
    return _c64(ref_r), _c64(ref_a) if ref_a is not None else None


def _filter(ref, peak):
    h = torch.empty_like(ref)
    B.sar_make_filter(ref, ref.numel(), peak, h)
    return h


def _geometry():
    g = synth.radar_geometry(APERTURE)
    return (g.range_cell_m, g.prf_hz, g.wavelength_m, g.speed_mps, g.centre_range_m)


def _spectral_inputs(case, seed):
    n, lines = case["n"], case["lines"]
    x = _lines((lines, n), seed, case["x"])
    rows = lines if case["per_line"] else 1
    h = torch.view_as_complex(torch.randn((rows, n, 2), device=DEV, generator=_gen(seed + 1)) * math.sqrt(0.5))
    if case["per_line"]:
        h[:, n // 8:n - n // 8] = 0          # the kept modes of a spectral layer
    return x, h.contiguous()


def _autofocus_inputs(case, seed):
    """Range-compressed lines with a defocusing phase error (as synth.range_compressed_scene), the
    azimuth reference and the current phase estimate."""
    n_az, n_rg = case["n_az"], case["n_rg"]
    rc = _noise((n_rg, n_az), 0.05, seed)
    chirp = _c64(synth.azimuth_chirp(_aperture(n_az)))
    ap = chirp.numel()
    for eta, r, a in _targets(n_az, n_rg, seed):
        e0, e1 = max(eta - ap // 2, 0), min(eta + ap // 2, n_az)
        rc[r, e0:e1] += a * chirp[e0 - (eta - ap // 2):e1 - (eta - ap // 2)]
    err = torch.from_numpy(synth.phase_error(n_az, seed=seed)).to(DEV)
    rc *= torch.polar(torch.ones_like(err), err).to(torch.complex64)
    phi = torch.from_numpy((synth.phase_error(n_az, seed=seed, noise_rad=0.0) * 0.5).astype("float32")).to(DEV)
    _, ref_a = _references(n_az, 1024)
    return _to_storage(rc, case["rc"]), ref_a, phi


def _uneven_layout(case):
    """Lengths of the mixed batch (the plan's, whatever the data) and where each line starts."""
    lengths = synth.uneven_lengths(case["count"], seed=3)
    offsets = lengths.cumsum() - lengths
    return lengths, offsets


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fft":
        n, batch, st = case["n"], case["batch"], STORAGE[case["storage"]]
        fwd = B.bfpfft_plan_create(n, batch, st, B.FORWARD)
        inv = B.bfpfft_plan_create(n, batch, st, B.INVERSE)
        if case["arith"] != "f32":
            B.bfpfft_plan_set_arith(fwd, ARITH[case["arith"]])
            B.bfpfft_plan_set_arith(inv, ARITH[case["arith"]])
        x = _lines((batch, n), seed, case["storage"])
        return case, fwd, inv, x, torch.empty_like(x), torch.empty_like(x)
    if kind == "uneven":
        lengths, offsets = _uneven_layout(case)
        x = _lines((int(lengths.sum()),), seed, case["storage"])
        plan = B.bfpfft_plan_create_many(lengths, offsets, STORAGE[case["storage"]], B.FORWARD)
        return case, plan, x, torch.empty_like(x)
    if kind == "sar":
        n_az, n_rg = case["n_az"], case["n_rg"]
        raw = _to_storage(_echo(n_az, n_rg, seed, False), case["raw"])
        ref_r, ref_a = _references(n_az if case["stage"] == "image" else 0, n_rg)
        hr = _filter(ref_r, False)
        ha = _filter(ref_a, True) if ref_a is not None else None
        rc = _empty((n_rg, n_az), case["out"])
        img = _empty((n_az, n_rg), case["out"]) if ha is not None else None
        return case, raw, hr, ha, rc, img
    if kind == "rda":
        n_az, n_rg = case["n_az"], case["n_rg"]
        raw = _echo(n_az, n_rg, seed, True)
        hr = _filter(_references(n_az, n_rg)[0], False)
        return case, raw, hr, _empty((n_az, n_rg), case["out"])
    if kind == "spectral":
        x, h = _spectral_inputs(case, seed)
        return case, x, h, _empty((case["lines"], case["n"]), case["out"])
    rc, ref_a, phi = _autofocus_inputs(case, seed)
    ha = _filter(ref_a, True)
    ws = GA.Workspace(case["n_az"], DEV, ARITH[case["arith"]])
    return case, rc, ha, phi.requires_grad_(True), ws


def run(state):
    case, kind = state[0], state[0]["kind"]
    if kind == "fft":
        _, fwd, inv, x, y, z = state
        B.bfpfft_exec(fwd, x, y)
        B.bfpfft_exec(inv, y, z)
        return y, z
    if kind == "uneven":
        _, plan, x, y = state
        B.bfpfft_exec(plan, x, y)
        return y
    if kind == "sar":
        _, raw, hr, ha, rc, img = state
        n_az, n_rg, arith = case["n_az"], case["n_rg"], ARITH[case["arith"]]
        out = STORAGE[case["out"]]
        B.sar_range_compress_arith(raw, STORAGE[case["raw"]], rc, out, hr, n_az, n_rg, True, arith)
        if img is None:
            return rc
        B.sar_azimuth_compress_arith(rc, out, 1, img, out, ha, n_az, n_rg, arith)
        return rc, img
    if kind == "rda":
        _, raw, hr, img = state
        flags = B.RDA_RCMC | B.RDA_RANGE_DEPENDENT | B.RDA_PEAK_NORMALISE
        B.sar_rda_image(raw, B.F32, img, STORAGE[case["out"]], hr, case["n_az"], case["n_rg"], _geometry(),
                        _aperture(case["n_az"]), flags)
        return img
    if kind == "spectral":
        _, x, h, y = state
        n = case["n"]
        B.bfp_spectral_filter(x, STORAGE[case["x"]], h, n if case["per_line"] else 0, y, STORAGE[case["out"]], n,
                              case["lines"], ARITH[case["arith"]])
        return y
    _, rc, ha, phi, ws = state
    e = GA.entropy(phi, rc, ha, STORAGE[case["rc"]], ws)
    grad, = torch.autograd.grad(e, phi)
    return e, grad


# ---- the exact results ---------------------------------------------------------------------------

def _matched(ref, peak):
    h = torch.fft.fft(ref.to(torch.complex128)).conj()
    return h / h.abs().max() if peak else h


def _exact_rda(case, seed):
    n_az, n_rg = case["n_az"], case["n_rg"]
    cell, prf, lam, v, r0 = _geometry()
    raw = _echo(n_az, n_rg, seed, True).to(torch.complex128)
    rc = torch.fft.ifft(torch.fft.fft(raw, dim=1) * _matched(_references(n_az, n_rg)[0], False)[None, :], dim=1)
    del raw
    s_rd = torch.fft.fft(rc, dim=0)
    del rc
    k = torch.arange(n_az, device=DEV, dtype=torch.float64)
    f = torch.where(k >= n_az // 2, k - n_az, k) * prf / n_az
    s = r0 * (1 / torch.sqrt(1 - (lam * f / (2 * v)) ** 2) - 1) / cell
    q = torch.arange(n_rg, device=DEV, dtype=torch.float64)
    q = torch.where(q > n_rg // 2, q - n_rg, q)
    ph = 2 * math.pi * q[None, :] * s[:, None] / n_rg
    ramp = torch.polar(torch.ones_like(ph), ph)
    ramp[:, n_rg // 2] = torch.cos(math.pi * s).to(torch.complex128)
    s_rd = torch.fft.ifft(torch.fft.fft(s_rd, dim=1) * ramp, dim=1)
    del ramp, ph
    ap = _aperture(n_az)
    r_m = r0 + (torch.arange(n_rg, device=DEV, dtype=torch.float64) - n_rg / 2) * cell
    ka = 2 * v * v / (lam * r_m * prf * prf)
    n = torch.arange(ap, device=DEV, dtype=torch.float64) - ap / 2
    refs = torch.zeros((n_rg, n_az), dtype=torch.complex128, device=DEV)
    ph = -math.pi * ka[:, None] * n[None, :] ** 2
    refs[:, (torch.arange(ap, device=DEV) - ap // 2) % n_az] = torch.polar(torch.ones_like(ph), ph)
    h = torch.fft.fft(refs, dim=1).conj()
    h = h / h.abs().amax(dim=1, keepdim=True)
    return _like(torch.fft.ifft(s_rd * h.T, dim=0), case["out"])


def _exact_autofocus(case, seed):
    rc, ref_a, phi = _autofocus_inputs(case, seed)
    h = _matched(ref_a, True)[None, :]
    p = phi.to(torch.float64)
    v = _values(rc) * torch.polar(torch.ones_like(p), -p)[None, :]
    i = torch.fft.ifft(torch.fft.fft(v, dim=1) * h, dim=1)
    q = i.real ** 2 + i.imag ** 2
    s = q.sum()
    ln = torch.where(q > 0, q.clamp_min(1e-300).log(), torch.zeros_like(q))
    e = torch.log(s) - (q * ln).sum() / s
    g = torch.where(q > 0, -(ln - torch.log(s) + e) / s, torch.zeros_like(q)) * i
    del i, q, ln
    b = torch.fft.ifft(torch.fft.fft(g, dim=1) * h.conj(), dim=1)
    return e, 2 * (b.conj() * v).imag.sum(dim=0)


def exact(case, seed):
    kind = case["kind"]
    if kind == "fft":
        x = _values(_lines((case["batch"], case["n"]), seed, case["storage"]))
        y = torch.fft.fft(x, dim=1)
        if case["storage"] in FP8:           # the plan's block exponent: stored X 2^-ceil(log2(n) / 2)
            y *= 2.0 ** -((int(math.log2(case["n"])) + 1) // 2)
        return _like(y, case["storage"]), _like(x, case["storage"])
    if kind == "uneven":
        lengths, offsets = _uneven_layout(case)
        y = _values(_lines((int(lengths.sum()),), seed, case["storage"]))
        for n in sorted(set(int(v) for v in lengths)):
            off = torch.from_numpy(offsets[lengths == n]).to(DEV)
            scale = 2.0 ** -((int(math.log2(n)) + 1) // 2) if case["storage"] in FP8 else 1.0
            step = max(1, (1 << 25) // n)
            for at in range(0, off.numel(), step):
                idx = off[at:at + step, None] + torch.arange(n, device=DEV)[None, :]
                y[idx] = torch.fft.fft(y[idx], dim=1) * scale
        return _like(y, case["storage"])
    if kind == "sar":
        n_az, n_rg = case["n_az"], case["n_rg"]
        raw = _values(_to_storage(_echo(n_az, n_rg, seed, False), case["raw"]))
        ref_r, ref_a = _references(n_az if case["stage"] == "image" else 0, n_rg)
        rc = torch.fft.ifft(torch.fft.fft(raw, dim=1) * _matched(ref_r, False)[None, :], dim=1).T.contiguous()
        if ref_a is None:
            return _like(rc, case["out"])
        img = torch.fft.ifft(torch.fft.fft(rc, dim=1) * _matched(ref_a, True)[None, :], dim=1).T.contiguous()
        return _like(rc, case["out"]), _like(img, case["out"])
    if kind == "rda":
        return _exact_rda(case, seed)
    if kind == "spectral":
        x, h = _spectral_inputs(case, seed)
        return _like(torch.fft.ifft(torch.fft.fft(_values(x), dim=1) * h.to(torch.complex128), dim=1), case["out"])
    return _exact_autofocus(case, seed)


# ---- what a pass cannot do without -----------------------------------------------------------------

def _fft_flops(lines, n):
    return 5.0 * lines * n * math.log2(n)


def work(case):
    kind = case["kind"]
    if kind == "fft":
        pts = float(case["n"]) * case["batch"]
        return {"bytes": 4 * pts * POINT_BYTES[case["storage"]], "flops": 2 * _fft_flops(case["batch"], case["n"])}
    if kind == "uneven":
        lengths, _ = _uneven_layout(case)
        return {"bytes": 2.0 * float(lengths.sum()) * POINT_BYTES[case["storage"]],
                "flops": sum(_fft_flops(1, int(n)) * int((lengths == n).sum()) for n in set(lengths.tolist()))}
    if kind == "spectral":
        pts = float(case["n"]) * case["lines"]
        h = 8 * (pts if case["per_line"] else case["n"])
        return {"bytes": pts * (POINT_BYTES[case["x"]] + POINT_BYTES[case["out"]]) + h,
                "flops": 2 * _fft_flops(case["lines"], case["n"]) + 6 * pts}
    n_az, n_rg = case["n_az"], case["n_rg"]
    pts = float(n_az) * n_rg
    if kind == "sar":
        ob = POINT_BYTES[case["out"]]
        w = {"bytes": pts * (POINT_BYTES[case["raw"]] + ob), "flops": 2 * _fft_flops(n_az, n_rg) + 6 * pts}
        if case["stage"] == "image":
            w["bytes"] += 2 * pts * ob       # rc is an output of one call and the input of the next
            w["flops"] += 2 * _fft_flops(n_rg, n_az) + 6 * pts
        return w
    if kind == "rda":
        # range compression, azimuth DFT, RCMC (two transforms), the bin's filter and the inverse
        return {"bytes": pts * (8 + POINT_BYTES[case["out"]]),
                "flops": 4 * _fft_flops(n_az, n_rg) + 3 * _fft_flops(n_rg, n_az) + 18 * pts}
    # autofocus: the image, its weights, the adjoint
    return {"bytes": pts * POINT_BYTES[case["rc"]], "flops": 4 * _fft_flops(n_rg, n_az) + 40 * pts}
