"""The calls whose speed counts: what a user of the beamformer has it do.

A case is one call of a public entry point on one set of sizes:

``op`` "beamform"  ``beamform`` on frames resident in device memory
``op`` "host"      ``beamform_host`` on frames in pinned host memory, images back in pinned memory
``op`` "metrics"   ``image_metrics`` on resident envelope images

``listed`` names the cases, ``draw`` gives others of the same ranges: 24 to
256 elements, 400 to 4096 samples, lateral grids on the element lattice
(``m`` columns a pitch) or off it (``m`` = 0, full delay table), 48 to 1024
depth rows at 0.7 to 4 RF samples a row, orders 1 to 8, FP32 / BF16 / FP16
RF, plain or compensated sums, linear or nearest samples, full aperture or
dynamic Hann aperture, 1 to 64 frames a call, any stages and outputs.
"""

import math

import numpy as np
import torch

import paper_2203_14906_gb300 as pa

RAW, ENV, LOG = pa.PA_STAGE_RAW, pa.PA_STAGE_ENV, pa.PA_STAGE_LOG
ALL_OUT = pa.PA_OUT_DAS | pa.PA_OUT_DMAS | pa.PA_OUT_HODMAS

PITCH, C, F0, DYN = 0.3e-3, 1540.0, 5e6, 60.0
TORCH_TYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


def _bf(name, **kw):
    c = dict(op="beamform", n_elem=128, n_samples=2048, fs_hz=40e6, nx=512, nz=512, m=4, z0_m=0.0,
             depth_m=40e-3, k=3, dtype="f32", compensated=False, f_number=0.0, interp="linear",
             outputs=ALL_OUT, stages=LOG, frames=1)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one frame of a 64-element probe on a quick-look grid, as a
        # pre-scan or an alignment loop makes it; launches and latency count
        _bf("quicklook_frame", n_elem=64, n_samples=1024, nx=128, nz=128, m=2, depth_m=20e-3),
        # live imaging: every frame is beamformed as it arrives, envelope kept next to the display
        _bf("live_frame", stages=ENV | LOG),
        # the same from and to host memory, the highest order alone: a scanner's
        # acquisition buffer in, the screen's image out
        _bf("live_frame_host", op="host", outputs=pa.PA_OUT_HODMAS),
        # a served batch of small requests: 16-bit frames of one probe, compensated sums
        _bf("served_batch_256", n_elem=64, nx=256, nz=256, k=2, dtype="bf16", compensated=True,
            frames=6),
        # offline reconstruction of a recorded sequence, the paper's order 3 (benchmark workload)
        _bf("sequence_512_k3", frames=32),
        # the order study's highest order of the paper, all stages kept for comparison
        _bf("order_study_k5", k=5, frames=8, stages=RAW | ENV | LOG),
        # integer delays as Eq. 1 writes them, raw images for a later filter
        _bf("nearest_raw_k2", k=2, frames=16, interp="nearest", stages=RAW),
        # large aperture, fine grid, 16-bit storage with compensated sums
        _bf("precision_1024", n_elem=256, n_samples=4096, fs_hz=50e6, nx=1024, nz=1024,
            depth_m=60e-3, dtype="bf16", compensated=True, frames=4, stages=ENV),
        # a lateral grid that is no multiple of the pitch: the full delay table
        _bf("off_lattice_400", nx=400, m=0, frames=12),
        # odd sizes throughout: odd aperture and record, ragged tiles, odd batch
        _bf("ragged_odd", n_elem=97, n_samples=1501, nx=291, nz=333, m=3, z0_m=1.5e-3,
            depth_m=22e-3, k=4, dtype="f16", frames=5, stages=ENV | LOG),
        # throughput reconstruction: dynamic aperture, 64 frames of 1024 x 1024
        _bf("throughput_apodised", nx=1024, nz=1024, m=8, k=4, dtype="bf16", compensated=True,
            f_number=1.5, frames=64),
        # image quality of a finished study: every target on every envelope image
        dict(name="study_metrics", op="metrics", n_elem=128, nx=512, nz=512, z0_m=0.0,
             depth_m=40e-3, images=96, rois=10),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    if rng.random() < 0.1:
        return dict(op="metrics", n_elem=128, nx=_log_uniform(rng, 100, 800),
                    nz=_log_uniform(rng, 100, 800), z0_m=0.0, depth_m=rng.uniform(20e-3, 50e-3),
                    images=_log_uniform(rng, 1, 96), rois=rng.randint(1, 16))
    limit = _cost(next(c for c in listed() if c["name"] == "throughput_apodised"))
    while True:
        n = _log_uniform(rng, 24, 256)
        ns = _log_uniform(rng, 400, 4096)
        if rng.random() < 0.6:
            ns = (ns + 7) // 8 * 8  # records are mostly padded to whole words
        m = rng.choice([0, 1, 2, 3, 4, 4, 6, 8])
        nx = rng.randint(max(24, n), 4 * n) if m == 0 else n * m
        nz = _log_uniform(rng, 48, 1024)
        # pixels finer than 0.7 samples a row are not asked for, nor images deeper than the record
        fs = 40e6
        per_row = min(rng.uniform(0.7, 4.0), 0.95 * ns / nz)
        dtype = rng.choice(["f32", "f32", "bf16", "f16"])
        c = _bf(None, op="host" if rng.random() < 0.12 else "beamform", n_elem=n, n_samples=ns,
                fs_hz=fs, nx=min(nx, 1024), nz=nz, m=m if nx <= 1024 else 0,
                z0_m=rng.choice([0.0, 0.0, rng.uniform(0.5e-3, 3e-3)]),
                depth_m=nz * per_row * C / fs, k=rng.choice([1, 2, 2, 3, 3, 3, 4, 4, 5, 5, 6, 7, 8]),
                dtype=dtype, compensated=rng.random() < (0.25 if dtype == "f32" else 0.7),
                f_number=rng.choice([0.0, 0.0, 0.0, rng.uniform(1.0, 2.5)]),
                interp=rng.choice(["linear", "linear", "linear", "nearest"]),
                outputs=rng.choice([ALL_OUT, ALL_OUT, ALL_OUT, pa.PA_OUT_HODMAS,
                                    pa.PA_OUT_DAS | pa.PA_OUT_DMAS]),
                stages=rng.choice([RAW, ENV, LOG, LOG, ENV | LOG, RAW | ENV | LOG]),
                frames=_log_uniform(rng, 1, 64))
        if c["op"] == "host":
            c["frames"] = min(c["frames"], 2)  # the live path; longer calls tune their schedule
        if c["m"] == 0 and n * c["nx"] * nz > 1 << 25:
            continue  # a full table of at most some hundred megabytes
        if c["k"] <= c["n_elem"] and _cost(c) <= limit:
            return c


# ------------------------------------------------------------------ geometry


def _grid(case):
    half = case["n_elem"] * PITCH / 2
    return dict(nx=case["nx"], nz=case["nz"], x0_m=-half, x1_m=half, z0_m=case["z0_m"],
                z1_m=case["z0_m"] + case["depth_m"])


def _axes(case, device):
    g = _grid(case)
    dx, dz = (g["x1_m"] - g["x0_m"]) / g["nx"], (g["z1_m"] - g["z0_m"]) / g["nz"]
    x = g["x0_m"] + (torch.arange(g["nx"], dtype=torch.float64, device=device) + 0.5) * dx
    z = g["z0_m"] + (torch.arange(g["nz"], dtype=torch.float64, device=device) + 0.5) * dz
    e = (torch.arange(case["n_elem"], dtype=torch.float64, device=device)
         - 0.5 * (case["n_elem"] - 1)) * PITCH
    return x, z, e


def _stage_list(stages):
    return [s for s in (RAW, ENV, LOG) if stages & s]


def _output_list(outputs):
    return [o for o in (pa.PA_OUT_DAS, pa.PA_OUT_DMAS, pa.PA_OUT_HODMAS) if outputs & o]


def _pairs(case):
    """(pixel, channel) pairs of one frame inside the aperture."""
    full = case["nx"] * case["nz"] * case["n_elem"]
    if not case["f_number"]:
        return full
    x, z, e = (v.numpy() for v in _axes(case, "cpu"))
    half = z / (2 * case["f_number"])
    total = 0
    for xc in x:
        d = np.sort(np.abs(xc - e))
        total += int(np.searchsorted(d, half, side="right").sum())
    return total


def work(case):
    if case["op"] == "metrics":
        px = sum(int(_inside(r, case, "cpu").sum()) for pair in _rois(case) for r in pair)
        record = 12 * 8  # bytes of one result record
        return {"bytes": 4 * px * case["images"] + record * case["images"] * case["rois"],
                "flops": 4 * px * case["images"]}
    elt = 4 if case["dtype"] == "f32" else 2
    n_out, stages = len(_output_list(case["outputs"])), _stage_list(case["stages"])
    px = case["nx"] * case["nz"]
    per_frame = case["n_elem"] * case["n_samples"] * elt + 4 * px * n_out * len(stages)
    # interpolation, roots, power sums of the order and of DAS and DMAS
    flops = _pairs(case) * (2 * case["k"] + 7)
    if case["stages"] & (ENV | LOG):
        size = 1 << max(0, (case["nz"] - 1).bit_length())
        flops += case["nx"] * n_out * 1.5 * 5 * size * max(1, size.bit_length() - 1)
    return {"bytes": per_frame * case["frames"], "flops": flops * case["frames"]}


def _cost(case):
    """Work of a case for draw()'s limit (the full aperture counted)."""
    return case["nx"] * case["nz"] * case["frames"] * (case["n_elem"] * (2 * case["k"] + 7)
                                                       * (0.4 if case["f_number"] else 1.0) + 200)


# -------------------------------------------------------------------- inputs


def _rf(case, seed):
    """RF [frames][N][Ns] of point absorbers (derivative-of-Gaussian pulses, 1/r
    amplitudes) plus noise, scaled to unit RMS, in the case's storage type."""
    dev = "cuda"
    f, n, ns = case["frames"], case["n_elem"], case["n_samples"]
    g = _grid(case)
    pos = np.random.default_rng([seed, 7])
    points = 12
    xs = torch.tensor(pos.uniform(0.9 * g["x0_m"], 0.9 * g["x1_m"], (points, f)), device=dev)
    span = g["z1_m"] - g["z0_m"]
    zs = torch.tensor(pos.uniform(g["z0_m"] + 0.1 * span, g["z0_m"] + 0.95 * span, (points, f)),
                      device=dev)
    amp = torch.tensor(10 ** (-pos.uniform(0, 1.5, (points, f))), device=dev)
    e = _axes(case, dev)[2]
    t = torch.arange(ns, dtype=torch.float32, device=dev) / case["fs_hz"]
    sigma = 1.0 / (2 * math.pi * F0)
    rf = torch.zeros((f, n, ns), dtype=torch.float32, device=dev)
    for p in range(points):
        r = torch.sqrt((xs[p][:, None] - e) ** 2 + zs[p][:, None] ** 2)
        u = (t - (r / C)[..., None].float()) / sigma
        rf -= (amp[p][:, None] * 1e-3 / r)[..., None].float() * u * torch.exp(0.5 - 0.5 * u * u)
    gen = torch.Generator(device=dev).manual_seed(seed)
    rf += 0.03 * rf.abs().amax() * torch.randn(rf.shape, generator=gen, device=dev)
    rf /= rf.square().mean().sqrt()
    return rf.to(TORCH_TYPES[case["dtype"]])


def _rois(case):
    """Disc targets spread over the image, each with an annulus around it as background."""
    g = _grid(case)
    out = []
    for i in range(case["rois"]):
        xc = g["x0_m"] * 0.8 + 1.6 * g["x1_m"] * (i + 0.5) / case["rois"]
        zc = g["z0_m"] + case["depth_m"] * (0.15 + 0.7 * ((i * 0.618034) % 1.0))
        out.append((dict(shape="disc", xc_m=xc, zc_m=zc, a_m=1.2e-3),
                    dict(shape="annulus", xc_m=xc, zc_m=zc, a_m=1.6e-3, b_m=2.8e-3)))
    return out


def _images(case, seed):
    """Envelope images: speckle with a bright blob on every target."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x, z, _ = _axes(case, "cuda")
    shape = (case["images"], case["nx"], case["nz"])
    img = torch.rand(shape, generator=gen, device="cuda").clamp_(min=1e-7).log_().mul_(-2).sqrt_()
    width = torch.empty(case["images"], device="cuda").uniform_(0.3e-3, 0.8e-3, generator=gen)
    for target, _ in _rois(case):
        d2 = ((x - target["xc_m"])[:, None] ** 2 + (z - target["zc_m"])[None, :] ** 2).float()
        img += 12.0 * torch.exp(-d2 / (2 * width[:, None, None] ** 2))
    return img


def prepare(case, seed):
    if case["op"] == "metrics":
        return dict(op="metrics", images=_images(case, seed), grid=_grid(case), rois=_rois(case))
    wl = dict(n_elem=case["n_elem"], pitch_m=PITCH, c_m_s=C, fs_hz=case["fs_hz"], t0_s=0.0,
              n_samples=case["n_samples"], order_k=case["k"], f_number=case["f_number"], f0_hz=F0,
              dyn_range_db=DYN, rf_dtype=case["dtype"], compensated=int(case["compensated"]),
              interp=case["interp"], **_grid(case))
    plan = pa.Plan(pa.make_desc(wl, outputs=case["outputs"], max_batch=case["frames"]))
    rf = _rf(case, seed)
    shape = plan.out_shape(case["frames"], case["stages"])
    if case["op"] == "host":
        rf = rf.cpu().pin_memory()
        out = torch.empty(shape, dtype=torch.float32, pin_memory=True)
    else:
        out = torch.empty(shape, dtype=torch.float32, device="cuda")
    return dict(op=case["op"], plan=plan, rf=rf, out=out, stages=case["stages"])


def run(state):
    if state["op"] == "metrics":
        return pa.image_metrics(state["images"], state["grid"], state["rois"])
    call = pa.beamform_host if state["op"] == "host" else pa.beamform
    return call(state["plan"], state["rf"], state["stages"], out=state["out"])


# ---------------------------------------------------------------- in 64 bits


def _band_mask(case, even, size, device):
    """Band-pass (f0 +- f0/2, around 2 f0 for even orders; raised-cosine roll-off f0/4,
    clipped at the axial Nyquist rate) times the analytic-signal weights."""
    dz = case["depth_m"] / case["nz"]
    nyquist = C / (2 * dz)
    lo, hi, roll = (1.5 * F0 if even else 0.5 * F0), (2.5 * F0 if even else 1.5 * F0), 0.25 * F0
    b = torch.arange(size, dtype=torch.float64, device=device)
    analytic = torch.where((b == 0) | (2 * b == size), 1.0, torch.where(2 * b < size, 2.0, 0.0))
    if lo >= nyquist:  # nothing of the band is left: only the mean goes
        return torch.where(b == 0, 0.0, 1.0) * analytic
    freq = C * b / (size * dz)
    off = torch.maximum(torch.clamp(lo - freq, min=0), torch.clamp(freq - min(hi, nyquist), min=0))
    band = torch.where(off < roll, 0.5 * (1 + torch.cos(math.pi * off / roll)),
                       torch.zeros_like(off))
    return band * analytic


def _exact_raw(case, rf):
    """DAS, DMAS and DMAS-k of every frame: [outputs][frames][nx][nz] in 64 bits."""
    k, n, ns = case["k"], case["n_elem"], case["n_samples"]
    x, z, e = _axes(case, rf.device)
    f, px = rf.shape[0], case["nx"] * case["nz"]
    rf = rf.double()
    das = torch.zeros((f, px), dtype=torch.float64, device=rf.device)
    q1, q2 = torch.zeros_like(das), torch.zeros_like(das)
    p = [torch.zeros_like(das) for _ in range(k)]
    for i in range(n):
        dxv = (x - e[i])[:, None]
        tau = (case["fs_hz"] * torch.sqrt(dxv * dxv + z * z) / C).reshape(-1)
        if case["interp"] == "nearest":
            idx = torch.floor(tau + 0.5).long()
            ok = (idx >= 0) & (idx <= ns - 1)
            s = rf[:, i].index_select(1, idx.clamp(0, ns - 1))
        else:
            idx = torch.floor(tau).long()
            ok = (idx >= 0) & (idx + 1 <= ns - 1)
            idx0 = idx.clamp(0, ns - 2)
            r0 = rf[:, i].index_select(1, idx0)
            s = rf[:, i].index_select(1, idx0 + 1).sub_(r0).mul_(tau - idx0).add_(r0)
        weight = ok.double()
        if case["f_number"]:
            half = z / (2 * case["f_number"])
            w = torch.where(dxv.abs() <= half, torch.cos(math.pi * dxv / (2 * half)) ** 2,
                            torch.zeros_like(dxv * z))
            weight = weight * w.reshape(-1)
        s = s * weight
        das += s
        a = s.abs()
        q2 += a
        sign = torch.sign(s)
        q1 += sign * a.sqrt()
        root = sign * a.pow(1.0 / k)
        power = root
        for j in range(k):
            p[j] += power
            if j + 1 < k:
                power = power * root
    el = [torch.ones_like(das)]
    for j in range(1, k + 1):  # Newton's identities
        acc = torch.zeros_like(das)
        for t in range(1, j + 1):
            acc += (-1) ** (t - 1) * el[j - t] * p[t - 1]
        el.append(acc / j)
    dmas = 0.5 * (q1 * q1 - q2)
    by_output = {pa.PA_OUT_DAS: das, pa.PA_OUT_DMAS: dmas,
                 pa.PA_OUT_HODMAS: das if k == 1 else dmas if k == 2 else el[k]}
    shape = (f, case["nx"], case["nz"])
    return [by_output[o].reshape(shape) for o in _output_list(case["outputs"])]


def _exact_images(case, rf):
    out = []
    size = 1 << max(0, (case["nz"] - 1).bit_length())
    even_of = {pa.PA_OUT_DAS: False, pa.PA_OUT_DMAS: True, pa.PA_OUT_HODMAS: case["k"] % 2 == 0}
    for o, raw in zip(_output_list(case["outputs"]), _exact_raw(case, rf)):
        by_stage = {RAW: raw}
        if case["stages"] & (ENV | LOG):
            mask = _band_mask(case, even_of[o], size, raw.device)
            env = torch.fft.ifft(torch.fft.fft(raw, n=size, dim=-1) * mask, dim=-1).abs()
            env = env[..., : case["nz"]]
            by_stage[ENV] = env
            peak = env.amax(dim=(1, 2), keepdim=True)
            log = 20 * torch.log10(env / peak)
            by_stage[LOG] = torch.nan_to_num(log, nan=-DYN, neginf=-DYN).clamp(-DYN, 0.0)
        out.append(torch.stack([by_stage[s] for s in _stage_list(case["stages"])], dim=1))
    return torch.stack(out, dim=2)  # [frames][stages][outputs][nx][nz]


def _inside(region, case, device):
    x, z, _ = _axes(case, device)
    d2 = (x - region["xc_m"])[:, None] ** 2 + (z - region["zc_m"])[None, :] ** 2
    if region["shape"] == "disc":
        return d2 <= region["a_m"] ** 2
    return (d2 > region["a_m"] ** 2) & (d2 <= region["b_m"] ** 2)


def _exact_metrics(case, images):
    cols = {name: [] for name in ("mu_in", "mu_out", "sigma_out", "snr_db", "cr_db", "peak")}
    for target, background in _rois(case):
        inner = images[:, _inside(target, case, images.device)].double()
        outer = images[:, _inside(background, case, images.device)].double()
        mu, mo = inner.mean(1), outer.mean(1)
        sd = (outer - mo[:, None]).square().mean(1).sqrt()
        for name, v in (("mu_in", mu), ("mu_out", mo), ("sigma_out", sd),
                        ("snr_db", 20 * torch.log10(mu / sd)), ("cr_db", 20 * torch.log10(mu / mo)),
                        ("peak", inner.amax(1))):
            cols[name].append(v)
    full = {name: torch.stack(v, dim=1).cpu().numpy() for name, v in cols.items()}
    # the histogram overlap and the walk along a row are defined in their own arithmetic
    for name in ("gcnr", "fwhm_m", "n_in", "n_out", "peak_j", "peak_l"):
        full[name] = None
    return full


def exact(case, seed):
    if case["op"] == "metrics":
        return _exact_metrics(case, _images(case, seed))
    parts = []
    rf = _rf(case, seed)
    step = max(1, (1 << 25) // (case["nx"] * case["nz"]))
    for f in range(0, case["frames"], step):
        images = _exact_images(case, rf[f:f + step])
        parts.append(images.cpu() if case["op"] == "host" else images)
    return torch.cat(parts)
