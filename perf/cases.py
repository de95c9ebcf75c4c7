"""Performance cases of the library: what its users run, from the smallest call to the largest.

Every case goes through the public binding (`hdr.Context`, `hdr.Server`). Scenes, rigs and sizes
follow the package's own seeded recipes (`synth`): log-uniform HDR scenes of smooth shading and
straight edges, RGGB sensors behind neutral-density filters, Poisson and read noise, 12-bit
clipping. The frames are rendered on the GPU here, so that a fresh one takes milliseconds.

A case is a dict of plain values; `kind` says which entry point it calls:
  frame      one frame from device buffers
  adaptive   one frame with steered windows (gradients, steering matrices, steered fit)
  structure  the gradient and steering-matrix passes alone
  batch      uneven frames in one graph launch
  serve      one frame of every concurrent video stream through the request loop, host buffers
  stats      per-pixel mean and variance of a calibration stack
"""
import math

import numpy as np
import torch

from paper_1308_4908_gb300 import hdr, synth

PAPER_ND = (1.0, 1 / 16, 1 / 256, 1 / 4096)   # the paper-scale rig's filters and the camera's
LADDER_ND = (1.0, 1 / 8, 1 / 64, 1 / 512)     # the batching recipe's filters

FRAME = {"kind": "frame", "n": 3, "w": 0, "h": 0, "ow": 0, "oh": 0, "order": 2, "scales": 4, "sigma": 0.7,
         "shift": 1.5, "rot": 0.2, "zoom": 1e-3, "paper_nd": True, "half": False, "comp": False, "calibrated": False,
         "camera": False, "rig": 1}


def _case(name, **over):
    return {**FRAME, **over, "name": name}


def listed():
    return [
        # The smallest call: a 64 x 64 region of two sensors, order 0, one window (previews, tests,
        # regions of interest). Launches and host work are most of it.
        _case("tiny-m0", n=2, w=64, h=64, ow=64, oh=64, order=0, scales=1, shift=1.0, rot=0.0, zoom=0.0,
              paper_nd=False),
        # One 720p video stream of two sensors, order 2 with four scales: the smallest stream served.
        _case("stream720-m2", n=2, w=1280, h=720, ow=1280, oh=720, rig=2),
        # The paper-scale frame: three 2048 x 2048 sensors with affine misalignment, order 2 with the
        # interval rule over four scales. The library's headline workload.
        _case("paper-m2", w=2048, h=2048, ow=2048, oh=2048, rig=3),
        # Full HD at 1.5 times the sensor resolution, order 1 with four scales: a resampled output,
        # whose pixels see the sensors at varying fractions.
        _case("hd-up-m1", w=1920, h=1080, ow=2880, oh=1620, order=1, paper_nd=False, rig=4),
        # Two sensors enlarged twofold to 4096 x 4096, order 0, one window, stored as FP16: output-heavy.
        _case("upsample-m0-half", n=2, w=2048, h=2048, ow=4096, oh=4096, order=0, scales=1, shift=1.0, rot=0.0,
              zoom=0.0, paper_nd=False, half=True, rig=5),
        # The paper's own camera: four 2336 x 1752 sensors displaced by a few pixels, order 0, one
        # window, tabulated window weights.
        _case("camera-m0", n=4, w=2336, h=1752, ow=2336, oh=1752, order=0, scales=1, shift=3.0, rot=0.0, zoom=0.0,
              camera=True, rig=6),
        # A laboratory rig with per-pixel calibration frames and odd sizes, order 2 at one fixed
        # window, compensated sums: the precise setting.
        _case("lab-m2-comp", w=1021, h=769, ow=1019, oh=767, scales=1, sigma=1.2, comp=True, calibrated=True, rig=7),
        # Adaptive (steered) windows on a 1-megapixel frame, order 2 with four scales: best quality,
        # the most work per pixel.
        _case("adaptive-m2", kind="adaptive", w=1024, h=1024, ow=1024, oh=1024, rig=8),
        # Structure analysis alone at full HD: the gradients and steering matrices that a program
        # computes once and uses for several reconstructions of a frame.
        _case("structure-hd", kind="structure", w=1920, h=1080, ow=1920, oh=1080, paper_nd=False, rig=9),
        # Sixteen uneven frames (512 x 512 to 2048 x 2048, two to four sensors, orders 0 to 2, 1x or
        # 1.5x) in one graph launch: offline processing of mixed material.
        {"name": "batch-16", "kind": "batch", "spec": 1004, "frames": 16, "cap": 2048},
        # One frame of each of eight concurrent video streams, 720p to 2048 x 2048 -> 3840 x 2160,
        # submitted together from pinned host buffers and polled: the request loop at its work.
        {"name": "serve-8", "kind": "serve", "streams": 8, "cap": 4096, "rig": 10},
        # Calibration of one sensor of the paper's camera: 64 flat-field frames to per-pixel mean and
        # variance; a width that is no multiple of the vector width.
        {"name": "stats-64", "kind": "stats", "frames": 64, "w": 2330, "h": 1752, "level": 900.0},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["single", "single", "single", "scales", "scales", "scales", "camera", "adaptive", "structure",
                       "batch", "serve", "stats"])
    rig = rng.randrange(1, 1000)
    if kind == "single":  # one window: any size, order, enlargement and storage
        order = rng.choice([0, 0, 1, 2])
        w, h = _log(rng, 48, 2048), _log(rng, 48, 2048)
        up = rng.choice([1.0, 1.0, 1.5, 2.0])
        ow, oh = max(1, int(w * up) - rng.randrange(3)), max(1, int(h * up) - rng.randrange(3))
        cal = w * h <= 1 << 20 and rng.random() < 0.3
        still = rng.random() < 0.5
        return {**FRAME, "n": rng.randint(2, 4), "w": w, "h": h, "ow": ow, "oh": oh, "order": order, "scales": 1,
                "sigma": 0.7 if order == 0 else 1.2, "shift": 1.0, "rot": 0.0 if still else 0.2,
                "zoom": 0.0 if still else 1e-3, "paper_nd": rng.random() < 0.5, "half": rng.random() < 0.3,
                "comp": rng.random() < 0.3, "calibrated": cal, "rig": rig}
    if kind == "scales":  # the interval rule over four scales: video-sized frames
        w, h = _log(rng, 512, 2048), _log(rng, 512, 2048)
        up = rng.choice([1.0, 1.0, 1.5])
        still = rng.random() < 0.3
        return {**FRAME, "n": rng.randint(2, 4), "w": w, "h": h, "ow": int(w * up), "oh": int(h * up),
                "order": rng.randint(0, 2), "rot": 0.0 if still else 0.2, "zoom": 0.0 if still else 1e-3,
                "paper_nd": rng.random() < 0.5, "half": rng.random() < 0.2, "rig": rig}
    if kind == "camera":  # the four-sensor camera, its translations or small rotations
        w, h = _log(rng, 640, 2336), _log(rng, 480, 1752)
        return {**FRAME, "n": 4, "w": w, "h": h, "ow": w, "oh": h, "order": 0, "scales": 1, "shift": 3.0,
                "rot": rng.choice([0.0, 0.3]), "zoom": 0.0, "camera": True, "rig": rig}
    if kind == "adaptive":
        w, h = _log(rng, 512, 1280), _log(rng, 512, 1280)
        return {**FRAME, "kind": "adaptive", "w": w, "h": h, "ow": w, "oh": h, "order": rng.randint(0, 2), "rig": rig}
    if kind == "structure":
        w, h = _log(rng, 128, 2048), _log(rng, 128, 2048)
        return {**FRAME, "kind": "structure", "n": rng.randint(2, 3), "w": w, "h": h, "ow": w, "oh": h, "rig": rig}
    if kind == "batch":
        return {"kind": "batch", "spec": rng.randrange(1, 100000), "frames": rng.randint(3, 8),
                "cap": _log(rng, 512, 1920)}
    if kind == "serve":
        return {"kind": "serve", "streams": rng.randint(2, 6), "cap": _log(rng, 640, 1920), "rig": rig}
    return {"kind": "stats", "frames": _log(rng, 4, 96), "w": _log(rng, 256, 2336), "h": _log(rng, 256, 1752),
            "level": float(rng.randint(60, 1200))}


# ------------------------------------------------------------------------------------------ inputs

def _rig(c):
    """The sensors of a frame case: their placement and calibration are the case's, whatever the seed."""
    r = np.random.default_rng([c["rig"], c["n"]])
    nds = PAPER_ND if c["paper_nd"] else LADDER_ND
    sensors = []
    for s in range(c["n"]):
        tx, ty = r.uniform(-c["shift"], c["shift"], 2)
        rot = r.uniform(-c["rot"], c["rot"]) if c["rot"] else 0.0
        zoom = 1.0 + (r.uniform(-c["zoom"], c["zoom"]) if c["zoom"] else 0.0)
        more = dict(gain=0.27, exposure=2.0 / 0.27, read_var=(72.0 * 0.27) ** 2) if c["camera"] else {}
        sen = synth.Sensor(c["w"], c["h"], nds[s], synth.affine_about_center(c["w"], c["h"], tx, ty, rot, zoom), **more)
        if c["calibrated"]:
            shape = (c["h"], c["w"])
            sen.bias_frame = (64.0 + r.normal(0.0, 2.0, shape)).astype(np.float32)
            sen.prnu_frame = r.uniform(0.95, 1.05, shape).astype(np.float32)
            sen.read_var_frame = r.uniform(6.0, 14.0, shape).astype(np.float32)
            sen.sat_frame = r.integers(3900, 4096, shape).astype(np.uint16)
        sensors.append(sen)
    return sensors


def _params(c):
    return synth.Params(order=c["order"], sigmas=synth.PAPER_SCALES if c["scales"] == 4 else (c["sigma"],),
                        out_w=c["ow"], out_h=c["oh"], out_affine=synth.output_affine(c["w"], c["h"], c["ow"], c["oh"]),
                        out_dtype=int(c["half"]), accum=int(c["comp"]))


def _render(scene, sen, seed, index):
    """The raw frame [height, pitch] of `scene` through `sen`: what synth.simulate_raw does, on the GPU."""
    dev = "cuda"
    g = torch.Generator(device=dev).manual_seed(1000003 * int(seed) + index)
    x = torch.arange(sen.width, device=dev, dtype=torch.float64)[None, :]
    y = torch.arange(sen.height, device=dev, dtype=torch.float64)[:, None]
    m = sen.affine
    u = (m[0, 0] * x + m[0, 1] * y + m[0, 2]) / scene.width
    v = (m[1, 0] * x + m[1, 1] * y + m[1, 2]) / scene.height
    acc, norm = torch.zeros_like(u), 0.0
    for amp, ang, _ in scene.ramps:
        acc += amp * (math.cos(ang) * (u - 0.5) + math.sin(ang) * (v - 0.5))
        norm += abs(amp) * 0.75
    for amp, fx, px, fy, py in scene.cosines:
        acc += amp * torch.cos(2 * math.pi * (fx * u + px)) * torch.cos(2 * math.pi * (fy * v + py))
        norm += abs(amp)
    xi, yi = x.long() & 1, y.long() & 1
    colour = torch.where((xi == 0) & (yi == 0), 0, torch.where((xi == 1) & (yi == 1), 2, 1))
    level = -2.0 + 6.0 * (0.5 + 1.25 * acc / norm).clamp(0.0, 1.0)
    level += torch.tensor(scene.base_tint, device=dev)[colour]
    for k, (px, py, ang, jump) in enumerate(scene.edges):
        side = torch.where(math.cos(ang) * (u - px) + math.sin(ang) * (v - py) > 0, 0.5, -0.5)
        level += side * (jump + torch.tensor(scene.edge_tint[k], device=dev)[colour])
    f = torch.pow(10.0, level.clamp(-2.0, 4.0))
    pick = lambda frame, scalar: scalar if frame is None else torch.from_numpy(frame).to(dev).double()  # noqa: E731
    e = torch.poisson((sen.exposure * sen.nd * f * pick(sen.prnu_frame, 1.0)).float(), generator=g)
    noise = torch.randn(e.shape, device=dev, generator=g) * pick(sen.read_var_frame, torch.tensor(sen.read_var)).sqrt()
    dn = torch.round(sen.gain * e + noise + pick(sen.bias_frame, sen.black)).clamp(0, synth.CLIP_DN)
    raw = torch.zeros((sen.height, sen.pitch), device=dev, dtype=torch.int16)
    raw[:, : sen.width] = dn.to(torch.int16)
    return raw.view(torch.uint16)


def _inputs(c, seed):
    """(sensors, parameters, raw frames on the GPU) of one frame case."""
    sensors = _rig(c)
    scene = synth.make_scene(seed, c["w"], c["h"])
    return sensors, _params(c), [_render(scene, s, seed, k) for k, s in enumerate(sensors)]


def _frames(c):
    """The frame cases that a batch, or one frame of every served stream, is made of."""
    if c["kind"] == "batch":
        return [{**FRAME, "n": n, "w": w, "h": h, "ow": round(w * up), "oh": round(h * up), "order": order,
                 "paper_nd": False, "rig": c["spec"] + k}
                for _, k, n, w, h, order, up in synth.batching_specs(c["spec"], c["frames"], c["cap"])]
    got = []
    for k in range(c["streams"]):
        w, h, n, ow, oh = synth.SERVING_STREAMS[k if c["streams"] == 8 else (c["rig"] + 3 * k) % 8]
        sx, sy = min(1.0, c["cap"] / w), min(1.0, c["cap"] / h)
        got.append({**FRAME, "n": n, "w": int(w * sx) // 8 * 8, "h": int(h * sy) // 2 * 2, "ow": int(ow * sx) // 8 * 8,
                    "oh": int(oh * sy) // 2 * 2, "rig": c["rig"] + k})
    return got


def _stack(c, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    pitch = synth.pitch_for(c["w"])
    frames = torch.zeros((c["frames"], c["h"], pitch), device="cuda", dtype=torch.int16)
    mean = torch.full((c["h"], c["w"]), c["level"], device="cuda")
    for k in range(c["frames"]):
        e = torch.poisson(mean, generator=g)
        dn = synth.GAIN_DN_PER_E * e + synth.READ_SIGMA_DN * torch.randn(e.shape, device="cuda", generator=g)
        frames[k, :, : c["w"]] = torch.round(dn + synth.BLACK_DN).clamp(0, synth.CLIP_DN).to(torch.int16)
    return frames.view(torch.uint16)


def _pinned(t):
    return t.cpu().view(torch.int16).pin_memory().numpy().view(np.uint16)


# ------------------------------------------------------------------------------------------ the calls

def prepare(case, seed):
    kind = case["kind"]
    ctx = hdr.Context(0)
    if kind == "stats":
        return {"kind": kind, "ctx": ctx, "frames": _stack(case, seed), "w": case["w"]}
    if kind in ("batch", "serve"):
        parts, keep = [], []
        for k, c in enumerate(_frames(case)):
            sensors, p, raws = _inputs(c, seed * 64 + k)
            ctx.set_rig(k, sensors)
            hp = hdr.params_struct(p)
            if kind == "batch":
                out = torch.empty((3, p.out_h, p.out_w), device="cuda")
                parts.append((ctx.frame(k, hp, raws, out, None, keep), out))
                keep.append(raws)
            else:
                out = torch.empty((3, p.out_h, p.out_w)).pin_memory().numpy()
                parts.append((k, hp, [_pinned(r) for r in raws], out))
        state = {"kind": kind, "ctx": ctx, "parts": parts, "keep": keep}
        if kind == "serve":
            state["server"] = hdr.Server(ctx)
        return state
    sensors, p, raws = _inputs(case, seed)
    ctx.set_rig(0, sensors)
    out = torch.empty((3, p.out_h, p.out_w), device="cuda", dtype=torch.float16 if p.out_dtype else torch.float32)
    return {"kind": kind, "ctx": ctx, "params": hdr.params_struct(p), "raws": raws, "out": out,
            "calpa": hdr.hdr_calpa_params_default(),
            "grad": torch.empty((p.out_h, p.out_w, 2), device="cuda") if kind == "structure" else None,
            "metric": torch.empty((p.out_h, p.out_w, 3), device="cuda") if kind == "structure" else None}


def run(state):
    kind, ctx = state["kind"], state["ctx"]
    if kind == "frame":
        return ctx.reconstruct(0, state["params"], state["raws"], out=state["out"])
    if kind == "adaptive":
        return ctx.reconstruct_adaptive(0, state["params"], state["calpa"], state["raws"], out=state["out"])
    if kind == "structure":
        grad = ctx.calpa_gradients(0, state["params"], state["calpa"], state["raws"], grad=state["grad"])
        return [grad, ctx.calpa_metric(state["calpa"], grad, metric=state["metric"])]
    if kind == "batch":
        ctx.reconstruct_batch([f for f, _ in state["parts"]])
        return [out for _, out in state["parts"]]
    if kind == "serve":
        tickets = [state["server"].submit(rig, p, raws, out, stream_id=rig) for rig, p, raws, out in state["parts"]]
        for t in tickets:
            state["server"].poll(t)
        return [out for _, _, _, out in state["parts"]]
    return list(ctx.calib_stack_stats(state["frames"], state["w"]))


# ------------------------------------------------------------------------------------------ the work

FLOPS_PER_PAIR = (7, 37, 88)  # the sums of one sample at one scale, by order: value and variance


def _work_frame(c, extra_bytes=0, scales=None, order=None, channels=(1.0, 1.0, 1.0)):
    sig = scales or (synth.PAPER_SCALES if c["scales"] == 4 else (c["sigma"],))
    px = c["ow"] * c["oh"]
    # samples of one channel inside a window: its density (1/4, 1/2, 1/4) times the window's area (green: half of it)
    pairs = sum(0.25 * math.pi * (3.0 * s) ** 2 for s in sig) * c["n"] * sum(channels)
    raw = 2 * c["w"] * c["h"] * c["n"] * (8 if c["calibrated"] else 1)
    return {"bytes": raw + px * (extra_bytes or 3 * (2 if c["half"] else 4)),
            "flops": px * pairs * FLOPS_PER_PAIR[c["order"] if order is None else order]}


def work(case):
    kind = case["kind"]
    if kind == "stats":
        px = case["w"] * case["h"]
        return {"bytes": 2 * px * case["frames"] + 8 * px, "flops": 3 * px * case["frames"]}
    if kind in ("batch", "serve"):
        parts = [_work_frame(c) for c in _frames(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    px = case["ow"] * case["oh"]
    pass1 = _work_frame(case, extra_bytes=20, scales=(1.2,), order=1, channels=(0.0, 1.0, 0.0))
    pass2 = px * 29 * 6
    if kind == "structure":
        return {"bytes": pass1["bytes"], "flops": pass1["flops"] + pass2}
    w = _work_frame(case)
    if kind == "adaptive":  # the steered windows are larger where the image is flat: counted at the isotropic size
        return {"bytes": w["bytes"], "flops": w["flops"] + pass1["flops"] + pass2}
    return w


# ------------------------------------------------------------------------------------------ in 64 bits

MONO = [(t - b, b) for t in range(5) for b in range(t + 1)]  # exponents of the moments, by degree
UNKNOWNS = (1, 3, 6)


def _converted(sen, raw):
    """(radiance, inverse variance) of every sample in FP64; inverse variance 0 where saturated."""
    get = lambda frame, scalar: scalar if frame is None else torch.from_numpy(frame.astype(np.float64)).cuda()  # noqa: E731
    y = raw.view(torch.int16)[:, : sen.width].double()
    a, gtn = get(sen.prnu_frame, 1.0), sen.gain * sen.exposure * sen.nd
    e = y - get(sen.bias_frame, sen.black)
    f = e / (gtn * a)
    iv = gtn ** 2 * a ** 2 / (sen.gain * e.clamp(min=0.0) + get(sen.read_var_frame, sen.read_var))
    return f, torch.where(y < get(sen.sat_frame, float(sen.sat)), iv, torch.zeros_like(iv))


def _fit(a, b, count, kv, P, min_pivot):
    """The weighted fit of P unknowns from its moments a, b, kv [moment][...]: (C_0, variance, coefficients, usable)."""
    at = {e: i for i, e in enumerate(MONO)}
    A = [[a[at[MONO[i][0] + MONO[j][0], MONO[i][1] + MONO[j][1]]] for j in range(P)] for i in range(P)]
    L, D, ok = [[None] * P for _ in range(P)], [], count >= P
    for j in range(P):
        d = A[j][j].clone()
        for q in range(j):
            d -= L[j][q] ** 2 * D[q]
        ok = ok & (A[j][j] > 0) & (d / A[j][j].clamp(min=1e-300) > min_pivot)
        D.append(torch.where(d > 0, d, torch.ones_like(d)))
        for i in range(j + 1, P):
            t = A[i][j].clone()
            for q in range(j):
                t -= L[i][q] * L[j][q] * D[q]
            L[i][j] = t / D[j]

    def solve(rhs):
        x = []
        for i in range(P):
            x.append(rhs[i] - sum(L[i][q] * x[q] for q in range(i)))
        x = [x[i] / D[i] for i in range(P)]
        for i in reversed(range(P)):
            x[i] = x[i] - sum(L[q][i] * x[q] for q in range(i + 1, P))
        return x

    zero = torch.zeros_like(D[0])
    l = solve([zero + 1.0] + [zero] * (P - 1))
    var = None if kv is None else sum(
        l[i] * l[j] * kv[at[MONO[i][0] + MONO[j][0], MONO[i][1] + MONO[j][1]]] for i in range(P) for j in range(P))
    coef = solve([b[i] for i in range(P)])
    return coef[0], var, coef, ok


def _reference(sensors, p, raws, metric=None, reach=1.0, gradient_sigma=None):
    """The reconstruction [3, H, W] in FP64, or the green gradients [H, W, 2] at gradient_sigma."""
    order = p.order if gradient_sigma is None else 1
    sigmas = p.sigmas if gradient_sigma is None else (gradient_sigma,)
    NA, P, J = len([e for e in MONO if sum(e) <= 2 * order]), UNKNOWNS[order], len(sigmas)
    taper = math.exp(-0.5 * p.trunc_k ** 2)
    samples = [_converted(s, r) for s, r in zip(sensors, raws)]
    out = torch.zeros((p.out_h, p.out_w, 2) if gradient_sigma else (3, p.out_h, p.out_w), device="cuda", dtype=torch.float64)
    rows = max(1, (1 << 19) // p.out_w)
    oa = p.out_affine
    for v0 in range(0, p.out_h, rows):
        v1 = min(p.out_h, v0 + rows)
        v, u = torch.meshgrid(torch.arange(v0, v1, device="cuda").double(), torch.arange(p.out_w, device="cuda").double(),
                              indexing="ij")
        u, v = u.reshape(-1), v.reshape(-1)
        X, Y = oa[0, 0] * u + oa[0, 1] * v + oa[0, 2], oa[1, 0] * u + oa[1, 1] * v + oa[1, 2]
        C = None if metric is None else metric[v0:v1].reshape(-1, 3)
        for c in ((1,) if gradient_sigma else (0, 1, 2)):
            sg = torch.tensor([s * (p.green_ratio if c == 1 else 1.0) for s in sigmas], device="cuda", dtype=torch.float64)[:, None]
            new = lambda *n: torch.zeros((*n, u.numel()), device="cuda", dtype=torch.float64)  # noqa: E731
            a, b, kv, count = new(J, NA), new(J, P), new(J, NA), new(J)
            R = p.trunc_k * float(sg[-1])
            for sen, (f, iv) in zip(sensors, samples):
                T = sen.affine
                inv = np.linalg.inv(T[:, :2])
                qx, qy = (float(inv[i, 0]) * (X - T[0, 2]) + float(inv[i, 1]) * (Y - T[1, 2]) for i in (0, 1))
                hx, hy = (reach * R * math.hypot(*inv[i]) for i in (0, 1))
                for ox, oy in {0: [(0, 0)], 1: [(1, 0), (0, 1)], 2: [(1, 1)]}[c]:
                    bx, by = ((qx - ox) / 2).floor().long(), ((qy - oy) / 2).floor().long()
                    for j in range(-math.ceil(hy / 2), math.ceil(hy / 2) + 2):
                        for i in range(-math.ceil(hx / 2), math.ceil(hx / 2) + 2):
                            x, y = ox + 2 * (bx + i), oy + 2 * (by + j)
                            inside = (x >= 0) & (x < sen.width) & (y >= 0) & (y < sen.height)
                            at = y.clamp(0, sen.height - 1) * sen.width + x.clamp(0, sen.width - 1)
                            dx = T[0, 0] * x + T[0, 1] * y + T[0, 2] - X
                            dy = T[1, 0] * x + T[1, 1] * y + T[1, 2] - Y
                            r2 = dx * dx + dy * dy
                            if C is not None:
                                r2 = C[:, 0] * dx * dx + 2 * C[:, 1] * dx * dy + C[:, 2] * dy * dy
                            w = iv.reshape(-1)[at] * inside
                            hold = (r2 < (p.trunc_k * sg) ** 2) & (w > 0)
                            K = (torch.exp(-r2 / (2 * sg * sg)) - taper) * hold
                            px, py = [torch.ones_like(dx), dx], [torch.ones_like(dy), dy]
                            for _ in range(2 * order - 1):
                                px.append(px[-1] * dx)
                                py.append(py[-1] * dy)
                            m = torch.stack([px[s] * py[t] for s, t in MONO[:NA]])
                            K = K[:, None, :]
                            a.addcmul_(K * w, m)
                            b.addcmul_(K * (w * f.reshape(-1)[at]), m[:P])
                            if J > 1:
                                kv.addcmul_(K * K * w, m)
                            count += hold
            fits = [_fit(a[j], b[j], count[j], kv[j], P, p.min_pivot) for j in range(J)]
            if gradient_sigma:
                _, _, coef, ok = fits[0]
                out[v0:v1] = (torch.stack(coef[1:3], 1) * ok[:, None]).reshape(v1 - v0, p.out_w, 2)
                continue
            val, done = torch.full_like(u, math.nan), torch.zeros_like(u, dtype=torch.bool)
            lo, hi = torch.full_like(u, -math.inf), torch.full_like(u, math.inf)
            for c0, var, _, ok in fits:  # the last scale whose running intersection is not empty
                half = p.ici_gamma * var.clamp(min=0.0).sqrt()
                nlo, nhi = torch.maximum(lo, c0 - half), torch.minimum(hi, c0 + half)
                take = ok & ~done & ~(nlo > nhi)
                done = done | (ok & (nlo > nhi))
                lo, hi, val = torch.where(take, nlo, lo), torch.where(take, nhi, hi), torch.where(take, c0, val)
            for lower in range(order - 1, -1, -1):  # no usable scale: a lower order at the largest one
                c0, _, _, ok = _fit(a[-1], b[-1], count[-1], None, UNKNOWNS[lower], p.min_pivot)
                val = torch.where(val.isnan() & ok, c0, val)
            out[c, v0:v1] = val.reshape(v1 - v0, p.out_w)
    return out


def _reference_metric(grad, k):
    """Steering matrices [H, W, 3] of gradients [H, W, 2] in FP64 with the default adaptive parameters k."""
    H, W = grad.shape[:2]
    g = grad * k.grad_scale
    prod = torch.stack([g[..., 0] * g[..., 0], g[..., 0] * g[..., 1], g[..., 1] * g[..., 1], torch.ones_like(g[..., 0])])
    r = int(math.floor(3.0 * k.window_sigma))
    T = torch.zeros_like(prod)
    for dj in range(-r, r + 1):
        for di in range(-r, r + 1):
            if di * di + dj * dj > (3.0 * k.window_sigma) ** 2:
                continue
            w = math.exp(-(di * di + dj * dj) / (2.0 * k.window_sigma ** 2))
            y0, y1, x0, x1 = max(0, -dj), min(H, H - dj), max(0, -di), min(W, W - di)
            cut = prod[:, y0 + dj:y1 + dj, x0 + di:x1 + di]
            T[:3, y0:y1, x0:x1] += w * cut[:3]
            T[3, y0:y1, x0:x1] += 1.0
    a, b, c, M = T
    h, d = 0.5 * (a + c), torch.sqrt((0.5 * (a - c)) ** 2 + b * b)
    l1, l2 = h + d, (h - d).clamp(min=0.0)
    first = (b * b + (l1 - a) ** 2) >= ((l1 - c) ** 2 + b * b)
    ux, uy = torch.where(first, b, l1 - c), torch.where(first, l1 - a, b)
    n = torch.sqrt(ux * ux + uy * uy)
    ux, uy = torch.where(n > 0, ux / n, torch.ones_like(n)), torch.where(n > 0, uy / n, torch.zeros_like(n))
    s1, s2 = l1.sqrt(), l2.sqrt()
    e = (s1 + k.lambda1) / (s2 + k.lambda1)
    gamma = ((s1 * s2 + k.lambda2) / M) ** k.alpha
    ea, eb = (gamma * e).clamp(k.min_eig, k.max_eig), (gamma / e).clamp(k.min_eig, k.max_eig)
    return torch.stack([ea * ux * ux + eb * uy * uy, (ea - eb) * ux * uy, ea * uy * uy + eb * ux * ux], 2)


def exact(case, seed):
    kind = case["kind"]
    if kind == "stats":
        y = _stack(case, seed).view(torch.int16)[:, :, : case["w"]]
        n = y.shape[0]
        s1, s2 = torch.zeros(y.shape[1:], device="cuda", dtype=torch.int64), torch.zeros(y.shape[1:], device="cuda", dtype=torch.int64)
        for f in y:
            s1 += f.long()
            s2 += f.long() ** 2
        return [s1.double() / n, (n * s2 - s1 * s1).double() / (n * (n - 1.0))]
    if kind in ("batch", "serve"):
        return [_reference(*_inputs(c, seed * 64 + k)) for k, c in enumerate(_frames(case))]
    sensors, p, raws = _inputs(case, seed)
    if kind == "frame":
        return _reference(sensors, p, raws)
    k = hdr.hdr_calpa_params_default()
    grad = _reference(sensors, p, raws, gradient_sigma=k.grad_sigma)
    metric = _reference_metric(grad, k)
    if kind == "structure":
        return [grad, metric]
    return _reference(sensors, p, raws, metric=metric, reach=1.0 / math.sqrt(k.min_eig))
