"""The calls a user of this library makes, as cases that can be timed and checked.

Each case is one pass through the public entry points of ``paper_1904_06017_gb300``: the
per-frame pipeline (row-shift warp, cost / aggregation / WTA, disparity transformation) at
several frame sizes and storage types, the LR check, a batch of uneven pairs, the FP32 volumes
in device memory, the self-estimated warp, the differentiable disparity without and with its
backward pass, and the roll-angle energy and refinement.

Inputs are synthetic road pairs drawn on the GPU from the seed: a blurred-noise texture, a road
disparity quadratic in the rotated row coordinate with elliptical potholes, a target rendered
from it with noise, and the row-shift table that follows the road's centre line.  ``exact``
states the same equations in 64-bit PyTorch operations.
"""
import math

import torch
import torch.nn.functional as F

import paper_1904_06017_gb300 as sg
from paper_1904_06017_gb300 import diff as sgd

DTYPES = {"f32": sg.STEREO_F32, "f16": sg.STEREO_F16, "bf16": sg.STEREO_BF16}


def _frame(name, width, height, disp, win, bil, sigma0, sigma1, dtype, warp=True):
    return dict(name=name, kind="frame", width=width, height=height, disp=disp, win=win, bil=bil,
                sigma0=sigma0, sigma1=sigma1, dtype=dtype, warp=warp)


def _soft(name, kind, batch, width, height, disp, win, bil, linear):
    return dict(name=name, kind=kind, batch=batch, width=width, height=height, disp=disp, win=win, bil=bil,
                sigma0=3.0, sigma1=10.0, temperature=0.1, linear=linear)


def listed():
    return [
        # A small camera frame without a warp model: the smallest pipeline call, where the seven
        # launches and their latencies count.
        _frame("frame_320x240", 320, 240, 64, 7, 9, 3.0, 10.0, "f32", warp=False),
        # The paper's own throughput example (695 x 361, d_max = 30) with the paper's filter: odd
        # sizes and a search range off every chunk size.
        _frame("frame_695x361", 695, 361, 30, 9, 11, 1.5, 5.5, "f32"),
        # A full-HD frame at the benchmark's settings: the ordinary production call.
        _frame("frame_1080p", 1920, 1080, 128, 9, 11, 3.0, 10.0, "f32"),
        # Full HD with the widest windows and range, costs stored in 16 bits: the precision
        # workload's reduced-precision form.
        _frame("frame_1080p_f16", 1920, 1080, 192, 9, 13, 3.0, 10.0, "f16"),
        # Reference view, target view and consistency mask of a 1024 x 768 road frame.
        dict(name="lr_1024x768", kind="lr", width=1024, height=768, disp=32, win=9, bil=11, sigma0=3.0,
             sigma1=10.0),
        # Frames of several cameras in one launch: sizes and ranges cycle through the batch
        # workload's (640 x 480 ... 1920 x 1080, D = 32, 64, 128).
        dict(name="batch_12_pairs", kind="batch", pairs=12, scale=1.0, win=9, bil=11, sigma0=3.0, sigma1=10.0),
        # The stage-per-call form: a program that wants the cost volume and the aggregated volume
        # in device memory (its own post-processing between the stages).
        dict(name="volumes_640x360", kind="volumes", width=640, height=360, disp=32, win=9, bil=11, sigma0=1.5,
             sigma1=5.5),
        # The warp model estimated from the pair itself, as on the first frame of a sequence.
        dict(name="warp_est_1024x768", kind="warp_est", width=1024, height=768, disp=128, factor=4),
        # Sub-pixel disparity of one frame by soft-argmin, without gradients (inference).
        _soft("soft_1280x720", "soft", 1, 1280, 720, 64, 9, 11, False),
        # Forward and backward over image crops with the interpolating warp, the shift table's
        # gradient included: the small training / calibration step.
        _soft("grad_96x64_linear", "grad", 1, 96, 64, 32, 9, 11, True),
        # Forward and backward of a training batch: the differentiation workload.
        _soft("grad_8x960x540", "grad", 8, 960, 540, 64, 9, 11, False),
        # Energy of the road model with its gradients and 50 roll refinement steps, on a batch of
        # disparity maps.
        dict(name="roll_8x960x540", kind="roll", batch=8, width=960, height=540, steps=50, masked=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "lr", "batch", "volumes", "warp_est", "soft", "grad", "grad", "roll"])
    win, bil = rng.choice([5, 7, 9, 9, 11]), rng.choice([7, 9, 11, 11, 13])
    if kind == "frame":
        w = _log(rng, 160, 1920)
        h = max(100, int(w * rng.uniform(0.45, 0.8)))
        h = min(h, 1080)
        d = max(16, min(_log(rng, 16, 192), w // 4))
        s0, s1 = rng.choice([(3.0, 10.0), (1.5, 5.5)])
        c = _frame("", w, h, d, win, bil, s0, s1, rng.choice(["f32", "f32", "f16", "bf16"]))
    elif kind == "lr":
        w = _log(rng, 320, 1280)
        c = dict(kind=kind, width=w, height=max(100, int(w * rng.uniform(0.45, 0.8))), disp=min(_log(rng, 16, 96), w // 4),
                 win=win, bil=bil, sigma0=3.0, sigma1=10.0)
    elif kind == "batch":
        c = dict(kind=kind, pairs=rng.randint(2, 12), scale=round(rng.uniform(0.4, 1.0), 3), win=win, bil=bil, sigma0=3.0,
                 sigma1=10.0)
    elif kind == "volumes":
        w = _log(rng, 160, 1024)
        c = dict(kind=kind, width=w, height=max(100, int(w * rng.uniform(0.45, 0.7))), disp=min(_log(rng, 16, 64), w // 4),
                 win=win, bil=bil, sigma0=1.5, sigma1=5.5)
    elif kind == "warp_est":
        w = _log(rng, 480, 1920)
        c = dict(kind=kind, width=w, height=int(w * rng.uniform(0.5, 0.75)), disp=min(_log(rng, 64, 192), w // 4),
                 factor=rng.choice([2, 4]))
    elif kind in ("soft", "grad"):
        lo, hi = (160, 1280) if kind == "soft" else (64, 960)
        w = _log(rng, lo, hi)
        h = max(48, int(w * rng.uniform(0.45, 0.7)))
        d = max(16, min(_log(rng, 16, 128), w // 3))
        b = max(1, min(rng.randint(1, 8), 8 * 960 * 540 * 64 // (w * h * d)))
        c = _soft("", kind, b, w, h, d, win, bil, rng.random() < 0.4)
    else:
        w = _log(rng, 160, 960)
        c = dict(kind=kind, batch=rng.randint(1, 8), width=w, height=max(90, int(w * rng.uniform(0.45, 0.7))),
                 steps=rng.randint(10, 50), masked=rng.random() < 0.5)
    c.pop("name", None)
    return c


# ------------------------------------------------------------------------------------ inputs

def _scene(width, height, disp, seed, warp=True):
    """One road pair on the GPU: (ref, tgt) uint8 [H][W], row shifts float32 [H], roll."""
    g = torch.Generator(device="cuda").manual_seed(1904060170 + seed)
    host = torch.Generator().manual_seed(1904060170 + seed)
    dev = torch.device("cuda")
    t = torch.arange(-4, 5, device=dev, dtype=torch.float32)
    k = torch.exp(-0.5 * t * t)
    k = k / k.sum()
    x = torch.randn(1, 1, height + 8, width + 8, generator=g, device=dev)
    x = F.conv2d(F.conv2d(x, k.view(1, 1, 9, 1)), k.view(1, 1, 1, 9))[0, 0]
    ref = (128.0 + 40.0 * (x - x.mean()) / x.std()).round().clamp(0.0, 255.0)

    r = torch.rand(32, generator=host, dtype=torch.float64).tolist()
    roll = math.radians(6.0 * (2.0 * r[0] - 1.0))
    depth = max(1.0, min(3.0 + 5.0 * r[1], 0.12 * disp))
    # the road's slope, bounded so that the disparities searched (after the warp, or all of them
    # where there is none) stay inside the range
    span = 0.5 * width * abs(math.sin(roll)) + 1.0
    if warp:
        a0, a1 = 5.0, min(0.12, 0.3 * disp / span)
    else:
        a0, a1 = 5.0, min(0.12, (0.75 * disp - 6.0) / (height + span))
    a2 = 1e-4 * a1 / 0.12
    uc = 0.5 * (width - 1)
    holes = []
    for i in range(4):
        q = r[2 + 5 * i:7 + 5 * i]
        holes.append(((0.15 + 0.7 * q[0]) * width, (0.35 + 0.5 * q[1]) * height, (0.04 + 0.06 * q[2]) * width,
                      (0.03 + 0.05 * q[3]) * height, (0.4 + 0.6 * q[4]) * depth))
    v = torch.arange(height, device=dev, dtype=torch.float64)[:, None]
    u = torch.arange(width, device=dev, dtype=torch.float64)[None, :]

    def road(uu):
        y = v * math.cos(roll) - (uu - uc) * math.sin(roll)
        return a0 + a1 * y + a2 * y * y

    def disparity(uu):
        d = road(uu)
        for pu, pv, ra, rb, dep in holes:
            d = d - dep * (1.0 - ((uu - pu) / ra) ** 2 - ((v - pv) / rb) ** 2).clamp(min=0.0)
        return d

    uu = u + disparity(u)
    for _ in range(4):
        uu = u + disparity(uu)
    uu = uu.clamp(0.0, width - 1.0)
    u0 = uu.floor().long()
    f = uu - u0
    refd = ref.double()
    smp = (1.0 - f) * refd.gather(1, u0) + f * refd.gather(1, (u0 + 1).clamp(max=width - 1))
    smp = smp + 2.0 * torch.randn(height, width, generator=g, device=dev)
    tgt = smp.round().clamp(0.0, 255.0)
    if warp:
        centre = road(torch.full((1, 1), uc, device=dev, dtype=torch.float64))[:, 0]
        below = span * (a1 + 2.0 * a2 * height) + depth
        shift = (centre - (math.ceil(below) + 2.0)).float()
    else:
        shift = torch.zeros(height, device=dev)
    return ref.to(torch.uint8), tgt.to(torch.uint8), shift.contiguous(), roll


def _image(a):
    """The image with its rows padded to a multiple of 16 bytes."""
    h, w = a.shape
    out = torch.zeros(h, (w + 15) // 16 * 16, dtype=torch.uint8, device="cuda")
    out[:, :w] = a
    return out


def _maps(h, w):
    return dict(disp=torch.empty(h, w, device="cuda"), wta=torch.empty(h, w, dtype=torch.int32, device="cuda"),
                valid=torch.empty(h, w, dtype=torch.uint8, device="cuda"))


def _batch_pairs(case):
    sizes, ranges = ((640, 480), (960, 540), (1280, 720), (1920, 1080)), (32, 64, 128)
    return [(int(sizes[i % 4][0] * case["scale"]), int(sizes[i % 4][1] * case["scale"]), ranges[(i + i // 4) % 3])
            for i in range(case["pairs"])]


def _float_scenes(case, seed):
    """Batched float images [B, H, W] and shifts [B, H] of the differentiable path."""
    s = [_scene(case["width"], case["height"], case["disp"], 1000 * seed + b) for b in range(case["batch"])]
    return (torch.stack([x[0] for x in s]).float(), torch.stack([x[1] for x in s]).float(),
            torch.stack([x[2] for x in s]))


def _roll_inputs(case, seed):
    """Noisy rolled-road disparity maps, the model's angle and line near them, a mask, and dS/dE."""
    g = torch.Generator(device="cuda").manual_seed(77 + seed)
    b, h, w = case["batch"], case["height"], case["width"]
    psi = 0.2 * (torch.rand(b, generator=g, device="cuda", dtype=torch.float64) - 0.5)
    a1 = 0.06 + 0.06 * torch.rand(b, generator=g, device="cuda", dtype=torch.float64)
    v = torch.arange(h, device="cuda", dtype=torch.float64)[None, :, None]
    u = torch.arange(w, device="cuda", dtype=torch.float64)[None, None, :]
    y = v * torch.cos(psi)[:, None, None] - u * torch.sin(psi)[:, None, None]
    noise = torch.randn(b, h, w, generator=g, device="cuda", dtype=torch.float64)
    disp = (5.0 + a1[:, None, None] * y + 0.3 * noise).float()
    theta = torch.stack([psi + 0.01, torch.full_like(psi, 4.9), 1.02 * a1], 1)
    mask = (torch.rand(b, h, w, generator=g, device="cuda") > 0.15).to(torch.uint8) if case["masked"] else None
    gain = 0.5 + torch.rand(b, generator=g, device="cuda", dtype=torch.float64)
    return disp, theta, mask, gain


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind in ("frame", "lr", "volumes"):
        w, h, d = case["width"], case["height"], case["disp"]
        ref, tgt, shift, _ = _scene(w, h, d, 1000 * seed, case.get("warp", True))
        s.update(ref=_image(ref), tgt=_image(tgt), shift=shift, **_maps(h, w))
        s["tw"] = torch.zeros_like(s["tgt"])
        s["stereo"] = sg.Stereo(w, h, d, win=case["win"], bil=case["bil"], sigma0=case["sigma0"], sigma1=case["sigma1"],
                                cost_dtype=DTYPES[case.get("dtype", "f32")])
        if kind == "frame":
            s["out"] = torch.empty_like(s["disp"])
            s["res"] = torch.zeros(48, dtype=torch.uint8, device="cuda")
        elif kind == "lr":
            s["ok"] = torch.empty_like(s["valid"])
            s["wta_tgt"] = torch.empty_like(s["wta"])
        else:
            s["cost"] = torch.empty(h, w, d, device="cuda")
            s["agg"] = torch.empty_like(s["cost"])
            s["best2"] = torch.empty(h, w, 2, device="cuda")
    elif kind == "batch":
        s["pairs"] = []
        for i, (w, h, d) in enumerate(_batch_pairs(case)):
            ref, tgt, shift, _ = _scene(w, h, d, 1000 * seed + i)
            p = dict(ref=_image(ref), tgt=_image(tgt), shift=shift, max_disp=d, **_maps(h, w))
            p["tgt_warped"] = torch.zeros_like(p["tgt"])
            p["disp_out"] = torch.empty_like(p["disp"])
            p["res"] = torch.zeros(48, dtype=torch.uint8, device="cuda")
            s["pairs"].append(p)
        s["batch"] = sg.StereoBatch(s["pairs"], win=case["win"], bil=case["bil"], sigma0=case["sigma0"],
                                    sigma1=case["sigma1"])
    elif kind == "warp_est":
        ref, tgt, _, _ = _scene(case["width"], case["height"], case["disp"], 1000 * seed, False)
        s.update(ref=_image(ref), tgt=_image(tgt), coef=torch.empty(3, dtype=torch.float64, device="cuda"),
                 shift=torch.empty(case["height"], device="cuda"))
        s["est"] = sg.WarpEstimator(case["width"], case["height"], case["disp"], factor=case["factor"])
    elif kind in ("soft", "grad"):
        s["ref"], s["tgt"], s["shift"] = _float_scenes(case, seed)
        if kind == "grad":
            for k in ("ref", "tgt") + (("shift",) if case["linear"] else ()):
                s[k].requires_grad_()
            g = torch.Generator(device="cuda").manual_seed(5 + seed)
            s["upstream"] = torch.randn(s["ref"].shape, generator=g, device="cuda")   # dS/dl of the loss behind it
    else:
        s["disp"], s["theta"], s["mask"], s["gain"] = _roll_inputs(case, seed)
        s["disp"].requires_grad_()
        s["theta"].requires_grad_()
    return s


# -------------------------------------------------------------------------------------- calls

def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "frame":
        st = s["stereo"]
        if case["warp"]:
            st.warp_target(s["tgt"], s["shift"], s["tw"])
        tw = s["tw"] if case["warp"] else s["tgt"]
        st.cost_aggregate_wta(s["ref"], tw, s["shift"], s["disp"], s["wta"], s["valid"])
        st.disparity_transform(s["disp"], s["valid"], 0.0, 0.0, s["out"], res=s["res"])
        return dict(disp=s["disp"], wta=s["wta"], valid=s["valid"], out=s["out"], fit=s["res"][:32].view(torch.float64),
                    counts=s["res"][32:].view(torch.int32))
    if kind == "lr":
        st = s["stereo"]
        st.warp_target(s["tgt"], s["shift"], s["tw"])
        st.cost_aggregate_wta(s["ref"], s["tw"], s["shift"], s["disp"], s["wta"], s["valid"])
        st.lr_check(s["ref"], s["tw"], s["shift"], s["wta"], s["ok"], s["wta_tgt"])
        return dict(disp=s["disp"], wta=s["wta"], valid=s["valid"], ok=s["ok"], wta_tgt=s["wta_tgt"])
    if kind == "volumes":
        st = s["stereo"]
        st.warp_target(s["tgt"], s["shift"], s["tw"])
        st.cost_volume(s["ref"], s["tw"], s["cost"])
        st.aggregate_volume(s["ref"], s["cost"], s["agg"])
        st.wta_volume(s["agg"], s["shift"], s["disp"], s["wta"], s["best2"])
        return dict(cost=s["cost"], agg=s["agg"], disp=s["disp"], wta=s["wta"], best2=s["best2"])
    if kind == "batch":
        s["batch"].run()
        return [dict(disp=p["disp"], wta=p["wta"], valid=p["valid"], out=p["disp_out"]) for p in s["pairs"]]
    if kind == "warp_est":
        s["est"].run(s["ref"], s["tgt"], s["coef"], s["shift"], 4.0)
        return dict(coef=s["coef"], shift=s["shift"])
    if kind in ("soft", "grad"):
        mode = sgd.STEREO_WARP_LINEAR if case["linear"] else sgd.STEREO_WARP_ROUND
        a = (s["ref"], s["tgt"], s["shift"], case["disp"], case["win"], case["bil"], case["sigma0"], case["sigma1"],
             case["temperature"], mode)
        if kind == "soft":
            with torch.no_grad():
                return dict(disp=sgd.soft_argmin_disparity(*a))
        disp = sgd.soft_argmin_disparity(*a)
        wanted = [s["ref"], s["tgt"]] + ([s["shift"]] if case["linear"] else [])
        grads = torch.autograd.grad(disp, wanted, s["upstream"])
        return dict(disp=disp.detach(), grads=list(grads))
    energy = sgd.dt_energy(s["disp"], s["theta"], s["mask"])
    gd, gt = torch.autograd.grad(energy, [s["disp"], s["theta"]], s["gain"])
    traj = sgd.refine_roll(s["disp"].detach(), s["mask"], 0.0, case["steps"])
    return dict(energy=energy.detach(), grad_disp=gd, grad_theta=gt, trajectory=traj)


# ------------------------------------------------------------------------- what a pass needs

def work(case):
    """Each input read once, each output written once; and the arithmetic of the equations:
    11 per pixel and disparity for the cost from window sums, 2 k^2 for the aggregation (the
    weights 2 k^2 per pixel), and as much again for each adjoint."""
    kind = case["kind"]
    if kind == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for w, h, d in _batch_pairs(case):
            one = work(dict(case, kind="frame", width=w, height=h, disp=d, warp=True))
            total = {k: total[k] + one[k] for k in total}
        return total
    w, h = case["width"], case["height"]
    px = w * h
    if kind == "roll":
        n = case["batch"] * px
        return {"bytes": n * (4 + 4 + (1 if case["masked"] else 0)), "flops": n * (8.0 + 14.0 + 20.0)}
    if kind == "warp_est":
        f = case["factor"]
        wc, hc, dc = w // f, h // f, -(-case["disp"] // f)
        return {"bytes": 2 * px + 4 * h, "flops": 2.0 * px + wc * hc * (dc * (2 * 49 + 12) + 2 * 49)}
    d, k2 = case["disp"], case["bil"] ** 2
    view = px * (d * (2 * k2 + 12) + 2 * k2)
    if kind == "frame":
        return {"bytes": px * (2 + (1 if case["warp"] else 0) + 4 + 4 + 1 + 4) + 4 * h, "flops": view}
    if kind == "lr":
        return {"bytes": px * (2 + 1 + 4 + 4 + 1 + 1 + 4) + 4 * h, "flops": 2 * view}
    if kind == "volumes":
        return {"bytes": px * (2 + 1 + 8 * d + 4 + 4 + 8) + 4 * h, "flops": view}
    b = case["batch"]
    if kind == "soft":
        return {"bytes": 12 * b * px, "flops": b * view}
    return {"bytes": 24 * b * px, "flops": b * (view + px * d * (4 * k2 + 40))}


# ------------------------------------------------------------- the same equations in 64 bits

def _box(x, w):
    """Sums over w consecutive entries of the last two dimensions."""
    n = x.shape[-1] - w + 1
    x = sum(x[..., i:i + n] for i in range(w))
    n = x.shape[-2] - w + 1
    return sum(x[..., i:i + n, :] for i in range(w))


def _edge(x, left, right, top, bottom):
    return F.pad(x[None, None], (left, right, top, bottom), mode="replicate")[0, 0]


def _flat(x, w):
    hi, lo = F.max_pool2d(x[None, None], w, 1)[0, 0], F.max_pool2d(-x[None, None], w, 1)[0, 0]
    return hi == -lo


def _costs(ref, tgt, disp, win):
    """1 - NCC, [D][H][W]: population statistics, clamp-to-edge reads, 1 where a block is flat."""
    r, n = win // 2, float(win * win)
    a = _edge(ref - 128.0, r, r, r, r)
    b = _edge(tgt - 128.0, r + disp - 1, r, r, r)
    wa = a.shape[1]
    sa, sb = _box(a, win), _box(b, win)
    va, vb = n * _box(a * a, win) - sa * sa, n * _box(b * b, win) - sb * sb
    fa, fb = _flat(a.detach(), win), _flat(b.detach(), win)
    va = torch.where(fa, torch.ones_like(va), va)
    vb = torch.where(fb, torch.ones_like(vb), vb)
    w = ref.shape[1]

    def at(x, d, n):   # the columns d to the left
        return x[:, disp - 1 - d:disp - 1 - d + n]

    s = _box(torch.stack([a * at(b, d, wa) for d in range(disp)]), win)
    sbd = torch.stack([at(sb, d, w) for d in range(disp)])
    vbd = torch.stack([at(vb, d, w) for d in range(disp)])
    flat = fa[None] | torch.stack([at(fb, d, w) for d in range(disp)])
    c = 1.0 - (n * s - sa[None] * sbd) / torch.sqrt(va[None] * vbd)
    return torch.where(flat, torch.ones_like(c), c)


def _aggregate(ref, cost, bil, sigma0, sigma1):
    """Bilateral aggregation guided by ref, neighbours outside the image left out."""
    r = bil // 2
    h, w = ref.shape
    guide = F.pad(ref, (r, r, r, r))
    inside = F.pad(torch.ones_like(ref), (r, r, r, r))
    wide = F.pad(cost, (r, r, r, r))
    total, z = torch.zeros_like(cost), torch.zeros_like(ref)
    for dy in range(bil):
        for dx in range(bil):
            di = guide[dy:dy + h, dx:dx + w] - ref
            k = torch.exp(-((dx - r) ** 2 + (dy - r) ** 2) / sigma0 ** 2 - di * di / sigma1 ** 2)
            k = k * inside[dy:dy + h, dx:dx + w]
            z = z + k
            total = total + k * wide[:, dy:dy + h, dx:dx + w]
    return total / z


def _rounded(shift):
    return torch.floor(shift.double() + 0.5)


def _warped(tgt, shift):
    h, w = tgt.shape
    x = torch.arange(w, device=tgt.device)[None, :] - _rounded(shift).long()[:, None]
    return tgt.gather(1, x.clamp(0, w - 1))


def _wta(e, shift):
    """Lowest minimum, parabola step, the shift added back: (d*, disparity, best, second)."""
    n = e.shape[0]
    idx = torch.arange(n, device=e.device)[:, None, None]
    best = e.amin(0)
    win = torch.where(e == best, idx, n).amin(0)
    other = torch.where(idx == win, math.inf, e).amin(0)
    m1 = e.gather(0, (win - 1).clamp(min=0)[None])[0]
    p1 = e.gather(0, (win + 1).clamp(max=n - 1)[None])[0]
    den = 2.0 * m1 + 2.0 * p1 - 4.0 * best
    step = torch.where((win > 0) & (win < n - 1) & (den > 0), (m1 - p1) / den, torch.zeros_like(den))
    return win, win + step + _rounded(shift)[:, None], best, other


def _valid(w, h, disp, m, shift):
    s = _rounded(shift)
    ok = torch.zeros(h, w, dtype=torch.bool, device=shift.device)
    if h < 2 * m + 1:
        return ok
    win = s.unfold(0, 2 * m + 1, 1)
    lo, hi = win.amin(1).clamp(max=0.0), win.amax(1).clamp(min=0.0)
    u = torch.arange(w, device=shift.device, dtype=torch.float64)[None, :]
    ok[m:h - m] = (u >= (m + disp - 1 + hi)[:, None]) & (u <= (w - 1 - m + lo)[:, None])
    return ok


def _plane(disp, ok):
    """The least-squares road of a map: (psi, alpha0, alpha1, energy)."""
    h, w = disp.shape
    v, u = torch.nonzero(ok, as_tuple=True)
    d = disp[v, u]
    uc, vc = 0.5 * (w - 1), 0.5 * (h - 1)
    m = torch.stack([torch.ones_like(d), u - uc, v - vc], 1)
    a, b, c = torch.linalg.solve(m.T @ m, m.T @ d).tolist()
    e = float((d - m @ torch.tensor([a, b, c], dtype=torch.float64, device=d.device)).square().sum())
    psi = math.atan2(-b, c) if c >= 0 else math.atan2(b, -c)
    return psi, a - b * uc - c * vc, c / math.cos(psi), e


def _transformed(disp, psi, a0, a1):
    h, w = disp.shape
    v = torch.arange(h, device=disp.device, dtype=torch.float64)[:, None]
    u = torch.arange(w, device=disp.device, dtype=torch.float64)[None, :]
    return disp - a0 + a1 * (u * math.sin(psi) - v * math.cos(psi))


def _frame_exact(ref, tgt, shift, disp, case):
    """(disparity, transformed disparity, fit) of one frame."""
    tw = _warped(tgt.double(), shift)
    e = _aggregate(ref.double(), _costs(ref.double(), tw, disp, case["win"]), case["bil"], case["sigma0"], case["sigma1"])
    l = _wta(e, shift)[1]
    del e
    h, w = ref.shape
    ok = _valid(w, h, disp, case["win"] // 2 + case["bil"] // 2, shift)
    if int(ok.sum()) < 3:
        return l, None, None
    psi, a0, a1, en = _plane(l, ok)
    return l, _transformed(l, psi, a0, a1), torch.tensor([psi, a0, a1, en], dtype=torch.float64)


def _soft_exact(ref, tgt, shift, case):
    """Soft-argmin disparity of one pair, differentiable in all three inputs."""
    h, w = ref.shape
    if case["linear"]:
        col = torch.arange(w, device=ref.device)[None, :]
        k = torch.floor(-shift.detach())
        f = -shift - k
        x = (col + k.long()[:, None])
        t0, t1 = tgt.gather(1, x.clamp(0, w - 1)), tgt.gather(1, (x + 1).clamp(0, w - 1))
        tw, back = t0 + f[:, None] * (t1 - t0), shift
    else:
        tw, back = _warped(tgt, shift), _rounded(shift.detach())
    e = _aggregate(ref, _costs(ref, tw, case["disp"], case["win"]), case["bil"], case["sigma0"], case["sigma1"])
    p = torch.softmax(-e / case["temperature"], 0)
    d = torch.arange(case["disp"], device=ref.device, dtype=torch.float64)[:, None, None]
    return (p * d).sum(0) + back[:, None]


def exact(case, seed):
    kind = case["kind"]
    if kind == "frame":
        ref, tgt, shift, _ = _scene(case["width"], case["height"], case["disp"], 1000 * seed, case["warp"])
        l, out, fit = _frame_exact(ref, tgt, shift, case["disp"], case)
        return dict(disp=l, wta=None, valid=None, out=out, fit=fit, counts=None)
    if kind == "lr":
        ref, tgt, shift, _ = _scene(case["width"], case["height"], case["disp"], 1000 * seed)
        l, _, _ = _frame_exact(ref, tgt, shift, case["disp"], case)
        return dict(disp=l, wta=None, valid=None, ok=None, wta_tgt=None)
    if kind == "volumes":
        ref, tgt, shift, _ = _scene(case["width"], case["height"], case["disp"], 1000 * seed)
        tw = _warped(tgt.double(), shift)
        c = _costs(ref.double(), tw, case["disp"], case["win"])
        e = _aggregate(ref.double(), c, case["bil"], case["sigma0"], case["sigma1"])
        _, l, best, other = _wta(e, shift)
        return dict(cost=c.permute(1, 2, 0).contiguous(), agg=e.permute(1, 2, 0).contiguous(), disp=l, wta=None,
                    best2=torch.stack([best, other], 2))
    if kind == "batch":
        outs = []
        for i, (w, h, d) in enumerate(_batch_pairs(case)):
            ref, tgt, shift, _ = _scene(w, h, d, 1000 * seed + i)
            l, out, _ = _frame_exact(ref, tgt, shift, d, case)
            outs.append(dict(disp=l, wta=None, valid=None, out=out))
        return outs
    if kind == "warp_est":
        f = case["factor"]
        ref, tgt, _, _ = _scene(case["width"], case["height"], case["disp"], 1000 * seed, False)
        h, w, dc = case["height"] // f, case["width"] // f, -(-case["disp"] // f)

        def coarse(a):
            s = a[:h * f, :w * f].long().view(h, f, w, f).sum((1, 3))
            return ((s + f * f // 2) // (f * f)).double()

        cr, ct, zero = coarse(ref), coarse(tgt), torch.zeros(h, device="cuda")
        e = _aggregate(cr, _costs(cr, ct, dc, 5), 7, 3.0, 10.0)
        l = _wta(e, zero)[1]
        ok = _valid(w, h, dc, 5, zero)
        v = torch.nonzero(ok, as_tuple=True)[0].double()
        m = torch.stack([torch.ones_like(v), v], 1)
        a, b = torch.linalg.solve(m.T @ m, m.T @ (f * l[ok])).tolist()
        c1 = b / f
        c0 = a - c1 * (f - 1) / 2.0
        rows = torch.arange(case["height"], dtype=torch.float64)
        return dict(coef=torch.tensor([c0, c1, float(v.numel())], dtype=torch.float64), shift=c0 + c1 * rows - 4.0)
    if kind in ("soft", "grad"):
        ref, tgt, shift = (x.double() for x in _float_scenes(case, seed))
        disp, grads = [], []
        up = None
        if kind == "grad":
            g = torch.Generator(device="cuda").manual_seed(5 + seed)
            up = torch.randn(ref.shape, generator=g, device="cuda").double()
        for b in range(case["batch"]):
            x = [ref[b].clone(), tgt[b].clone(), shift[b].clone()]
            if up is None:
                with torch.no_grad():
                    disp.append(_soft_exact(*x, case))
                continue
            wanted = x if case["linear"] else x[:2]
            for t in wanted:
                t.requires_grad_()
            l = _soft_exact(*x, case)
            grads.append(torch.autograd.grad(l, wanted, up[b]))
            disp.append(l.detach())
        out = dict(disp=torch.stack(disp))
        if up is not None:
            out["grads"] = [torch.stack(list(g)) for g in zip(*grads)]
        return out
    disp, theta, mask, gain = _roll_inputs(case, seed)
    h, w = case["height"], case["width"]
    d = disp.double().requires_grad_()
    th = theta.clone().requires_grad_()
    v = torch.arange(h, device="cuda", dtype=torch.float64)[None, :, None]
    u = torch.arange(w, device="cuda", dtype=torch.float64)[None, None, :]
    keep = torch.ones_like(d, requires_grad=False) if mask is None else mask.double()
    psi, a0, a1 = (th[:, i, None, None] for i in range(3))
    energy = (keep * (d - a0 - a1 * (v * torch.cos(psi) - u * torch.sin(psi))).square()).sum((1, 2))
    gd, gt = torch.autograd.grad(energy, [d, th], gain)
    return dict(energy=energy.detach(), grad_disp=gd, grad_theta=gt, trajectory=None)
