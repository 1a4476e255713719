"""The work whose speed is measured: calls a user of the encoder makes, over the sizes they make them at.

Each case is one kind of call (`KINDS`) at one size.  Inputs are synthetic and seeded: video-conferencing frames (a
smooth background, an elliptical subject of about 30 % of the frame with band-limited texture) and Gaussian sets of the
two shapes the encoder meets, the region-of-interest initialisation ("roi": an even tiling of the subject, wide faint
Gaussians elsewhere) and the random initialisation ("random").
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2505_09324_gb300 import _native as nat
from paper_2505_09324_gb300.autograd import rasterize
from paper_2505_09324_gb300.learned import LearnedInitializer, Trainer, packaged
from paper_2505_09324_gb300.quant import DEFAULT_BITS, Quantizer, frame_bits
from paper_2505_09324_gb300.raster import BatchRasterizer, GaussianRasterizer, RasterConfig, roi_init

KINDS = ("decode", "grad", "encode", "fit", "upload", "batch", "pframe", "roi", "network", "train", "code")
ROI_FRAC = 0.7
SIGMA_CUT, ALPHA_MIN, DET_EPS = 4.5, 1.0 / 255.0, 1e-8
RESOLUTIONS = ((640, 360), (1280, 720), (1920, 1080))


def listed():
    hd = {"width": 1920, "height": 1080, "n": 20000}
    return [
        # a decoder showing a thumbnail-sized frame: the smallest call, all latency
        {"name": "decode_256", "kind": "decode", "width": 256, "height": 256, "n": 2000, "init": "random", "tile": 16, "stage": 64},
        # a decoder showing a full frame, default settings
        {"name": "decode_1080p", "kind": "decode", **hd, "init": "roi", "tile": 16, "stage": 64},
        # a torch program training through the rasterizer (forward and backward by autograd), ragged sizes
        {"name": "grad_719p", "kind": "grad", "width": 1279, "height": 719, "n": 9001, "init": "roi", "tile": 16, "stage": 64},
        # a whole small fit from random Gaussians, one call
        {"name": "encode_256", "kind": "encode", "width": 256, "height": 256, "n": 2000, "init": "random", "iters": 32, "tile": 16, "stage": 64},
        # the encoder's hot loop: iterations of a running fit with the schedule the autotuner picks at this size
        {"name": "fit_1080p", "kind": "fit", **hd, "init": "roi", "iters": 8, "tile": 32, "stage": 128},
        # one iteration driven from the host: 8-bit frame and Gaussians up, Gaussians down
        {"name": "upload_1080p", "kind": "upload", **hd, "init": "roi", "tile": 32, "stage": 128},
        # an offline encoder fitting many clips of mixed sizes in one launch per step
        {"name": "batch_12", "kind": "batch", "clips": 12, "iters": 4, "tile": 32, "stage": 128},
        # one P-frame of a sequence: reference render, selection, selective fit
        {"name": "pframe_1080p", "kind": "pframe", **hd, "iters": 8, "tile": 16, "stage": 64},
        # the superpixel initialisation of an I-frame
        {"name": "roi_1080p", "kind": "roi", **hd},
        # the learned initialisation of a batch of I-frames (shipped weights)
        {"name": "network_1080p", "kind": "network", **hd, "batch": 8},
        # one training step of the learned initialiser at its training size
        {"name": "train_1080p", "kind": "train", **hd, "batch": 8},
        # coding a fitted frame: quantisation and its size in bits
        {"name": "code_1080p", "kind": "code", **hd, "select": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _log_size(rng, lo, hi):
    """A frame of lo to hi pixels a side across, of a usual shape, seldom a multiple of anything."""
    w = _log_int(rng, lo, hi)
    return w, max(64, int(w * rng.choice((9 / 16, 3 / 4, 1.0, 9 / 16))) + rng.randint(-3, 3))


def draw(rng):
    kind = rng.choice(KINDS)
    w, h = _log_size(rng, 160, 1920)
    h = min(h, 1088)
    n = _log_int(rng, max(300, w * h // 1000), max(600, min(30000, w * h // 30)))
    c = {"kind": kind, "width": w, "height": h, "n": n}
    if kind in ("decode", "grad", "encode", "fit", "upload", "pframe"):
        c["tile"], c["stage"] = rng.choice(((16, 64), (16, 64), (32, 128), (32, 64), (16, 128), (8, 64)))
    if kind in ("decode", "grad", "encode", "fit", "upload"):
        c["init"] = rng.choice(("roi", "roi", "random"))
    if kind == "encode":
        c["iters"] = rng.randint(8, 32)
    if kind in ("fit", "pframe"):
        c["iters"] = rng.randint(4, 8)
    if kind == "batch":
        c = {"kind": kind, "clips": rng.randint(2, 12), "iters": rng.randint(2, 4), "tile": 32, "stage": 128}
    if kind in ("network", "train"):
        w, h = _log_size(rng, 160, 1280)
        w = w // 16 * 16 if rng.random() < 0.7 else w
        slots = 10 * (-(-w // 32)) * (-(-h // 32))
        c.update(width=w, height=h, batch=rng.randint(1, 8 if kind == "network" else 4), n=rng.randint(slots // 4, slots))
    if kind == "code":
        c["select"] = rng.random() < 0.5
    return c


# ---------------------------------------------------------------------------------------------------------------------
# Inputs


def _waves(xs, ys, kx, ky, phase, amp):
    """sum_j amp_j sin(kx_j x + ky_j y + phase_j) on a grid, as one matrix product."""
    a, b = kx[:, None] * xs[None], ys[:, None] * ky[None] + phase[None]
    return torch.cat([b.cos(), b.sin()], 1) @ torch.cat([amp[:, None] * a.sin(), amp[:, None] * a.cos()])


def _uniform(gen, lo, hi, *shape):
    return (lo + (hi - lo) * torch.rand(*shape, generator=gen, dtype=torch.float64)).cuda()


def _normal(gen, *shape):
    return torch.randn(*shape, generator=gen, dtype=torch.float64).cuda()


def _scene(gen, w, h):
    """A conferencing frame [3, h, w] float32 and its subject mask [h, w] uint8."""
    xs = torch.arange(w, device="cuda", dtype=torch.float64) + 0.5
    ys = torch.arange(h, device="cuda", dtype=torch.float64) + 0.5
    a = math.sqrt(0.3 * w * h / (math.pi * 1.3))
    ox, oy = (xs - w / 2)[None] / a, (ys - h / 2)[:, None] / (1.3 * a)
    rho = (ox * ox + oy * oy).sqrt()
    s = ((1.0 - rho) * a / 3.0 + 0.5).clamp(0, 1)
    alpha = s * s * (3 - 2 * s)
    frame = torch.empty(3, h, w, device="cuda", dtype=torch.float64)
    for ch in range(3):
        cyc = torch.randint(-3, 4, (2, 8), generator=gen).double().cuda()
        amp = _uniform(gen, 0.2, 1.0, 8)
        back = 0.5 + 0.25 * _waves(xs, ys, 2 * math.pi * cyc[0] / w, 2 * math.pi * cyc[1] / h, _uniform(gen, 0, 6.28, 8), amp) / amp.sum()
        lam, ang, amp = _uniform(gen, 24, 96, 64), _uniform(gen, 0, 6.28, 64), _uniform(gen, 0, 1, 64)
        k = 2 * math.pi / lam
        tex = _waves(xs, ys, k * ang.cos(), k * ang.sin(), _uniform(gen, 0, 6.28, 64), 0.15 * amp / amp.sum())
        frame[ch] = alpha * (_uniform(gen, 0.3, 0.7, 1) + tex) + (1 - alpha) * back
    return frame.float(), (rho <= 1.0).to(torch.uint8)


def _outside(gen, mask, n):
    """n positions spread over the pixels outside the mask (float64 [2, n])."""
    free = torch.nonzero(mask.reshape(-1) == 0).reshape(-1)
    pick = free[(torch.rand(n, generator=gen, dtype=torch.float64).cuda() * free.numel()).long().clamp(max=free.numel() - 1)]
    w = mask.shape[1]
    return torch.stack([pick % w, pick // w]).double() + _uniform(gen, 0, 1, 2, n)


def _colours(frame, xy):
    _, h, w = frame.shape
    return frame[:, xy[1].long().clamp(0, h - 1), xy[0].long().clamp(0, w - 1)].double()


def _gaussians(gen, frame, mask, n, init):
    """A Gaussian set [9, n] float32 as an early fit of the frame has it."""
    _, h, w = frame.shape
    p = torch.empty(9, n, device="cuda", dtype=torch.float64)
    if init == "random":
        p[0], p[1] = _uniform(gen, 0, w, n), _uniform(gen, 0, h, n)
        p[2], p[4] = (_uniform(gen, 0, math.log(8), n).exp() for _ in range(2))
        p[3], p[5:8], p[8] = _normal(gen, n), _uniform(gen, 0, 1, 3, n), _uniform(gen, 0.2, 1, n)
        return p.float()
    area = float(mask.sum())
    step = max(1.0, math.sqrt(area / (ROI_FRAC * n)))
    gx, gy = math.ceil(w / step), math.ceil(h / step)
    cell = torch.arange(gx * gy, device="cuda")
    xy = torch.stack([cell % gx + 0.5, cell // gx + 0.5]) * step
    inside = (xy[0] < w) & (xy[1] < h)
    inside &= mask[xy[1].long().clamp(max=h - 1), xy[0].long().clamp(max=w - 1)] != 0
    xy = xy[:, inside][:, :n]
    m = xy.shape[1]
    xy = xy + step * _uniform(gen, -0.2, 0.2, 2, m)
    l1, l3 = (step / math.sqrt(3) * (0.15 * _normal(gen, m)).exp() for _ in range(2))
    p[0:2, :m], p[2, :m], p[3, :m], p[4, :m] = xy, l1, 0.1 * step * _normal(gen, m), l3
    p[8, :m] = step * step / (2 * math.pi * l1 * l3)
    if m < n:
        xy = _outside(gen, mask, n - m)
        size = math.sqrt(4 * max(1.0, (w * h - area) / (n - m)) / (2 * math.pi))
        p[0:2, m:] = xy
        p[2, m:], p[4, m:] = (size * (0.1 * _normal(gen, n - m)).exp() for _ in range(2))
        p[3, m:], p[8, m:] = 0.05 * size * _normal(gen, n - m), 0.25 * (0.1 * _normal(gen, n - m)).exp()
    p[5:8] = _colours(frame, p[0:2]) + 0.02 * _normal(gen, 3, n)
    return p.float()


def _moments(gen, w, h, n):
    """Adam moments of a fit that has run for a while: the mean small against the root mean square."""
    scale = torch.tensor([0.2, 0.2, 0.2, 0.2, 0.2, 1.0, 1.0, 1.0, 1.0], device="cuda", dtype=torch.float64)[:, None] / (w * h)
    v = (scale * (0.5 * _normal(gen, 9, n)).exp()).square()
    return (0.1 * v.sqrt() * _normal(gen, 9, n)).float(), (0.2 * v).float()


def _clip_sizes(gen, count):
    pick = torch.randint(0, len(RESOLUTIONS), (count,), generator=gen).tolist()
    n = torch.exp(torch.rand(count, generator=gen) * math.log(25) + math.log(2000)).round().int().tolist()
    return [(*RESOLUTIONS[k], m) for k, m in zip(pick, n)]


def _batch_sizes(case):
    """The clip table of a batch: fixed by the case, so that its work does not vary with the inputs."""
    return _clip_sizes(torch.Generator().manual_seed(1000 + case["clips"]), case["clips"])


def _changed(gen, frame):
    """The next frame of a sequence: the texture of a part of the subject has moved."""
    _, h, w = frame.shape
    ys, xs = torch.meshgrid(torch.arange(h, device="cuda"), torch.arange(w, device="cuda"), indexing="ij")
    cx, cy = w * float(_uniform(gen, 0.45, 0.55, 1)), h * float(_uniform(gen, 0.4, 0.6, 1))
    near = ((xs - cx) / (0.2 * w)) ** 2 + ((ys - cy) / (0.4 * h)) ** 2 < 1
    ang = _uniform(gen, 0, 6.28, 3)
    wave = torch.sin(0.11 * (xs[None] * ang.cos()[:, None, None] + ys[None] * ang.sin()[:, None, None]) + ang[:, None, None])
    return (frame.double() + 0.08 * wave * near).float()


def _config(case):
    return RasterConfig(tile=case["tile"], stage=case["stage"])


RESUME_STEP = 200


def _net(case):
    w, h, n, b = case["width"], case["height"], case["n"], case["batch"]
    return packaged(w, h, n, b) or LearnedInitializer(w, h, n, b, seed=3)


def _inputs(case, seed):
    """The inputs of a case, by name (the same for prepare and exact)."""
    gen = torch.Generator().manual_seed(int(seed))
    kind = case["kind"]
    if kind == "batch":
        scenes = [(_scene(gen, w, h), w, h, n) for w, h, n in _batch_sizes(case)]
        return {"frames": [s[0] for s, _, _, _ in scenes], "params": [_gaussians(gen, *s, n, "roi") for s, _, _, n in scenes]}
    w, h, n = case["width"], case["height"], case["n"]
    if kind in ("network", "train"):
        scenes = [_scene(gen, w, h) for _ in range(case["batch"])]
        d = {"frames": torch.stack([s[0] for s in scenes]), "masks": torch.stack([s[1] for s in scenes])}
        if kind == "train":
            d["targets"] = torch.cat([_gaussians(gen, *s, n, "roi") for s in scenes], 1).contiguous()
        return d
    frame, mask = _scene(gen, w, h)
    if kind == "roi":
        return {"frame": frame, "mask": mask, "bg": _outside(gen, mask, n).float().contiguous()}
    d = {"frame": frame, "params": _gaussians(gen, frame, mask, n, case.get("init", "roi"))}
    if kind == "grad":
        d["dimg"] = (_normal(gen, 3, h, w) / (3 * h * w)).float()
    if kind == "fit":
        d["m"], d["v"] = _moments(gen, w, h, n)
    if kind == "upload":
        d["rgb"] = (frame.clamp(0, 1) * 255).round().to(torch.uint8).permute(1, 2, 0).contiguous().cpu()
    if kind == "pframe":
        d["frame"] = _changed(gen, _Splat(d["params"], w, h).image().float())
    if kind == "code":
        d["selected"] = (torch.rand(n, generator=gen) < 0.45).to(torch.uint8).cuda()
    return d


def prepare(case, seed):
    kind, d = case["kind"], _inputs(case, seed)
    state = {"case": dict(case), **d}
    if kind in ("decode", "grad", "encode", "fit", "upload", "pframe"):
        state["rast"] = GaussianRasterizer(case["width"], case["height"], case["n"], config=_config(case))
        state["adam"] = (torch.empty_like(d["params"]), torch.empty_like(d["params"]))
        state["work"] = d["params"].clone()
    if kind in ("encode", "batch", "pframe"):
        state["side"] = torch.cuda.Stream()
    if kind == "fit":
        b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
        state["checkpoint"] = {"params": d["params"], "m": d["m"], "v": d["v"], "step": RESUME_STEP, "beta1_pow": b1**RESUME_STEP,
                               "beta2_pow": b2**RESUME_STEP, "decay_pow": 1.0}
    if kind == "upload":
        w, h = case["width"], case["height"]
        state["rgb"], state["up"] = d["rgb"].pin_memory(), d["params"].cpu().pin_memory()
        state["down"] = torch.empty_like(state["up"]).pin_memory()
        state["rgb_dev"], state["frame_dev"] = torch.empty(h, w, 3, dtype=torch.uint8, device="cuda"), torch.empty(3, h, w, device="cuda")
    if kind == "batch":
        state["rast"] = BatchRasterizer(_batch_sizes(case), config=_config(case))
        state["targets"], state["params"] = state["rast"].pack_images(d["frames"]), state["rast"].pack_params(d["params"])
        state["frames"] = None
    if kind in ("network", "train"):
        state["net"] = _net(case)
    if kind == "train":
        state["trainer"] = Trainer(state["net"])
    if kind == "code":
        lo, hi = d["params"].amin(1), d["params"].amax(1)
        state["quantizer"] = Quantizer(DEFAULT_BITS, lo.tolist(), hi.tolist())
    torch.cuda.synchronize()
    return state


def run(state):
    return globals()["_run_" + state["case"]["kind"]](state, state["case"])


def _run_decode(s, case):
    s["rast"].prepare(s["params"])
    return s["rast"].render_fwd()


def _run_grad(s, case):
    p = s["params"].detach().requires_grad_()
    img = rasterize(p, s["rast"])
    (grad,) = torch.autograd.grad(img, p, s["dimg"])
    return {"image": img.detach(), "grad": grad}


def _run_encode(s, case):
    s["side"].wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s["side"]):
        s["work"].copy_(s["params"])
        r = s["rast"].encode_frame(s["frame"], s["work"], case["iters"], check_every=8, adam_state=s["adam"])
    torch.cuda.current_stream().wait_stream(s["side"])
    return {"params": s["work"], "iters": r["iters"], "trace": r["trace"]}


def _run_fit(s, case):
    s["rast"].fit_restore(s["checkpoint"], s["work"], s["adam"])
    for _ in range(case["iters"]):
        s["rast"].fit_step(s["frame"], s["work"], s["adam"])
    return {"params": s["work"], "m": s["adam"][0], "v": s["adam"][1]}


def _run_upload(s, case):
    m, v = s["adam"]
    s["rast"].fit_reset(s["adam"])
    nat.fit_step_rgb8(s["rast"].plan, s["rast"].ws_ptr, s["rgb"].data_ptr(), s["rgb_dev"].data_ptr(), s["frame_dev"].data_ptr(),
                      s["up"].data_ptr(), s["work"].data_ptr(), m.data_ptr(), v.data_ptr(), s["down"].data_ptr(),
                      int(torch.cuda.current_stream().cuda_stream))
    return {"params": s["down"], "m": m, "v": v, "frame": s["frame_dev"]}


def _run_batch(s, case):
    s["side"].wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s["side"]):
        p = s["params"].clone()
        psnr = s["rast"].encode_batch(s["targets"], p, case["iters"])
    torch.cuda.current_stream().wait_stream(s["side"])
    return {"params": p, "psnr": np.array(psnr, np.float32)}


def _run_pframe(s, case):
    s["side"].wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s["side"]):
        s["work"].copy_(s["params"])
        s["rast"].prepare(s["work"])
        ref = s["rast"].render_fwd()
        sel, count = s["rast"].select_changed(ref, s["frame"], 0.02)
        psnr = s["rast"].encode_pframe(s["frame"], s["work"], sel, case["iters"], adam_state=s["adam"])
    torch.cuda.current_stream().wait_stream(s["side"])
    return {"reference": ref, "selected": sel, "count": count, "params": s["work"], "psnr": np.array([psnr], np.float32)}


def _run_roi(s, case):
    params, n_roi = roi_init(s["frame"], s["mask"], case["n"], ROI_FRAC, s["bg"])
    return {"params": params, "n_roi": n_roi}


def _run_network(s, case):
    params = s["net"].forward(s["frames"], s["masks"], keep_col=False)
    return {"out": s["net"].out, "params": params, "slots": s["net"].sel}


def _run_train(s, case):
    loss, chamfer = s["trainer"].step(s["frames"], s["masks"], s["targets"])
    return {"loss": loss, "chamfer": chamfer, "grads": list(s["net"].dw)}


def _run_code(s, case):
    codes, values, ranges = s["quantizer"].quantize(s["params"])
    bits = frame_bits(s["quantizer"], s["params"], s["selected"] if case["select"] else None)
    return {"codes": codes.view(torch.int16), "values": values, "ranges": ranges, "bits": np.array([bits])}


# ---------------------------------------------------------------------------------------------------------------------
# What a pass cannot do without


def _hits(w, h, n, init):
    """(pixel, Gaussian) pairs inside the cut-off: the ellipses' area."""
    if init == "random":
        return n * 2 * math.pi * 4.45 * (7 / math.log(8)) ** 2
    return 0.3 * w * h * 2 * math.pi * SIGMA_CUT / 3 + 0.7 * w * h * 4 * math.log(255 / 4)


FWD, BWD = 14, 26  # arithmetic of one pair: distance, exponential, colours; the gradient sums (a multiply-add counts 2)


def _net_flops(case):
    h, w, ch, flops = case["height"], case["width"], (8, 32, 64, 128, 256, 384), 0
    acts = [4 * 3 * h * w + h * w]
    for ci, co in zip(ch, ch[1:]):
        h, w = (h + 1) // 2, (w + 1) // 2
        flops += 2 * h * w * co * (9 * ci + 1)
        acts.append(2 * h * w * co)
    flops += 2 * h * w * 96 * 385
    return case["batch"] * flops, case["batch"] * (2 * sum(acts) - acts[0] + 4 * h * w * 96)


def work(case):
    kind, it = case["kind"], case.get("iters", 1)
    if kind == "batch":
        both = [(w * h, n, _hits(w, h, n, "roi")) for w, h, n in _batch_sizes(case)]
        px, n, hits = (sum(x[k] for x in both) for k in range(3))
        return {"bytes": it * (12 * px + 216 * n), "flops": it * hits * (FWD + BWD)}
    w, h, n = case["width"], case["height"], case["n"]
    px, hits = w * h, _hits(w, h, n, case.get("init", "roi"))
    if kind == "decode":
        return {"bytes": 36 * n + 12 * px, "flops": hits * FWD}
    if kind == "grad":
        return {"bytes": 72 * n + 24 * px, "flops": hits * (2 * FWD + BWD)}
    if kind in ("encode", "fit"):
        return {"bytes": it * (12 * px + 216 * n), "flops": it * hits * (FWD + BWD)}
    if kind == "upload":
        return {"bytes": 3 * px + 12 * px + 216 * n, "flops": hits * (FWD + BWD)}
    if kind == "pframe":  # selection over the whole frame, fitting over about half of it
        return {"bytes": 36 * px + it * (6 * px + 130 * n), "flops": hits * (FWD + it * 0.5 * (FWD + BWD))}
    if kind == "roi":  # ten passes over the subject, 25 candidates a pixel
        return {"bytes": 13 * px + 44 * n, "flops": 10 * 0.3 * px * 25 * 12}
    if kind in ("network", "train"):
        flops, moved = _net_flops(case)
        if kind == "network":
            return {"bytes": moved, "flops": flops}
        hits *= case["batch"]
        return {"bytes": 3 * moved + case["batch"] * (12 * px + 144 * n), "flops": 3 * flops + hits * (FWD + BWD)}
    return {"bytes": (36 + 18 + 36 + 18) * n, "flops": 9 * n * 8}


# ---------------------------------------------------------------------------------------------------------------------
# The same results in 64 bits


class _Splat:
    """The accumulated-sum render of a Gaussian set and its gradient in 64 bits, over blocks of 32 x 32 pixels."""

    T, CHUNK = 32, 4096

    def __init__(self, params, w, h):
        self.p, self.w, self.h = params.double(), w, h
        mx, my, l1, l2, l3 = self.p[:5]
        wt = self.p[8].abs()
        ok = torch.isfinite(self.p).all(0) & ((l1 * l3) ** 2 > DET_EPS) & (wt >= ALPHA_MIN)
        self.tau = torch.log(wt.clamp(min=ALPHA_MIN) / ALPHA_MIN).clamp(max=SIGMA_CUT)
        rx = (2 * self.tau).sqrt() * l1.abs() + 1e-6
        ry = (2 * self.tau).sqrt() * (l2 * l2 + l3 * l3).sqrt() + 1e-6
        self.tx, self.ty = -(-w // self.T), -(-h // self.T)

        def span(c, r, count):
            lo = ((c - r) / self.T).floor().clamp(0, count).nan_to_num().long()
            hi = (((c + r) / self.T).floor() + 1).clamp(0, count).nan_to_num().long()
            return lo, torch.where(ok, (hi - lo).clamp(min=0), 0)

        (x0, nx), (y0, ny) = span(mx, rx, self.tx), span(my, ry, self.ty)
        count = nx * ny
        self.g = torch.repeat_interleave(torch.arange(self.p.shape[1], device=params.device), count)
        j = torch.arange(self.g.numel(), device=params.device) - torch.repeat_interleave(count.cumsum(0) - count, count)
        self.x, self.y = x0[self.g] + j % nx[self.g], y0[self.g] + j // nx[self.g]

    def _pairs(self):
        grid = torch.arange(self.T, device=self.p.device, dtype=torch.float64) + 0.5
        for k in range(0, self.g.numel(), self.CHUNK):
            g, x, y = (t[k : k + self.CHUNK] for t in (self.g, self.x, self.y))
            mx, my, l1, l2, l3 = (self.p[r, g][:, None] for r in range(5))
            u1 = ((x[:, None] * self.T + grid - mx) / l1)[:, None, :]
            u2 = ((y[:, None] * self.T + grid - my)[:, :, None] - l2[:, :, None] * u1) / l3[:, :, None]
            sig = 0.5 * (u1 * u1 + u2 * u2)
            yield g, y * self.tx + x, u1, u2, torch.where(sig <= self.tau[g][:, None, None], torch.exp(-sig), 0.0)

    def _blocks(self, img):
        img = F.pad(img, (0, self.tx * self.T - self.w, 0, self.ty * self.T - self.h))
        return img.view(3, self.ty, self.T, self.tx, self.T).permute(1, 3, 0, 2, 4).reshape(-1, 3, self.T * self.T)

    def image(self):
        acc = torch.zeros(self.tx * self.ty, 3, self.T * self.T, device=self.p.device, dtype=torch.float64)
        col = (self.p[5:8] * self.p[8]).T
        for g, tile, _, _, e in self._pairs():
            acc.index_add_(0, tile, col[g][:, :, None] * e.reshape(len(g), 1, -1))
        img = acc.view(self.ty, self.tx, 3, self.T, self.T).permute(2, 0, 3, 1, 4).reshape(3, self.ty * self.T, self.tx * self.T)
        return img[:, : self.h, : self.w].contiguous()

    def grad(self, dimg):
        blocks, p = self._blocks(dimg.double()), self.p
        s = torch.zeros(p.shape[1], 8, device=p.device, dtype=torch.float64)
        col = (p[5:8] * p[8]).T
        for g, tile, u1, u2, e in self._pairs():
            ge = blocks[tile] * e.reshape(len(g), 1, -1)
            sv = torch.einsum("pck,pc->pk", ge, col[g]).view_as(e)
            su1, su2 = sv * u1, sv * u2
            s.index_add_(0, g, torch.stack([*ge.sum(2).T, *(t.sum((1, 2)) for t in (su1, su2, su1 * u1, su1 * u2, su2 * u2))], 1))
        r = p[3] / p[4]
        out = torch.empty_like(p)
        out[0], out[1] = (s[:, 3] - r * s[:, 4]) / p[2], s[:, 4] / p[4]
        out[2], out[3], out[4] = (s[:, 5] - r * s[:, 6]) / p[2], s[:, 6] / p[4], s[:, 7] / p[4]
        out[5:8] = p[8] * s[:, :3].T
        out[8] = (p[5:8] * s[:, :3].T).sum(0)
        return out


def _fit64(frame, params, m, v, step, iters, every=0, select=None):
    """Adam on the mean squared error: (params, m, v, psnr of the renders at each check) after `iters` iterations."""
    frame, p, m, v = frame.double(), params.double(), m.double(), v.double()
    _, h, w = frame.shape
    b1, b2, lr = (float(np.float32(x)) for x in (0.9, 0.999, 1e-2))
    trace = []
    for k in range(iters):
        sp = _Splat(p, w, h)
        img = sp.image()
        if every and ((k + 1) % every == 0 or k + 1 == iters):
            trace.append(_psnr(img, frame))
        g = sp.grad(2 * (img - frame) / (3 * h * w))
        nm, nv = b1 * m + (1 - b1) * g, b2 * v + (1 - b2) * g * g
        t = step + k + 1
        np_ = p - lr * (nm / (1 - b1**t)) / ((nv / (1 - b2**t)).sqrt() + 1e-8)
        on = torch.ones_like(p, dtype=torch.bool) if select is None else (select != 0).expand_as(p)
        p, m, v = torch.where(on, np_, p), torch.where(on, nm, m), torch.where(on, nv, v)
    return p, m, v, trace


def _psnr(img, frame):
    return -10 * math.log10(float((img.clamp(0, 1) - frame.double()).square().mean()))


def exact(case, seed):
    return globals()["_exact_" + case["kind"]](case, _inputs(case, seed))


def _exact_decode(case, d):
    return _Splat(d["params"], case["width"], case["height"]).image()


def _exact_grad(case, d):
    sp = _Splat(d["params"], case["width"], case["height"])
    return {"image": sp.image(), "grad": sp.grad(d["dimg"])}


def _exact_encode(case, d):
    zero = torch.zeros_like(d["params"])
    p, _, _, trace = _fit64(d["frame"], d["params"], zero, zero, 0, case["iters"], every=8)
    return {"params": p, "iters": None, "trace": trace}


def _exact_fit(case, d):
    p, m, v, _ = _fit64(d["frame"], d["params"], d["m"], d["v"], RESUME_STEP, case["iters"])
    return {"params": p, "m": m, "v": v}


def _exact_upload(case, d):
    zero = torch.zeros_like(d["params"])
    frame = d["rgb"].cuda().permute(2, 0, 1).double() / 255
    p, m, v, _ = _fit64(frame, d["params"], zero, zero, 0, 1)
    return {"params": p.cpu(), "m": m, "v": v, "frame": frame}


def _exact_batch(case, d):
    ps, psnr = [], []
    for frame, params in zip(d["frames"], d["params"]):
        zero = torch.zeros_like(params)
        p = _fit64(frame, params, zero, zero, 0, case["iters"])[0]
        ps.append(p)
        psnr.append(_psnr(_Splat(p, frame.shape[2], frame.shape[1]).image(), frame))
    return {"params": torch.cat(ps, 1), "psnr": np.array(psnr)}


def _exact_pframe(case, d):
    return {"reference": _Splat(d["params"], case["width"], case["height"]).image()}


def _exact_roi(case, d):
    """Ten K-means passes over the subject's pixels, then a Gaussian for each segment and for each background position."""
    w, h, n = case["width"], case["height"], case["n"]
    frame, mask = d["frame"].double(), d["mask"] != 0
    area, f64 = float(mask.sum()), {"device": "cuda", "dtype": torch.float64}
    S = max(1.0, math.sqrt(area / round(ROI_FRAC * n)))
    gx, gy = math.ceil(w / S), math.ceil(h / S)
    cell = torch.arange(gx * gy, device="cuda")
    cx, cy = (cell % gx + 0.5).double() * S, (cell // gx + 0.5).double() * S
    seed = (cx.floor() < w) & (cy.floor() < h)
    seed &= mask[cy.long().clamp(max=h - 1), cx.long().clamp(max=w - 1)]
    M = min(n, int(seed.sum()))
    index = torch.where(seed, seed.long().cumsum(0) - 1, -1)
    index = torch.where(index < M, index, -1)
    q = torch.stack([cx[seed][:M], cy[seed][:M]])
    cen = torch.cat([frame[:, q[1].long(), q[0].long()], q])
    ys, xs = torch.nonzero(mask, as_tuple=True)
    pix = torch.cat([frame[:, ys, xs], (xs + 0.5)[None].double(), (ys + 0.5)[None].double()])
    px, py = (pix[3] / S).floor().long(), (pix[4] / S).floor().long()
    for _ in range(10):
        best, lab = torch.full_like(pix[0], math.inf), torch.full_like(px, -1)
        for dj in range(-2, 3):
            for di in range(-2, 3):
                jx, jy = px + di, py + dj
                inside = (jx >= 0) & (jx < gx) & (jy >= 0) & (jy < gy)
                c = torch.where(inside, index[(jy * gx + jx).clamp(0, gx * gy - 1)], -1)
                diff = pix - cen[:, c.clamp(min=0)]
                dist = diff[:3].square().sum(0) + (0.2 / S) ** 2 * diff[3:].square().sum(0)
                take = (c >= 0) & (diff[3:].abs().amax(0) <= S) & (dist < best)
                best, lab = torch.where(take, dist, best), torch.where(take, c, lab)
        on = lab >= 0
        rows = torch.cat([torch.ones_like(pix[:1]), pix, pix[3:4] ** 2, pix[3:4] * pix[4:5], pix[4:5] ** 2])[:, on]
        s = torch.zeros(9, M, **f64).index_add_(1, lab[on], rows)
        mean = s[1:] / s[0].clamp(min=1)
        lim = torch.minimum(torch.maximum(mean[3:5], q - S), q + S)
        cen = torch.where(s[0] > 0, torch.cat([mean[:3], lim]), cen)
    out = torch.empty(9, n, **f64)
    vxx, vxy, vyy = mean[5] - mean[3] ** 2 + 1 / 12, mean[6] - mean[3] * mean[4], mean[7] - mean[4] ** 2 + 1 / 12
    c1 = vxx.sqrt()
    c3 = (vyy - (vxy / c1) ** 2).sqrt()
    full = torch.cat([mean[3:5], 2 * torch.stack([c1, vxy / c1, c3]), mean[:3], (s[0] / (8 * math.pi * c1 * c3))[None]])
    side = torch.full_like(c1, 2 * S / math.sqrt(12))
    bare = torch.cat([q, torch.stack([side, 0 * side, side]), frame[:, q[1].long(), q[0].long()], torch.ones_like(side)[None]])
    out[:, :M] = torch.where(s[0] > 0, full, bare)
    if M < n:
        xy = d["bg"].double()[:, : n - M]
        size = math.sqrt(4 * max(1.0, (w * h - area) / (n - M)) / (2 * math.pi))
        out[0:2, M:], out[2, M:], out[3, M:], out[4, M:], out[8, M:] = xy, size, 0, size, 0.25
        out[5:8, M:] = frame[:, xy[1].long().clamp(0, h - 1), xy[0].long().clamp(0, w - 1)]
    return {"params": out, "n_roi": None}


def _half(x):
    """x rounded to bfloat16, as the network stores it; the gradient passes."""
    return x + (x.detach().bfloat16().double() - x.detach())


def _network64(weights, frame, mask):
    """The head's output [cells, columns] of one frame; `weights`: per layer [co, columns], the bias in column ks^2 ci."""
    x = _half(torch.cat([frame.double(), (mask != 0).double()[None], torch.zeros(4, *mask.shape, device="cuda", dtype=torch.float64)]))
    for k, wt in enumerate(weights):
        ci, ks = x.shape[0], 3 if k + 1 < len(weights) else 1
        ho, wo = ((x.shape[1] + 1) // 2, (x.shape[2] + 1) // 2) if ks == 3 else x.shape[1:]
        col = F.unfold(x[None], ks, padding=ks // 2, stride=2 if ks == 3 else 1)[0]
        wk = wt[:, : ks * ks * ci].view(-1, ks * ks, ci).permute(0, 2, 1).reshape(wt.shape[0], -1)
        z = wk @ col + wt[:, ks * ks * ci, None]
        x = _half(F.relu(z)).view(-1, ho, wo) if ks == 3 else z
    return x.T


def _weights64(case):
    return [w.bfloat16().double() for w in _net(case).w32]


def _exact_network(case, d):
    weights = _weights64(case)
    return {"out": torch.cat([_network64(weights, f, m) for f, m in zip(d["frames"], d["masks"])]), "params": None, "slots": None}


def _decode64(out, w, h, n, slots=10, cell=32, scale=6.0):
    """The n Gaussians of largest |weight| of one frame's head output, in slot order."""
    gw = -(-w // cell)
    o = out[:, : 9 * slots].reshape(-1, 9)
    keep = (0.25 + o[:, 8]).detach().abs().sort(descending=True, stable=True).indices[:n].sort().values
    o, c, s = o[keep], keep // slots, keep % slots
    q = math.ceil(math.sqrt(slots))
    r = -(-slots // q)
    mx = ((c % gw) + (s % q + 0.5) / q) * cell + cell / 2 * torch.tanh(o[:, 0])
    my = ((c // gw) + (s // q + 0.5) / r) * cell + cell / 2 * torch.tanh(o[:, 1])
    l1, l3 = (scale * torch.exp(o[:, k].clamp(-4, 3)) for k in (2, 4))
    return torch.stack([mx, my, l1, scale * o[:, 3], l3, *(0.5 + o[:, 5:8]).T, 0.25 + o[:, 8]])


def _chamfer64(p, t):
    """The Chamfer distance of two sets of means and its gradient towards the first."""
    dist = torch.cdist(p.T, t.T, compute_mode="donot_use_mm_for_euclid_dist")
    (d1, j1), (d2, j2) = dist.min(1), dist.min(0)
    g = 2 * (p - t[:, j1]) / p.shape[1]
    g.index_add_(1, j2, 2 * (p[:, j2] - t) / t.shape[1])
    return float(d1.square().mean() + d2.square().mean()), g


def _exact_train(case, d):
    w, h, n, weights = case["width"], case["height"], case["n"], [x.requires_grad_() for x in _weights64(case)]
    loss, clamped, chamfer = 0.0, 0.0, []
    for b, (frame, mask) in enumerate(zip(d["frames"], d["masks"])):
        params = _decode64(_network64(weights, frame, mask), w, h, n)
        p = params.detach()
        sp = _Splat(p, w, h)
        img = sp.image()
        loss += float((img - frame).square().mean())
        clamped += float((img.clamp(0, 1) - frame).square().mean())
        g = sp.grad(2 * (img - frame) / (3 * h * w))
        far, push = _chamfer64(p[:2], d["targets"][:2, b * n : (b + 1) * n].double())
        chamfer.append(far)
        g[:2] += 1e-5 * push
        params.backward(g)
    return {"loss": np.array([loss, clamped]), "chamfer": np.array(chamfer), "grads": [x.grad for x in weights]}


def _exact_code(case, d):
    x = d["params"]
    n, bits = case["n"], DEFAULT_BITS
    lo, hi = x.amin(1).double()[:, None], x.amax(1).double()[:, None]
    top = torch.tensor([float((1 << b) - 1) for b in bits], device="cuda", dtype=torch.float64)[:, None]
    code = ((x.double() - lo) * top / (hi - lo)).round().clamp(min=0).minimum(top)
    on = d["selected"] != 0 if case["select"] else torch.ones(n, device="cuda", dtype=torch.bool)
    total = int(on.sum())
    size = total * math.ceil(math.log2(max(n, 2))) if case["select"] else 0
    for row in code[:, on]:
        c = row.unique(return_counts=True)[1].double()
        size += total * math.log2(total) - float((c * c.log2()).sum())
    return {"codes": None, "values": lo + code * (hi - lo) / top, "ranges": torch.stack([lo[:, 0], hi[:, 0]]), "bits": None}
