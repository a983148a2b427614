"""Measured workloads of the denoiser: what its users call, over the sizes and options they use.

Kinds of case:
  frame    one frame of a running sequence through ``Denoiser.denoise_frame`` (the ordinary call);
           ``export`` adds the checkpoint of the temporal state that a program takes with it
  cut      the first frame of a sequence or the one after a camera cut: no history, so every pixel's
           variance comes from its spatial neighbourhood
  stages   the same frame stage by stage (temporal stage, then each a-trous pass) in 16-bit or FP32
           storage, as a program does that composites on the tone-mapped colour itself
  batch    one frame of several streams of uneven sizes in one ``Batch`` call replayed as a graph
  learned  one frame with the kernel-predicting network in place of a-trous passes 1.., with or
           without the per-tile fallback to the plain passes
  train    one resumed Adam step of that network on a batch of crops
  host     a few frames given and returned in pinned host memory, pipelined

Frames are the package's procedural scenes (40 spheres, one moving 8 px a frame, a 0.5 px pan; 6
spheres in small frames), as in its benchmark.  A running sequence's state is imported: the colour history and
moments a sequence holds after some frames, with patches of short history that earlier
disocclusions left.
"""
import math
import struct

import numpy as np
import torch
import torch.nn.functional as F

from paper_2312_06827_gb300 import scene, svgf

LUMA = (0.2126, 0.7152, 0.0722)
PRECISION = {"fp32": svgf.FP32, "fp16": svgf.FP16, "bf16": svgf.BF16}
HISTORY_KINDS = ("frame", "stages", "batch", "learned")


def listed():
    return [
        # the smallest scene of the tests: seven launches of little work, so latency is what counts
        {"name": "frame_128", "kind": "frame", "w": 128, "h": 128, "mode": "5x5", "channel": "specular",
         "rectify": "clamp", "budget": False, "export": False},
        # a ragged window: the shadow channel with clipping and the roughness-adapted pass count,
        # and the state saved with the frame
        {"name": "frame_ragged_shadow", "kind": "frame", "w": 1283, "h": 717, "mode": "5x5", "channel": "shadow",
         "rectify": "clip", "budget": True, "export": True},
        # the ordinary frame: 1080p at the defaults
        {"name": "frame_1080p", "kind": "frame", "w": 1920, "h": 1080, "mode": "5x5", "channel": "specular",
         "rectify": "clamp", "budget": False, "export": False},
        # the same with the separable passes
        {"name": "frame_1080p_separable", "kind": "frame", "w": 1920, "h": 1080, "mode": "separable",
         "channel": "specular", "rectify": "clamp", "budget": False, "export": False},
        # the largest frame
        {"name": "frame_4k", "kind": "frame", "w": 3840, "h": 2160, "mode": "5x5", "channel": "specular",
         "rectify": "clamp", "budget": False, "export": False},
        # the largest frame in 16-bit storage, stage by stage
        {"name": "stages_4k_fp16", "kind": "stages", "w": 3840, "h": 2160, "mode": "5x5", "precision": "fp16"},
        # a camera cut at 1440p
        {"name": "cut_1440p", "kind": "cut", "w": 2560, "h": 1440, "mode": "5x5"},
        # eight streams of 640x360 to 2560x1440 served together
        {"name": "batch_8", "kind": "batch", "streams": 8, "scale": 1.0, "mode": "5x5"},
        # the learned form at 1080p, network only
        {"name": "learned_1080p", "kind": "learned", "w": 1920, "h": 1080, "mode": "5x5", "fallback": False},
        # the learned form at 720p with its per-tile fallback
        {"name": "learned_720p_fallback", "kind": "learned", "w": 1280, "h": 720, "mode": "5x5", "fallback": True},
        # the training step of the package's own recipe: 16 crops of 256 x 256
        {"name": "train_16x256", "kind": "train", "b": 16, "w": 256, "h": 256},
        # three 720p frames from and to host memory
        {"name": "host_720p", "kind": "host", "w": 1280, "h": 720, "frames": 3, "mode": "5x5"},
    ]


def _size(rng, lo, hi):
    """A width and height (odd ones among them) of lo to hi pixels, spread over the logarithm."""
    px = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    w = min(3840, max(24, int(math.sqrt(px * rng.uniform(1.0, 2.2)))))
    h = min(2160, max(24, int(px / w)))
    return w, h


def draw(rng):
    kind = rng.choice(("frame", "frame", "frame", "stages", "cut", "batch", "learned", "train", "host"))
    mode = rng.choice(("5x5", "5x5", "separable"))
    if kind == "batch":
        return {"kind": kind, "streams": rng.randint(2, 8), "scale": round(rng.uniform(0.2, 1.0), 3), "mode": mode}
    if kind == "train":
        return {"kind": kind, "b": rng.randint(1, 16), "w": rng.randint(40, 256), "h": rng.randint(40, 256)}
    big = {"frame": 8.2e6, "stages": 8.2e6, "cut": 3.6e6, "learned": 2.0e6, "host": 2.0e6}[kind]
    w, h = _size(rng, 3e3, big)
    c = {"kind": kind, "w": w, "h": h, "mode": mode}
    if kind == "frame":
        c.update(channel=rng.choice(("specular", "specular", "shadow")), rectify=rng.choice(("clamp", "clamp", "clip")),
                 budget=rng.random() < 0.25, export=rng.random() < 0.25)
    elif kind == "stages":
        c["precision"] = rng.choice(("fp32", "fp16", "bf16"))
    elif kind == "learned":
        c["fallback"] = rng.random() < 0.5
    elif kind == "host":
        c["frames"] = rng.randint(1, 4)
    return c


# ---- inputs ------------------------------------------------------------------------------------

def _sizes(case):
    """The frame sizes of a case: one, or one per stream of a batch."""
    if case["kind"] != "batch":
        return [(case["w"], case["h"])]
    s = case["scale"]
    four = [(640, 360), (1280, 720), (1920, 1080), (2560, 1440)]
    return [(max(24, int(w * s) + i % 2), max(24, int(h * s) + i % 3)) for i, (w, h) in
            enumerate(four[i % 4] for i in range(case["streams"]))]


def _config(case, w, h):
    channel = svgf.CHANNEL_SHADOW if case.get("channel") == "shadow" else svgf.CHANNEL_INDIRECT_SPECULAR
    c = svgf.channel_config(channel, w, h)
    c.spatial_mode = svgf.SEPARABLE if case["mode"] == "separable" else svgf.ATROUS_5X5
    c.precision = PRECISION[case.get("precision", "fp32")]
    c.rectify_mode = svgf.RECTIFY_CLIP if case.get("rectify") == "clip" else svgf.RECTIFY_CLAMP
    if case.get("budget"):
        # pass counts by roughness; the shadow channel's "roughness" is the light's angle in degrees
        c.iter_by_roughness, c.iter_count1 = 1, 2
        c.iter_rough_t0, c.iter_rough_t1 = (4.0, 5.0) if case.get("channel") == "shadow" else (0.1, 0.3)
    return c


def _frames(case, seed, w, h, count, stream=0):
    """`count` consecutive frames of a scene and the G-buffer of the frame before them (numpy)."""
    sc = scene.SceneConfig(w, h, n_spheres=40 if w * h > 1 << 17 else 6, moving_sphere=True, seed=seed, stream=stream)
    t0 = 3 + seed % 40
    keys = ["noisy", "gt", "gbuf_nz", "motion", "roughness", "albedo"]
    shadow = case.get("channel") == "shadow"
    if shadow:
        keys += ["shadow_noisy", "shadow_angle"]
    prev = scene.render_frame(sc, t0 - 1, ["gt", "gbuf_nz"])
    out = []
    for t in range(t0, t0 + count):
        f = scene.render_frame(sc, t, keys)
        if shadow:
            f["noisy"] = np.repeat(f["shadow_noisy"][..., None], 3, axis=2)
            f["roughness"] = f["shadow_angle"]
        out.append(f)
    return out, prev


def _history(case, seed, prev, tonemapped):
    """The temporal state of a running sequence: the previous frame's colour with the noise that is
    left in it, the luminance moments of its samples, and history lengths of 4 to 40 frames with
    patches of 1 to 3 (numpy float32: history [H, W, 4], moments [H, W, 4])."""
    rng = np.random.default_rng([seed, 77])
    gt = prev["gt"]
    h, w = gt.shape[:2]
    if tonemapped:
        clean = gt / (1.0 + (gt @ np.array(LUMA, np.float32))[..., None])
    else:
        clean = np.repeat(np.clip(gt[..., 1:2], 0.0, 1.0), 3, axis=2)
    noise = rng.standard_normal((h, w, 1), dtype=np.float32)
    hist = np.zeros((h, w, 4), np.float32)
    hist[..., :3] = clean * (1.0 + 0.05 * noise)
    luma = hist[..., :3] @ np.array(LUMA, np.float32)
    mom = np.zeros((h, w, 4), np.float32)
    mom[..., 0] = luma
    mom[..., 1] = (0.3 * luma) ** 2 * rng.uniform(0.2, 1.8, (h, w)).astype(np.float32) + 1e-6
    th, tw = -(-h // 16), -(-w // 16)
    patch = np.where(rng.random((th, tw)) < 0.01, rng.integers(1, 4, (th, tw)), rng.integers(4, 41, (th, tw)))
    mom[..., 2] = np.kron(patch, np.ones((16, 16)))[:h, :w]
    return hist, mom


def _upload(f):
    return {k: torch.from_numpy(f[k]).cuda() for k in ("noisy", "gbuf_nz", "motion", "roughness", "albedo")}


def _crops(case, seed):
    """Features, pass-0 colour and target of a batch of crops, as training takes them."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    b, h, w = case["b"], case["h"], case["w"]
    rnd = lambda *s: torch.rand(*s, generator=g, device="cuda")
    smooth = lambda x: F.interpolate(x, size=(h, w), mode="bilinear", align_corners=False).permute(0, 2, 3, 1)
    clean = smooth(rnd(b, 3, max(2, h // 16), max(2, w // 16))) * 0.8
    c0 = torch.zeros(b, h, w, 4, device="cuda")
    c0[..., :3] = clean * (0.9 + 0.2 * rnd(b, h, w, 1))
    c0[..., 3] = 1e-3 * rnd(b, h, w)
    target = torch.zeros(b, h, w, 4, device="cuda")
    target[..., :3] = clean
    feats = torch.zeros(b, h, w, 16, device="cuda")
    feats[..., :3] = c0[..., :3]
    feats[..., 3] = c0[..., 3].sqrt()
    feats[..., 4] = 2.0 + 2.0 * smooth(rnd(b, 1, 4, 4))[..., 0]
    feats[..., 5:7] = 2.0 * smooth(rnd(b, 2, 4, 4)) - 1.0
    feats[..., 7:10] = 0.1 + 0.8 * smooth(rnd(b, 3, 4, 4))
    return feats.bfloat16(), c0, target


def _weights(seed):
    """Kaiming-normal weights with small biases, the last layer scaled by 0.1 (numpy float32)."""
    rng = np.random.default_rng([seed, 5])
    parts = []
    for l, (ci, co) in enumerate(zip(svgf.KPN_CIN, svgf.KPN_COUT)):
        w = rng.standard_normal(co * 9 * ci) * math.sqrt(2.0 / (9 * ci)) * (0.1 if l == 3 else 1.0)
        parts += [w, 0.02 * rng.standard_normal(co)]
    return np.concatenate(parts).astype(np.float32)


ADAM_STEPS, LR = 500, 1e-3


def _checkpoint(seed):
    """A training checkpoint in the library's layout: parameters and Adam moments after 500 steps."""
    rng = np.random.default_rng([seed, 6])
    p = _weights(seed)
    v = (1e-3 * rng.uniform(0.5, 1.5, p.size)) ** 2
    m = 3e-4 * rng.standard_normal(p.size)
    head = struct.pack("<IIIIQ", 0x504B5653, 1, svgf.KPN_PARAM_COUNT, 1, ADAM_STEPS)
    return p, m.astype(np.float32), v.astype(np.float32), head


# ---- the call ----------------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "train":
        st["feats"], st["c0"], st["target"] = _crops(case, seed)
        k = svgf.KPN(case["b"] * case["h"] * case["w"], train=True)
        p, m, v, head = _checkpoint(seed)
        k.load(head + p.tobytes() + m.tobytes() + v.tobytes())
        st["kpn"], st["feats"] = k, st["feats"].view(torch.int16)
        return st
    streams = []
    for i, (w, h) in enumerate(_sizes(case)):
        cfg = _config(case, w, h)
        d = svgf.Denoiser(cfg)
        fs, prev = _frames(case, seed, w, h, case.get("frames", 1), i)
        s = {"d": d, "w": w, "h": h}
        if kind == "host":
            d.enable_host_staging()
            pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory()
            s["host"] = [{k: pin(f[k]) for k in ("noisy", "gbuf_nz", "motion", "roughness")} for f in fs]
            s["outs"] = [torch.empty(h, w, 4).pin_memory() for _ in fs]
        else:
            dv = _upload(fs[0])
            s["albedo"] = dv["albedo"]
            has = kind in HISTORY_KINDS
            s["prev"] = torch.from_numpy(prev["gbuf_nz"]).cuda() if has else None
            s["frame"] = svgf.make_frame(dv["noisy"], dv["gbuf_nz"], dv["motion"], dv["roughness"], s["prev"])
            s["out"] = torch.empty(h, w, 4, device="cuda")
            if has:
                hist, mom = _history(case, seed + i, prev, cfg.tonemap)
                d.history_import(torch.from_numpy(hist).cuda(), torch.from_numpy(mom).cuda())
            if case.get("export"):
                s["state"] = [torch.empty(h, w, 4, device="cuda") for _ in range(2)]
        streams.append(s)
    st["streams"] = streams
    if kind == "stages":
        t = torch.float32 if case["precision"] == "fp32" else torch.int16
        st["cv"] = [torch.empty(case["h"], case["w"], 4, dtype=t, device="cuda") for _ in range(2)]
    if kind == "batch":
        st["batch"] = svgf.Batch([s["d"] for s in streams])
        st["batch"].use_graph(True)
        st["stream"] = torch.cuda.Stream()
    if kind == "learned":
        st["kpn"] = svgf.KPN(case["w"] * case["h"], train=False)
        st["kpn"].set_params(torch.from_numpy(_weights(seed)))
    torch.cuda.synchronize()
    return st


FALLBACK_STD = 0.06    # luminance spread above which a tile falls back: about 10 % of a 720p frame's tiles


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "train":
        k = st["kpn"]
        loss = k.train_step(st["feats"], st["c0"], st["target"], LR)
        return {"loss": loss, "grad": k.grad, "params": k.params, "adam_m": k.adam_m, "adam_v": k.adam_v}
    s = st["streams"][0]
    d = s["d"]
    if kind == "batch":
        outs = [x["out"] for x in st["streams"]]
        st["batch"].denoise([x["frame"] for x in st["streams"]], outs, stream=st["stream"])
        return outs
    if kind == "host":
        for f, o in zip(s["host"], s["outs"]):
            d.submit_host(f["noisy"], f["gbuf_nz"], f["motion"], f["roughness"], o)
        d.wait_host()
        return s["outs"]
    if kind == "learned":
        t = FALLBACK_STD if case["fallback"] else math.inf
        n = st["kpn"].denoise_frame(d, s["frame"], s["albedo"], s["out"], detail_threshold=t)
        return {"rgb": s["out"], "fallback_tiles": n}
    if kind == "stages":
        cv = st["cv"]
        d.reproject_accumulate(s["frame"], cv[0])
        for i in range(d.cfg.atrous_iters):
            d.atrous(i, s["frame"], cv[i & 1], cv[(i + 1) & 1])
        last = cv[d.cfg.atrous_iters & 1]
        if case["precision"] == "fp32":
            return {"colour": last[..., :3], "variance": last[..., 3]}
        # a record is three FP16 (or BF16) colours and a BF16 variance
        colour = torch.float16 if case["precision"] == "fp16" else torch.bfloat16
        return {"colour": last.view(colour)[..., :3], "variance": last.view(torch.bfloat16)[..., 3]}
    if kind == "cut":
        d.reset_history()
    d.denoise_frame(s["frame"], s["out"])
    if case.get("export"):
        d.history_export(*s["state"])
        return {"rgb": s["out"], "history": s["state"][0], "moments": s["state"][1]}
    return s["out"]


# ---- what a pass cannot do without ---------------------------------------------------------------

TAP_OPS = 24           # operations of one edge-stopping tap: the normal, depth and luminance terms, the sums
KPN_MACS = 9 * (10 * 32 + 32 * 32 + 32 * 32 + 32 * 25)


def work(case):
    kind = case["kind"]
    if kind == "train":
        n = case["b"] * case["h"] * case["w"]
        # forward, data gradient (not of the first layer) and weight gradient; features, colours in
        macs = 3 * KPN_MACS - 9 * 10 * 32
        return {"bytes": n * (32 + 16 + 16) + 7 * 4 * svgf.KPN_PARAM_COUNT, "flops": n * (2 * macs + 2 * 2 * 25 * 8)}
    px = sum(w * h for w, h in _sizes(case))
    rec = 8 if case.get("precision", "fp32") != "fp32" else 16
    taps = 8 if case["mode"] == "separable" else 24
    passes = 5
    b, f = 12 + 16 + 8 + 4, 150                # noisy colour, G-buffer, motion, roughness; the temporal stage
    b += 2 * rec                               # history and moments out
    b += rec if kind == "stages" else 16       # the result
    if kind in HISTORY_KINDS:
        b += 16 + 2 * rec                      # previous G-buffer, history and moments in
    if kind == "cut":
        f += 48 * TAP_OPS                      # the 7x7 variance estimate
    if kind == "learned":
        b += 12
        f += taps * TAP_OPS + 2 * KPN_MACS + 2 * 25 * 7
    else:
        f += passes * taps * TAP_OPS
    if case.get("export"):
        b += 2 * 16
    return {"bytes": px * b * case.get("frames", 1), "flops": px * f * case.get("frames", 1)}


# ---- the same in 64 bits -------------------------------------------------------------------------

def _luma(c):
    return LUMA[0] * c[0] + LUMA[1] * c[1] + LUMA[2] * c[2]


def _grad(z):
    """Central-difference depth gradient, one-sided at the borders, 0 along an axis of extent 1."""
    gx, gy = torch.zeros_like(z), torch.zeros_like(z)
    if z.shape[1] > 1:
        gx[:, 1:-1] = 0.5 * (z[:, 2:] - z[:, :-2])
        gx[:, 0], gx[:, -1] = z[:, 1] - z[:, 0], z[:, -1] - z[:, -2]
    if z.shape[0] > 1:
        gy[1:-1] = 0.5 * (z[2:] - z[:-2])
        gy[0], gy[-1] = z[1] - z[0], z[-1] - z[-2]
    return gx, gy


def _padded(x, r):
    return F.pad(x[None], (r, r, r, r))[0]


def _edge(g, gq, grad, dx, dy, c):
    """Normal and depth weight of the tap at offset (dx, dy) as its logarithm."""
    t = 0.5 * ((g[0] - gq[0]) ** 2 + (g[1] - gq[1]) ** 2 + (g[2] - gq[2]) ** 2)
    e = c["sigma_n"] * torch.log1p(-torch.clamp(t, max=1.0))
    return e - (gq[3] - g[3]).abs() / (c["sigma_z"] * (grad[0] * dx + grad[1] * dy).abs() + c["eps"])


def _box(x, n):
    """Mean over the in-image 3x3 neighbourhood (n: the number of its pixels)."""
    p = _padded(x, 1)
    h, w = x.shape[-2:]
    return sum(p[:, 1 + j:1 + j + h, 1 + i:1 + i + w] for j in (-1, 0, 1) for i in (-1, 0, 1)) / n


def _temporal(f, prev_g, hist, mom, c):
    """Accumulated colour and variance [4, H, W] and moments [3, H, W] (mean, variance, length)."""
    noisy, g, mv = f["noisy"], f["g"], f["mv"]
    h, w = g.shape[-2:]
    col = noisy / (1.0 + c["luma_k"] * _luma(noisy)) if c["tonemap"] else noisy
    yy, xx = torch.meshgrid(torch.arange(h, device=g.device), torch.arange(w, device=g.device), indexing="ij")
    zero = torch.zeros_like(g[0])
    valid = torch.zeros_like(g[0], dtype=torch.bool)
    hc, m1, s2, n = torch.zeros_like(col), zero, zero, zero
    if hist is not None:
        fl = torch.floor(-mv)
        fr = -mv - fl
        bx, by = xx + fl[0].long(), yy + fl[1].long()
        taps = []
        for j in (0, 1):
            for i in (0, 1):
                tx, ty = bx + i, by + j
                wt = (fr[0] if i else 1 - fr[0]) * (fr[1] if j else 1 - fr[1])
                ok = (tx >= 0) & (ty >= 0) & (tx < w) & (ty < h) & (wt > 0)
                q = (ty.clamp(0, h - 1) * w + tx.clamp(0, w - 1)).reshape(-1)
                at = lambda img: img.reshape(img.shape[0], -1)[:, q].reshape(img.shape[0], h, w)
                gp = at(prev_g)
                ok &= (gp[3] - g[3]).abs() <= c["depth_rel_tol"] * g[3]
                ok &= ((g[:3] - gp[:3]) ** 2).sum(0) <= 2.0 * (1.0 - c["normal_cos_tol"])
                taps.append((torch.where(ok, wt, zero), at(hist), at(mom)))
        sw = sum(t[0] for t in taps)
        valid = sw >= c["disocclusion_weight"]
        rs = torch.where(valid, 1.0 / sw.clamp(min=1e-300), zero)
        hc = sum(t[0] * t[1][:3] for t in taps) * rs
        m1 = sum(t[0] * t[2][0] for t in taps) * rs
        s2 = sum(t[0] * (t[2][1] + (t[2][0] - m1) ** 2) for t in taps) * rs
        n = torch.stack([torch.where(t[0] > 0, t[2][2], zero) for t in taps]).amax(0)
    if c["clamp_enable"]:
        cnt = _box(torch.ones_like(col[:1]), 1.0)
        mean = _box(col, cnt)
        p, pc = _padded(col, 1), _padded(torch.ones_like(col[:1]), 1)
        var = sum(((p[:, 1 + j:1 + j + h, 1 + i:1 + i + w] - mean) ** 2) * pc[:, 1 + j:1 + j + h, 1 + i:1 + i + w]
                  for j in (-1, 0, 1) for i in (-1, 0, 1)) / cnt
        ext = c["clamp_gamma"] * var.sqrt()
        dlt = hc - mean
        if c["rectify_mode"] == svgf.RECTIFY_CLIP:
            t = torch.where(dlt == 0, torch.zeros_like(dlt), dlt.abs() / ext).amax(0)
            hc = torch.where(t > 1, mean + dlt / t.clamp(min=1.0), hc)
        else:
            hc = torch.minimum(torch.maximum(hc, mean - ext), mean + ext)
    nn = torch.where(valid, (n + 1).clamp(max=c["max_history"]), torch.ones_like(n))
    a, am = (1.0 / nn).clamp(min=c["alpha"]), (1.0 / nn).clamp(min=c["alpha_moments"])
    out = torch.where(valid, hc + a * (col - hc), col)
    l = _luma(col)
    dl = l - m1
    mu = torch.where(valid, m1 + am * dl, l)
    sv = torch.where(valid, (1 - am) * (s2 + am * dl * dl), zero)
    short = nn < c["min_temporal_frames"]
    var = torch.where(short, zero, sv.clamp(min=0))
    if bool(short.any()):
        r = c["spatial_var_radius"]
        pg, pm, inside = _padded(g, r), _padded(torch.stack([mu, sv]), r), _padded(torch.ones_like(g[:1]), r)[0]
        grad = _grad(g[3])
        cut = lambda x, i, j: x[..., r + j:r + j + h, r + i:r + i + w]

        def weight(i, j):
            wt = torch.exp(_edge(g, cut(pg, i, j), grad, float(i), float(j), c))
            return wt * cut(inside, i, j)
        offs = [(i, j) for j in range(-r, r + 1) for i in range(-r, r + 1)]
        ws = sm = ss = torch.zeros_like(zero)
        for i, j in offs:
            wt, q = weight(i, j), cut(pm, i, j)
            ws, sm, ss = ws + wt, sm + wt * q[0], ss + wt * q[1]
        mean = sm / ws
        vv = torch.zeros_like(zero)
        for i, j in offs:
            vv = vv + weight(i, j) * (cut(pm, i, j)[0] - mean) ** 2
        var = torch.where(short, ((ss + vv) / ws).clamp(min=0), var)
    return torch.cat([out, var[None]]), torch.stack([mu, sv, nn])


def _filter(cv, guide_var, f, step, offs, c, with_var):
    """One weighted pass over the tap offsets `offs` at dilation `step`."""
    g, grad, l = f["g"], f["grad"], _luma(cv)
    h, w = l.shape
    r = 2 * step
    pc, pg, inside = _padded(cv, r), _padded(g, r), _padded(torch.ones_like(g[:1]), r)[0]
    b3 = {0: 0.375, 1: 0.25, 2: 0.0625}
    den = c["sigma_l"] * guide_var.sqrt() + c["eps"]
    sw, sc, sv = torch.zeros_like(l), torch.zeros_like(cv[:3]), torch.zeros_like(l)
    for j, k in offs:
        dx, dy = j * step, k * step
        cut = lambda x: x[..., r + dy:r + dy + h, r + dx:r + dx + w]
        q = cut(pc)
        e = _edge(g, cut(pg), grad, float(dx), float(dy), c) - (_luma(q) - l).abs() / den
        hw = (b3[abs(j)] if any(o[0] for o in offs) else 1.0) * (b3[abs(k)] if any(o[1] for o in offs) else 1.0)
        wt = hw * torch.exp(e) * cut(inside)
        sw, sc, sv = sw + wt, sc + wt * q[:3], sv + wt * wt * q[3]
    return torch.cat([sc / sw, (sv / (sw * sw) if with_var else cv[3])[None]])


def _atrous(cv, f, it, c):
    # the luminance guide: [1 2 1] x [1 2 1] / 16 of the variance, in-image taps renormalised
    k3 = torch.tensor([0.25, 0.5, 0.25], dtype=torch.float64, device=cv.device)
    ker = (k3[:, None] * k3[None, :])[None, None]
    vf = F.conv2d(cv[3][None, None], ker, padding=1) / F.conv2d(torch.ones_like(cv[3])[None, None], ker, padding=1)
    vf = vf[0, 0].clamp(min=0)
    res = None
    for lvl in ((0, 1) if c["adaptive_start"] else (0,)):
        step = 1 << (it + lvl)
        if c["spatial_mode"] == svgf.SEPARABLE:
            o = _filter(cv, vf, f, step, [(j, 0) for j in range(-2, 3)], c, False)
        else:
            o = _filter(cv, vf, f, step, [(j, k) for k in range(-2, 3) for j in range(-2, 3)], c, True)
        res = o if res is None else torch.where(f["rough"] > c["roughness_threshold"], o, res)
    active = _budget(f, c) > it
    res = torch.where(active, res, cv)
    if c["spatial_mode"] == svgf.SEPARABLE:
        mid, res = res, None
        for lvl in ((0, 1) if c["adaptive_start"] else (0,)):
            o = _filter(mid, vf, f, 1 << (it + lvl), [(0, k) for k in range(-2, 3)], c, True)
            res = o if res is None else torch.where(f["rough"] > c["roughness_threshold"], o, res)
        res = torch.where(active, res, mid)
    return res


def _budget(f, c):
    full = torch.full_like(f["rough"], float(c["atrous_iters"]))
    if not c["iter_by_roughness"]:
        return full
    r = f["rough"]
    return torch.where(r <= c["iter_rough_t0"], full * 0 + c["iter_count0"],
                       torch.where(r <= c["iter_rough_t1"], full * 0 + c["iter_count1"], full))


def _inverse(cv, c):
    if not c["tonemap"]:
        return cv
    return torch.cat([cv[:3] / (1.0 - c["luma_k"] * _luma(cv)).clamp(min=1e-6), cv[3:]])


def _f64(x):
    t = torch.from_numpy(np.ascontiguousarray(x)).cuda().double()
    return t.permute(2, 0, 1).contiguous() if t.dim() == 3 else t


def _inputs64(f):
    g = _f64(f["gbuf_nz"])
    return {"noisy": _f64(f["noisy"]), "g": g, "mv": _f64(f["motion"]), "rough": _f64(f["roughness"]), "grad": _grad(g[3]),
            "albedo": _f64(f["albedo"])}


def _plain64(f, prev_g, hist, mom, c):
    """Every a-trous pass of one frame: accumulated colour, the passes' outputs, moments."""
    acc, mom = _temporal(f, prev_g, hist, mom, c)
    outs = [acc]
    for it in range(c["atrous_iters"]):
        outs.append(_atrous(outs[-1], f, it, c))
    return outs, mom


def _hwc(x):
    return x.permute(1, 2, 0).contiguous()


def _layers64(p):
    """The flat parameters as conv2d weights and biases."""
    out, o = [], 0
    for ci, co in zip(svgf.KPN_CIN, svgf.KPN_COUT):
        w = p[o:o + co * 9 * ci].reshape(co, 3, 3, ci).permute(0, 3, 1, 2)
        o += co * 9 * ci
        out.append((w, p[o:o + co]))
        o += co
    return out


def _apply64(k, c, d):
    """The per-pixel 5x5 kernels k [B, 25, H, W] applied to c [B, 3, H, W] at dilation d."""
    h, w = c.shape[-2:]
    p, ones = F.pad(c, (2 * d,) * 4), F.pad(torch.ones_like(c[:, :1]), (2 * d,) * 4)
    num = den = 0.0
    for i in range(25):
        y, x = (i // 5) * d, (i % 5) * d
        num = num + k[:, i:i + 1] * p[..., y:y + h, x:x + w]
        den = den + k[:, i:i + 1] * ones[..., y:y + h, x:x + w]
    return num / den


def _network64(x, p):
    for l, (w, b) in enumerate(_layers64(p)):
        x = F.conv2d(x, w, b, padding=1)
        x = F.relu(x) if l < 3 else x
    return torch.softmax(x, dim=1)


def _train64(case, seed):
    feats, c0, target = _crops(case, seed)
    p, m, v, _ = (torch.from_numpy(a).cuda().double() if isinstance(a, np.ndarray) else a for a in _checkpoint(seed))
    x = feats[..., :10].double().permute(0, 3, 1, 2)
    c = c0[..., :3].double().permute(0, 3, 1, 2)
    t = target[..., :3].double().permute(0, 3, 1, 2)
    q = p.clone().requires_grad_(True)
    k = _network64(x, q)
    loss = ((_apply64(k, _apply64(k, c, 1), 4) - t) ** 2).mean()
    loss.backward()
    g, n = q.grad, ADAM_STEPS + 1
    m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    p = p - LR * (m / (1 - 0.9 ** n)) / ((v / (1 - 0.999 ** n)).sqrt() + 1e-8)
    return {"loss": loss.detach().reshape(1), "grad": g, "params": p, "adam_m": m, "adam_v": v}


def _learned64(case, seed, f, outs, c):
    cv, g = outs[1], f["g"]
    s = g[:3].abs().sum(0)
    o = g[:2] / s
    folded = (1.0 - o.flip(0).abs()) * torch.where(o >= 0, 1.0, -1.0)
    o = torch.where(g[2] < 0, folded, o)
    x = torch.cat([cv[:3], cv[3:].clamp(min=0).sqrt(), g[3:].clamp(min=1e-20).log2(), o, f["albedo"]])
    k = _network64(x[None], torch.from_numpy(_weights(seed)).cuda().double())
    c1 = _apply64(k, cv[None, :3], 1)
    res = _inverse(torch.cat([_apply64(k, c1, 4)[0], cv[3:]]), c)
    n = 0
    if case["fallback"]:
        l = _luma(cv)
        h, w = l.shape
        for y in range(0, h, 32):
            for x0 in range(0, w, 32):
                if float(l[y:y + 32, x0:x0 + 32].std(unbiased=False)) > FALLBACK_STD:
                    res[:, y:y + 32, x0:x0 + 32] = _inverse(outs[-1][:, y:y + 32, x0:x0 + 32], c)
                    n += 1
    return {"rgb": _hwc(res), "fallback_tiles": n}


def exact(case, seed):
    kind = case["kind"]
    with torch.backends.cudnn.flags(enabled=False):    # plain FP64 convolutions
        if kind == "train":
            return _train64(case, seed)
        res = []
        for i, (w, h) in enumerate(_sizes(case)):
            cfg = _config(case, w, h)
            c = {k: (float(np.float32(v)) if isinstance(v, float) else v) for k, v in vars(cfg).items()}
            fs, prev = _frames(case, seed, w, h, case.get("frames", 1), i)
            hist = mom = prev_g = None
            if kind in HISTORY_KINDS:
                hist, mom = (_f64(a) for a in _history(case, seed + i, prev, cfg.tonemap))
                prev_g = _f64(prev["gbuf_nz"])
            for fr in fs:
                f = _inputs64(fr)
                outs, mom = _plain64(f, prev_g, hist, mom, c)
                prev_g, hist = f["g"], outs[1]          # the first pass's output is the colour history
                if kind == "learned":
                    return _learned64(case, seed, f, outs, c)
                if kind == "stages":
                    return {"colour": _hwc(outs[-1][:3]), "variance": outs[-1][3]}
                rgb = _hwc(_inverse(outs[-1], c))
                if case.get("export"):
                    pad = lambda x: _hwc(torch.cat([x[:3], torch.zeros_like(x[:1])]))
                    return {"rgb": rgb, "history": pad(hist), "moments": pad(mom)}
                res.append(rgb.cpu() if kind == "host" else rgb)
    return res if kind in ("batch", "host") else res[0]
