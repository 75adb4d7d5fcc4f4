"""The framework's performance cases: what its users have it do, pass by pass.

A pass is one frame (of one stream, or of every stream of a batch) pushed
through the public entry points into reservoirs that already hold a running
session's history. Frames, gazes, motion and depth are made on the GPU from
the seed: a broadband scene of gratings and hard-edged disks, foveated around
a gaze that fixates and jitters.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

import paper_2510_03964_gb300 as wrs

DISTINCT = 8  # frames of a session, pushed cyclically: two fixations of four jittered gazes


def _case(name, kind, width, height, K, fp16=False, bias=1, rule=0, flush=False, age=0,
          filter="bilinear"):
    return {"name": name, "kind": kind, "width": width, "height": height, "K": K, "fp16": fp16,
            "bias": bias, "rule": rule, "flush": flush, "age": age, "filter": filter}


def listed():
    return [
        # a thumbnail-sized stream: the smallest call, where launches and latency count
        _case("tiny_k4", "push", 256, 256, 4, age=8),
        # one HD stream, four slots, FP32 colour
        _case("hd_k4", "push", 1920, 1080, 4, age=120),
        # the headline: one 4K stream, eight slots, FP32 colour
        _case("uhd_k8", "push", 3840, 2160, 8, age=240),
        # the same stream with FP16 slot colours (what serving stores)
        _case("uhd_k8_fp16", "push", 3840, 2160, 8, fp16=True, age=240),
        # the paper's own reservoir: one slot, the literal n = 1 rule, at its display's size
        _case("uhd_k1_literal", "push", 3840, 2160, 1, rule=1, age=240),
        # one eye of a headset under the full temporal bias (lightness difference)
        _case("vr_k8_fp16_bias2", "push", 2064, 2208, 8, fp16=True, bias=2, age=120),
        # a desktop window of odd size, with disoccluded pixels flushed
        _case("window_k4_flush", "push", 1365, 767, 4, flush=True, age=60),
        # a moving camera: every reservoir gathered through motion vectors and a depth test
        _case("uhd_pan_k8", "reproject", 3840, 2160, 8, age=60),
        # the foveation post-process alone: mip levels of a new image, then the foveated frame
        _case("uhd_foveate", "foveate", 3840, 2160, 0),
        # a rendered image foveated on read inside the update (the serving frame loop)
        _case("uhd_k8_fp16_foveated", "push_foveated", 3840, 2160, 8, fp16=True, age=120),
        # eight viewers of four resolutions and mixed slot counts in one batched launch
        _case("batch8_fp16", "batch", 3840, 2160, 8, fp16=True, age=60),
        # frames and results in pinned host memory, uploads and downloads overlapped
        _case("hd_k4_host", "host", 1920, 1080, 4, age=16),
    ]


def draw(rng):
    kind = rng.choice(["push"] * 6 + ["reproject", "foveate", "push_foveated", "batch", "host"])
    pixels = math.exp(rng.uniform(math.log(128 * 96), math.log(3840 * 2160)))
    aspect = math.exp(rng.uniform(math.log(0.75), math.log(2.0)))
    w = max(64, min(4096, round(math.sqrt(pixels * aspect))))
    h = max(48, min(2304, int(pixels / w)))
    if kind in ("push_foveated", "batch") or rng.random() < 0.5:
        w = (w + 3) // 4 * 4  # those two calls take widths divisible by 4; others any width
    if w * h > 3840 * 2160:
        h = 3840 * 2160 // w
    c = _case("", kind, w, h, 0)
    del c["name"]
    if kind == "foveate":
        c["filter"] = rng.choice(["box", "bilinear"])
        return c
    c["K"] = rng.choice([1, 2, 3, 4, 4, 4, 5, 6, 8, 8, 8] + ([16] if kind == "push" else []))
    c["rule"] = 1 if c["K"] == 1 and rng.random() < 0.6 else 0
    c["fp16"] = kind == "batch" or rng.random() < 0.5  # batches are the serving mix: FP16 colour
    c["bias"] = rng.choice([0, 1, 1, 1, 1, 2])
    c["flush"] = kind in ("push", "reproject") and rng.random() < 0.25
    c["filter"] = rng.choice(["box", "bilinear"])
    c["age"] = round(math.exp(rng.uniform(math.log(8), math.log(120))))
    return c


# ---------------------------------------------------------------- inputs

def _radii(w):
    r = float(max(8, round(w * 0.0525)))  # 200 px of 3840: the fovea, then 2.5 and 5 times it
    return (r, 2.5 * r, 5.0 * r)


def _gazes(w, h, seed):
    g = np.random.Generator(np.random.Philox(key=[seed & 0xFFFFFFFF, 2]))
    out = []
    for _ in range(2):
        fx, fy = g.uniform(0.2, 0.8) * w, g.uniform(0.2, 0.8) * h
        for _ in range(DISTINCT // 2):
            jx, jy = g.normal(0.0, 0.0016 * w, 2)
            out.append((float(np.float32(fx + jx)), float(np.float32(fy + jy))))
    return out


class _Scene:
    """Gratings at depth 10 behind disks at depths 2 to 6, seen by a camera
    that pans 3.25 px right and 0.75 px down per frame."""

    def __init__(self, w, h, seed):
        g = np.random.Generator(np.random.Philox(key=[seed & 0xFFFFFFFF, 1]))
        self.w, self.h, self.size = w, h, float(max(w, h))
        self.theta, self.freq = g.random(16) * np.pi, 2.0 + 46.0 * g.random(16)
        self.phase, self.amp = g.random(16) * 2.0 * np.pi, g.random((16, 3)) * 2.0 - 1.0
        self.c = g.random((8, 2)) * np.array([w, h])
        self.r, self.z = (0.03 + 0.09 * g.random(8)) * self.size, np.sort(2.0 + 4.0 * g.random(8))[::-1]
        self.col = g.random((8, 3))

    def view(self, t):
        """(image [H][W][3], motion [H][W][2], depth [H][W]) of frame t."""
        cx, cy = 3.25 * t, 0.75 * t
        xs = torch.arange(self.w, device="cuda", dtype=torch.float32)[None, :] + 0.5
        ys = torch.arange(self.h, device="cuda", dtype=torch.float32)[:, None] + 0.5
        img = torch.zeros((3, self.h, self.w), device="cuda")
        for i in range(16):
            k = 2.0 * math.pi * self.freq[i] / self.size
            s = torch.sin((k * math.cos(self.theta[i])) * (xs + cx) + (k * math.sin(self.theta[i])) * (ys + cy)
                          + float(self.phase[i]))
            for ch in range(3):
                img[ch].add_(s, alpha=float(self.amp[i, ch]))
        total = torch.tensor(np.abs(self.amp).sum(0), device="cuda", dtype=torch.float32)[:, None, None]
        img = (img + total) / (2.0 * total)
        depth = torch.full((self.h, self.w), 10.0, device="cuda")
        for i in range(8):
            s = 10.0 / self.z[i]
            dx, dy = (self.c[i, 0] - cx * s) % self.w, (self.c[i, 1] - cy * s) % self.h
            inside = (xs - dx) ** 2 + (ys - dy) ** 2 <= float(self.r[i]) ** 2
            colour = torch.tensor(self.col[i], device="cuda", dtype=torch.float32)[:, None, None]
            img = torch.where(inside, colour, img)
            depth = torch.where(inside, float(self.z[i]), depth)
        scale = 10.0 / depth
        motion = torch.stack((-3.25 * scale, -0.75 * scale), dim=-1)
        return img.clamp_(0.0, 1.0).permute(1, 2, 0).contiguous(), motion.contiguous(), depth


def _levels(w, h, gaze):
    """Ring level of every pixel."""
    xs = torch.arange(w, device="cuda", dtype=torch.float32)[None, :] + 0.5 - gaze[0]
    ys = torch.arange(h, device="cuda", dtype=torch.float32)[:, None] + 0.5 - gaze[1]
    d2 = xs * xs + ys * ys
    return sum((d2 > float(np.float32(r) * np.float32(r))).to(torch.uint8) for r in _radii(w))


def _means(img, level, dtype=torch.float32):
    """Block means [3][hb][wb] of one mip level."""
    b = 1 << level
    return F.avg_pool2d(img.to(dtype).permute(2, 0, 1)[None], b, b, ceil_mode=True, count_include_pad=False)[0]


def _shown(means, level, w, h, filter):
    """A level's means at full resolution, [3][h][w]."""
    if filter == "box":
        return means.repeat_interleave(1 << level, 1)[:, :h].repeat_interleave(1 << level, 2)[:, :, :w]

    def at(n, nb):
        u = ((torch.arange(n, device="cuda", dtype=means.dtype) + 0.5) / (1 << level) - 0.5).clamp_(0, nb - 1)
        i = u.floor().long()
        return i, (i + 1).clamp_(max=nb - 1), u - i

    x0, x1, fx = at(w, means.shape[2])
    y0, y1, fy = at(h, means.shape[1])
    rows = means[:, :, x0] * (1 - fx) + means[:, :, x1] * fx
    return rows[:, y0] * (1 - fy)[:, None] + rows[:, y1] * fy[:, None]


def _foveated(img, gaze, filter="box", dtype=torch.float32):
    h, w = img.shape[:2]
    lev = _levels(w, h, gaze)
    out = img.to(dtype)
    for L in (1, 2, 3):
        out = torch.where((lev == L)[..., None], _shown(_means(img, L, dtype), L, w, h, filter).permute(1, 2, 0), out)
    return out.contiguous()


def _flush_map(w, h, i):
    """0xFF in a band behind a moving object, 0 elsewhere."""
    m = torch.zeros((h, w), dtype=torch.uint8, device="cuda")
    x = (i * w) // DISTINCT
    m[h // 4: h // 4 + h // 2, x: x + max(1, w // 32)] = 0xFF
    return m


_CLASSES = ((3840, 2160), (2064, 2208), (1440, 1600), (1920, 1080))


def _streams(c):
    """(width, height, K) of the case's streams: one, or a batch's two of each
    resolution with K and 4 slots, scaled to the case's size."""
    if c["kind"] != "batch":
        return [(c["width"], c["height"], c["K"])]
    fx, fy = c["width"] / 3840.0, c["height"] / 2160.0
    out = []
    for w, h in _CLASSES:
        size = (max(4, round(w * fx / 4) * 4), max(1, round(h * fy)))
        out += [(*size, c["K"]), (*size, min(4, c["K"]))]
    return out


def _inputs(c, i, seed):
    """What stream i is fed: per frame of its cycle the frame (or the rendered
    image), gaze, flush map, motion, depth and previous depth."""
    w, h, _ = _streams(c)[i]
    scene, gazes = _Scene(w, h, seed * 64 + i), _gazes(w, h, seed * 64 + i)
    cycle, before, img = [], None, None
    if c["kind"] == "reproject":
        before = scene.view(-1)[2]
    for d in range(DISTINCT):
        f = {"gaze": gazes[d], "fov": _flush_map(w, h, d) if c["flush"] else None}
        if c["kind"] == "reproject":
            view, f["motion"], f["depth"] = scene.view(d)
            f["prev_depth"], before = before, f["depth"]
            f["frame"] = _foveated(view, gazes[d])
        elif c["kind"] in ("foveate", "push_foveated"):
            f["frame"] = img = scene.view(d)[0] if d % 2 == 0 else img  # a new image every other frame
        else:
            img = scene.view(0)[0] if img is None else img
            f["frame"] = _foveated(img, gazes[d])
        cycle.append(f)
    return cycle


# ---------------------------------------------------------------- the cases

def _planes(c, st, buf, K):
    """The stream's reservoirs as views of its state buffer (wrs_state_layout)."""
    lay, hw = st.layout, st.width * st.height
    pl = lay.plane_px

    def view(off, n, item, dtype, width=1):
        return buf[off: off + n * pl * item].view(dtype).view(n, pl, width)[:, :hw]

    out = {"W": view(lay.W_off, 1, 4, torch.float32), "idx": view(lay.idx_off, K, 4, torch.int32)}
    if not c["rule"]:  # the literal rule has no keys and no bias product
        out["P"] = view(lay.P_off, 1, 4, torch.float32)
        out["key"] = view(lay.key_off, K, 4, torch.float32)
    if c["fp16"]:  # colour halves and the weight's two halves, as bits
        out["rec"] = view(lay.col_off, K, 8, torch.int16, 4)
        out["wt_lo"] = view(lay.wt_off, K, 2, torch.int16)
    else:
        out["rec"] = view(lay.col_off, K, 16, torch.float32, 4)
    return out


def prepare(case, seed):
    c, s = case, {"case": case, "t": 0, "streams": [], "cycle": [], "out": [], "planes": []}
    for i, (w, h, K) in enumerate(_streams(c)):
        s["cycle"].append(_inputs(c, i, seed))
        if c["kind"] == "foveate":
            continue
        st = wrs.Stream(w, h, K, _radii(w)[0], seed=seed, stream_id=i, color_fp16=c["fp16"],
                        temporal_bias=c["bias"], update_rule=c["rule"])
        s["streams"].append(st)
        s["out"].append(torch.empty((h, w, 3), device="cuda"))
        s["planes"].append([_planes(c, st, st.state, K)])
    if c["kind"] == "reproject":
        st = s["streams"][0]
        st.set_reprojection_buffer()
        s["planes"][0].append(_planes(c, st, st.spare, c["K"]))  # frames alternate between the two
    elif c["kind"] in ("foveate", "push_foveated"):
        cyc = s["cycle"][0]
        s["fov"] = [wrs.Foveation(f["frame"], _radii(c["width"]), filter=c["filter"]) if d % 2 == 0 else None
                    for d, f in enumerate(cyc)]
        s["fov"] = [s["fov"][d // 2 * 2] for d in range(DISTINCT)]
        s["mips"] = [wrs.mip_levels(f.mip, c["width"], c["height"], 4) for f in s["fov"]]
        if c["kind"] == "foveate":
            s["out"] = [torch.empty((c["height"], c["width"], 3), device="cuda")]
            s["ring"] = torch.empty((c["height"], c["width"]), dtype=torch.uint8, device="cuda")
    elif c["kind"] == "batch":
        s["batch"] = wrs.Batch(len(s["streams"]))
    elif c["kind"] == "host":
        s["pipe"] = wrs.HostPipeline(s["streams"][0])
        for f in s["cycle"][0]:
            f["frame"] = f["frame"].cpu().pin_memory()
        s["out"] = [torch.empty((c["height"], c["width"], 3)).pin_memory() for _ in range(4)]
        torch.cuda.synchronize()  # the pipeline runs on streams of its own
    for _ in range(c["age"]):
        run(s)
    return s


def run(s):
    c, t = s["case"], s["t"]
    s["t"] = t + 1
    d = t % DISTINCT
    kind, f = c["kind"], s["cycle"][0][d]
    if kind == "foveate":
        fov = s["fov"][d]
        fov.rebuild()
        fov.frame(f["gaze"], out=s["out"][0], ring_map=s["ring"])
        return {"frame": s["out"][0], "ring": s["ring"], "mip": s["mips"][d]}
    if kind == "batch":
        fs = [cyc[d] for cyc in s["cycle"]]
        s["batch"].push(s["streams"], [x["frame"] for x in fs], [x["gaze"] for x in fs], outs=s["out"])
        return {"out": s["out"], "state": [p[0] for p in s["planes"]]}
    st, out = s["streams"][0], s["out"][0]
    if kind == "push":
        st.push_frame(f["frame"], f["gaze"], fov_map=f["fov"], out=out)
    elif kind == "reproject":
        st.push_frame_reproject(f["frame"], f["gaze"], f["motion"], f["depth"], f["prev_depth"], 0.05,
                                fov_map=f["fov"], out=out)
        return {"out": out, "state": s["planes"][0][s["t"] % 2]}
    elif kind == "push_foveated":
        s["fov"][d].rebuild()
        st.push_foveated(s["fov"][d], f["gaze"], out=out)
        return {"out": out, "state": s["planes"][0][0], "mip": s["mips"][d]}
    elif kind == "host":
        out = s["out"][t % 4]
        s["pipe"].push(f["frame"], f["gaze"], out)
    return {"out": out, "state": s["planes"][0][0]}


def _rate(c, K):
    """Share of pixels whose reservoir takes the new sample at the case's age:
    K slots against a biased weight sum of about sqrt(2 t) samples."""
    t = c["age"] + 1.0
    return min(1.0, K / (1.0 + (math.sqrt(2.0 * t) if c["bias"] else t)))


def work(case):
    c, b, n = case, 0.0, 0.0
    for w, h, K in _streams(c):
        px = float(w * h)
        if c["kind"] in ("foveate", "push_foveated"):
            b += px * (12.0 + 16.0 * (1 / 4 + 1 / 16 + 1 / 64))  # the image read, three levels written
            n += px * 16.0
        if c["kind"] == "foveate":
            b += px * 13.0  # frame and ring map written
            n += px * 40.0
            continue
        rec = 10.0 if c["fp16"] else 16.0
        key = 0.0 if c["rule"] else 4.0
        sums = 8.0 if c["rule"] else 16.0  # W (and P) read and written
        b += px * (12.0 + sums + (1.0 if c["flush"] else 0.0))  # output written
        if c["kind"] != "push_foveated":
            b += px * 12.0  # frame read
        else:
            n += px * 40.0  # foveated from the image above
        if c["kind"] == "reproject":
            b += px * (2.0 * K * (rec + key + 4.0) + 16.0)  # every slot read and written; motion, depths
        else:
            b += px * (K * (rec + key) + _rate(c, K) * (rec + key + 4.0))
        n += px * (120.0 + 12.0 * K + (150.0 if c["bias"] == 2 else 0.0))
    return {"bytes": b, "flops": n}


# ---------------------------------------------------------------- the same in 64 bits

def _uniforms(hw, t, stream_id, seed):
    """Philox4x32-10: counter (pixel / 4, t, stream, 0), key the seed; word pixel % 4."""
    m = 0xFFFFFFFF
    c0 = torch.arange((hw + 3) // 4, device="cuda", dtype=torch.int64)
    c1, c2, c3 = torch.full_like(c0, t), torch.full_like(c0, stream_id), torch.zeros_like(c0)
    k0, k1 = seed & m, (seed >> 32) & m
    for _ in range(10):
        a, b = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((b >> 32) & m) ^ c1 ^ k0, b & m, ((a >> 32) & m) ^ c3 ^ k1, a & m
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    x = torch.stack((c0, c1, c2, c3), dim=1).reshape(-1)[:hw]
    return ((x >> 8) | 1).double() * 2.0 ** -24


def _density(e):
    q = (1.0 + e / 1.058) ** 2
    return (0.9851 + (1.0 - 0.9851) * torch.exp(-e / 22.14) * q) / (q * (1.0 + e / 41.03))


def _weights(w, h, gaze, r_f):
    x = torch.arange(w, device="cuda", dtype=torch.float64)[None, :] + 0.5 - gaze[0]
    y = torch.arange(h, device="cuda", dtype=torch.float64)[:, None] + 0.5 - gaze[1]
    d = torch.sqrt(x * x + y * y)
    edge = _density(torch.tensor(2.5, dtype=torch.float64, device="cuda"))
    far = (_density((d * (2.5 / r_f)).clamp_(max=180.0)) / edge).clamp_(max=1.0)
    return torch.where(d <= r_f, 1.0, far).reshape(-1)


def _lightness(rgb):
    y = (0.2126 * rgb[..., 0] + 0.7152 * rgb[..., 1] + 0.0722 * rgb[..., 2]).clamp_(0.0, 1.0)
    return torch.where(y > 216 / 24389, 116.0 * y.clamp(min=1e-30) ** (1 / 3) - 16.0, (24389 / 27) * y)


def _resolve(rec):
    """[hw][3] weighted mean of the slots of rec [K][hw][4] = {w, r, g, b}."""
    num = (rec[..., :1] * rec[..., 1:]).sum(0)
    den = rec[..., :1].sum(0)
    return torch.where(den > 0, num / torch.where(den > 0, den, 1.0), 0.0)


def _session(c, i, seed):
    """Stream i's reservoirs and resolved frame after its history and one pass."""
    w, h, K = _streams(c)[i]
    hw, r_f = w * h, _radii(w)[0]
    cycle = _inputs(c, i, seed)
    f64 = {"device": "cuda", "dtype": torch.float64}
    W, P = torch.zeros(hw, **f64), torch.ones(hw, **f64)
    key, rec = torch.full((K, hw), math.inf, **f64), torch.zeros((K, hw, 4), **f64)
    shown = {}
    for t in range(c["age"] + 1):
        d = t % DISTINCT
        f = cycle[d]
        if d not in shown:
            frame = f["frame"] if c["kind"] != "push_foveated" else _foveated(f["frame"], f["gaze"], c["filter"],
                                                                             torch.float64)
            shown[d] = frame.double().reshape(hw, 3)
        rgb = shown[d]
        drop = torch.zeros(hw, dtype=torch.bool, device="cuda") if f["fov"] is None else f["fov"].reshape(-1) == 0xFF
        if c["kind"] == "reproject":
            x = torch.arange(w, device="cuda", dtype=torch.float32)[None, :] + 0.5 - f["motion"][..., 0]
            y = torch.arange(h, device="cuda", dtype=torch.float32)[:, None] + 0.5 - f["motion"][..., 1]
            ok = ((x >= 0) & (x < w) & (y >= 0) & (y < h)).reshape(-1)
            q = (y.floor().long().clamp_(0, h - 1) * w + x.floor().long().clamp_(0, w - 1)).reshape(-1)
            q = torch.where(ok, q, torch.arange(hw, device="cuda"))
            z, z0 = f["depth"].reshape(-1).double(), f["prev_depth"].reshape(-1).double()[q]
            drop = drop | ~ok | ((z0 - z).abs() > float(np.float32(0.05)) * z)
            W, P, key, rec = W[q], P[q], key[:, q], rec[:, q]
        wt = _weights(w, h, f["gaze"], r_f)
        u = _uniforms(hw, t, i, seed)
        factor = 1.0
        if c["bias"] == 2:
            old = rec[..., :1].sum(0)[:, 0] > 0
            dl = ((_lightness(_resolve(rec)) - _lightness(rgb)).abs() * 0.01).clamp_(max=1.0)
            factor = torch.where(old, 1.0 - dl, 1.0)
            drop = drop | ((factor <= 0) & (W > 0))
        W, P = torch.where(drop, 0.0, W), torch.where(drop, 1.0, P)
        key.masked_fill_(drop, math.inf)
        rec.masked_fill_(drop[:, None], 0.0)
        if c["bias"]:
            fade = torch.where(W > 0, W / (W + wt) * factor, 1.0)
            W, P = W * fade, P * fade
        if c["rule"]:
            take, at = u * (W + wt) > W, torch.zeros(hw, dtype=torch.int64, device="cuda")
        else:
            small = P < 2.0 ** -64
            P = torch.where(small, P * 2.0 ** 64, P)
            key = torch.where(small & torch.isfinite(key), (key * 2.0 ** 64).clamp(max=3.4028234663852886e38), key)
            new = -torch.log(u) / wt * P
            largest, at = key.max(dim=0)
            take = new < largest
        W = W + wt
        p = take.nonzero()[:, 0]
        colour = rgb[p].half().double() if c["fp16"] else rgb[p]
        rec[at[p], p] = torch.cat((wt[p, None], colour), dim=1)
        if not c["rule"]:
            key[at[p], p] = new[p]
    state = {"W": W.view(1, hw, 1), "idx": None, "rec": None if c["fp16"] else rec}
    if not c["rule"]:
        state.update(P=P.view(1, hw, 1), key=key.view(K, hw, 1))
    if c["fp16"]:
        state["wt_lo"] = None
    return _resolve(rec).view(h, w, 3), state


def exact(case, seed):
    c = case
    mip = None
    if c["kind"] in ("foveate", "push_foveated"):
        f = _inputs(c, 0, seed)[c["age"] % DISTINCT]
        mip = [F.pad(_means(f["frame"], L, torch.float64).permute(1, 2, 0), (0, 1)) for L in (1, 2, 3)]
    if c["kind"] == "foveate":
        return {"frame": _foveated(f["frame"], f["gaze"], c["filter"], torch.float64), "ring": None, "mip": mip}
    got = [_session(c, i, seed) for i in range(len(_streams(c)))]
    if c["kind"] == "batch":
        return {"out": [o for o, _ in got], "state": [s for _, s in got]}
    out = {"out": got[0][0], "state": got[0][1]}
    if mip is not None:
        out["mip"] = mip
    return out
