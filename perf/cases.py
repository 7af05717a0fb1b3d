"""Timed cases of the BDIS library: what its users have it do, by public entry point.

Inputs are seeded surgical-like stereo pairs made on the GPU (the recipe of
the repository's 640x480 workload: smoothed-noise texture with a shading
ramp, textureless rectangles, dark ellipses, a plane-plus-bumps disparity
field of a tenth of the width, sensor noise, specular highlights in the right
view only).

A case is a dict of plain values; `kind` names the entry point:
  match    Matcher.match / match_warm / match_learned on device images;
  host     Matcher.match_host on pinned host images;
  plan     Plan.run over groups of several image sizes (one CUDA graph);
  stages   the method level by level through the step entry points;
  train    ProposalNet.gradient: loss and weight gradient of the proposal net.
"""
import math
import os

import numpy as np
import torch
import torch.nn.functional as F

import paper_2106_07136_gb300 as bd

DIS = 1  # BDIS_FUSION_DIS
BASE = dict(kind="match", start="plain", dtype="u8", w=640, h=480, count=1, ps=8, overlap=0.75,
            iters=12, coarsest=4, finest=0, window=5, step=0.5, gamma=0.75, normalize=1, fusion=0)


def _case(**kw):
    return dict(BASE, **kw)


def listed():
    return [
        # the smallest call: one 160x120 pair with half-overlapping patches (a
        # preview or a test image; launches and host time are what it costs)
        _case(name="small pair 160x120", w=160, h=120, overlap=0.5, iters=8, coarsest=2, gamma=0.25),
        # one camera frame at the paper's settings: the latency of a live loop
        _case(name="one pair 640x480"),
        # offline throughput at the paper's settings, the repository's benchmark batch
        _case(name="batch 512 x 640x480", count=512),
        # the paper's other patch size, an ordinary batch
        _case(name="patch 12, 64 x 640x480", ps=12, count=64),
        # the baseline fusion the paper compares against (inverse squared residual)
        _case(name="DIS fusion, 64 x 640x480", fusion=DIS, count=64),
        # settings off the paper's: a patch size and window of the user's own,
        # float images of odd size, a half-size result brought to full size
        _case(name="own settings, 24 x 501x375 f32", w=501, h=375, count=24, dtype="f32", ps=10,
              overlap=0.6, iters=10, coarsest=3, finest=1, window=7, step=0.4, gamma=0.5),
        # streams of 1280x1024 video, each frame seeded by its stream's last map
        _case(name="video, 4 x 1280x1024", start="warm", w=1280, h=1024, count=4),
        # learned start with the fewer iterations it allows
        _case(name="learned, 64 x 640x480", start="learned", iters=5, count=64),
        # a batch of mixed sizes, the coarsest scale raised with the width
        _case(name="mixed sizes, 32 pairs", kind="plan",
              groups="320x240x8,640x480x12,1280x720x8,1920x1080x4"),
        # images that come from and go to host memory, one blocking call
        _case(name="host, 64 x 640x480", kind="host", count=64),
        # level by level with every per-patch output, as label making and
        # evaluation programs run the method (large, ragged images)
        _case(name="stages, 2 x 1917x1079", kind="stages", w=1917, h=1079, count=2),
        # one training batch of the proposal network on its pyramid level
        _case(name="train, 64 x 40x30", kind="train", w=40, h=30, count=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pairs(c):
    """[(width, height, count)] of a case."""
    if c["kind"] == "plan":
        return [tuple(int(v) for v in g.split("x")) for g in c["groups"].split(",")]
    return [(c["w"], c["h"], c["count"])]


def draw(rng):
    kind = rng.choice(["match"] * 6 + ["host", "plan", "stages", "train"])
    c = _case(kind=kind)
    if kind == "train":
        c.update(w=_log_int(rng, 20, 120), h=_log_int(rng, 15, 90))
        c["count"] = max(1, min(_log_int(rng, 1, 256), 300000 // (c["w"] * c["h"])))
        return c
    c.update(ps=rng.choice([8, 8, 8, 12, 12, 16, 6, 10]), overlap=rng.choice([0.75, 0.75, 0.5, 0.6]),
             iters=rng.randint(4, 12), gamma=rng.choice([0.25, 0.5, 0.75]))
    if rng.random() < 0.2:
        c.update(window=rng.choice([3, 7]), step=rng.choice([0.4, 0.5, 1.0]))
    if rng.random() < 0.15:
        c["fusion"] = DIS
    if kind == "match":
        c["start"] = rng.choice(["plain", "plain", "warm", "learned"])
    if kind in ("match", "stages") and rng.random() < 0.25:
        c["dtype"] = "f32"
    w = _log_int(rng, 160, 1920)
    h = max(120, int(w * rng.uniform(0.55, 0.85)))
    if rng.random() < 0.5:
        w, h = w // 16 * 16, h // 16 * 16
    # a drawn case stays under a quarter of the largest listed one's pixels
    most = 512 * 640 * 480 // (4 if c["ps"] in (8, 12, 16) and c["window"] == 5 else 16)
    count = max(1, min(_log_int(rng, 1, 192), most // (w * h)))
    c.update(w=w, h=h, count=count)
    top = max(l for l in range(6) if min(w, h) / 2 ** l >= 2 * c["ps"])
    c["coarsest"] = rng.randint(max(1, top - 2), max(1, top))
    if rng.random() < 0.2 and c["coarsest"] > 1:
        c["finest"] = 1
    if kind == "plan":
        c["groups"] = ",".join("%dx%dx%d" % (max(160, int(w * s)), max(120, int(h * s)),
                                             max(1, int(count / 4)))
                               for s in (1.0, rng.uniform(0.4, 0.9), rng.uniform(0.4, 0.9)))
    return c


# ------------------------------------------------------------------ inputs

def _rows_at(img, xs):
    """Linear reads of each row of img (B, H, W) at xs, clamped."""
    n = img.shape[-1]
    xs = xs.clamp(0.0, n - 1.0)
    i0 = xs.floor().clamp(max=n - 2).long()
    t = xs - i0
    return (1 - t) * torch.gather(img, 2, i0) + t * torch.gather(img, 2, i0 + 1)


def _blur(s, dim):
    """Gaussian of sigma 2 along one dimension (13 taps, wrapped), by shifted adds."""
    k = [math.exp(-i * i / 8.0) for i in range(-6, 7)]
    out = torch.zeros_like(s)
    for i, v in zip(range(-6, 7), k):
        out += s.roll(i, dim) * (v / sum(k))
    return out


def _make(seed, w, h, n):
    """n pairs of w x h: float views in 0..255 and the disparity on the left grid."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def u(lo, hi):
        return torch.rand(n, 1, 1, generator=g, device="cuda") * (hi - lo) + lo

    yy, xx = torch.meshgrid(torch.arange(h, device="cuda", dtype=torch.float32),
                            torch.arange(w, device="cuda", dtype=torch.float32), indexing="ij")
    scene = _blur(_blur(torch.rand(n, h, w, generator=g, device="cuda"), 2), 1)
    scene = (scene - scene.mean()) / scene.std() * 40.0 + 128.0 + xx / w * 40.0
    flat = torch.zeros(n, h, w, dtype=torch.bool, device="cuda")
    for _ in range(9):
        rw, rh = u(0.08, 0.22) * w, u(0.08, 0.22) * h
        x0, y0 = u(0, 1) * (w - rw), u(0, 1) * (h - rh)
        inside = (xx >= x0) & (xx < x0 + rw) & (yy >= y0) & (yy < y0 + rh)
        scene = torch.where(inside, u(60.0, 200.0), scene)
        flat |= inside
    for _ in range(2):
        cx, cy, ax, ay = u(0, w), u(0, h), u(0.1, 0.22) * w, u(0.1, 0.22) * h
        scene = torch.where(((xx - cx) / ax) ** 2 + ((yy - cy) / ay) ** 2 <= 1.0, scene * 0.2, scene)
    dmax = w / 10.0
    lo, hi = u(0.1, 0.3) * dmax, u(0.45, 0.65) * dmax
    d = lo + (hi - lo) * xx / w + u(-0.1, 0.1) * dmax * (yy / h - 0.5)
    for _ in range(6):
        cx, cy, s = u(0, w), u(0, h), u(0.05, 0.12) * w
        d = d + u(-0.2, 0.2) * dmax * torch.exp(-((xx - cx) ** 2 + (yy - cy) ** 2) / (2 * s * s))
    d = d.clamp(0.0, dmax)

    def noise(std):
        return torch.randn(n, h, w, generator=g, device="cuda") * std

    x = xx.expand(n, h, w)
    right = _rows_at(scene, x + d) + noise(2.0)
    left = scene + noise(1.0) * flat
    for _ in range(10):
        cx, cy, s = u(0, w), u(0, h), u(3.0, 13.0)
        right = right + 400.0 * torch.exp(-((xx - cx) ** 2 + (yy - cy) ** 2) / (2 * s * s))
    dl = d
    for _ in range(6):
        dl = _rows_at(d, x - dl)
    return left.clamp(0, 255), right.clamp(0, 255), dl


def _images(case, seed, w, h, n, disparity=False):
    """(left, right[, last frame's map]) on the GPU, made a few pairs at a time."""
    dt = torch.uint8 if case["dtype"] == "u8" else torch.float32
    left = torch.empty(n, h, w, dtype=dt, device="cuda")
    right = torch.empty_like(left)
    prev = torch.empty(n, h, w, device="cuda") if disparity else None
    step = max(1, (64 << 20) // (w * h * 8))
    for i in range(0, n, step):
        k = min(step, n - i)
        a, b, d = _make((seed * 1000003 + i * 7919 + w) % (1 << 40), w, h, k)
        if dt == torch.uint8:
            a, b = a.round(), b.round()
        left[i:i + k] = a.to(dt)
        right[i:i + k] = b.to(dt)
        if disparity:
            # what the last frame left behind: the field moved by a pixel or
            # two, not estimated where the match fell outside the right view
            p = d.roll((2, 1), (2, 1)) + 0.7
            x = torch.arange(w, device="cuda", dtype=torch.float32)
            prev[i:i + k] = torch.where(x - p < 0, torch.full_like(p, float("nan")), p)
    return left, right, prev


def _params(case):
    return bd.default_params(patch_size=case["ps"], overlap=case["overlap"],
                             iterations=case["iters"], coarsest_scale=case["coarsest"],
                             finest_scale=case["finest"], window_samples=case["window"],
                             window_step=case["step"], gamma=case["gamma"],
                             normalize=case["normalize"], fusion=case["fusion"])


def _planes(case, seed):
    """Level planes and labels of a training batch: 1/16-size views, their disparity there."""
    w, h, n = case["w"], case["h"], case["count"]
    out = [torch.empty(n, h, w, device="cuda") for _ in range(3)]
    step = max(1, (64 << 20) // (w * h * 256 * 8))
    for i in range(0, n, step):
        k = min(step, n - i)
        a, b, d = _make((seed * 1000003 + i * 7919 + w) % (1 << 40), 16 * w, 16 * h, k)
        d = torch.where(torch.arange(16 * w, device="cuda") - d < 0,
                        torch.full_like(d, float("nan")), d)
        for o, v in zip(out, (a, b)):
            o[i:i + k] = F.avg_pool2d(v[:, None], 16)[:, 0]
        out[2][i:i + k] = d[:, ::16, ::16] / 16.0
    left, right, label = out
    step_right = torch.zeros_like(right)
    step_right[..., :-1] = right[..., 1:] - right[..., :-1]
    return left, torch.stack([right, step_right], -1).contiguous(), label


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "train":
        s["L"], s["R"], s["label"] = _planes(case, seed)
        s["weights"] = bd.net_init_weights(seed=seed % 1000)
        s["net"] = bd.ProposalNet(s["weights"])
        return s
    s["params"] = _params(case)
    if kind == "plan":
        s["groups"] = []
        for i, (w, h, n) in enumerate(_pairs(case)):
            left, right, _ = _images(case, seed + 131 * i, w, h, n)
            s["groups"].append((left, right, torch.empty(n, h, w, device="cuda")))
        # autotune=False: the tuner's choice may round differently from run to run
        s["plan"] = bd.Plan(s["groups"], s["params"], autotune=False, scale_to_width=True)
        return s
    w, h, n = _pairs(case)[0]
    s["left"], s["right"], s["prev"] = _images(case, seed, w, h, n, case["start"] == "warm")
    if kind == "host":
        s["left"], s["right"] = s["left"].cpu().pin_memory(), s["right"].cpu().pin_memory()
        s["out"] = torch.empty(n, h, w).pin_memory()
    elif kind == "match":
        s["out"] = torch.empty(n, h, w, device="cuda")
    if kind in ("match", "host"):
        s["matcher"] = bd.Matcher("cuda:0")
        if kind == "match":
            s["matcher"].reserve(w, h, n, s["params"])
    if case["start"] == "learned":
        path = os.path.join(os.path.dirname(bd.__file__), "weights", "proposal.bdisnet")
        s["net"] = bd.ProposalNet(bd.load_net_weights(path)[0])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "match":
        if case["start"] == "warm":
            return s["matcher"].match_warm(s["left"], s["right"], s["prev"], s["params"], s["out"])
        if case["start"] == "learned":
            return s["matcher"].match_learned(s["net"], s["left"], s["right"], s["params"],
                                              out=s["out"])
        return s["matcher"].match(s["left"], s["right"], s["params"], s["out"])
    if kind == "host":
        return s["matcher"].match_host(s["left"], s["right"], s["params"], s["out"])
    if kind == "plan":
        s["plan"].run()
        return [g[2] for g in s["groups"]]
    if kind == "train":
        loss, grad = s["net"].gradient(s["L"], s["R"], s["label"])
        return {"loss": loss, "grad": grad}
    p = s["params"]
    planes = [bd.prepare_level0(s["left"], s["right"])]
    for _ in range(p.coarsest_scale):
        planes.append(bd.pyramid_level(planes[-1][0], planes[-1][1]))
    coarse, levels = None, []
    for l in range(p.coarsest_scale, p.finest_scale - 1, -1):
        left, right, grad = planes[l]
        r = bd.search_level(left, right, grad, coarse, p)
        coarse = bd.densify_level(tuple(left.shape[1:]), p, r["d_star"], r["weight"], coarse,
                                  l == p.finest_scale, left, right)
        levels.append(dict(r, map=coarse))
    return {"planes": planes, "levels": levels}


# ------------------------------------------------------------------ work

NET = ((2, 32, 1), (32, 32, 2), (32, 32, 4), (32, 32, 4), (32, 32, 2), (32, 1, 1))


def work(case):
    """Bytes: images in, map out (stages: every output once). Flops: 8 per patch pixel and
    evaluation, window samples + 5 updates per patch (patches stop early; about 5 is the mean at
    the finest level), plus the network's multiply-adds."""
    net = sum(18.0 * a * b for a, b, _ in NET)
    if case["kind"] == "train":
        px = case["w"] * case["h"] * case["count"]
        count = sum(9 * a * b + b for a, b, _ in NET)
        return {"bytes": px * 16.0 + count * 8.0, "flops": px * 3 * net}
    es = 1 if case["dtype"] == "u8" else 4
    window = case["window"] if case["fusion"] == 0 else 0
    nbytes, flops = 0.0, 0.0
    for w, h, n in _pairs(case):
        nbytes += n * w * h * (2.0 * es + 4 + (4 if case["start"] == "warm" else 0))
        for l in range(case["coarsest"] + 1):
            lw, lh = bd.level_dims(w, h, l)
            if case["kind"] == "stages":
                nbytes += n * lw * lh * 16.0
            if case["start"] == "learned" and l == bd.proposal_level(case["coarsest"]):
                flops += n * lw * lh * net
            if l < case["finest"]:
                continue
            patches = float(n)
            for d in (lw, lh):
                patches *= bd.grid(d, case["ps"], case["overlap"])[1]
            flops += patches * case["ps"] ** 2 * 8 * (min(case["iters"], 5) + window)
            if case["kind"] == "stages":
                nbytes += patches * (22.0 + 4 * case["window"]) + (n * lw * lh * 4.0 if l else 0)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ 64-bit values

def _down(p):
    """5x5 binomial smoothing with a mirrored border, even samples kept."""
    k = torch.tensor([1.0, 4.0, 6.0, 4.0, 1.0], dtype=torch.float64, device=p.device) / 16.0
    p = F.conv2d(F.pad(p[:, None], (2, 2, 2, 2), mode="reflect"), k.view(1, 1, 1, 5))
    return F.conv2d(p, k.view(1, 1, 5, 1))[:, 0, ::2, ::2]


def _plane_outputs(left, right):
    step = torch.zeros_like(right)
    step[..., :-1] = right[..., 1:] - right[..., :-1]
    p = F.pad(left[:, None], (1, 1, 1, 1), mode="reflect")[:, 0]
    dx = p[..., 2:] - p[..., :-2]
    return left, torch.stack([right, step], -1), (dx[:, :-2] + 2 * dx[:, 1:-1] + dx[:, 2:]) / 8.0


def exact(case, seed):
    """64-bit values of the pyramid planes and of the network's loss and gradient. The searched
    maps have none: which patches are kept, and so which pixels are estimated at all, turns on
    ties and thresholds that another rounding decides otherwise."""
    if case["kind"] == "train":
        s = prepare(case, seed)
        w = torch.tensor(s["weights"], dtype=torch.float64, device="cuda", requires_grad=True)
        x = torch.stack([s["L"].double(), s["R"][..., 0].double()], 1)
        x = (x - 128.0) / 64.0
        at = 0
        for i, (a, b, dil) in enumerate(NET):
            k = w[at:at + 9 * a * b].view(b, 3, 3, a).permute(0, 3, 1, 2)
            bias = w[at + 9 * a * b:at + 9 * a * b + b]
            at += 9 * a * b + b
            x = F.conv2d(x, k, bias, padding=dil, dilation=dil)
            x = x.relu() if i < 5 else x
        label = s["label"].double()
        known = torch.isfinite(label)
        e = torch.where(known, x[:, 0] - torch.where(known, label, 0.0), 0.0)
        loss = torch.where(e.abs() <= 1, 0.5 * e * e, e.abs() - 0.5).mean()
        loss.backward()
        return {"loss": float(loss), "grad": np.asarray(w.grad.cpu())}
    if case["kind"] != "stages":
        return None
    left, right, _ = _images(case, seed, case["w"], case["h"], case["count"])
    left, right = left.double(), right.double()
    planes = []
    for l in range(case["coarsest"] + 1):
        if l:
            left, right = _down(left), _down(right)
        planes.append(_plane_outputs(left, right))
    return {"planes": planes}
