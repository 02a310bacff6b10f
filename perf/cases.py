"""The workloads that this framework's speed is judged by, as a program has them.

Three kinds of pass, each through the public entry points:

* ``frame``: one cooperative-perception frame on a context that the program
  keeps: the agents' payloads complete one after another, the program waits for
  the detections and reads the head output (the logits and box residuals).  The
  payload is the program's own array ("array"), was received straight into the
  library's pinned staging buffer ("staging"), or lies in device memory already
  ("resident").
* ``pillars``: the allocation-free pillarise / PFN / scatter pass on device
  arrays.
* ``nms``: rotated non-maximum suppression of a ranked list of boxes.

Networks are the two of the workload presets: the PointPillars network
(3 / 5 / 5 convolutions of 64 / 128 / 256 channels, a 3 x 128-channel neck; "pp")
and the small one (3 convolutions of 32 channels, no neck; "small").
"""
import math

import numpy as np
import torch

import synth
from paper_2608_08330_gb300 import rtcc as R

DEV = "cuda"
_PP = dict(net="pp", pillars=16000, boxes=256, absent=0, multiscale=False)


def listed():
    return [
        # the smallest frame: 2 agents, 64 x 64 cells; latency and launches count
        dict(name="frame_small_2", kind="frame", net="small", agents=2, w=64, h=64, points=2048,
             fusion="max", dtype="fp16", mode="rtcc", payload="array", pillars=2048, boxes=128,
             absent=0, multiscale=False),
        # a vehicle without partners: one branch on the long-range grid
        dict(_PP, name="frame_lone", kind="frame", agents=1, w=704, h=200, points=130000,
             fusion="max", dtype="fp16", mode="rtcc", payload="staging"),
        # the ordinary frame: 3 agents, 256 x 256 cells
        dict(_PP, name="frame_pp3", kind="frame", agents=3, w=256, h=256, points=110000,
             fusion="max", dtype="fp16", mode="rtcc", payload="staging", pillars=12000),
        # a ragged grid, payloads in the program's own arrays, one agent that did
        # not report, all branches held to the last arrival
        dict(_PP, name="frame_ragged_4", kind="frame", agents=4, w=328, h=184, points=70001,
             fusion="max", dtype="bf16", mode="barrier", payload="array", absent=1),
        # long range with attention fusion, 16-bit brain floats
        dict(_PP, name="frame_attn_5", kind="frame", agents=5, w=704, h=200, points=130000,
             fusion="attn", dtype="bf16", mode="rtcc", payload="staging"),
        # the multi-scale placement: the blocks' maps are fused before the neck
        dict(_PP, name="frame_scales_5", kind="frame", agents=5, w=704, h=200, points=130000,
             fusion="attn", dtype="bf16", mode="rtcc", payload="resident", multiscale=True),
        # the largest frame: 8 agents, released as they complete
        dict(_PP, name="frame_stress_8", kind="frame", agents=8, w=704, h=200, points=160000,
             fusion="max", dtype="fp16", mode="rtcc", payload="staging"),
        # the same in the multi-scale placement, payloads resident, held to the last arrival
        dict(_PP, name="frame_scales_8", kind="frame", agents=8, w=704, h=200, points=160000,
             fusion="max", dtype="fp16", mode="barrier", payload="resident", multiscale=True),
        # a plugin's pillarisation: a small sweep and a full one on an odd grid
        dict(name="pillars_small", kind="pillars", w=64, h=64, points=2048, ch=32, pts=16,
             pillars=2048, dtype="fp16"),
        dict(name="pillars_full", kind="pillars", w=301, h=211, points=130000, ch=64, pts=32,
             pillars=12000, dtype="bf16"),
        # suppression of a short and of the longest list
        dict(name="nms_128", kind="nms", n=128, iou=0.15, span=51.2),
        dict(name="nms_512", kind="nms", n=512, iou=0.15, span=40.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame"] * 6 + ["pillars"] * 2 + ["nms"])
    if kind == "nms":
        return dict(kind=kind, n=_log(rng, 8, 512), iou=round(rng.uniform(0.05, 0.6), 3),
                    span=round(rng.uniform(20.0, 140.0), 1))
    if kind == "pillars":
        w = _log(rng, 33, 704)
        return dict(kind=kind, w=w, h=_log(rng, 33, max(34, min(256, 65536 // w))),
                    points=_log(rng, 500, 131072), ch=rng.choice([32, 64]), pts=rng.randint(8, 32),
                    pillars=_log(rng, 1000, 16384), dtype=rng.choice(["fp16", "bf16"]))
    agents = rng.randint(1, 8)
    c = dict(kind=kind, agents=agents, fusion=rng.choice(["max", "max", "attn"]),
             dtype=rng.choice(["fp16", "bf16"]), mode=rng.choice(["rtcc", "barrier"]),
             payload=rng.choice(["array", "staging", "resident"]), boxes=rng.choice([128, 256, 300]),
             absent=rng.choice([0, 0, 1]) if agents > 1 else 0)
    if rng.random() < 0.2:
        return dict(c, net="small", w=_log(rng, 40, 300), h=_log(rng, 40, 200),
                    points=_log(rng, 2000, 60000), pillars=_log(rng, 2000, 12000), multiscale=False)
    # the PointPillars network halves the grid three times; 8 agents' arrays of
    # up to 60000 points cost no more than the largest frame
    return dict(c, net="pp", w=8 * _log(rng, 8, 88), h=8 * _log(rng, 8, 25),
                points=_log(rng, 5000, 60000 if c["payload"] == "array" else 160000), pillars=_log(rng, 4000, 16000),
                multiscale=rng.random() < 0.3)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _config(c, seed=0):
    """The workload description of a frame or pillars case."""
    pp = c.get("net", "pp") == "pp"
    hx, hy = 0.2 * c["w"], 0.2 * c["h"]
    clusters = min(20, c["points"] // 2000)
    return synth.get_config(
        "pp3" if pp else "tiny", n_agents=c.get("agents", 1), grid_w=c["w"], grid_h=c["h"],
        x_min=-hx, x_max=hx, y_min=-hy, y_max=hy, pts_x=(-hx, hx), pts_y=(-hy, hy),
        max_pillars=c["pillars"], fusion=c.get("fusion", "max"), dtype=c["dtype"],
        max_boxes=c.get("boxes", 256), n_uniform=c["points"] - 500 * clusters, n_clusters=clusters,
        cluster_pts=500, cluster_sigma=0.5, point_seed=seed, pfn_ch=c.get("ch", 64 if pp else 32),
        max_pts=c.get("pts", 32 if pp else 16))


_weights = {}


def _weights_for(c):
    """The trained model's stand-in: one set of weights per network and grid."""
    cfg = _config(c)
    key = (cfg.blocks, cfg.up_strides, cfg.pfn_ch, cfg.grid_w, cfg.grid_h)
    if key not in _weights:
        _weights[key] = synth.weights_for(cfg)
    return _weights[key]


def _points(c, seed):
    cfg = _config(c, seed)
    return [synth.points_for(cfg, 0, k) for k in range(cfg.n_agents)]


class Frame:
    def __init__(self, c, seed):
        self.cfg = cfg = _config(c)
        self.c = c
        R.load()
        flags = R.FLAG_MULTISCALE if c["multiscale"] else 0
        self.ctx = R.rtcc_init(R.model_config(cfg, flags=flags), synth.weight_blob(_weights_for(c)))
        R.rtcc_set_mode(self.ctx, R.MODE_BARRIER if c["mode"] == "barrier" else R.MODE_RTCC)
        self.points, self.frame = _points(c, seed), 0
        self.gone = set(range(1, 1 + c["absent"]))           # never agent 0, the ego
        for k in range(cfg.n_agents):
            if c["payload"] == "resident":
                R.rtcc_stage_resident(self.ctx, k, self.points[k])
            elif c["payload"] == "staging":
                buf = R.rtcc_staging_buffer(self.ctx, k)[:len(self.points[k])]
                buf[:] = self.points[k]
                self.points[k] = buf

    def __del__(self):
        if getattr(self, "ctx", None):
            R.rtcc_destroy(self.ctx)

    def run(self):
        ctx, cfg = self.ctx, self.cfg
        self.frame += 1
        R.rtcc_frame_begin(ctx, self.frame, 0.0)
        for k in range(cfg.n_agents):
            if k in self.gone:
                R.rtcc_payload_absent(ctx, k, float(k))
            elif self.c["payload"] == "resident":
                R.rtcc_payload_resident(ctx, k, float(k))
            else:
                R.rtcc_payload_complete(ctx, k, self.points[k], float(k))
        _, boxes, _ = R.rtcc_wait_detection(ctx, 10000)
        # which anchors hold a detection: a list in rank order would differ
        # wherever two nearly equal scores change places
        kept = np.zeros(cfg.feat_w * cfg.feat_h * cfg.anchors, dtype=np.uint8)
        kept[boxes["anchor"]] = 1
        return {"head": R.rtcc_get_head(ctx, cfg.feat_h, cfg.feat_w), "kept": kept}


class Pillars:
    def __init__(self, c, seed):
        R.load()
        self.cfg = cfg = _config(c)
        self.mc = R.model_config(cfg)
        w, b = _pfn_weights(c)
        i32 = dict(dtype=torch.int32, device=DEV)
        self.pts = torch.from_numpy(_points(c, seed)[0]).to(DEV)
        self.w, self.b = w.to(DEV), b.to(DEV)
        self.cell2pillar = torch.empty(cfg.grid_h * cfg.grid_w, **i32)
        self.pillar_cell = torch.zeros(cfg.max_pillars, **i32)
        self.count = torch.zeros(cfg.max_pillars, **i32)
        self.stats = torch.empty(8, **i32)
        self.image = torch.empty(cfg.grid_h, cfg.grid_w, cfg.pfn_ch, device=DEV,
                                 dtype=torch.bfloat16 if cfg.dtype == "bf16" else torch.float16)

    def run(self):
        R.rtcc_pillarise_noalloc(
            self.mc, self.pts.data_ptr(), self.pts.shape[0], self.w.data_ptr(), self.b.data_ptr(),
            self.cell2pillar.data_ptr(), self.pillar_cell.data_ptr(), self.count.data_ptr(),
            self.stats.data_ptr(), self.image.data_ptr(), torch.cuda.current_stream().cuda_stream)
        return {"cell2pillar": self.cell2pillar, "pillar_cell": self.pillar_cell,
                "count": self.count, "stats": self.stats, "image": self.image}


class Nms:
    """Ranked boxes as a detector's decode leaves them: a few per object, around
    it and turned a little, and strays."""

    def __init__(self, c, seed):
        R.load()
        self.iou, n = c["iou"], c["n"]
        rng = np.random.default_rng([seed, 11])
        obj = rng.uniform(-c["span"], c["span"], (max(1, n // 5), 2))
        at = obj[rng.integers(0, len(obj), n)] + rng.normal(0.0, 0.6, (n, 2))
        b = np.zeros(n, dtype=R.BOX_DTYPE)
        b["x"], b["y"], b["z"] = at[:, 0], at[:, 1], -1.0
        b["l"] = 3.9 * np.exp(rng.normal(0.0, 0.15, n))
        b["w"] = 1.6 * np.exp(rng.normal(0.0, 0.15, n))
        b["h"] = 1.56
        b["yaw"] = rng.integers(0, 2, n) * (math.pi / 2) + rng.normal(0.0, 0.3, n)
        b["score"] = np.sort(rng.uniform(0.5, 1.0, n))[::-1]
        b["anchor"] = rng.permutation(70400)[:n]
        self.boxes = b

    def run(self):
        # the kept boxes in rank order, in the list's own length: padded
        out = np.full(len(self.boxes), -1, dtype=R.BOX_DTYPE)
        got = R.rtcc_nms(self.boxes, self.iou)
        out[:len(got)] = got
        return {"anchor": out["anchor"],
                "box": out.view(np.float32).reshape(-1, 9)[:, :8]}


def prepare(case, seed):
    return {"frame": Frame, "pillars": Pillars, "nms": Nms}[case["kind"]](case, seed)


def run(state):
    return state.run()


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

def work(case):
    if case["kind"] == "nms":
        # every pair takes a few tens of operations; the boxes come in and go out
        return {"bytes": 2 * 36 * case["n"], "flops": 40 * case["n"] ** 2 / 2}
    cfg = _config(case)
    cells = cfg.grid_w * cfg.grid_h
    kept = min(case["pillars"], cells)
    pfn = 2.0 * 4 * cfg.pfn_ch * case["points"]
    if case["kind"] == "pillars":
        return {"bytes": 16 * case["points"] + cells * (2 * cfg.pfn_ch + 4) + 8 * kept, "flops": pfn}
    present = case["agents"] - case["absent"]
    conv, neck, weights = 0.0, 0.0, 9 * cfg.pfn_ch
    w, h, cin = cfg.grid_w, cfg.grid_h, cfg.pfn_ch
    for bi, (n, ch, st) in enumerate(cfg.blocks):
        w, h = w // st, h // st
        for _ in range(n):
            conv += 2.0 * w * h * ch * cin * 9
            weights += ch * cin * 9
            cin = ch
        if cfg.up_strides:
            neck += 2.0 * w * h * ch * cfg.up_ch * cfg.up_strides[bi] ** 2
            weights += ch * cfg.up_ch * cfg.up_strides[bi] ** 2
    out = cfg.feat_w * cfg.feat_h
    flops = present * (pfn + conv) + neck * (1 if case["multiscale"] else present) + 2.0 * out * cfg.feat_ch * 16
    return {"bytes": 16 * case["points"] * present + 2 * (weights + 16 * cfg.feat_ch) + out * 64 + out * 2,
            "flops": flops}


# Four times the error that the path shows against `exact`, which is its
# rounding of every stored activation to 16 bits (frames: 2.9e-4 to 5.1e-4 in
# fp16, 2.4e-3 to 3.9e-3 in bf16; the pillar image: 2.0e-4 and 1.6e-3); of the
# detections, what ties and near-ties in score or overlap can move.
def tolerance(case):
    if case["kind"] == "nms":
        return "exact"                         # boxes are copied, never computed
    half = case["dtype"] == "fp16"
    if case["kind"] == "pillars":
        return {"rel": 8e-4 if half else 6.4e-3, "differ": 0.0}
    return {"rel": 2e-3 if half else 1.6e-2, "differ": 0.005}


# --------------------------------------------------------------------------
# the same in 64 bits
# --------------------------------------------------------------------------

def _rounded(c, a):
    """The values the model is defined on: its weights in the storage type."""
    t = torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    return t.to(torch.bfloat16 if c["dtype"] == "bf16" else torch.float16).double()


def _pfn_weights(c):
    wt = _weights_for(c)
    return _rounded(c, wt["pfn.w"]).float(), _rounded(c, wt["pfn.b"]).float()


def _image64(c, cfg, pts):
    """Pillars in point order (at most max_pillars, max_pts points each), the 9
    features of each kept point, linear + ReLU + maximum, on the BEV grid."""
    p = torch.from_numpy(pts).to(DEV)
    n, W, H = p.shape[0], cfg.grid_w, cfg.grid_h
    f32 = lambda v: torch.tensor(v, dtype=torch.float32, device=DEV)  # noqa: E731
    ix = torch.floor((p[:, 0] - f32(cfg.x_min)) / f32(cfg.pillar))
    iy = torch.floor((p[:, 1] - f32(cfg.y_min)) / f32(cfg.pillar))
    ok = (p[:, 2] >= f32(cfg.z_min)) & (p[:, 2] < f32(cfg.z_max))
    ok &= (ix >= 0) & (ix < W) & (iy >= 0) & (iy < H)
    idx = torch.nonzero(ok).flatten()
    cell = (iy[idx] * W + ix[idx]).long()
    first = torch.full((W * H,), n, device=DEV).scatter_reduce(0, cell, idx, "amin")
    opened = torch.nonzero(first < n).flatten()
    opened = opened[torch.argsort(first[opened])][:cfg.max_pillars]
    pid = torch.full((W * H,), -1, device=DEV)
    pid[opened] = torch.arange(len(opened), device=DEV)
    own, order = torch.sort(pid[cell], stable=True)
    lo = torch.searchsorted(own, own)
    keep = (own >= 0) & (torch.arange(len(own), device=DEV) - lo < cfg.max_pts)
    own, order = own[keep], order[keep]
    q = p[idx[order]].double()
    cnt = torch.zeros(len(opened), dtype=torch.float64, device=DEV).index_add(0, own, torch.ones_like(q[:, 0]))
    mean = torch.zeros(len(opened), 3, dtype=torch.float64, device=DEV).index_add(0, own, q[:, :3])
    mean = (mean / cnt[:, None])[own]
    at = opened[own]
    xc = cfg.x_min + ((at % W).double() + 0.5) * cfg.pillar
    yc = cfg.y_min + ((at // W).double() + 0.5) * cfg.pillar
    f = torch.cat([q, q[:, :3] - mean, (q[:, 0] - xc)[:, None], (q[:, 1] - yc)[:, None]], 1)
    w, b = _pfn_weights(c)
    lin = torch.relu(f @ w.double().T + b.double())
    vec = torch.zeros(len(opened), cfg.pfn_ch, dtype=torch.float64, device=DEV)
    vec = vec.scatter_reduce(0, own[:, None].expand_as(lin), lin, "amax")
    img = torch.zeros(W * H, cfg.pfn_ch, dtype=torch.float64, device=DEV)
    img[opened] = vec
    return img.view(H, W, -1)


def _conv64(x, w, b, s):
    H, W, _ = x.shape
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
    y = b.expand((H // s) * (W // s), -1).clone()
    for t in range(9):
        dy, dx = divmod(t, 3)
        v = xp[dy:dy + s * (H // s - 1) + 1:s, dx:dx + s * (W // s - 1) + 1:s]
        y.addmm_(v.reshape(-1, x.shape[2]), w[:, :, dy, dx].T)
    return torch.relu(y).view(H // s, W // s, -1)


def _neck64(c, cfg, blocks):
    wt, ups = _weights_for(c), []
    for bi, s in enumerate(cfg.up_strides):
        w, b = _rounded(c, wt["up%d.w" % bi]), _rounded(c, wt["up%d.b" % bi])
        h, v, ci = blocks[bi].shape
        y = (blocks[bi].reshape(-1, ci) @ w.permute(0, 2, 3, 1).reshape(ci, -1)).view(h, v, s, s, -1)
        ups.append(torch.relu(y.permute(0, 2, 1, 3, 4).reshape(h * s, v * s, -1) + b))
    return torch.cat(ups, 2) if ups else blocks[-1]


def _fuse64(c, maps):
    x = torch.stack(maps)
    if c["fusion"] == "max":
        return x.amax(0)
    s = (x[:1] * x).sum(-1) / math.sqrt(x.shape[-1])
    return (torch.softmax(s, 0)[..., None] * x).sum(0)


def exact(case, seed):
    if case["kind"] == "nms":
        return None
    cfg, wt = _config(case), _weights_for(case)
    pts = _points(case, seed)
    if case["kind"] == "pillars":
        return {"cell2pillar": None, "pillar_cell": None, "count": None, "stats": None,
                "image": _image64(case, cfg, pts[0])}
    blocks = []
    for k in range(cfg.n_agents):
        if 1 <= k <= case["absent"]:
            continue
        x, outs = _image64(case, cfg, pts[k]), []
        for bi, (n, _, st) in enumerate(cfg.blocks):
            for li in range(n):
                x = _conv64(x, _rounded(case, wt["b%d.c%d.w" % (bi, li)]),
                            _rounded(case, wt["b%d.c%d.b" % (bi, li)]), st if li == 0 else 1)
            outs.append(x)
        blocks.append(outs)
    if case["multiscale"]:
        F = _neck64(case, cfg, [_fuse64(case, [b[i] for b in blocks]) for i in range(len(cfg.blocks))])
    else:
        F = _fuse64(case, [_neck64(case, cfg, b) for b in blocks])
    w, b = _rounded(case, wt["head.w"]), _rounded(case, wt["head.b"])
    return {"head": F @ w.T + b, "kept": None}
