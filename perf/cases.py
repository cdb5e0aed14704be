"""Workloads the filter is timed on, through its public entry points.

``listed()`` are twelve fixed workloads, ``draw(rng)`` gives others of the same
ranges; ``prepare`` makes a workload's inputs, table, network or batch;
``run`` is one pass; ``work`` is what a pass cannot do without; ``exact`` is
the pass's result in 64 bits, computed with plain torch.

Kinds of workload:

* ``frame``  one frame through ``Table.filter`` (build, insert, blend, lookup);
* ``noalloc``  one plain frame through ``pps_filter_noalloc``;
* ``batch``  one frame of several views through ``Batch.run``;
* ``train``  online training of the learned fallback on a filtered frame;
* ``infer``  the learned fallback's answers for the low-count vertices.

Every probe limit is large enough that no vertex exceeds it: which vertices
exceed a short one depends on the order of the atomics, so their results could
not be compared between two runs.
"""
from __future__ import annotations

import math
from dataclasses import dataclass
from typing import Dict, Optional

import numpy as np
import torch

from paper_1902_05942_gb300 import pps, scene
from paper_1902_05942_gb300.configs import BATCHED_SURVIVAL, BATCHED_VIEWS, FilterConfig

# Jitter frames a case goes through before it starts over (a renderer's frame
# number grows; a bounded cycle keeps the history's size bounded).
FRAME_CYCLE = 8
# Frames a temporal case has behind it before its first pass.
WARM_FRAMES = 2
# Vertices per cell, roughly, of the procedural scene at the default scale.
CELLS_PER_VERTEX = 0.47

FRAME = dict(kind="frame", paths=1, bounces=3, survival=0.8, scale=4.0, probes=64, fixed=False,
             hist=0, log2_hist=0, alpha=0.2, fallback="none", variants=False, migrate=False,
             cluster=0.0)


def _frame(name: str, width: int, height: int, log2_slots: int, **kw) -> dict:
    return dict(FRAME, name=name, width=width, height=height, log2_slots=log2_slots, **kw)


def listed():
    return [
        # a preview thumbnail inside a plug-in whose host owns the GPU memory:
        # the smallest call, all launch and latency
        dict(_frame("thumbnail_noalloc", 96, 80, 14, bounces=1), kind="noalloc"),
        # the small preset: primary hits of a 256 x 256 frame
        _frame("small", 256, 256, 18, bounces=1),
        # an interactive window of odd size: half-precision history, exact
        # integration over the frames
        _frame("window_fp16_history", 1279, 719, 21, bounces=2, hist=2, log2_hist=23, alpha=-1.0),
        # a full HD frame without history: offline or after a camera cut
        _frame("hd_plain", 1920, 1080, 23),
        # the headline: full HD, temporal blending
        _frame("hd_temporal", 1920, 1080, 23, hist=1, log2_hist=25),
        # order-independent sums (reproducible renders)
        _frame("hd_fixed_point", 1920, 1080, 23, fixed=True),
        # low-count vertices search their 3 x 3 x 3 neighborhood
        _frame("hd_neighbors", 1920, 1080, 23, hist=1, log2_hist=25, fallback="neighbors"),
        # path-length level of detail and a material word in the key
        _frame("720p_key_variants", 1280, 720, 22, hist=1, log2_hist=24, variants=True),
        # online training of the learned fallback, four Adam steps a frame
        dict(_frame("train_hd", 1920, 1080, 23), kind="train", batch=16384, steps=4),
        # the learned fallback answering for the low-count vertices of a frame
        dict(_frame("infer_hd", 1920, 1080, 23, hist=1, log2_hist=25), kind="infer"),
        # eight cameras (light-field or multi-user rendering), 37 M vertices
        dict(_frame("batched_views", 0, 0, 0, bounces=2, survival=BATCHED_SURVIVAL), kind="batch",
             views=8, shrink=1.0),
        # 4K, two paths per pixel, six bounces, most vertices in a corner of
        # the scene, a table far larger than L2
        _frame("stress_4k", 3840, 2160, 26, paths=2, bounces=6, scale=0.5, probes=512, hist=2,
               log2_hist=28, cluster=0.8),
    ]


def _log_uniform(rng, lo: float, hi: float) -> float:
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng) -> dict:
    kind = rng.choice(["frame", "frame", "frame", "frame", "noalloc", "batch", "train", "infer"])
    pixels = _log_uniform(rng, 4800, 500_000 if kind == "noalloc" else 2_200_000)
    width = max(8, round(math.sqrt(pixels * rng.uniform(0.8, 2.2))))
    height = max(8, int(pixels / width))
    bounces = 1 if kind == "noalloc" else rng.randint(1, 3)
    scale = rng.choice([2.0, 4.0, 4.0, 8.0])
    c = _frame("", width, height, 0, bounces=bounces, scale=scale)
    del c["name"]
    c["kind"] = kind
    if kind == "batch":
        c.update(bounces=2, survival=BATCHED_SURVIVAL, scale=4.0, width=0, height=0,
                 views=rng.randint(2, 8), shrink=round(_log_uniform(rng, 0.1, 1.0), 3))
        return c
    c["log2_slots"] = max(12, math.ceil(math.log2(1.6 * _vertices(c))) + rng.choice([0, 0, 1]))
    if kind == "noalloc":
        c["log2_slots"] = min(c["log2_slots"], 20)
    if kind == "frame":
        c["fixed"] = rng.random() < 0.2
        c["hist"] = rng.choice([0, 1, 1, 2])
        c["fallback"] = rng.choice(["none", "none", "none", "coarse", "neighbors"])
        c["alpha"] = rng.choice([0.2, 0.2, -1.0])
        if c["fallback"] == "none":
            c["variants"] = rng.random() < 0.15
            c["migrate"] = bool(c["hist"]) and not c["variants"] and rng.random() < 0.15
        if c["hist"]:
            c["log2_hist"] = c["log2_slots"] + 2
    if kind == "infer":
        c["hist"], c["log2_hist"] = 1, c["log2_slots"] + 2
    if kind == "train":
        c["batch"], c["steps"] = 128 * rng.randint(16, 160), rng.randint(1, 6)
    return c


# ---------------------------------------------------------------- sizes
def _views(case) -> list:
    """(width, height, log2_slots, eye or None) of each view of the case."""
    if case["kind"] != "batch":
        return [(case["width"], case["height"], case["log2_slots"], None)]
    out = []
    for i in range(case["views"]):
        w, h = (max(8, round(x * case["shrink"])) for x in BATCHED_VIEWS[i])
        a = 2.0 * math.pi * i / case["views"]
        out.append((w, h, max(12, math.ceil(math.log2(1.7 * w * h))),
                    (12.4 * math.sin(a), 3.0, -12.4 * math.cos(a))))
    return out


def _view_vertices(case, width: int, height: int) -> int:
    """Vertices of one view: what Russian roulette leaves on average."""
    paths = width * height * case["paths"]
    return round(paths * sum(case["survival"] ** k for k in range(case["bounces"])))


def _vertices(case) -> int:
    return sum(_view_vertices(case, w, h) for w, h, _, _ in _views(case))


# Multiply-adds of the network per sample: 80 x 64 + 2 x 64 x 64 + 64 x 3.
_MACS = 80 * 64 + 2 * 64 * 64 + 64 * 3


def work(case) -> dict:
    n = _vertices(case)
    if case["kind"] == "train":
        # each sample's vertex (24 B), target and count (16 B); forward, deltas, gradients;
        # weights, moments and gradients of each step
        s = case["batch"] * case["steps"]
        return {"bytes": s * 40 + case["steps"] * _MACS * 24, "flops": 6 * _MACS * s}
    if case["kind"] == "infer":
        # every count and status once; a listed vertex's 24 B in and 13 B out
        low = 0.13 * n
        return {"bytes": 5 * n + 37 * low, "flops": 2 * _MACS * low}
    # nine streams in; r, g, b, count and status out; a history entry (value
    # and fingerprint) read and written per cell
    b = n * (36 + 17) + (n * 8 if case["variants"] else 0)
    if case["hist"]:
        b += n * CELLS_PER_VERTEX * 2 * (20 if case["hist"] == 1 else 12)
    return {"bytes": b, "flops": 0}


# ---------------------------------------------------------------- inputs
def _spec(case, view: scene.View, seed: int, index: int) -> scene.StreamSpec:
    # a little more survival than the case has: the stream is then cut to the
    # case's vertex count, the same for every seed
    return scene.StreamSpec(view=view, bounces=case["bounces"], survival=case["survival"] + 0.03,
                            scene_seed=1 + seed, path_seed=1000 * seed + 2 + 101 * index,
                            radiance_seed=1000 * seed + 3 + 101 * index,
                            cluster_fraction=case["cluster"])


def _inputs(case, seed: int) -> list:
    """Per view: the vertex streams, the camera position and the filter's options."""
    out = []
    for i, (w, h, log2, eye) in enumerate(_views(case)):
        view = scene.View(w, h, paths_per_pixel=case["paths"])
        if eye:
            view.eye, view.target = eye, (0.0, 0.5, 0.0)
        s = scene.trace_stream(_spec(case, view, seed, i), 0, "cuda")
        n = _view_vertices(case, w, h)
        if s["px"].numel() < n:
            raise RuntimeError(f"{s['px'].numel()} vertices traced, {n} wanted")
        v = {k: s[k][:n] for k in scene.STREAMS}
        if case["variants"]:
            g = torch.Generator(device="cuda").manual_seed(seed + 7)
            p = torch.stack([v["px"], v["py"], v["pz"]], 1)
            d = (p - torch.tensor(view.eye, device="cuda")).norm(dim=1)
            first = s["bounce_counts"][0]
            # the length of the path so far: longer than the camera distance
            # from the second vertex on
            d[first:] += 4.0 * torch.rand(d.numel() - first, generator=g, device="cuda")
            v["dist"] = d.contiguous()
            v["extra"] = torch.randint(0, 4, (d.numel(),), generator=g, device="cuda",
                                       dtype=torch.int32)
        cfg = FilterConfig(log2_slots=log2, max_probes=case["probes"], voxel_scale=case["scale"],
                           pixel_angle=view.pixel_angle(), accum_fixed=case["fixed"],
                           hist_mode=case["hist"], log2_hist_slots=case["log2_hist"],
                           fallback=case["fallback"], hist_migrate=case["migrate"])
        out.append((v, view.eye, cfg))
    return out


def _weights(seed: int) -> np.ndarray:
    rng = np.random.RandomState(seed % (1 << 31))
    parts = []
    for fan, out in ((80, 64), (64, 64), (64, 64), (64, 3)):
        parts += [rng.standard_normal(out * fan) * math.sqrt(2.0 / fan), np.zeros(out)]
    return np.concatenate(parts).astype(np.float32)


def prepare(case, seed):
    views = _inputs(case, seed)
    s = {"case": case, "frame": WARM_FRAMES}
    if case["kind"] == "batch":
        s["views"] = [(pps.Table(cfg), v, pps.empty_output(v["px"].numel())) for v, _, cfg in views]
        s["cams"] = [eye for _, eye, _ in views]
        s["batch"] = pps.Batch(s["views"])
        return s
    v, eye, cfg = views[0]
    s.update(v=v, eye=eye, out=pps.empty_output(v["px"].numel()))
    if case["kind"] == "noalloc":
        n = v["px"].numel()
        s.update(n=n, params=pps.make_params(cfg), vertices=pps.make_vertices(v, n),
                 output=pps.make_output(s["out"], n))
        return s
    s["table"] = pps.Table(cfg)
    if case["kind"] == "frame":
        if case["hist"]:
            for f in range(WARM_FRAMES):
                s["table"].filter(v, eye, f, blend=True, alpha=case["alpha"], out=s["out"])
        return s
    # the learned fallback works on a filtered frame
    for f in range(WARM_FRAMES if case["hist"] else 1):
        s["table"].filter(v, eye, f, blend=bool(case["hist"]), alpha=case["alpha"], out=s["out"])
    torch.cuda.synchronize()
    s.pop("table").close()
    kw = dict(batch=case["batch"], steps=case["steps"]) if case["kind"] == "train" else {}
    s["net"] = pps.MLP(pps.mlp_params(seed=seed & 0xFFFF, **kw), init=_weights(seed))
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    frame = s["frame"]
    s["frame"] = WARM_FRAMES + (frame - WARM_FRAMES + 1) % FRAME_CYCLE
    if kind == "batch":
        s["batch"].run(s["cams"], frame)
        return [out for _, _, out in s["views"]]
    if kind == "noalloc":
        pps.pps_filter_noalloc(s["params"], pps.camera(s["eye"]), frame, s["vertices"], s["n"],
                               s["output"])
        return s["out"]
    if kind == "train":
        s["net"].train(s["v"], s["out"], frame)
        return s["net"].get_weights()
    if kind == "infer":
        s["net"].infer(s["v"], s["out"])
        return s["out"]
    return s["table"].filter(s["v"], s["eye"], frame, blend=bool(case["hist"]),
                             alpha=case["alpha"], out=s["out"])


# ---------------------------------------------------------------- the same in 64 bits
_M32 = 0xFFFFFFFF
_JITTER_SEED = 0x0051F15E
_LOD = 24
_LOWCOUNT = 4


def _philox(c0, c1, c2, k0: int, k1: int):
    """First two words of Philox4x32-10 (Salmon et al. 2011), counter (c0, c1, c2, 0)."""
    x = [c0, c1, c2, torch.zeros_like(c0)]
    for r in range(10):
        p0, p1 = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57  # low 64 bits of the products
        a, b = (k0 + r * 0x9E3779B9) & _M32, (k1 + r * 0xBB67AE85) & _M32
        x = [((p1 >> 32) & _M32) ^ x[1] ^ a, p1 & _M32, ((p0 >> 32) & _M32) ^ x[3] ^ b, p0 & _M32]
    return x[0], x[1]


def _pow2(e: torch.Tensor) -> torch.Tensor:
    return ((e + 127) << 23).to(torch.int32).view(torch.float32)


def _distance(cam, x, y, z):
    dx, dy, dz = cam[0] - x, cam[1] - y, cam[2] - z
    return torch.sqrt((dx * dx + dy * dy) + dz * dz)


def _level(k, d):
    e = ((k * d).view(torch.int32) >> 23).bitwise_and(255).to(torch.int64) - 127
    return e.clamp(-_LOD, _LOD)


@dataclass
class _Words:
    """Quantized keys: voxel, level, packed normal and extra word (int64)."""

    X: torch.Tensor
    Y: torch.Tensor
    Z: torch.Tensor
    L: torch.Tensor
    N: torch.Tensor
    E: torch.Tensor

    def at(self, sel) -> "_Words":
        return _Words(*(getattr(self, f)[sel] for f in "XYZLNE"))

    def hashed(self) -> torch.Tensor:
        """One 64-bit word per key (two of 10^8 keys agree with probability < 10^-3)."""
        h = torch.full_like(self.X, 0x243F6A8885A308D3)
        for w in (self.X, self.Y, self.Z, self.L, self.N, self.E):
            h = (h ^ w) * 0x2545F4914F6CDD1D
            h = h ^ ((h >> 31) & 0x1FFFFFFFF)
            h = h * 0x5851F42D4C957F2D
            h = h ^ ((h >> 29) & 0x7FFFFFFFF)
        return h


def _keys(v, eye, cfg, frame: int, scale: float) -> _Words:
    """Algorithm 1's quantized keys, in the FP32 steps that define them."""
    f32 = dict(dtype=torch.float32, device=v["px"].device)
    cam = torch.tensor(eye, **f32)
    # fl32(s * theta), each operand rounded to FP32 first
    k = torch.tensor(scale, **f32) * torch.tensor(cfg.pixel_angle, **f32)
    px, py, pz, nx, ny, nz = (v[c] for c in ("px", "py", "pz", "nx", "ny", "nz"))
    dist = v.get("dist")
    d0 = _distance(cam, px, py, pz)
    l0 = _level(k, d0 if dist is None else dist)
    i = torch.arange(px.numel(), device=px.device)
    a0, a1 = _philox(i, torch.zeros_like(i), torch.zeros_like(i), _JITTER_SEED, frame)
    u = (a0 >> 8).to(torch.float32) * 2.0 ** -24 - 0.5
    w = (a1 >> 8).to(torch.float32) * 2.0 ** -24 - 0.5
    # tangent frame of Duff et al. 2017
    s = torch.copysign(torch.ones_like(nz), nz)
    a = -torch.reciprocal(s + nz)
    q = (nx * ny) * a
    t = (1.0 + s * ((nx * nx) * a), s * q, -(s * nx))
    b = (q, s + (ny * ny) * a, -ny)
    e = _pow2(l0)
    x, y, z = (p + (u * t[j] + w * b[j]) * e for j, p in enumerate((px, py, pz)))
    d1 = _distance(cam, x, y, z)
    l1 = _level(k, d1 if dist is None else (dist - d0) + d1)
    inv = _pow2(-l1)
    X, Y, Z = (torch.floor(c * inv).to(torch.int64) for c in (x, y, z))
    n8 = [torch.floor((c + 1.0) * 128.0).clamp(0, 255).to(torch.int64) for c in (nx, ny, nz)]
    ex = v["extra"].to(torch.int64) if "extra" in v else torch.zeros_like(X)
    return _Words(X, Y, Z, l1, n8[0] | (n8[1] << 8) | (n8[2] << 16), ex)


@dataclass
class _Cells:
    """Cells of one frame or of a history: sorted hashes, values (n, 3), counts."""

    h: torch.Tensor
    c: torch.Tensor
    n: torch.Tensor

    def find(self, h):
        """Index of each hash and whether it is there."""
        if not self.h.numel():
            z = torch.zeros_like(h)
            return z, z.bool()
        j = torch.searchsorted(self.h, h).clamp_max(self.h.numel() - 1)
        return j, self.h[j] == h


class _Filter:
    """The filter of one resolution over successive frames of one stream."""

    def __init__(self, case, v, eye, cfg, scale):
        self.case, self.v, self.eye, self.cfg, self.scale = case, v, eye, cfg, scale
        self.rgb = torch.stack([v[c] for c in "rgb"], 1).double()
        z = torch.zeros(0, dtype=torch.int64, device=self.rgb.device)
        self.hist = _Cells(z, self.rgb[:0], z.double())

    def frame(self, number: int):
        """Per-vertex values and counts of frame `number`."""
        case = self.case
        words = _keys(self.v, self.eye, self.cfg, number, self.scale)
        h, inv = torch.unique(words.hashed(), return_inverse=True)
        n = torch.zeros(h.numel(), dtype=torch.float64, device=h.device)
        n.index_add_(0, inv, torch.ones_like(self.rgb[:, 0]))
        c = torch.zeros((h.numel(), 3), dtype=torch.float64, device=h.device)
        c.index_add_(0, inv, self.rgb)
        c /= n[:, None]
        if case["hist"]:
            j, there = self.hist.find(h)
            if self.hist.h.numel():
                old = torch.where(there, self.hist.n[j], torch.zeros_like(n))
                a = old / (old + n) if case["alpha"] < 0 else torch.full_like(
                    n, float(np.float32(case["alpha"])))
                a = torch.where(there, a, torch.zeros_like(a))[:, None]
                c = a * self.hist.c[j] + (1.0 - a) * c
                n = n + old
                self.hist.c[j[there]] = c[there]
                self.hist.n[j[there]] = n[there]
            new = ~there
            allh = torch.cat([self.hist.h, h[new]])
            order = torch.argsort(allh)
            self.hist = _Cells(allh[order], torch.cat([self.hist.c, c[new]])[order],
                               torch.cat([self.hist.n, n[new]])[order])
        value, count = c[inv], n[inv]
        if case["fallback"] == "neighbors":
            self._pool(words, _Cells(h, c, n), value, count)
        return value, count

    @staticmethod
    def _pool(words, cells, value, count):
        low = torch.nonzero(count < _LOWCOUNT).flatten()
        w = words.at(low)
        sv = torch.zeros((low.numel(), 3), dtype=torch.float64, device=low.device)
        sn = torch.zeros(low.numel(), dtype=torch.float64, device=low.device)
        for o in range(27):
            d = _Words(w.X + o // 9 - 1, w.Y + o // 3 % 3 - 1, w.Z + o % 3 - 1, w.L, w.N, w.E)
            j, there = cells.find(d.hashed())
            n = torch.where(there, cells.n[j], torch.zeros_like(sn))
            sv += n[:, None] * cells.c[j]
            sn += n
        value[low] = sv / sn[:, None]
        count[low] = sn


def _filtered(case, v, eye, cfg, frames):
    """Values (n, 3) and counts after the given frame numbers."""
    fine = _Filter(case, v, eye, cfg, case["scale"])
    coarse = _Filter(case, v, eye, cfg, 2.0 * case["scale"]) if case["fallback"] == "coarse" else None
    for f in frames:
        value, count = fine.frame(f)
        if coarse is not None:
            cv, cn = coarse.frame(f)
            low = count < _LOWCOUNT
            value = torch.where(low[:, None], cv, value)
            count = torch.where(low, cn, count)
    return value, count


def _encode(v, j) -> torch.Tensor:
    cols = []
    for c in ("px", "py", "pz"):
        p = ((v[c][j].double() + 100.0) / 200.0).clamp(0.0, 1.0)
        for k in range(12):
            cols += [torch.sin(math.pi * 2 ** k * p), torch.cos(math.pi * 2 ** k * p)]
    cols += [v[c][j].double() for c in ("nx", "ny", "nz")]
    cols += [torch.zeros_like(cols[0])] * 5
    return torch.stack(cols, 1)


def _layers(w: torch.Tensor) -> list:
    out, o = [], 0
    for fan, m in ((80, 64), (64, 64), (64, 64), (64, 3)):
        out.append((w[o:o + m * fan].view(m, fan), w[o + m * fan:o + m * fan + m]))
        o += m * fan + m
    return out


def _network(w, x) -> torch.Tensor:
    for i, (a, b) in enumerate(_layers(w)):
        x = x @ a.T + b
        if i < 3:
            x = torch.relu(x)
    return x


def _samples(case, seed, frame, step, count):
    """The training samples of one step: the first of 16 Philox candidates with
    a count of at least 8 (-1: none)."""
    i = torch.arange(case["batch"], device=count.device)
    pick = torch.full_like(i, -1)
    for tr in reversed(range(16)):
        x, _ = _philox(i, torch.full_like(i, step), torch.full_like(i, tr), seed & 0xFFFF, frame)
        j = (x * count.numel()) >> 32
        pick = torch.where(count[j] >= 8, j, pick)
    return pick


def _trained(case, seed, v, value, count):
    w = torch.from_numpy(_weights(seed)).double().to(value.device).requires_grad_()
    m, q = torch.zeros_like(w), torch.zeros_like(w)
    for step in range(case["steps"]):
        j = _samples(case, seed, WARM_FRAMES, step, count)
        j = j[j >= 0]
        loss = (_network(w, _encode(v, j)) - value[j]).square().sum() / (2 * case["batch"])
        g, = torch.autograd.grad(loss, w)
        m, q = 0.9 * m + 0.1 * g, 0.999 * q + 0.001 * g * g
        t = step + 1
        u = 1e-3 * (m / (1 - 0.9 ** t)) / ((q / (1 - 0.999 ** t)).sqrt() + 1e-8)
        w = (w.detach() - u).requires_grad_()
    return w.detach().cpu().numpy()


def _result(value) -> Dict[str, Optional[torch.Tensor]]:
    return {"r": value[:, 0], "g": value[:, 1], "b": value[:, 2], "count": None, "status": None}


def exact(case, seed):
    if case["migrate"]:
        return None  # the history's moves between levels have no short form
    views = _inputs(case, seed)
    if case["kind"] == "batch":
        return [_result(_filtered(case, v, eye, cfg, [WARM_FRAMES])[0]) for v, eye, cfg in views]
    v, eye, cfg = views[0]
    if case["kind"] in ("frame", "noalloc"):
        frames = range(WARM_FRAMES + 1) if case["hist"] else [WARM_FRAMES]
        return _result(_filtered(case, v, eye, cfg, frames)[0])
    value, count = _filtered(case, v, eye, cfg, range(WARM_FRAMES if case["hist"] else 1))
    if case["kind"] == "train":
        return _trained(case, seed, v, value, count)
    w = torch.from_numpy(_weights(seed)).double().to(value.device)
    for j in torch.nonzero(count < _LOWCOUNT).flatten().split(1 << 20):
        value[j] = _network(w, _encode(v, j))
    return _result(value)
