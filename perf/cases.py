"""Performance cases of the rasterizer: what its users have it do, through the public entry points.

  listed()            the named cases
  draw(rng)           one more case of the same ranges
  prepare(case, seed) scene, cameras, frame and buffers, on the GPU, from the seed alone
  run(state)          one pass
  work(case)          bytes and operations that one pass cannot do without
  exact(case, seed)   what run() returns, by the definitions (Eq. 2, Eq. 7 and their chain rule) in plain 64-bit torch

Kinds of pass:
  forward   binning, sort, render into buffers that the program keeps
  sensor    the same with the simulator's sensor outputs (depth, median depth, normals, instance mask)
  train     one optimisation step's device work: binning, sort + render + loss, backward
  autograd  render() under torch.autograd, the gradients of features and colour coming from the user's own head
  labels    query-guided instance labels of a whole scene

Scenes: "room" is the indoor stand-in of paper_2604_10951_gb300/scenes.py (thin surfels on the walls and objects of a
6 x 3 x 5 m room, seen from a circle inside it), "box" its small cloud in front of one camera; both drawn on the GPU.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2604_10951_gb300 import _lib as L
from paper_2604_10951_gb300 import raster, scenes

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
ROOM = (3.0, 1.5, 2.5)   # half sizes of the room (y down)
W_FEAT, W_RGB = 1.0, 1.0  # loss weights of a training step


def _case(kind, scene, n, views, c, dtype, k, stop="tmin", tile=16, sched="grid", sh=-1, lowpass=False, renorm=False):
    return dict(kind=kind, scene=scene, n=n, views=views, c=c, dtype=dtype, k=k, stop=stop, tile=tile, sched=sched,
                sh=sh, lowpass=lowpass, renorm=renorm)


def _labels(n, nq, dim, dtype):
    return dict(kind="labels", n=n, nq=nq, dim=dim, dtype=dtype)


def listed():
    mixed = ",".join(["320x240", "640x480", "1280x720"] * 4)
    return [
        # a viewer's frame of a small object: the smallest call, latency and launches
        dict(_case("forward", "box", 2000, "128x128", 16, "f32", 4), name="tiny_forward"),
        # fine-tuning on a preview-sized, ragged view through autograd
        dict(_case("autograd", "room", 100_000, "321x243", 32, "bf16", 8), name="preview_autograd"),
        # rendering FP32 features of a room from a Kinect-like camera
        dict(_case("forward", "room", 500_000, "640x480", 64, "f32", 8), name="room_forward_f32"),
        # the training step of the room: BF16 features, Top-K 8, exact stop
        dict(_case("train", "room", 500_000, "640x480", 64, "bf16", 8, "exact_topk"), name="room_train_bf16"),
        # the same step with full accumulation in FP32 (Eq. 2 without the selection), the accuracy baseline
        dict(_case("train", "room", 500_000, "640x480", 64, "f32", 0), name="room_train_full_f32"),
        # 16-d semantic features with the paper's K = 24 at the ScanNet colour resolution (968 rows: a ragged last tile row)
        dict(_case("autograd", "room", 500_000, "1296x968", 16, "f32", 24), name="scannet_autograd_k24"),
        # features of a dense scene at 720p
        dict(_case("forward", "room", 1_500_000, "1280x720", 128, "bf16", 8, "exact_topk"), name="large_forward_bf16"),
        # one step over twelve views of mixed size in one call: the largest
        dict(_case("train", "room", 1_000_000, mixed, 128, "bf16", 8, "exact_topk"), name="batched_train_bf16"),
        # a simulator's sensor frame: 32-d instance labels as features, their mask, depth images and normals
        dict(_case("sensor", "room", 500_000, "640x480", 32, "bf16", 8), name="sensor_frame"),
        # view-dependent colours (degree 3) with the low-pass filter and renormalised selection
        dict(_case("autograd", "room", 300_000, "640x480", 32, "f32", 8, sh=3, lowpass=True, renorm=True),
             name="sh_lowpass_autograd"),
        # instance labels of a room's Gaussians for 32 queries, for BF16 rendering
        dict(_labels(500_000, 32, 32, "bf16"), name="instance_labels"),
        # ... and of a dense scene for many queries with wide features, in FP32
        dict(_labels(1_200_001, 112, 64, "f32"), name="instance_labels_wide"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "forward", "sensor", "train", "train", "autograd", "autograd", "labels"])
    dtype = rng.choice(["f32", "bf16"])
    if kind == "labels":
        while True:
            c = _labels(_log_int(rng, 2000, 1_500_000), 16 * rng.randint(1, 12), 16 * rng.randint(1, 8), dtype)
            if c["n"] * c["nq"] <= 150_000_000:
                return c
    scene = rng.choice(["room", "room", "room", "box"])
    if scene == "box":
        n = _log_int(rng, 1000, 20_000)
        w = _log_int(rng, 48, 256)
        views = "%dx%d" % (w, max(16, int(w * rng.uniform(0.6, 1.2))))
    else:
        n = _log_int(rng, 50_000, 1_500_000)
        nv = rng.choice([1, 1, 1, 2, 5])
        sizes = []
        for _ in range(nv):
            w = _log_int(rng, 160, 1296 if nv == 1 else 640)
            sizes.append("%dx%d" % (w, int(w * rng.choice([0.75, 0.75, 0.5625, 1.0]))))
        views = ",".join(sizes)
        n = n if nv == 1 else min(n, 600_000)
    step = 8 if dtype == "bf16" else 4
    c = min(128, max(step, step * round(_log_int(rng, 8, 128) / step)))
    k = rng.choice([0, 3, 4, 8, 8, 8, 12, 16, 24, 32])
    if k == 0:
        c = min(c, 64)
    npx = sum(w * h for w, h in _sizes(dict(views=views)))
    while c > step and npx * c * (k or 25) > 1_500_000_000:  # well below the largest listed case
        c -= step
    stop = "tmin" if k == 0 else rng.choice(["tmin", "exact_topk"])
    variant = kind == "autograd" and rng.random() < 0.4
    return _case(kind, scene, n, views, c, dtype, k, stop, rng.choice([16, 16, 16, 8, 32]),
                 rng.choice(["grid", "grid", "persistent"]), rng.choice([0, 1, 2, 3]) if variant else -1,
                 variant and rng.random() < 0.5, variant and k > 0 and rng.random() < 0.5)


# ---- inputs ---------------------------------------------------------------------------------------------------------

def _sizes(case):
    return [tuple(int(x) for x in v.split("x")) for v in case["views"].split(",")]


def _unit(g, n, dev):
    q = torch.randn(n, 4, generator=g, device=dev)
    return q / q.norm(dim=1, keepdim=True)


def _room(n, c, g, rng, dev):
    """85 % of the surfels on the walls in proportion to their area, 15 % on 40 ellipsoids clear of the cameras' circle,
    normals along the surface; features and colours around one of 40 centres."""
    half = np.array(ROOM)
    blobs, radii = [], []
    while len(blobs) < 40:
        r = np.full(3, rng.uniform(0.15, 0.5)) if rng.random() < 0.5 else rng.uniform(0.15, 0.5, 3)
        m = 0.5 + r.max()
        for _ in range(10_000):
            p = rng.uniform(-half + m, half - m)
            if math.hypot(math.hypot(p[0], p[2]) - 1.0, p[1]) >= m:
                break
        blobs.append(p)
        radii.append(r)
    t = lambda a: torch.as_tensor(np.asarray(a, np.float32), device=dev)
    area = np.array([half[1] * half[2], half[1] * half[2], half[0] * half[2], half[0] * half[2], half[0] * half[1],
                     half[0] * half[1]])
    prob = np.concatenate([0.85 * area / area.sum(), np.full(40, 0.15 / 40)])
    part = torch.multinomial(t(prob), n, replacement=True, generator=g)
    wall = part < 6
    axis, sign = (part.clamp(max=5) // 2), (part % 2).float() * 2 - 1
    on = torch.nn.functional.one_hot(axis, 3).bool()
    h = t(half)
    p = (torch.rand(n, 3, generator=g, device=dev) * 2 - 1) * h
    flat = sign[:, None] * h + 0.002 * torch.randn(n, 3, generator=g, device=dev)
    p_wall = torch.where(on, flat, p)
    n_wall = torch.where(on, -sign[:, None].expand(n, 3), torch.zeros_like(p))
    b = (part - 6).clamp(min=0)
    d = torch.randn(n, 3, generator=g, device=dev)
    d = d / d.norm(dim=1, keepdim=True)
    rb = t(radii)[b]
    p_blob, n_blob = t(blobs)[b] + d * rb, d / rb
    means = torch.where(wall[:, None], p_wall, p_blob)
    nrm = torch.where(wall[:, None], n_wall, n_blob)
    nrm = nrm / nrm.norm(dim=1, keepdim=True)
    al = torch.stack([1 + nrm[:, 2], -nrm[:, 1], nrm[:, 0], torch.zeros_like(nrm[:, 0])], 1)
    al = torch.where((al[:, :1] < 1e-6), t([0.0, 1.0, 0.0, 0.0]).expand(n, 4), al)
    al = al / al.norm(dim=1, keepdim=True)
    phi = torch.rand(n, generator=g, device=dev) * math.pi
    cw, cz = torch.cos(phi), torch.sin(phi)
    w, x, y, z = al.unbind(1)
    quats = torch.stack([w * cw - z * cz, x * cw + y * cz, y * cw - x * cz, w * cz + z * cw], 1)
    scales = torch.exp(-4.5 + 0.6 * torch.randn(n, 2, generator=g, device=dev))
    opac = torch.sigmoid(1.0 + 1.5 * torch.randn(n, generator=g, device=dev))
    cl = torch.where(wall, part, b)
    centres = torch.randn(40, c, generator=g, device=dev)
    feats = 0.1 * torch.randn(n, c, generator=g, device=dev)
    feats += centres[cl]
    base = torch.rand(40, 3, generator=g, device=dev)
    rgb = (base[cl] + 0.05 * torch.randn(n, 3, generator=g, device=dev)).clamp_(0, 1)
    return means, scales, quats, opac, rgb, feats


def _box(n, c, g, dev):
    """Surfels uniform in [-1, 1]^3 with random rotations."""
    means = torch.rand(n, 3, generator=g, device=dev) * 2 - 1
    scales = torch.exp(-3.0 + 0.5 * torch.randn(n, 2, generator=g, device=dev))
    opac = torch.sigmoid(torch.randn(n, generator=g, device=dev))
    return (means, scales, _unit(g, n, dev), opac, torch.rand(n, 3, generator=g, device=dev),
            torch.randn(n, c, generator=g, device=dev))


def _cameras(case, rng):
    """(fx, fy, cx, cy, w, h, 3x4 world->camera, near) per view: box, from 3 m in front; room, on the 1 m circle looking
    outward with a 30 degree turn and 10 degrees down, field of view as a Kinect's."""
    out = []
    sizes = _sizes(case)
    for i, (w, h) in enumerate(sizes):
        if case["scene"] == "box":
            vm = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 1, 3.0]], np.float32)
            out.append((float(w), float(w), w / 2.0, h / 2.0, w, h, vm, 0.2))
            continue
        th = 2 * math.pi * ((i + rng.uniform(0, 1)) / len(sizes))
        yaw, pitch = th + math.radians(30.0), math.radians(10.0)
        f = np.array([math.cos(pitch) * math.cos(yaw), math.sin(pitch), math.cos(pitch) * math.sin(yaw)])
        r = np.cross([0.0, 1.0, 0.0], f)
        r /= np.linalg.norm(r)
        rot = np.stack([r, np.cross(f, r), f])
        pos = np.array([math.cos(th), 0.0, math.sin(th)])
        fx = float(np.float32(525.0 / 640.0 * w if w * 9 != h * 16 else 900.0 / 1280.0 * w))
        out.append((fx, fx, w / 2.0, h / 2.0, w, h, np.concatenate([rot, -rot @ pos[:, None]], 1).astype(np.float32),
                    0.2))
    return out


def _render_inputs(case, seed):
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed * 7919 + 11)
    rng = np.random.default_rng(seed)
    dt = DTYPES[case["dtype"]]
    n, c = case["n"], case["c"]
    means, scales, quats, opac, rgb, feats = _room(n, c, g, rng, dev) if case["scene"] == "room" else _box(n, c, g, dev)
    s = dict(means=means, scales=scales, quats=quats, opac=opac, rgb=rgb, feats=feats.to(dt), cams=_cameras(case, rng))
    if case["sh"] >= 0:  # colour coefficients: the base colour, then falling higher orders
        nb = (case["sh"] + 1) ** 2
        k = 0.15 * torch.randn(n, nb, 3, generator=g, device=dev)
        k[:, 0] = (rgb - 0.5) / 0.28209479177387814
        s["rgb"] = k.contiguous()
    npx = sum(w * h for w, h in _sizes(case))
    if case["kind"] == "train":
        s["f_tgt"] = torch.randn(npx, c, generator=g, device=dev, dtype=torch.float32).to(dt)
        s["rgb_tgt"] = torch.rand(npx, 3, generator=g, device=dev)
    elif case["kind"] == "autograd":  # what the user's head and colour loss send back
        s["d_feat"] = (torch.randn(npx, c, generator=g, device=dev) / (npx * c)).to(dt)
        s["d_rgb"] = torch.randn(npx, 3, generator=g, device=dev).sign_() / (3 * npx)
    return s


def _label_inputs(case, seed):
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed * 7919 + 13)
    n, nq, dim = case["n"], case["nq"], case["dim"]
    h = torch.tensor(ROOM, device=dev)
    means = (torch.rand(n, 3, generator=g, device=dev) * 2 - 1) * h
    p_q = (torch.rand(nq, 3, generator=g, device=dev) * 2 - 1) * (h - 0.5)
    sig = 0.4 + 0.8 * torch.rand(nq, 3, generator=g, device=dev)
    rot = _rotation(_unit(g, nq, dev).double())
    prec = rot @ torch.diag_embed(sig.double() ** -2) @ rot.transpose(1, 2)
    prec = torch.stack([prec[:, 0, 0], prec[:, 1, 1], prec[:, 2, 2], prec[:, 0, 1], prec[:, 0, 2], prec[:, 1, 2]], 1)
    f_q = 3.0 / math.sqrt(dim) * torch.randn(nq, dim, generator=g, device=dev)
    near = torch.cat([torch.cdist(m, p_q).argmin(1) for m in means.split(1 << 18)])
    f_ins = f_q[near] + 0.3 / math.sqrt(dim) * torch.randn(n, dim, generator=g, device=dev)
    return dict(means=means, f_ins=f_ins.bfloat16(), f_q=f_q.bfloat16(), p_q=p_q, prec=prec.float().contiguous())


# ---- passes ---------------------------------------------------------------------------------------------------------

def prepare(case, seed):
    if case["kind"] == "labels":
        s = _label_inputs(case, seed)
        s.update(case=case, err=torch.zeros(1, dtype=torch.int32, device="cuda"))
        return s
    s = _render_inputs(case, seed)
    s["case"] = case
    dt = DTYPES[case["dtype"]]
    cams = [scenes.Camera(*c) for c in s["cams"]]
    params = raster.make_params(C=case["c"], K=case["k"], tile_size=case["tile"], stop_rule=case["stop"], feat_dtype=dt,
                                schedule=case["sched"], lowpass=case["lowpass"], renorm=case["renorm"],
                                sh_degree=case["sh"] if case["sh"] >= 0 else None)
    fr = raster.Frame(cams, case["n"], params, pair_capacity=1 << 12, deferred=True)
    geo = (s["means"], s["scales"], s["quats"], s["opac"])
    fr.grow(fr.bin_and_sort(*geo))  # a workspace for this scene, with margin
    s["frame"] = fr
    npx, dev = fr.total_pix, fr.device
    if case["kind"] == "autograd":
        for k in ("means", "scales", "quats", "opac", "rgb", "feats"):
            s[k].requires_grad_(True)
        return s
    s["out"] = fr.new_outputs()
    if case["kind"] == "sensor":
        s["aux"] = (torch.empty(npx, device=dev), torch.empty(npx, device=dev), torch.empty(npx, 3, device=dev))
        s["label"] = torch.empty(npx, dtype=torch.int32, device=dev)
    elif case["kind"] == "train":
        s["d_feat"] = torch.empty_like(s["out"][0])
        s["d_rgb"] = torch.empty_like(s["out"][1])
        s["loss"] = torch.zeros(1, dtype=torch.float64, device=dev)
        s["grads"] = [torch.empty_like(s[k]) for k in ("means", "scales", "quats", "opac", "rgb", "feats")]
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "labels":
        return raster.query_labels(s["f_ins"], s["means"], s["f_q"], s["p_q"], s["prec"],
                                   out_dtype=DTYPES[case["dtype"]], err=s["err"])
    fr = s["frame"]
    geo = (s["means"], s["scales"], s["quats"], s["opac"])
    if case["kind"] == "autograd":
        F, rgb, T, ids = raster.render(*geo, s["rgb"], s["feats"], fr)
        grads = torch.autograd.grad([F, rgb], [*geo, s["rgb"], s["feats"]], [s["d_feat"], s["d_rgb"]])
        return [F, rgb, T, ids, list(grads)]
    F, rgb, T, ids = s["out"]
    fr.project_bin(*geo)
    if case["kind"] == "train":
        fr.sort_render_forward_loss(s["rgb"], s["feats"], F, rgb, T, ids, s["f_tgt"], s["rgb_tgt"], W_FEAT, W_RGB,
                                    s["d_feat"], s["d_rgb"], s["loss"])
        fr.render_backward(*geo, s["rgb"], s["feats"], T, s["d_feat"], s["d_rgb"], None, *s["grads"])
        return [F, rgb, T, ids, s["loss"], s["grads"]]
    fr.sort()
    if case["kind"] == "sensor":
        d, dm, nrm = s["aux"]
        fr.render_forward_aux(s["rgb"], s["feats"], F, rgb, T, ids, d, dm, nrm, label=s["label"])
        return [F, rgb, T, ids, d, dm, nrm, s["label"]]
    fr.render_forward(s["rgb"], s["feats"], F, rgb, T, ids)
    return [F, rgb, T, ids]


# ---- work -----------------------------------------------------------------------------------------------------------

def work(case):
    """Bytes: every surfel's geometry, the colours and feature rows of the visible surfels (all of a box; about one in
    sixteen of a room per view), every per-pixel input and output once, every gradient once.  Operations: about 60
    surfels meet a pixel (some 30 operations each, twice that for the replay), then 2 C per selected surfel and pass."""
    s = 2 if case["dtype"] == "bf16" else 4
    if case["kind"] == "labels":
        n, nq, dim = case["n"], case["nq"], case["dim"]
        return {"bytes": n * (2 * dim + 12 + nq * s) + nq * (2 * dim + 36), "flops": n * nq * (2 * dim + 25)}
    n, c, k = case["n"], case["c"], case["k"]
    sizes = _sizes(case)
    npx = sum(w * h for w, h in sizes)
    vis = n if case["scene"] == "box" else min(n, n * len(sizes) // 16)
    col = 12 if case["sh"] < 0 else 12 * (case["sh"] + 1) ** 2
    sel = k if k else 25
    b = n * 40 + vis * (col + c * s) + npx * (c * s + 16 + 4 * k)
    f = npx * (60 * 30 + 2 * c * sel)
    if case["kind"] == "sensor":
        b += npx * 24
    if case["kind"] == "train":
        b += npx * (2 * c * s + 24 + 8)  # targets, and their gradients
    if case["kind"] == "autograd":
        b += npx * (c * s + 12)
    if case["kind"] in ("train", "autograd"):
        b += n * (40 + col + c * s)
        f += npx * (60 * 60 + 4 * c * sel)
    return {"bytes": b, "flops": f}


# ---- the definitions in 64 bits -------------------------------------------------------------------------------------

def _rotation(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)], 1),
                        torch.stack([2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)], 1),
                        torch.stack([2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1)], 1)


def _harmonics(deg, d):
    """Real spherical harmonics without the Condon-Shortley sign, b = l^2 + l + m."""
    x, y, z = d.unbind(1)
    pi = math.pi
    Y = [torch.full_like(x, 0.5 * math.sqrt(1 / pi))]
    if deg >= 1:
        a = math.sqrt(3 / (4 * pi))
        Y += [a * y, a * z, a * x]
    if deg >= 2:
        a = 0.5 * math.sqrt(15 / pi)
        Y += [a * x * y, a * y * z, 0.25 * math.sqrt(5 / pi) * (3 * z * z - 1), a * x * z, a / 2 * (x * x - y * y)]
    if deg >= 3:
        a, b, c = 0.25 * math.sqrt(35 / (2 * pi)), 0.5 * math.sqrt(105 / pi), 0.25 * math.sqrt(21 / (2 * pi))
        Y += [a * y * (3 * x * x - y * y), b * x * y * z, c * y * (5 * z * z - 1),
              0.25 * math.sqrt(7 / pi) * z * (5 * z * z - 3), c * x * (5 * z * z - 1), b / 2 * z * (x * x - y * y),
              a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, 1)


class _View:
    """One view: the contributions of every pixel in depth order (no gradients), then the outputs from the leaves."""

    def __init__(self, case, leaf, cam):
        fx, fy, cx, cy, self.w, self.h, vm, self.near = cam
        f32 = lambda v: float(np.float32(v))
        dev = leaf["means"].device
        self.case, self.leaf, self.npx = case, leaf, self.w * self.h
        self.R = torch.as_tensor(vm[:, :3].astype(np.float64), device=dev)
        self.t = torch.as_tensor(vm[:, 3].astype(np.float64), device=dev)
        self.Kc = torch.tensor([[f32(fx), 0, f32(cx)], [0, f32(fy), f32(cy)], [0, 0, 1]], dtype=torch.float64,
                               device=dev)
        self.vm32, self.near = vm, f32(self.near)
        self.amin, self.amax, self.tmin = f32(1.0 / 255.0), f32(0.99), f32(1e-4)

    def rows(self, idx):
        """Homography of the surfels idx: its adjugate's rows [n, 9], determinant, projected centre, camera centre."""
        lf = self.leaf
        rot = _rotation(lf["quats"][idx])
        tu = lf["scales"][idx, 0:1] * rot[:, :, 0] @ self.R.T
        tv = lf["scales"][idx, 1:2] * rot[:, :, 1] @ self.R.T
        pc = lf["means"][idx] @ self.R.T + self.t
        c0, c1, c2 = tu @ self.Kc.T, tv @ self.Kc.T, pc @ self.Kc.T
        a0, a1, a2 = (torch.linalg.cross(c1, c2), torch.linalg.cross(c2, c0), torch.linalg.cross(c0, c1))
        return torch.cat([a0, a1, a2], 1), (c0 * a0).sum(1), c2[:, :2] / c2[:, 2:], pc

    def hit(self, m, ctr, o, x, y):
        c = [m[:, 3 * r] * x + m[:, 3 * r + 1] * y + m[:, 3 * r + 2] for r in range(3)]
        rho = (c[0] * c[0] + c[1] * c[1]) / (c[2] * c[2])
        scr = torch.zeros_like(rho, dtype=torch.bool)
        if self.case["lowpass"]:
            rs = 2 * ((x - ctr[:, 0]) ** 2 + (y - ctr[:, 1]) ** 2)
            scr = ~(rho <= rs)
            rho = torch.where(scr, rs, rho)
        return o * torch.exp(-0.5 * rho), c[2], scr

    @torch.no_grad()
    def contributions(self):
        lf, v = self.leaf, self.vm32
        m32 = lf["means"].float()
        z32 = (m32[:, 0] * float(v[2, 0]) + m32[:, 1] * float(v[2, 1])) + m32[:, 2] * float(v[2, 2]) + float(v[2, 3])
        pc = lf["means"] @ self.R.T + self.t
        idx = ((pc[:, 2] > self.near) & (lf["opac"] >= self.amin)).nonzero()[:, 0]
        m, det, ctr, pc = self.rows(idx)
        lim = 1e-3 * self.Kc[0, 0] * self.Kc[1, 1] * lf["scales"][idx].prod(1) * pc.norm(dim=1)
        keep = det.abs() > lim
        idx, m, det, ctr = idx[keep], m[keep], det[keep], ctr[keep]
        # pixel box of the disc u^2 + v^2 <= k^2 (a little widened), all pixels where the conic is no ellipse
        kb = 2 * torch.log(lf["opac"][idx] / self.amin) * 1.001 + 1e-9
        sh = torch.stack([m[:, 3 * r] * ctr[:, 0] + m[:, 3 * r + 1] * ctr[:, 1] + m[:, 3 * r + 2] for r in range(3)], 1)
        a = torch.stack([m.view(-1, 3, 3)[:, :, 0], m.view(-1, 3, 3)[:, :, 1], sh], 2)  # about the centre
        a = a / a.abs().amax((1, 2), keepdim=True)
        q = lambda i, j: a[:, 0, i] * a[:, 0, j] + a[:, 1, i] * a[:, 1, j] - kb * a[:, 2, i] * a[:, 2, j]
        A, B, C, D, E, F = q(0, 0), q(0, 1), q(1, 1), q(0, 2), q(1, 2), q(2, 2)
        gd = A * C - B * B
        ell = (A > 0) & (gd > 0)
        X, Y = (B * E - C * D) / gd, (B * D - A * E) / gd
        fp = -(F + D * X + E * Y)
        hx, hy = (fp * C / gd).clamp(min=0).sqrt(), (fp * A / gd).clamp(min=0).sqrt()
        none = ell & ~(fp > 0)
        lo, hi = torch.stack([X - hx, Y - hy], 1), torch.stack([X + hx, Y + hy], 1)
        if self.case["lowpass"]:
            r = (0.5 * kb).sqrt()[:, None]
            lo = torch.where(none[:, None], -r, torch.minimum(lo, -r))
            hi = torch.where(none[:, None], r, torch.maximum(hi, r))
            none = torch.zeros_like(none)
        size = torch.tensor([self.w, self.h], dtype=torch.float64, device=m.device)
        lo = torch.where(ell[:, None], (lo + ctr - 0.5).ceil(), torch.zeros_like(lo))
        hi = torch.where(ell[:, None], (hi + ctr - 0.5).floor(), size - 1)
        lo, hi = lo.clamp(min=0), torch.minimum(hi, size - 1)
        n_box = ((hi - lo + 1).clamp(min=0)).prod(1)
        keep = (n_box > 0) & ~none
        idx, m, det, ctr, lo, hi, n_box = (t[keep] for t in (idx, m, det, ctr, lo, hi, n_box))
        order = torch.argsort(z32[idx], stable=True)  # idx ascends: ties by index
        idx, m, det, ctr, lo, hi, n_box = (t[order] for t in (idx, m, det, ctr, lo, hi, n_box))
        n_box, x0, y0 = n_box.long(), lo[:, 0].long(), lo[:, 1].long()
        bw = (hi[:, 0] - lo[:, 0] + 1).long()
        total = torch.cumsum(n_box, 0)
        got, at, done = [(idx[:0].int(), idx[:0].int())], 0, 0
        while at < idx.numel():
            end = max(at + 1, int(torch.searchsorted(total, done + (1 << 25), right=True)))
            j = torch.repeat_interleave(torch.arange(at, end, device=m.device), n_box[at:end])
            k = torch.arange(j.numel(), device=m.device) - (total[j] - n_box[j] - done)
            px, py = x0[j] + k % bw[j], y0[j] + k // bw[j]
            x, y = px + 0.5, py + 0.5
            al, c2, scr = self.hit(m[j], ctr[j], lf["opac"][idx[j]], x, y)
            ok = (al >= self.amin) & (scr | (det[j] / c2 > self.near))
            got.append((j[ok].int(), (py[ok] * self.w + px[ok]).int()))
            done, at = int(total[end - 1]), end
        sid, pix = torch.cat([g[0] for g in got]), torch.cat([g[1] for g in got])
        pix, o = torch.sort(pix, stable=True)
        return idx, sid[o].long(), pix.long()

    @torch.no_grad()
    def traverse(self, idx, sid, pix):
        """Which contributions are composited (stop rules), and the selected ones of each pixel [npx, K] (-1: none)."""
        case, K, dev = self.case, self.case["k"], sid.device
        m, _, ctr, _ = self.rows(idx)
        al = torch.empty(sid.numel(), dtype=torch.float64, device=dev)
        for a in range(0, sid.numel(), 1 << 24):
            j, p = sid[a:a + (1 << 24)], pix[a:a + (1 << 24)]
            al[a:a + (1 << 24)] = self.hit(m[j], ctr[j], self.leaf["opac"][idx[j]], p % self.w + 0.5,
                                           p // self.w + 0.5)[0].clamp(max=self.amax)
        cnt = torch.bincount(pix, minlength=self.npx)
        start = torch.cumsum(cnt, 0) - cnt
        inc = torch.zeros(sid.numel(), dtype=torch.bool, device=dev)
        T = torch.ones(self.npx, dtype=torch.float64, device=dev)
        tw = torch.full((self.npx, max(K, 1)), -math.inf, dtype=torch.float64, device=dev)
        ti = torch.full((self.npx, max(K, 1)), -1, dtype=torch.int64, device=dev)
        act, d = (cnt > 0).nonzero()[:, 0], 0
        while act.numel():
            i = start[act] + d
            a, Ta = al[i], T[act]
            Tn = Ta * (1 - a)
            go = Tn >= self.tmin
            act, i, a, Ta, Tn = act[go], i[go], a[go], Ta[go], Tn[go]
            inc[i] = True
            T[act] = Tn
            more = cnt[act] > d + 1
            if K:
                w = a * Ta
                low, slot = tw[act].min(1)
                put = w > low
                tw[act[put], slot[put]] = w[put]
                ti[act[put], slot[put]] = i[put]
                if case["stop"] == "exact_topk":
                    more &= ~(self.amax * Tn <= tw[act].min(1).values)
            act, d = act[more], d + 1
        new = torch.cumsum(inc, 0) - 1
        return sid[inc], pix[inc], torch.where(ti >= 0, new[ti.clamp(min=0)], ti)

    def colours(self, idx):
        lf = self.leaf
        if self.case["sh"] < 0:
            return lf["rgb"][idx]
        d = lf["means"][idx] + self.R.T @ self.t
        Y = _harmonics(self.case["sh"], d / d.norm(dim=1, keepdim=True))
        return (0.5 + torch.einsum("nb,nbc->nc", Y, lf["rgb"][idx])).clamp(min=0)

    def outputs(self):
        """[F, rgb, T] and the sensor images, differentiable with respect to the leaves."""
        case, lf, npx = self.case, self.leaf, self.npx
        idx, sid, pix = self.contributions()
        sid, pix, sel = self.traverse(idx, sid, pix)
        m, det, ctr, pc = self.rows(idx)
        x, y = pix % self.w + 0.5, pix // self.w + 0.5
        raw, c2, scr = self.hit(m.index_select(0, sid), ctr.index_select(0, sid),
                                lf["opac"][idx].index_select(0, sid), x, y)
        al = raw.clamp(max=self.amax)
        lg = torch.log1p(-al)
        cs = torch.cumsum(lg, 0)
        cnt = torch.bincount(pix, minlength=npx)
        first = torch.cumsum(cnt, 0) - cnt
        before = torch.cat([torch.zeros_like(cs[:1]), cs])  # sum over all earlier contributions
        logT = before[:-1] - before.index_select(0, first).index_select(0, pix)
        w = al * torch.exp(logT)
        zero = lambda *s: torch.zeros(*s, dtype=torch.float64, device=sid.device)
        T = torch.exp(zero(npx).index_add(0, pix, lg))
        rgb = zero(npx, 3).index_add(0, pix, w[:, None] * self.colours(idx).index_select(0, sid))
        feats = lf["feats"]
        if case["k"]:
            ww = torch.cat([w, zero(1)])[sel]  # -1: the zero at the end
            if case["renorm"]:
                s = ww.sum(1, keepdim=True)
                ww = torch.where(s > 0, ww / torch.where(s > 0, s, torch.ones_like(s)), ww)
            rows = idx[sid][sel.clamp(min=0)]
            parts = []
            for c0 in range(0, feats.shape[1], 32):
                fc = feats[:, c0:c0 + 32]
                parts.append(torch.einsum("pk,pkc->pc", ww, fc.index_select(0, rows.reshape(-1)).view(*rows.shape, -1)))
            F = torch.cat(parts, 1)
        else:
            F = torch.cat([zero(npx, min(16, feats.shape[1] - c0)).index_add(
                0, pix, w[:, None] * feats[:, c0:c0 + 16].index_select(0, idx).index_select(0, sid))
                for c0 in range(0, feats.shape[1], 16)], 1)
        out = [F, rgb, T]
        if case["kind"] == "sensor":
            z = torch.where(scr, pc[sid, 2], det[sid] / c2)
            half = (T_after := torch.exp(logT + lg)) < 0.5
            ahead = torch.cumsum(half, 0) - half.long()
            firsts = half & (ahead == torch.cat([ahead, ahead[-1:]])[first][pix])
            med = zero(npx)
            med[pix[firsts]] = z[firsts]
            rot = _rotation(lf["quats"][idx])
            n = torch.linalg.cross(rot[:, :, 0], rot[:, :, 1]) @ self.R.T
            n = torch.where(((n * pc).sum(1) > 0)[:, None], -n, n)
            del T_after
            out += [zero(npx).index_add(0, pix, w * z), med, zero(npx, 3).index_add(0, pix, w[:, None] * n[sid])]
        return out


def _exact_labels(case, seed):
    s = _label_inputs(case, seed)
    out = torch.empty(case["n"], case["nq"], dtype=torch.float64, device="cuda")
    fq, pq, p = s["f_q"].double(), s["p_q"].double(), s["prec"].double()
    P = torch.stack([p[:, [0, 3, 4]], p[:, [3, 1, 5]], p[:, [4, 5, 2]]], 1)
    for a in range(0, case["n"], 1 << 17):
        b = slice(a, a + (1 << 17))
        sim = torch.sigmoid(s["f_ins"][b].double() @ fq.T)
        d = s["means"][b].double()[:, None] - pq[None]
        prox = torch.exp(-0.5 * torch.einsum("nqi,qij,nqj->nq", d, P, d))
        out[b] = torch.softmax(sim * prox, 1)
    return out


def exact(case, seed):
    if case["kind"] == "labels":
        return _exact_labels(case, seed)
    s = _render_inputs(case, seed)
    names = ("means", "scales", "quats", "opac", "rgb", "feats")
    grad = case["kind"] in ("train", "autograd")
    leaf = {k: s[k].double().requires_grad_(grad) for k in names}
    npx = sum(w * h for w, h in _sizes(case))
    outs, loss, at = [], torch.zeros(1, dtype=torch.float64, device="cuda"), 0
    for cam in s["cams"]:  # a view at a time: the gradients add up in the leaves
        v = _View(case, leaf, cam)
        with torch.set_grad_enabled(grad):
            o = v.outputs()
        px = slice(at, at + v.npx)
        at += v.npx
        if case["kind"] == "train":
            part = (W_FEAT * ((o[0] - s["f_tgt"][px].double()) ** 2).sum() / (npx * case["c"]) +
                    W_RGB * (o[1] - s["rgb_tgt"][px].double()).abs().sum() / (3 * npx))
            part.backward()
            loss += part.detach()
        elif case["kind"] == "autograd":
            torch.autograd.backward([o[0], o[1]], [s["d_feat"][px].double(), s["d_rgb"][px].double()])
        outs.append([t.detach() for t in o])
    o = [torch.cat(t) for t in zip(*outs)]
    got = [o[0], o[1], o[2], None]
    if case["kind"] == "sensor":
        return got + o[3:] + [None]
    if grad:
        g = [leaf[k].grad if leaf[k].grad is not None else torch.zeros_like(leaf[k]) for k in names]
        got += ([loss] if case["kind"] == "train" else []) + [g]
    return got
