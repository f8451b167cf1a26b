"""The work a user has this library do, as cases that can be timed and compared.

A case is one call chain through the public entry points (raster.Frame / Adam / rasterize, train.PlainTrainer,
train.BatchedTrainer, init.*), on synthetic Richtmyer-Meshkov-like interfaces: the workloads of bench.py and of the
tests, from one 64x64 image of 500 Gaussians to the merged 4K render of 100M.  Inputs are made on the device from the
seed alone; ground-truth images and masks are point splats drawn by plain torch, so no input depends on a kernel.

exact() restates what a case computes in 64 bits with torch alone: projection, per-tile lists, blending and its
gradient (autograd), loss, Adam, nearest neighbours and the initialiser network.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import synth
from paper_2509_12138_gb300 import init as ginit
from paper_2509_12138_gb300.raster import Adam, Frame, Owned, Units, pack_cameras, rasterize
from paper_2509_12138_gb300.train import BatchedTrainer, PlainTrainer

BG = (1.0, 1.0, 1.0)
LAM = 0.2                      # weight of 1 - SSIM (bench.py)
Y00 = 0.28209479177387814
T0 = 1000                      # optimiser steps behind a training case
LR_STEPS = 7000
SLABS = (0.5, 1.5, 2.5, 3.5, 4.0, 4.5, 5.5, 6.0)  # relative x-slab populations of the partitioned scene
DEV = "cuda"


def listed():
    return [
        # the gradient check of a small scene through autograd: 500 Gaussians, all 59 parameters, 64x64 (latency)
        dict(name="autograd-500", kind="autograd", n=500, w=64, h=64, deg=3),
        # the small training workload: 2,000 Gaussians on a sphere, 8 views of 128x128 as units of one call, then
        # the projection backward summed over the views and a separate Adam step
        dict(name="views-2k", kind="views", n=2000, w=128, h=128, deg=0, views=8),
        # one training step of PlainTrainer, quick-check size (bench.py iso200k-540p)
        dict(name="train-200k-540p", kind="train", n=200_000, modes=8, w=960, h=540, deg=3, sparse=False),
        # one training step of PlainTrainer at 1M Gaussians (bench.py iso1M-1080p)
        dict(name="train-1M-1080p", kind="train", n=1_000_000, modes=8, w=1920, h=1080, deg=3, sparse=False),
        # the headline step: 10M Gaussians at 1080p, the next view's projection inside the Adam kernel
        dict(name="train-10M-1080p", kind="train_next", n=10_000_000, modes=16, w=1920, h=1080, deg=3),
        # bitwise reproducible gradients (fixed-point accumulation), a ragged image and SH degree 2
        dict(name="grads-det-700k", kind="grads", n=700_000, modes=8, w=1011, h=757, deg=2),
        # forward only: viewing a trained 10M scene (bench.py's render metric)
        dict(name="render-10M-1080p", kind="render", n=10_000_000, modes=16, w=1920, h=1080, deg=3, whole=False),
        # the merged render of 8 ghost-celled partitions at 4K (bench.py merge100M-4k)
        dict(name="merge-100M-4k", kind="merge", n=100_000_000, modes=32, w=3840, h=2160, deg=3, parts=8),
        # one graph-captured step of 8 uneven partitions (bench.py batched28M-1080p at a tenth of its points)
        dict(name="batched-2.8M-1080p", kind="batched", n=2_800_000, modes=8, w=1920, h=1080, deg=3, parts=8, vps=1),
        # learned initialisation of 1M points: 16 nearest neighbours, then the network
        dict(name="init-1M", kind="init", n=1_000_000, modes=8),
        # one step of the network's fit on the 2M-point subset the 30M experiment uses
        dict(name="fit-2M", kind="fit", n=2_000_000, modes=8),
        # the masked loss and its image gradient alone, one image of the paper's larger square size
        dict(name="loss-2048sq", kind="loss", w=2048, h=2048, units=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["autograd", "views", "train", "train", "train_next", "grads", "render", "merge", "batched",
                       "init", "fit", "loss"])
    if kind == "autograd":
        return dict(kind=kind, n=_log_int(rng, 50, 3000), w=rng.randint(24, 200), h=rng.randint(24, 200),
                    deg=rng.randint(0, 3))
    if kind == "views":
        return dict(kind=kind, n=_log_int(rng, 500, 20_000), w=rng.randint(48, 256), h=rng.randint(48, 256),
                    deg=rng.randint(0, 3), views=rng.randint(1, 8))
    w, h = rng.randint(400, 2048), rng.randint(300, 1440)
    modes = rng.choice([8, 16, 32])
    if kind == "train":
        return dict(kind=kind, n=_log_int(rng, 40_000, 6_000_000), modes=modes, w=w, h=h, deg=rng.randint(0, 3),
                    sparse=rng.random() < 0.25)
    if kind == "train_next":
        return dict(kind=kind, n=_log_int(rng, 300_000, 10_000_000), modes=modes, w=w, h=h, deg=3)
    if kind == "grads":
        return dict(kind=kind, n=_log_int(rng, 40_000, 3_000_000), modes=modes, w=w, h=h, deg=rng.randint(0, 3))
    if kind == "render":
        return dict(kind=kind, n=_log_int(rng, 100_000, 10_000_000), modes=modes, w=w, h=h, deg=rng.randint(0, 3),
                    whole=rng.random() < 0.4)
    if kind == "merge":
        return dict(kind=kind, n=_log_int(rng, 3_000_000, 40_000_000), modes=modes, w=rng.randint(1000, 3840),
                    h=rng.randint(700, 2160), deg=3, parts=rng.choice([2, 4, 8]))
    if kind == "batched":
        return dict(kind=kind, n=_log_int(rng, 200_000, 4_000_000), modes=modes, w=w, h=h, deg=3,
                    parts=rng.randint(2, 8), vps=rng.randint(1, 2))
    if kind == "init":
        return dict(kind=kind, n=_log_int(rng, 20_000, 2_000_000), modes=modes)
    if kind == "fit":
        return dict(kind=kind, n=_log_int(rng, 30_000, 2_500_000), modes=modes)
    return dict(kind=kind, w=rng.randint(200, 2048), h=rng.randint(200, 2048), units=rng.randint(1, 4))


# ---------------------------------------------------------------- inputs
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1_000_003 + salt) & 0x7FFFFFFF)
    return g


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device=DEV)


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device=DEV)


def _bits2(v):
    q = (v.double() * 65535.0).long()
    for s, m in ((8, 0x00FF00FF), (4, 0x0F0F0F0F), (2, 0x33333333), (1, 0x55555555)):
        q = (q | (q << s)) & m
    return q


def _planes(deg):
    return 3 + (3 * (deg + 1) ** 2 + 3) // 4


def _surface(n, modes, seed, strips=None):
    """Points [n, 3] of the interface z = 0.5 + 0.1 sum_k a_k sin(2 pi (kx x + ky y) + phi_k) in the Z-order an
    extraction emits, with unit normals, Lambert colours and the mean distance to the three nearest neighbours.
    strips (edges, counts): that many points in each x-strip instead of a uniform density; their strip comes too."""
    r = np.random.default_rng([int(seed), 77])
    k = np.arange(1, modes + 1)
    th = r.uniform(0, 2 * math.pi, modes)
    t = lambda a: torch.tensor(a, dtype=torch.float32, device=DEV)  # noqa: E731
    amp, kx, ky, ph = t(r.uniform(0, 1, modes) / k), t(k * np.cos(th)), t(k * np.sin(th)), t(r.uniform(0, 2 * math.pi, modes))
    g = _gen(seed, 1)
    x, y = _rand(g, n), _rand(g, n)
    strip = None
    if strips is not None:
        edges = t(strips[0])
        strip = torch.repeat_interleave(torch.arange(len(strips[1]), device=DEV), torch.tensor(strips[1], device=DEV))
        x = edges[strip] + x * (edges[strip + 1] - edges[strip])
    o = torch.argsort(_bits2(x) | (_bits2(y) << 1), stable=True)
    x, y = x[o], y[o]
    strip = None if strip is None else strip[o]
    del o
    p = torch.empty((n, 3), device=DEV)
    nrm = torch.empty((n, 3), device=DEV)
    col = torch.empty((n, 3), device=DEV)
    area = 0.0
    for a in range(0, n, 1 << 22):
        b = min(n, a + (1 << 22))
        arg = 2 * math.pi * (x[a:b, None] * kx + y[a:b, None] * ky) + ph
        c = 0.2 * math.pi * torch.cos(arg) * amp
        hx, hy = (c * kx).sum(1), (c * ky).sum(1)
        z = 0.5 + 0.1 * (torch.sin(arg) * amp).sum(1)
        p[a:b, 0], p[a:b, 1], p[a:b, 2] = x[a:b], y[a:b], z
        il = 1.0 / torch.sqrt(hx * hx + hy * hy + 1.0)
        nrm[a:b, 0], nrm[a:b, 1], nrm[a:b, 2] = -hx * il, -hy * il, il
        area += (1.0 / il).sum()
        zn = ((z - 0.2) / 0.6).clamp(0, 1)
        shade = 0.2 + 0.8 * ((-0.3 * hx - 0.5 * hy + 0.8) * il / math.sqrt(0.98)).abs()
        col[a:b] = (torch.stack([0.2 + 0.75 * zn, 0.4 + 0.2 * zn, 0.9 - 0.7 * zn], 1) * shade[:, None]).clamp(0, 1)
    spacing = (0.5 + 0.75 + 0.9375) / 3.0 / math.sqrt(n / (float(area) / n))
    return (p, nrm, col, spacing) if strips is None else (p, nrm, col, spacing, strip)


def _splats(pts, nrm, col, spacing, deg, seed, age):
    """Parameter planes: "mid" = some way into training, "trained" = opaque, flattened splats along the surface."""
    n = pts.shape[0]
    g = _gen(seed, 2)
    P = torch.zeros((_planes(deg), n, 4), device=DEV)
    P[0, :, :3] = pts + 0.2 * spacing * _randn(g, n, 3)
    trained = age == "trained"
    P[1, :, :3] = math.log(spacing) + (0.1 if trained else 0.0) + (0.3 if trained else 0.2) * _randn(g, n, 3)
    P[1, :, 3] = (0.3 if trained else -1.3) + (1.3 if trained else 0.8) * _randn(g, n)
    if trained:  # the short axis along the normal
        P[1, :, 2] -= 1.0
        P[2, :, 0], P[2, :, 1], P[2, :, 2] = 1.0 + nrm[:, 2], -nrm[:, 1], nrm[:, 0]
    else:
        P[2, :, 0] = 1.0
    P[2] += 0.1 * _randn(g, n, 4)
    nc = 3 * (deg + 1) ** 2
    P[3, :, :3] = (col - 0.5) / Y00
    if deg > 0:
        P[3, :, 3] = 0.04 * _randn(g, n)
        for q in range(4, P.shape[0]):
            w = min(4, nc - 4 * (q - 3))
            P[q, :, :w] = 0.04 * _randn(g, n, w)
    return P


def _cams(w, h, seed, views):
    all_ = synth.orbital_cameras(64, 1.5, center=(0.5, 0.5, 0.5), width=w, height=h)
    return all_.subset([(11 * int(seed) + 7 + 23 * j) % 64 for j in range(views)])


def _look(pts, col, cams, w, h, seed):
    """Ground truth [V, 3, h, w] and mask [V, h, w] of every view: the nearest point per cell on a grid coarse
    enough to leave few holes, white elsewhere."""
    n, V = pts.shape[0], len(cams)
    s = 1
    while n * s * s < 0.8 * w * h and s < 16:
        s *= 2
    gw, gh = (w + s - 1) // s, (h + s - 1) // s
    gt = torch.empty((V, 3, h, w), device=DEV)
    mask = torch.empty((V, h, w), dtype=torch.uint8, device=DEV)
    for v in range(V):
        M = torch.tensor(cams.viewmat[v], device=DEV)
        c = pts @ M[:, :3].T + M[:, 3]
        px = ((c[:, 0] / c[:, 2] * float(cams.fx[v]) + float(cams.cx[v])) / s).round().long()
        py = ((c[:, 1] / c[:, 2] * float(cams.fy[v]) + float(cams.cy[v])) / s).round().long()
        ok = (c[:, 2] > 0.2) & (px >= 0) & (px < gw) & (py >= 0) & (py < gh)
        key = (c[:, 2].contiguous().view(torch.int32).long() << 32) | torch.arange(n, device=DEV)
        cell = torch.full((gw * gh,), 1 << 62, dtype=torch.int64, device=DEV)
        cell.scatter_reduce_(0, (py * gw + px)[ok], key[ok], "amin")
        hit = cell < (1 << 62)
        img = torch.ones((gw * gh, 3), device=DEV)
        img[hit] = col[cell[hit] & 0xFFFFFFFF]
        up = lambda t: t.reshape(gh, gw, -1).repeat_interleave(s, 0).repeat_interleave(s, 1)[:h, :w]  # noqa: E731
        gt[v] = up(img).permute(2, 0, 1)
        mask[v] = up(hit.to(torch.uint8))[..., 0]
    return gt, mask


def _moments(P, seed, std):
    """Adam state T0 steps into a run: gradients of about `std` so far."""
    g = _gen(seed, 3)
    m, v = torch.empty_like(P), torch.empty_like(P)
    for k in range(P.shape[0]):
        m[k] = 0.3 * std * _randn(g, *P.shape[1:])
        v[k] = (std * (0.5 + _rand(g, *P.shape[1:]))) ** 2
    return {"m": m, "v": v, "step": torch.full((1,), T0, dtype=torch.int32, device=DEV)}


def _small(case, seed):
    """The small scenes: random Gaussians (autograd) or a unit sphere's points (views)."""
    g, n, deg = _gen(seed, 4), case["n"], case["deg"]
    P = torch.zeros((_planes(deg), n, 4), device=DEV)
    nc = 3 * (deg + 1) ** 2
    if case["kind"] == "autograd":
        P[0, :, :3] = 2 * _rand(g, n, 3) - 1
        P[1, :, :3] = -3.5 + 1.5 * _rand(g, n, 3)
        P[1, :, 3] = -2 + 5 * _rand(g, n)
        P[2] = _randn(g, n, 4)
    else:
        d = _randn(g, n, 3)
        P[0, :, :3] = d / d.norm(dim=1, keepdim=True)
        P[1, :, :3] = math.log(math.sqrt(4 * math.pi / n) * 0.73) + 0.1 * _randn(g, n, 3)
        P[1, :, 3] = -2 + _randn(g, n)
        P[2, :, 0] = 1.0
    flat = 0.2 * _randn(g, n, 4 * (P.shape[0] - 3))
    flat[:, nc:] = 0
    flat[:, :3] = 2 * _rand(g, n, 3) - 1
    P[3:] = flat.reshape(n, -1, 4).permute(1, 0, 2)
    views = case.get("views", 1)
    cams = synth.orbital_cameras(max(views, 8), 3.0, width=case["w"], height=case["h"])
    cams = cams.subset([(int(seed) + j) % len(cams) for j in range(views)])
    shape = (views, 3, case["h"], case["w"])
    return dict(P=P, cams=cams, gt=0.1 + 0.8 * _rand(g, *shape), dimg=_randn(g, *shape) / shape[2] / shape[3],
                mask=(_rand(g, views, case["h"], case["w"]) < 0.7).to(torch.uint8))


def _scene(case, seed, age, views):
    pts, nrm, col, sp = _surface(case["n"], case["modes"], seed)
    cams = _cams(case["w"], case["h"], seed, views)
    gt, mask = _look(pts, col, cams, case["w"], case["h"], seed) if age == "mid" else (None, None)
    return dict(P=_splats(pts, nrm, col, sp, case["deg"], seed, age), cams=cams, gt=gt, mask=mask)


def _grad_std(case):
    return 0.5 / (case["w"] * case["h"])


def _parts(case, seed):
    """The surface cut into x-slabs with 5% ghost layers: planes of all partitions one after another, their
    offsets and each partition's own ground truth and masks."""
    k, V = case["parts"], 3
    # strips of each slab: its left and right ghost layers' sources and the rest, with the same counts for every seed
    density = np.asarray(SLABS[:k] if case["kind"] == "batched" else [1.0] * k)
    share = np.outer(density / density.sum(), [0.05, 0.9, 0.05]).reshape(-1)
    share[0], share[-1] = share[0] + share[1], share[-1] + share[-2]  # the outer slabs have one ghost layer each
    share[1], share[-2] = 0.0, 0.0
    counts = np.floor(share * case["n"]).astype(np.int64)
    counts[np.argmax(counts)] += case["n"] - counts.sum()
    edges = np.linspace(0.0, 1.0, k + 1)
    cuts = (edges[:-1, None] + np.array([0.0, 0.05, 0.95]) / k).reshape(-1)
    cuts[1], cuts[-1] = cuts[2], cuts[-2] if k > 1 else cuts[-1]
    cuts = np.append(cuts, 1.0)
    pts, nrm, col, sp, strip = _surface(case["n"], case["modes"], seed, (cuts, counts))
    off, rows = [0], []
    for p in range(k):
        mine = (strip >= 3 * p - (1 if p else 0)) & (strip < 3 * p + 3 + (1 if p < k - 1 else 0))
        rows.append(torch.nonzero(mine).squeeze(1))
        off.append(off[-1] + rows[-1].numel())
    cams = _cams(case["w"], case["h"], seed, V)
    gt = mask = None
    if case["kind"] == "batched":
        both = [_look(pts[r], col[r], cams, case["w"], case["h"], seed) for r in rows]
        gt, mask = torch.stack([b[0] for b in both]), torch.stack([b[1] for b in both])
        del both
    order = torch.cat(rows)
    del rows
    pts, nrm, col = pts[order], nrm[order], col[order]
    del order
    P = _splats(pts, nrm, col, sp, case["deg"], seed, "mid" if case["kind"] == "batched" else "trained")
    boxes = np.zeros((k, 6), np.float32)
    boxes[:, 0], boxes[:, 3] = edges[:-1], edges[1:]
    boxes[0, 0], boxes[-1, 3] = -1e30, 1e30
    boxes[:, 1:3], boxes[:, 4:] = -1e30, 1e30
    return dict(P=P, off=np.asarray(off, np.int64), cams=cams, gt=gt, mask=mask, boxes=boxes)


def _weights(seed):
    """Network weights as a fit leaves them: He-initialised layers, a small output layer around the plain form."""
    w = ginit.init_weights(int(seed) % 1000, DEV)
    g = _gen(seed, 5)
    w[7168 + 64 + 4096 + 64:7168 + 64 + 4096 + 64 + 512] = 0.05 * _randn(g, 512)
    return w


def _targets(n, seed):
    g = _gen(seed, 6)
    t = 0.3 * _randn(g, n, 8)
    t[:, 3] += 1.0
    t[:, 7] -= 1.0
    return t


def _images(case, seed):
    """A rendered image near its ground truth (smooth fields and noise) and a mask of one large blob per unit."""
    g, U, w, h = _gen(seed, 7), case["units"], case["w"], case["h"]
    up = lambda c, a, b: torch.nn.functional.interpolate(_rand(g, U, c, a, b), (h, w), mode="bilinear")  # noqa: E731
    gt = (0.8 * up(3, 24, 24) + 0.2 * _rand(g, U, 3, h, w)).clamp(0, 1)
    img = gt + 0.1 * (up(3, 40, 40) - 0.5) + 0.02 * _randn(g, U, 3, h, w)
    yy, xx = torch.meshgrid(torch.linspace(-1, 1, h, device=DEV), torch.linspace(-1, 1, w, device=DEV), indexing="ij")
    m = (xx * xx + yy * yy)[None] < 0.55 + 0.4 * up(1, 9, 9)[:, 0]
    return img.contiguous(), gt.contiguous(), m.to(torch.uint8)


# ---------------------------------------------------------------- the calls
def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind, t=0)
    if kind == "autograd":
        s = _small(case, seed)
        st.update(P=s["P"].requires_grad_(True), cams=pack_cameras(s["cams"], DEV), dimg=s["dimg"],
                  frame=Frame(case["n"], Units.single(case["n"]), case["w"], case["h"], case["deg"], DEV))
        st["frame"].fit_capacity(s["P"].detach(), st["cams"])
    elif kind == "views":
        s = _small(case, seed)
        fr = Frame(case["n"], Units.single(case["n"], case["views"]), case["w"], case["h"], case["deg"], DEV)
        st.update(P=s["P"], cams=pack_cameras(s["cams"], DEV), gt=s["gt"], mask=s["mask"], frame=fr,
                  opt=Adam(s["P"], case["deg"], lr_steps=LR_STEPS))
        st["opt"].load_state_dict(_moments(s["P"], seed, _grad_std(case)))
        fr.fit_capacity(s["P"], st["cams"])
    elif kind in ("train", "train_next"):
        s = _scene(case, seed, "mid", 3)
        cams = pack_cameras(s["cams"], DEV)
        tr = PlainTrainer(s["P"], case["deg"], cams, s["gt"], s["mask"], range(3), lr_steps=LR_STEPS, lam=LAM, bg=BG)
        tr.opt.load_state_dict(_moments(s["P"], seed, _grad_std(case)))
        tr.opt.sparse = case.get("sparse", False)
        st.update(tr=tr)
        if kind == "train_next":
            tr.frame.preprocess(tr.params, tr.cam(0))
    elif kind == "grads":
        s = _scene(case, seed, "mid", 1)
        fr = Frame(case["n"], Units.single(case["n"]), case["w"], case["h"], case["deg"], DEV, deterministic=True)
        st.update(P=s["P"], cams=pack_cameras(s["cams"], DEV), gt=s["gt"], mask=s["mask"], frame=fr)
        fr.fit_capacity(s["P"], st["cams"])
    elif kind == "render":
        s = _scene(case, seed, "trained", 1)
        fr = Frame(case["n"], Units.single(case["n"]), case["w"], case["h"], case["deg"], DEV, with_backward=False,
                   with_loss=False, max_instances=3 * case["n"])
        fr.walk_whole_lists = case["whole"]
        st.update(P=s["P"], cams=pack_cameras(s["cams"], DEV), frame=fr)
        fr.fit_capacity(s["P"], st["cams"])
    elif kind == "merge":
        s = _parts(case, seed)
        n = int(s["off"][-1])
        closed = np.full(case["parts"], 0b110, np.int32)
        closed[-1] |= 1
        own = Owned(s["off"], s["boxes"], closed)
        fr = Frame(n, Units.single(n), case["w"], case["h"], case["deg"], DEV, with_backward=False, with_loss=False,
                   max_instances=2 * n)
        fr.walk_whole_lists = True  # the mode bench.py picks for this render
        cams = pack_cameras(s["cams"].subset([0]), DEV)
        fr.fit_capacity(s["P"], cams, own)
        st.update(P=s["P"], cams=cams, frame=fr, own=own)
    elif kind == "batched":
        s = _parts(case, seed)
        tr = BatchedTrainer(s["P"], case["deg"], s["off"], pack_cameras(s["cams"], DEV), s["gt"], s["mask"], range(3),
                            case["vps"], lr_steps=LR_STEPS, lam=LAM, bg=BG)
        tr.opt.load_state_dict(_moments(s["P"], seed, _grad_std(case)))
        tr.t = T0
        st.update(tr=tr)
    elif kind in ("init", "fit"):
        pts, nrm, _, sp = _surface(case["n"], case["modes"], seed)
        st.update(pts=pts, nrm=nrm, w=_weights(seed))
        if kind == "init":
            st["P"] = torch.zeros((_planes(3), case["n"], 4), device=DEV)
        else:
            st["idx"], st["dist"] = ginit.knn(pts, 16)
            st["target"] = _targets(case["n"], seed)
            st["fit"] = ginit.MLPTrainer(st["w"])
            mo = _moments(st["w"].reshape(1, -1, 4), seed, 0.02)
            st["fit"].m.copy_(mo["m"].reshape(-1))
            st["fit"].v.copy_(mo["v"].reshape(-1))
            st["fit"].step_dev.fill_(T0)
    else:
        img, gt, mask = _images(case, seed)
        fr = Frame(1, Units.single(1, case["units"]), case["w"], case["h"], 0, DEV)
        fr.img.copy_(img)
        st.update(frame=fr, gt=gt, mask=mask)
    return st


def run(st):
    kind = st["kind"]
    if kind == "autograd":
        st["P"].grad = None
        img = rasterize(st["P"], st["frame"], st["cams"], BG)
        img.backward(st["dimg"])
        return dict(img=img.detach(), grad=st["P"].grad)
    if kind == "views":
        fr = st["frame"]
        img = fr.forward(st["P"], st["cams"], BG)
        loss = fr.loss(st["gt"], st["mask"], LAM)
        grads = fr.backward(st["P"], st["cams"], BG)
        st["opt"].step(grads)
        return dict(img=img, loss=loss, grads=grads, P=st["P"], m=st["opt"].m, v=st["opt"].v)
    if kind == "train":
        tr = st["tr"]
        tr.step(st["t"] % 3)
        st["t"] += 1
        return _trained(tr)
    if kind == "train_next":
        tr, v = st["tr"], st["t"] % 3
        fr = tr.frame
        fr.sort()
        fr.render(BG)
        fr.loss(tr.gt[v:v + 1], tr.mask[v:v + 1], LAM)
        fr.blend_backward(BG)
        tr.opt.fused_step(fr, tr.cam(v), next_cams_dev=tr.cam((v + 1) % 3))
        st["t"] += 1
        return _trained(tr)
    if kind == "grads":
        fr = st["frame"]
        img = fr.forward(st["P"], st["cams"], BG)
        loss = fr.loss(st["gt"], st["mask"], LAM)
        return dict(img=img, loss=loss, grads=fr.backward(st["P"], st["cams"], BG))
    if kind == "render":
        fr = st["frame"]
        return dict(img=fr.forward(st["P"], st["cams"], BG), final_T=fr.final_T)
    if kind == "merge":
        fr = st["frame"]
        return dict(img=fr.merge_render(st["P"], st["cams"], BG, st["own"]), final_T=fr.final_T)
    if kind == "batched":
        st["tr"].step()
        return _trained(st["tr"])
    if kind == "init":
        idx, dist = ginit.knn(st["pts"], 16)
        ginit.init_gaussians(st["P"], st["pts"], st["nrm"], st["w"], idx, dist)
        return dict(idx=idx, dist=dist, P=st["P"])
    if kind == "fit":
        f = st["fit"]
        loss = f.step(st["pts"], st["nrm"], st["idx"], st["dist"], st["target"])
        return dict(loss=loss, grad=f.grad, w=f.w, m=f.m, v=f.v)
    fr = st["frame"]
    return dict(loss=fr.loss(st["gt"], st["mask"], LAM), dimg=fr.dimg)


def _trained(tr):
    fr = tr.frame
    return dict(img=fr.img, final_T=fr.final_T, loss=fr.loss_val, P=tr.params, m=tr.opt.m, v=tr.opt.v)


def work(case):
    """Bytes: inputs once, outputs once.  Flops: the per-Gaussian projection (about 600 forward, 1,500 backward), the
    separable SSIM windows (about 700 per pixel and channel) or the network (2 x 11.8k per point and pass); the
    blend's work depends on the data and is left out."""
    kind = case["kind"]
    if kind in ("init", "fit"):
        n = case["n"]
        if kind == "init":
            return {"bytes": n * (12 + 12 + 16 * 8 + 3 * 16), "flops": n * 2 * 11_776.0}
        return {"bytes": n * (24 + 16 * 8 + 32), "flops": 3 * n * 2 * 11_776.0}
    pix = case["w"] * case["h"]
    if kind == "loss":
        return {"bytes": case["units"] * pix * (12 + 12 + 1 + 12), "flops": case["units"] * pix * 3 * 700.0}
    n, par = case["n"], 16 * _planes(case["deg"])
    if kind == "merge":
        n = int(n * (1 + 0.1 * (case["parts"] - 1) / case["parts"]))
    units = case.get("views", 1) * case.get("vps", 1)
    img = units * pix * 16 * (case["parts"] if kind == "batched" else 1)
    fwd = {"bytes": n * par + img, "flops": 600.0 * n * units}
    if kind in ("render", "merge"):
        return fwd
    if kind in ("autograd", "grads"):
        return {"bytes": fwd["bytes"] + img + n * par, "flops": fwd["flops"] + 1500.0 * n * units}
    if kind == "batched":
        n = int(n * (1 + 0.1 * (case["parts"] - 1) / case["parts"]))
    return {"bytes": 6 * n * par + 2 * img, "flops": 2100.0 * n * units}


# ---------------------------------------------------------------- 64 bits
def _sh_basis(d, deg):
    x, y, z = d.unbind(1)
    c1 = math.sqrt(3 / (4 * math.pi))
    Y = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    if deg >= 1:
        Y += [-c1 * y, c1 * z, -c1 * x]
    if deg >= 2:
        a, b, c = 0.5 * math.sqrt(15 / math.pi), 0.25 * math.sqrt(5 / math.pi), 0.25 * math.sqrt(15 / math.pi)
        Y += [a * x * y, -a * y * z, b * (2 * z * z - x * x - y * y), -a * x * z, c * (x * x - y * y)]
    if deg >= 3:
        a, b, c = 0.25 * math.sqrt(35 / (2 * math.pi)), 0.5 * math.sqrt(105 / math.pi), 0.25 * math.sqrt(21 / (2 * math.pi))
        d_, e = 0.25 * math.sqrt(7 / math.pi), 0.25 * math.sqrt(105 / math.pi)
        xx, yy, zz = x * x, y * y, z * z
        Y += [-a * y * (3 * xx - yy), b * x * y * z, -c * y * (4 * zz - xx - yy), d_ * z * (2 * zz - 3 * xx - 3 * yy),
              -c * x * (4 * zz - xx - yy), e * z * (xx - yy), -a * x * (xx - 3 * yy)]
    return torch.stack(Y, 1)


def _project(P, cams, v, deg):
    """Records [n, 9] = (u, v, A, B, C, opacity, r, g, b), the depth and the 3-sigma radius (0: culled) of double
    planes P [planes, n, 4]."""
    f = lambda a: torch.tensor(np.asarray(a, np.float64), device=DEV)  # noqa: E731
    M = f(cams.viewmat[v])
    fx, fy, cx, cy = (float(getattr(cams, k)[v]) for k in ("fx", "fy", "cx", "cy"))
    mean, ls, lo, q = P[0, :, :3], P[1, :, :3], P[1, :, 3], P[2]
    t = mean @ M[:, :3].T + M[:, 3]
    z = t[:, 2]
    q = q / q.norm(dim=1, keepdim=True)
    w, x, y, k = q.unbind(1)
    R = torch.stack([1 - 2 * (y * y + k * k), 2 * (x * y - w * k), 2 * (x * k + w * y),
                     2 * (x * y + w * k), 1 - 2 * (x * x + k * k), 2 * (y * k - w * x),
                     2 * (x * k - w * y), 2 * (y * k + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)
    S = R * torch.exp(ls)[:, None, :]
    lx, ly = 1.3 * float(cams.tan_fovx[v]), 1.3 * float(cams.tan_fovy[v])
    xz, yz = (t[:, 0] / z).clamp(-lx, lx), (t[:, 1] / z).clamp(-ly, ly)
    T0r = (fx / z)[:, None] * M[0, :3] - (fx * xz / z)[:, None] * M[2, :3]
    T1r = (fy / z)[:, None] * M[1, :3] - (fy * yz / z)[:, None] * M[2, :3]
    a0, a1 = (T0r[:, None, :] @ S)[:, 0], (T1r[:, None, :] @ S)[:, 0]
    a, b, c = (a0 * a0).sum(1) + 0.3, (a0 * a1).sum(1), (a1 * a1).sum(1) + 0.3
    det = a * c - b * b
    mid = 0.5 * (a + c)
    with torch.no_grad():
        rad = torch.ceil(3 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp_min(0.1))))
        rad = torch.where((z > cams.znear) & (det > 0), rad, torch.zeros_like(rad)).long()
    d = mean - f(cams.campos[v])
    Y = _sh_basis(d / d.norm(dim=1, keepdim=True), deg)
    sh = P[3:].permute(1, 0, 2).reshape(P.shape[1], -1)[:, :3 * (deg + 1) ** 2].reshape(-1, (deg + 1) ** 2, 3)
    rgb = ((Y[:, :, None] * sh).sum(1) + 0.5).clamp_min(0)
    u = torch.stack([fx * t[:, 0] / z + cx, fy * t[:, 1] / z + cy, c / det, -b / det, a / det, torch.sigmoid(lo)], 1)
    return torch.cat([u, rgb], 1), z, rad


def _lists(rec, z, rad, w, h):
    """Instances in (tile, float32 depth, index) order: record of each, first position and length per tile."""
    tx, ty = (w + 15) // 16, (h + 15) // 16
    fu, fv = torch.floor(rec[:, 0]).long(), torch.floor(rec[:, 1]).long()
    box = lambda f, r, m: torch.div(f + r, 16, rounding_mode="floor").clamp(0, m)  # noqa: E731
    x0, x1, y0, y1 = box(fu, -rad, tx), box(fu, rad + 15, tx), box(fv, -rad, ty), box(fv, rad + 15, ty)
    nt = torch.where(rad > 0, (x1 - x0) * (y1 - y0), torch.zeros_like(rad))
    o = torch.argsort(z.float(), stable=True)
    nt_o = nt[o]
    who = torch.repeat_interleave(o, nt_o)
    k = torch.arange(who.numel(), device=DEV) - torch.repeat_interleave(torch.cumsum(nt_o, 0) - nt_o, nt_o)
    wd = (x1 - x0)[who]
    tile = (y0[who] + torch.div(k, wd, rounding_mode="floor")) * tx + x0[who] + k % wd
    del k, wd
    o = torch.argsort(tile.to(torch.int32), stable=True)
    length = torch.bincount(tile, minlength=tx * ty)
    return who[o], torch.cumsum(length, 0) - length, length


def _blend(rec, lists, w, h, dimg=None, budget=40_000_000):
    """Image [3, h, w] and final transmittance [h, w]; with dimg, the gradient of rec instead."""
    who, first, length = lists
    tx = (w + 15) // 16
    th = (h + 15) // 16
    px, py = torch.arange(256, device=DEV) % 16, torch.arange(256, device=DEV) // 16
    leaf = rec.detach().requires_grad_(dimg is not None)
    img = torch.empty((th * 16, tx * 16, 4), dtype=torch.float64, device=DEV)
    img[..., :3], img[..., 3] = torch.tensor(BG, dtype=torch.float64, device=DEV), 1.0
    img = img.reshape(th, 16, tx, 16, 4).permute(0, 2, 1, 3, 4).reshape(th * tx, 256, 4).contiguous()
    if dimg is not None:
        d = torch.zeros((3, th * 16, tx * 16), dtype=torch.float64, device=DEV)
        d[:, :h, :w] = dimg
        d = d.reshape(3, th, 16, tx, 16).permute(1, 3, 2, 4, 0).reshape(th * tx, 256, 3)
    order = torch.argsort(length, descending=True)
    lens = length[order].tolist()
    a = 0
    while a < len(lens) and lens[a] > 0:
        b = a + max(1, budget // (lens[a] * 256))
        tiles = order[a:b]
        tiles = tiles[length[tiles] > 0]
        L = lens[a]
        pos = torch.arange(L, device=DEV)[None]
        there = pos < length[tiles][:, None]
        idx = who[(first[tiles][:, None] + pos).clamp_max(who.numel() - 1)]
        with torch.set_grad_enabled(dimg is not None):
            r = leaf[idx]
            dx = r[..., 0:1] - ((tiles % tx) * 16)[:, None, None] - px
            dy = r[..., 1:2] - (torch.div(tiles, tx, rounding_mode="floor") * 16)[:, None, None] - py
            power = -0.5 * (r[..., 2:3] * dx * dx + r[..., 4:5] * dy * dy) - r[..., 3:4] * dx * dy
            al = (r[..., 5:6] * torch.exp(power)).clamp_max(0.99)
            al = torch.where((power <= 0) & (al >= 1.0 / 255.0) & there[..., None], al, torch.zeros_like(al))
            lt = torch.cumsum(torch.log1p(-al), 1)
            kept = torch.exp(lt.detach()) >= 1e-4
            wgt = torch.where(kept, al * torch.exp(lt - torch.log1p(-al)), torch.zeros_like(al))
            rgb = torch.einsum("tlp,tlc->tpc", wgt, r[..., 6:9])
            T = 1.0 - wgt.sum(1)
            out = rgb + T[..., None] * torch.tensor(BG, dtype=torch.float64, device=DEV)
            if dimg is not None:
                out.backward(d[tiles])
        if dimg is None:
            img[tiles, :, :3], img[tiles, :, 3] = out, T
        a += tiles.numel()
    if dimg is not None:
        return leaf.grad
    img = img.reshape(th, tx, 16, 16, 4).permute(0, 2, 1, 3, 4).reshape(th * 16, tx * 16, 4)[:h, :w]
    return img[..., :3].permute(2, 0, 1).contiguous(), img[..., 3].contiguous()


STEP = 1 << 20  # Gaussians projected at a time


def _records(P, cams, v, deg, keep=None):
    got = [_project(P[:, a:a + STEP].double(), cams, v, deg) for a in range(0, P.shape[1], STEP)]
    rec, z, rad = (torch.cat([g[k] for g in got]) for k in range(3))
    return rec, z, rad if keep is None else torch.where(keep, rad, torch.zeros_like(rad))


def _record_grads(P, cams, v, deg, g, G):
    for a in range(0, P.shape[1], STEP):
        p = P[:, a:a + STEP].double().requires_grad_(True)
        _project(p, cams, v, deg)[0].backward(g[a:a + STEP])
        G[:, a:a + STEP] += p.grad


def _loss64(img, gt, mask):
    """The masked L1 + SSIM loss of one unit and dloss/dimg."""
    img = img.detach().double().requires_grad_(True)
    gt, m = gt.double(), mask != 0
    w = torch.exp(-torch.arange(-5, 6, dtype=torch.float64, device=DEV) ** 2 / 4.5)
    w = w / w.sum()

    def conv(x):
        x = torch.nn.functional.pad(x, (0, 0, 5, 5))
        x = sum(w[k] * x[:, k:k + img.shape[1]] for k in range(11))
        x = torch.nn.functional.pad(x, (5, 5, 0, 0))
        return sum(w[k] * x[:, :, k:k + img.shape[2]] for k in range(11))

    ux, uy = conv(img), conv(gt)
    vx, vy, c = conv(img * img) - ux * ux, conv(gt * gt) - uy * uy, conv(img * gt) - ux * uy
    s = (2 * ux * uy + 1e-4) * (2 * c + 9e-4) / ((ux * ux + uy * uy + 1e-4) * (vx + vy + 9e-4))
    n = int(m.sum())
    if n == 0:
        return img.new_zeros(()), torch.zeros_like(img)
    loss = (1 - LAM) * (img - gt).abs()[:, m].sum() / (3 * n) + LAM * (1 - s[:, m].mean())
    loss.backward()
    return loss.detach(), img.grad


def _adam64(P, G, mo, lr0, lr1, steps, eps, b=(0.9, 0.999)):
    t = T0 + 1
    m = b[0] * mo["m"].double() + (1 - b[0]) * G
    v = b[1] * mo["v"].double() + (1 - b[1]) * G * G
    lr = lr0 if steps <= 0 else torch.where((lr0 == lr1) | (lr0 <= 0), lr0,
                                            lr0 * (lr1 / lr0.clamp_min(1e-300)) ** (min(t, steps) / steps))
    return P.double() - lr * (m / (1 - b[0] ** t)) / (torch.sqrt(v / (1 - b[1] ** t)) + eps), m, v


def _rates(deg):
    """Learning rates at the start and at the end of the schedule, [planes, 1, 4] (the 3D-GS defaults)."""
    a = torch.zeros((_planes(deg), 1, 4), dtype=torch.float64, device=DEV)
    a[0, 0, :3], a[1, 0, :3], a[1, 0, 3], a[2] = 1.6e-4, 5e-3, 5e-2, 1e-3
    a[3:] = 2.5e-3 / 20
    a[3, 0, :3] = 2.5e-3
    b = a.clone()
    b[0, 0, :3] = 1.6e-6
    return a, b


def _knn64(p, k):
    """Exact k nearest neighbours of points on a height field: candidates of 3x3 cells in (x, y), brute force where
    the k-th distance reaches past them."""
    n = p.shape[0]
    p = p.double()
    dim = max(1, int(math.sqrt(n) / 8))
    cx, cy = ((p[:, c] * dim).long().clamp(0, dim - 1) for c in (0, 1))
    cell = cy * dim + cx
    o = torch.argsort(cell, stable=True)
    cnt = torch.bincount(cell, minlength=dim * dim)
    start = torch.cumsum(cnt, 0) - cnt
    idx = torch.empty((n, k), dtype=torch.int64, device=DEV)
    dist = torch.empty((n, k), dtype=torch.float64, device=DEV)
    most = int(cnt.max())

    def best(rows, cand, ok):
        d = (p[cand] - p[rows][:, None]).square().sum(2)
        d = torch.where(ok & (cand != rows[:, None]), d, torch.full_like(d, math.inf))
        d, j = torch.topk(d, k, dim=1, largest=False, sorted=True)
        return d.sqrt(), cand.gather(1, j)

    q = torch.arange(most, device=DEV)
    for a in range(0, n, 1 << 16):
        rows = o[a:a + (1 << 16)]
        cand, ok = [], []
        for ex in (-1, 0, 1):
            for ey in (-1, 0, 1):
                nx, ny = cx[rows] + ex, cy[rows] + ey
                inside = (nx >= 0) & (nx < dim) & (ny >= 0) & (ny < dim)
                c = torch.where(inside, ny * dim + nx, torch.zeros_like(nx))
                cand.append(o[(start[c][:, None] + q).clamp_max(n - 1)])
                ok.append(inside[:, None] & (q < cnt[c][:, None]))
        dist[rows], idx[rows] = best(rows, torch.cat(cand, 1), torch.cat(ok, 1))
    far = torch.nonzero(~(dist[:, -1] < 1.0 / dim)).squeeze(1)
    for a in range(0, far.numel(), 64):
        rows = far[a:a + 64]
        dist[rows], idx[rows] = best(rows, torch.arange(n, device=DEV)[None].expand(rows.numel(), n),
                                     torch.ones((1, 1), dtype=torch.bool, device=DEV))
    return idx, dist


def _net64(w, pts, nrm, idx, dist):
    n = idx.shape[0]
    W1, b1, W2, b2, W3, b3 = (x.reshape(s) for x, s in zip(torch.split(w, [7168, 64, 4096, 64, 512, 8]),
                                                          [(112, 64), (64,), (64, 64), (64,), (64, 8), (8,)]))
    off = (pts[idx] - pts[:n, None]) / dist.mean(1)[:, None, None].clamp_min(1e-12)
    X = torch.cat([off.reshape(n, 48), nrm[idx].reshape(n, 48), nrm[:n]], 1)
    return torch.relu(torch.relu(X @ W1[:99] + b1) @ W2 + b2) @ W3 + b3


def exact(case, seed):
    kind, deg = case["kind"], case.get("deg", 0)
    n_all = case.get("n", 0)
    if n_all > 12_000_000:
        return None  # 172M instances at 100M splats: 80 s
    grads = n_all <= 4_000_000  # billions of (pixel, splat) gradients in 64 bits: 40 s at 10M, 6 s for the image alone
    if kind == "loss":
        img, gt, mask = _images(case, seed)
        got = [_loss64(img[u], gt[u], mask[u]) for u in range(case["units"])]
        return dict(loss=torch.stack([g[0] for g in got]).mean().reshape(1),
                    dimg=torch.stack([g[1] for g in got]) / case["units"])
    if kind in ("init", "fit"):
        pts, nrm, _, _ = _surface(case["n"], case["modes"], seed)
        w = _weights(seed).double()
        idx, dist = _knn64(pts, 16)
        pts, nrm, n = pts.double(), nrm.double(), case["n"]
        if kind == "init":
            y = torch.cat([_net64(w, pts, nrm, idx[a:a + STEP], dist[a:a + STEP]) if a == 0 else
                           _net64(w, torch.cat([pts[a:a + STEP], pts]), torch.cat([nrm[a:a + STEP], nrm]),
                                  idx[a:a + STEP] + min(STEP, n - a), dist[a:a + STEP]) for a in range(0, n, STEP)])
            P = torch.zeros((_planes(3), n, 4), dtype=torch.float64, device=DEV)
            P[0, :, :3] = pts
            P[1, :, :3] = torch.log(dist[:, :3].mean(1)).clamp_min(math.log(1e-7))[:, None] + y[:, :3]
            P[1, :, 3], P[2] = y[:, 7], y[:, 3:7]
            return dict(idx=None, dist=dist, P=P)
        t = _targets(n, seed).double()
        w.requires_grad_(True)
        loss = 0.0
        for a in range(0, n, STEP):
            m = min(STEP, n - a)
            y = _net64(w, torch.cat([pts[a:a + m], pts]), torch.cat([nrm[a:a + m], nrm]), idx[a:a + m] + m, dist[a:a + m])
            part = (y - t[a:a + m]).square().sum() / (8 * n)
            part.backward()
            loss = loss + part.detach()
        mo = _moments(w.detach().float().reshape(1, -1, 4), seed, 0.02)
        mo = {k: v.reshape(-1) for k, v in mo.items()}
        lr = torch.full_like(mo["m"], 1e-3, dtype=torch.float64)
        w1, m1, v1 = _adam64(w.detach(), w.grad, mo, lr, lr, 0, 1e-8)
        return dict(loss=loss.reshape(1), grad=w.grad, w=w1, m=m1, v=v1)
    W, H = case["w"], case["h"]
    if kind in ("autograd", "views"):
        s = _small(case, seed)
    elif kind in ("batched", "merge"):
        s = _parts(case, seed)
    else:
        s = _scene(case, seed, "trained" if kind == "render" else "mid", 1 if kind in ("grads", "render") else 3)
    P, cams = s["P"], s["cams"]
    n = P.shape[1]
    # (Gaussians, view, ground truth, mask) of every unit of the pass
    if kind == "batched":
        k, vps = case["parts"], case["vps"]
        of = lambda p, j: (T0 * vps + j + p) % 3  # noqa: E731
        units = [(slice(int(s["off"][p]), int(s["off"][p + 1])), of(p, j), s["gt"][p, of(p, j)], s["mask"][p, of(p, j)])
                 for p in range(k) for j in range(vps)]
    else:
        views = case.get("views", 1)
        units = [(slice(0, n), v, None if s["gt"] is None else s["gt"][v], None if s["gt"] is None else s["mask"][v])
                 for v in range(views)]
    keep = None
    if kind == "merge":
        x, lo, hi = P[0, :, 0], s["boxes"][:, 0], s["boxes"][:, 3]
        part = torch.bucketize(torch.arange(n, device=DEV), torch.tensor(s["off"][1:-1], device=DEV), right=True)
        lo, hi = torch.tensor(lo, device=DEV)[part], torch.tensor(hi, device=DEV)[part]
        keep = (x >= lo) & (x < hi)
    G = torch.zeros_like(P, dtype=torch.float64 if grads else None) if kind not in ("render", "merge") else None
    imgs, Ts, losses = [], [], []
    for sl, v, gt, mask in units:
        rec, z, rad = _records(P[:, sl], cams, v, deg, keep)
        ls = _lists(rec, z, rad, W, H)
        img, T = _blend(rec, ls, W, H)
        imgs.append(img)
        Ts.append(T)
        if G is None:
            continue
        if not grads:
            losses.append(_loss64(img, gt, mask)[0])
            continue
        if kind == "autograd":
            d = s["dimg"][0].double()
        else:
            loss, d = _loss64(img, gt, mask)
            losses.append(loss)
            d = d / len(units)
        _record_grads(P[:, sl], cams, v, deg, _blend(rec, ls, W, H, d, 12_000_000), G[:, sl])
    img, T = torch.stack(imgs), torch.stack(Ts)
    if kind == "autograd":
        return dict(img=img, grad=G)
    if kind in ("render", "merge"):
        return dict(img=img, final_T=T)
    loss = torch.stack(losses).mean().reshape(1)
    if kind == "grads":
        return dict(img=img, loss=loss, grads=G)
    if not grads:
        return dict(img=img, final_T=T, loss=loss, P=None, m=None, v=None)
    a, b = _rates(deg)
    P1, m, v = _adam64(P, G, _moments(P, seed, _grad_std(case)), a, b, LR_STEPS, 1e-15)
    if kind == "views":
        return dict(img=img, loss=loss, grads=G, P=P1, m=m, v=v)
    if case.get("sparse", False):  # whether a gradient is zero is the kernels' own rounding
        P1 = m = v = None
    return dict(img=img, final_T=T, loss=loss, P=P1, m=m, v=v)
