"""Performance cases: calls that a program using this library makes, over the sizes, precisions and forms it is used with.

listed() gives the named cases and draw() more of the same ranges; prepare() makes what a caller has in hand (images or
descriptors on the GPU, a context, a workspace, output buffers), run() makes one pass through the public entry points,
work() says what that pass cannot do without, and exact() gives its computed values in 64 bits (plain torch) where the
output is a number and not a decision: matches are the outcome of maxima over near-equal scores, so they have none.

Inputs are seeded and synthetic, of the kind the repository's tests and benchmark use: value noise and the same image
warped by a smooth displacement, with a gain and a little noise.
"""
import math
import weakref

import torch
import torch.nn.functional as F

from paper_1506_07656_gb300 import autograd, dm

PREC = {"fp32": dm.DM_FP32, "bf16": dm.DM_BF16, "fp8": dm.DM_FP8_E4M3}
DEV = "cuda"
MIXED = ((320, 240), (640, 480), (1024, 436), (1242, 375))


# --------------------------------------------------------------------------------------------------------------------
# The cases
# --------------------------------------------------------------------------------------------------------------------
def listed():
    def pair(kind, name, w, h, prec, **more):
        return dict(kind=kind, name=name, w1=w, h1=h, w2=w, h2=h, prec=prec, comp=True, **more)

    return [
        # one thumbnail pair at a time: the smallest call, bound by launches and latency
        pair("match", "match fp32 64x48", 64, 48, "fp32", disp=6.0),
        # the plain method where bit-exact FP32 results are wanted
        pair("match", "match fp32 512x224", 512, 224, "fp32", disp=40.0),
        # one video frame pair in the fast precision: the common single call
        pair("match", "match bf16 1024x436", 1024, 436, "bf16", disp=120.0),
        # one driving-scene pair (odd, wide, low) in the fastest precision
        pair("match", "match fp8 1242x375", 1242, 375, "fp8", disp=60.0),
        # a served queue of pairs of mixed sizes, resident on the device: two of each size in one call (the largest case)
        dict(kind="batch", name="batch bf16 mixed 8", n=8, shape=0, prec="bf16", comp=True, host=False, disp=60.0),
        # the same from page-locked host memory, images in and matches out inside the call
        dict(kind="batch", name="batch bf16 host 4x640x480", n=4, shape=2, prec="bf16", comp=True, host=True, disp=40.0),
        # descriptors and correlation pyramid alone, kept by a caller that reads the maps: ragged, unequal sizes
        dict(kind="pyramid", name="pyramid bf16 319x237/301x243", w1=319, h1=237, w2=301, h2=243, prec="bf16", comp=True,
             disp=10.0),
        # differentiable form: loss and both gradients of FP32 descriptor fields through autograd (forward + backward)
        pair("grad", "grad fp32 256x256", 256, 256, "fp32", disp=16.0),
        # approximate form: dictionary of patch prototypes, pyramid over the prototypes, backtracking
        pair("approx", "approx bf16 1024x436", 1024, 436, "bf16", disp=120.0, protos=1024, iters=10),
        # the earlier backtracking variant, entry points at every level
        pair("star", "star bf16 512x224", 512, 224, "bf16", disp=40.0),
        # scale and rotation invariant form: 72 warped pairs in one call
        pair("invariant", "invariant bf16 512x224", 512, 224, "bf16", disp=20.0),
        # variational flow refined from the matches of a frame pair
        pair("deepflow", "deepflow fp32 1024x436", 1024, 436, "fp32", disp=20.0),
    ]


def draw(rng):
    def size(lo, hi, most):
        """Sides spread over the logarithm of lo..hi, odd ones among them, at most `most` pixels."""
        w = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        h = int(round(min(w * rng.uniform(0.35, 1.1), most / w)))
        return w, max(h, 24)

    kind = rng.choice(("match", "match", "match", "batch", "pyramid", "grad", "approx", "star", "invariant", "deepflow"))
    prec = rng.choice(("fp32", "bf16", "bf16", "fp8"))
    comp = rng.random() < 0.8
    if kind == "batch":
        return dict(kind=kind, n=rng.randint(2, 6), shape=rng.randint(5, 60), prec=rng.choice(("bf16", "fp8")), comp=comp,
                    host=rng.random() < 0.5, disp=round(rng.uniform(4, 40), 1))
    if kind == "match":
        w1, h1 = size(48, 1242, 1024 * 436 if prec != "fp32" else 640 * 272)
    elif kind == "pyramid":
        w1, h1 = size(40, 320, 320 * 240)
    elif kind == "grad":
        w1, h1 = size(40, 256, 256 * 256)
        prec, comp = "fp32", True
    elif kind == "approx":
        w1, h1 = size(256, 1024, 1024 * 436)
        prec = rng.choice(("bf16", "fp8"))
    elif kind == "star":
        w1, h1 = size(64, 512, 512 * 224)
        prec = rng.choice(("fp32", "bf16"))
    elif kind == "invariant":
        w1, h1 = size(64, 448, 448 * 200)
        prec = rng.choice(("bf16", "fp8"))
    else:
        w1, h1 = size(48, 1024, 1024 * 436)
        prec, comp = "fp32", True
    w2, h2 = w1, h1
    if kind in ("match", "pyramid", "approx") and rng.random() < 0.4:   # images of two cameras, or a crop
        w2, h2 = max(32, int(w1 * rng.uniform(0.7, 1.0))), max(24, int(h1 * rng.uniform(0.7, 1.0)))
    c = dict(kind=kind, w1=w1, h1=h1, w2=w2, h2=h2, prec=prec, comp=comp, disp=round(rng.uniform(0.01, 0.12) * w1, 1))
    if kind == "approx":
        c["protos"], c["iters"] = rng.randint(64, 1024), rng.randint(4, 10)
    return c


def _sizes(case):
    """The (w, h) of a batch's pairs: two of each of the mixed sizes, one size for all, or sizes spread by `shape`."""
    n, s = case["n"], case["shape"]
    if s == 0:
        return [MIXED[k // 2 % 4] for k in range(n)]
    if s < 5:
        return [MIXED[s - 1]] * n
    return [(97 + (s * 41 * (k + 1)) % 540, 61 + (s * 29 * (k + 2)) % 300) for k in range(n)]


# --------------------------------------------------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------------------------------------------------
def _lattice(lat, w, h, cell):
    """Smoothstep interpolation of a random lattice on a w x h grid."""
    y, x = torch.arange(h, device=DEV, dtype=torch.float64) / cell, torch.arange(w, device=DEV, dtype=torch.float64) / cell
    y0, x0 = y.floor().long(), x.floor().long()
    ty, tx = y - y0, x - x0
    ty, tx = (ty * ty * (3 - 2 * ty))[:, None], (tx * tx * (3 - 2 * tx))[None, :]
    rows0, rows1 = lat[y0], lat[y0 + 1]
    top = rows0[:, x0] * (1 - tx) + rows0[:, x0 + 1] * tx
    bot = rows1[:, x0] * (1 - tx) + rows1[:, x0 + 1] * tx
    return top * (1 - ty) + bot * ty


def _noise(w, h, gen, octaves, cell):
    """Value noise of several octaves, scaled to [0, 1]."""
    out, amp = 0.0, 1.0
    for _ in range(octaves):
        lat = torch.rand((math.ceil(h / cell) + 2, math.ceil(w / cell) + 2), generator=gen, device=DEV, dtype=torch.float64)
        out = out + amp * _lattice(lat, w, h, cell)
        amp, cell = amp / 2, max(cell / 2, 1.0)
    return (out - out.min()) / (out.max() - out.min()).clamp_min(1e-12)


def _sample(img, x, y):
    """Bilinear samples of img [H][W], coordinates clamped to the image."""
    h, w = img.shape
    x, y = x.clamp(0, w - 1), y.clamp(0, h - 1)
    x0, y0 = x.floor(), y.floor()
    fx, fy = x - x0, y - y0
    x0, y0 = x0.long(), y0.long()
    x1, y1 = (x0 + 1).clamp_max(w - 1), (y0 + 1).clamp_max(h - 1)
    top = img[y0, x0] + fx * (img[y0, x1] - img[y0, x0])
    bot = img[y1, x0] + fx * (img[y1, x1] - img[y1, x0])
    return top + fy * (bot - top)


def _images(w1, h1, w2, h2, disp, seed):
    """Image 1, image 2 = image 1 displaced by a smooth field of at most `disp` pixels, brighter and noisy; the field."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    img1 = _noise(w1, h1, gen, 4, 16.0)
    cell = max(w2, h2) / 2.0
    dx, dy = (_noise(w2, h2, gen, 2, cell) * 2 - 1 for _ in range(2))
    s = disp / (dx * dx + dy * dy).sqrt().max().clamp_min(1e-12)
    dx, dy = dx * s, dy * s
    y, x = torch.meshgrid(torch.arange(h2, device=DEV, dtype=torch.float64),
                          torch.arange(w2, device=DEV, dtype=torch.float64), indexing="ij")
    img2 = 1.05 * _sample(img1, x * (w1 / w2) - dx, y * (h1 / h2) - dy)
    img2 = (img2 + 0.01 * torch.randn(img2.shape, generator=gen, device=DEV, dtype=torch.float64)).clamp(0, 1)
    return img1.float().contiguous(), img2.float().contiguous(), (dx, dy), gen


def _case_images(case, seed):
    return _images(case["w1"], case["h1"], case["w2"], case["h2"], case["disp"], seed)


def _matches(case, field, gen):
    """Rows (x1, y1, x2, y2, score) of a device match list with its count, as a matching call leaves them: two thirds of
    the atomic patches, in patch order, displaced by the field (to a pixel), one in twenty astray."""
    w, h = case["w1"], case["h1"]
    cy, cx = torch.meshgrid(torch.arange(2, h, 4, device=DEV), torch.arange(2, w, 4, device=DEV), indexing="ij")
    cx, cy = cx.reshape(-1), cy.reshape(-1)
    n0 = cx.numel()
    r = torch.rand((4, n0), generator=gen, device=DEV, dtype=torch.float64)
    astray = r[1] < 0.05
    tx = torch.where(astray, r[2] * (w - 1), cx + field[0][cy, cx]).round().clamp(0, w - 1)
    ty = torch.where(astray, r[3] * (h - 1), cy + field[1][cy, cx]).round().clamp(0, h - 1)
    score = 2.0 + 5.0 * torch.rand(n0, generator=gen, device=DEV, dtype=torch.float64)
    rows = torch.stack([cx.double(), cy.double(), tx, ty, score], 1)[r[0] < 0.67].float()
    out = torch.zeros((n0, 5), device=DEV)
    out[:rows.shape[0]] = rows
    return out, torch.tensor([rows.shape[0]], dtype=torch.int32, device=DEV)


def _descriptor_fields(case, seed):
    img1, img2, _, _ = _case_images(case, seed)
    return _descriptors64(img1).float().contiguous(), _descriptors64(img2).float().contiguous()


# --------------------------------------------------------------------------------------------------------------------
# prepare / run
# --------------------------------------------------------------------------------------------------------------------
class _Kept:
    """What a program keeps between calls: a context, and one workspace for all the inputs of a size."""

    def __init__(self, prec, comp):
        self.context = dm.Context(PREC[prec], compensated=comp)
        self.ctx = self.context.ctx
        self.ws = None


_KEPT = weakref.WeakValueDictionary()


def _kept(case, nbytes):
    key = tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "disp")))
    k = _KEPT.get(key)
    if k is None:
        k = _Kept(case["prec"], case["comp"])
        _KEPT[key] = k
        n = nbytes(k.ctx)
        k.ws = torch.empty(max(n, 256), dtype=torch.uint8, device=DEV) if n else None
    return k


def _out(w1, h1, w2, h2):
    n0 = dm.dm_geometry(w1, h1, w2, h2)["n_patch0"]
    return torch.zeros((n0, 5), device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "batch":
        sets = [_images(w, h, w, h, case["disp"], seed * 64 + k)[:2] for k, (w, h) in enumerate(_sizes(case))]
        outs = [_out(i1.shape[1], i1.shape[0], i2.shape[1], i2.shape[0]) for i1, i2 in sets]
        items = [(i1, i2, o, c) for (i1, i2), (o, c) in zip(sets, outs)]
        if case["host"]:
            items = [tuple(t.cpu().pin_memory() for t in it) for it in items]
            s["pairs"] = dm.make_pairs_host(items)
            s["kept"] = _kept(case, lambda ctx: dm.dm_batch_host_workspace_bytes(ctx, s["pairs"]))
        else:
            s["pairs"] = dm.make_pairs(items)
            s["kept"] = _kept(case, lambda ctx: dm.dm_batch_workspace_bytes(ctx, s["pairs"]))
        s["items"] = items
        return s
    size = (case["w1"], case["h1"], case["w2"], case["h2"])
    if kind == "grad":
        s["kept"] = _kept(case, lambda ctx: 0)
        s["d1"], s["d2"] = (d.requires_grad_() for d in _descriptor_fields(case, seed))
        return s
    s["i1"], s["i2"], field, gen = _case_images(case, seed)
    s["out"], s["count"] = _out(*size)
    if kind == "match":
        s["kept"] = _kept(case, lambda ctx: dm.dm_workspace_bytes(ctx, *size)["match"])
    elif kind == "star":
        s["kept"] = _kept(case, lambda ctx: dm.dm_star_workspace_bytes(ctx, *size)["match"])
    elif kind == "invariant":
        s["kept"] = _kept(case, lambda ctx: dm.dm_invariant_workspace_bytes(ctx, *size))
    elif kind == "deepflow":
        s["matches"], s["n"] = _matches(case, field, gen)
        s["prm"] = dm.dm_flow_params()
        s["kept"] = _kept(case, lambda ctx: dm.dm_deepflow_workspace_bytes(ctx, size[0], size[1], s["matches"].shape[0], s["prm"]))
        s["u"], s["v"] = torch.zeros_like(s["i1"]), torch.zeros_like(s["i1"])
    else:
        geo = dm.dm_geometry(*size)
        s["d1"] = torch.empty((case["h1"], case["w1"], 9), device=DEV)
        s["d2"] = torch.empty((case["h2"], case["w2"], 9), device=DEV)
        if kind == "pyramid":
            s["kept"] = _kept(case, lambda ctx: dm.dm_workspace_bytes(ctx, *size)["desc"])
            # the pyramid is the output: its own memory, zero where no patch exists
            n = dm.dm_workspace_bytes(s["kept"].ctx, *size)["pyramid"]
            s["pyr"] = torch.zeros(n, dtype=torch.uint8, device=DEV)
            s["levels"] = geo["L"] + 1
        else:
            def total(ctx):
                b = dm.dm_workspace_bytes(ctx, *size)
                return b["desc"] + b["pyramid"] + b["backtrack"] + 1024

            s["kept"] = _kept(case, total)
            b = dm.dm_workspace_bytes(s["kept"].ctx, *size)
            cut = [-(-b[k] // 256) * 256 for k in ("desc", "pyramid")]
            ws = s["kept"].ws
            s["ws_desc"], s["ws_pyr"], s["ws_bt"] = ws[:b["desc"]], ws[cut[0]:cut[0] + b["pyramid"]], ws[cut[0] + cut[1]:]
            D = min(case["protos"], geo["n_patch0"])
            s["protos"] = torch.zeros((D, 144), device=DEV)
            s["assign"] = torch.zeros(geo["n_patch0"], dtype=torch.int32, device=DEV)
            s["ws_k"] = torch.empty(dm.dm_prototypes_workspace_bytes(s["kept"].ctx, size[0], size[1], D), dtype=torch.uint8,
                                    device=DEV)
    return s


def _level(pyr, ws, level):
    """Device views of one level: values [n][rows][columns] and argmax codes (None at the top)."""
    i = dm.dm_pyramid_level(pyr, level)
    n, mh, pitch = i["n"], i["mh"], i["pitch"]
    at = i["vals"] - ws.data_ptr()
    vals = ws[at:at + n * mh * pitch * 4].view(torch.float32).view(n, mh, pitch)[:, :, :i["mw"]]
    if not i["argmax"]:
        return vals, None
    at = i["argmax"] - ws.data_ptr()
    return vals, ws[at:at + n * mh * pitch].view(n, mh, pitch)[:, :, :i["mw"]]


def run(s):
    case, k = s["case"], s["kept"]
    kind = case["kind"]
    if kind == "match":
        dm.dm_match(k.ctx, s["i1"], s["i2"], k.ws, s["out"], s["count"])
        return s["out"], s["count"]
    if kind == "batch":
        (dm.dm_match_batch_host if case["host"] else dm.dm_match_batch)(k.ctx, s["pairs"], k.ws)
        return [it[2:] for it in s["items"]]
    if kind == "star":
        dm.dm_match_star(k.ctx, s["i1"], s["i2"], k.ws, s["out"], s["count"])
        return s["out"], s["count"]
    if kind == "invariant":
        dm.dm_match_invariant(k.ctx, s["i1"], s["i2"], k.ws, s["out"], s["count"])
        return s["out"], s["count"]
    if kind == "deepflow":
        dm.dm_deepflow(k.ctx, s["i1"], s["i2"], s["matches"], s["n"], s["u"], s["v"], k.ws, s["prm"])
        return s["u"], s["v"]
    if kind == "grad":
        loss = autograd.top_max_loss(s["d1"], s["d2"], k.context)
        return loss.detach(), *torch.autograd.grad(loss, (s["d1"], s["d2"]))
    ws = k.ws if kind == "pyramid" else s["ws_desc"]
    dm.dm_descriptors(k.ctx, s["i1"], s["d1"], ws)
    dm.dm_descriptors(k.ctx, s["i2"], s["d2"], ws)
    if kind == "pyramid":
        pyr = dm.dm_correlate_pyramid(k.ctx, s["d1"], s["d2"], s["pyr"])
        levels = [_level(pyr, s["pyr"], i) for i in range(s["levels"])]
        dm.dm_pyramid_free(pyr)
        return {"desc": (s["d1"], s["d2"]), "vals": [v for v, _ in levels], "argmax": [a for _, a in levels if a is not None]}
    dm.dm_prototypes(k.ctx, s["d1"], s["protos"].shape[0], case["iters"], s["protos"], s["assign"], s["ws_k"])
    pyr = dm.dm_correlate_pyramid_approx(k.ctx, s["protos"], s["assign"], case["w1"], case["h1"], s["d2"], s["ws_pyr"])
    dm.dm_backtrack(k.ctx, pyr, s["ws_bt"], s["out"], s["count"])
    dm.dm_pyramid_free(pyr)
    return s["protos"], s["assign"], s["out"], s["count"]


# --------------------------------------------------------------------------------------------------------------------
# work
# --------------------------------------------------------------------------------------------------------------------
def _patches(w, h):
    return ((w - 3) // 4 + 1 if w >= 3 else 0) * ((h - 3) // 4 + 1 if h >= 3 else 0)


def _match_work(w1, h1, w2, h2, maps=None):
    """Images in, matches out; level-0 products of `maps` patches (all of them by default), and per position of every
    level above four additions and a power of the pooled value."""
    n0 = _patches(w1, h1)
    levels = max(1, math.ceil(math.log2(max(w1, h1) / 4)))
    lattice = -(-w1 // 4) * -(-h1 // 4)
    flops = 288.0 * (n0 if maps is None else maps) * w2 * h2 + sum(6.0 * lattice * w2 * h2 / 4 ** l for l in range(1, levels + 1))
    return {"bytes": 4.0 * (w1 * h1 + w2 * h2) + 20.0 * n0, "flops": flops}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        each = [_match_work(w, h, w, h) for w, h in _sizes(case)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    size = (case["w1"], case["h1"], case["w2"], case["h2"])
    w1, h1, w2, h2 = size
    if kind in ("match", "star"):
        return _match_work(*size)
    if kind == "approx":
        n0 = _patches(w1, h1)
        D = min(case["protos"], n0)
        w = _match_work(*size, maps=D)
        return {"bytes": w["bytes"] + 576.0 * D + 4.0 * n0, "flops": w["flops"] + 288.0 * n0 * D * (case["iters"] + 1)}
    if kind == "invariant":
        total = {"bytes": 4.0 * (w1 * h1 + w2 * h2) + 20.0 * _patches(w1, h1), "flops": 0.0}
        for i in range(9):
            sg = -2 + 0.5 * i
            s1, s2 = max(1.0, 2.0 ** sg), max(1.0, 2.0 ** -sg)
            for k in range(8):
                c, d = abs(math.cos(k * math.pi / 4)), abs(math.sin(k * math.pi / 4))
                wr, hr = int((c * w2 + d * h2) / s2 + 0.5), int((d * w2 + c * h2) / s2 + 0.5)
                total["flops"] += _match_work(int(w1 / s1 + 0.5), int(h1 / s1 + 0.5), wr, hr)["flops"]
        return total
    if kind == "deepflow":
        px = sum(w * h for w, h in _flow_sizes(w1, h1))
        return {"bytes": 16.0 * w1 * h1 + 20.0 * _patches(w1, h1), "flops": px * 5.0 * (25 * 45 + 90)}
    w = _match_work(*size)
    if kind == "grad":   # both fields in, both gradients out
        return {"bytes": 72.0 * (w1 * h1 + w2 * h2), "flops": w["flops"]}
    # images in, descriptors and every level's pooled values and argmax codes out
    levels = max(1, math.ceil(math.log2(max(w1, h1) / 4)))
    stored = sum((_patches(w1, h1) if l == 0 else -(-w1 // 4) * -(-h1 // 4)) * -(-w2 // 2 ** (l + 1)) * -(-h2 // 2 ** (l + 1))
                 for l in range(levels))
    return {"bytes": 40.0 * (w1 * h1 + w2 * h2) + 5.0 * stored, "flops": w["flops"]}


# --------------------------------------------------------------------------------------------------------------------
# exact: the method in 64 bits, plain torch
# --------------------------------------------------------------------------------------------------------------------
def _smooth64(x, sigma):
    """Gaussian smoothing of [H][W][C], taps to ceil(3 sigma), replicated border."""
    R = math.ceil(3 * sigma)
    t = torch.exp(-torch.arange(-R, R + 1, device=DEV, dtype=torch.float64) ** 2 / (2 * sigma * sigma))
    t = t / t.sum()
    y = x.permute(2, 0, 1)[:, None]
    y = F.conv2d(F.pad(y, (R, R, 0, 0), mode="replicate"), t.view(1, 1, 1, -1))
    y = F.conv2d(F.pad(y, (0, 0, R, R), mode="replicate"), t.view(1, 1, -1, 1))
    return y[:, 0].permute(1, 2, 0)


def _dx(f):
    return 0.5 * (torch.cat([f[:, 1:], f[:, -1:]], 1) - torch.cat([f[:, :1], f[:, :-1]], 1))


def _dy(f):
    return 0.5 * (torch.cat([f[1:], f[-1:]], 0) - torch.cat([f[:1], f[:-1]], 0))


def _descriptors64(img):
    """Pixel descriptors: smooth, gradient, eight half-wave projections, smooth, sigmoid, smooth, append mu, normalise."""
    g = _smooth64(255.0 * img.double()[..., None], 1.0)[..., 0]
    gx, gy = _dx(g), _dy(g)
    ang = torch.arange(8, device=DEV, dtype=torch.float64) * (math.pi / 4)
    ch = (gx[..., None] * torch.cos(ang) + gy[..., None] * torch.sin(ang)).clamp_min(0)
    ch = 2 / (1 + torch.exp(-0.2 * _smooth64(ch, 1.0))) - 1
    ch = _smooth64(ch, 1.0)
    d = torch.cat([ch, torch.full_like(ch[..., :1], 0.3)], -1)
    return d / d.norm(dim=-1, keepdim=True)


def _grid(w1, h1, level):
    if level == 0:
        return (w1 - 3) // 4 + 1, (h1 - 3) // 4 + 1
    return -(-w1 // 4), -(-h1 // 4)


def _children(w1, h1, level):
    """[4][patches] indices at level - 1 of the children (-1 outside the grid), in the order (-1,-1), (-1,1), (1,-1), (1,1)."""
    gx, gy = _grid(w1, h1, level)
    cgx, cgy = _grid(w1, h1, level - 1)
    iy, ix = torch.meshgrid(torch.arange(gy, device=DEV), torch.arange(gx, device=DEV), indexing="ij")
    got = []
    for ox in (-1, 1):
        for oy in (-1, 1):
            ax, ay = ((ox - 1) // 2, (oy - 1) // 2) if level == 1 else (ox * 2 ** (level - 2), oy * 2 ** (level - 2))
            cx, cy = ix + ax, iy + ay
            ok = (cx >= 0) & (cy >= 0) & (cx < cgx) & (cy < cgy)
            got.append(torch.where(ok, cy * cgx + cx, torch.full_like(cx, -1)).reshape(-1))
    return torch.stack(got)


def _pyramid64(d1, d2, lam=1.4):
    """Every level's stored maps (zero where no patch exists): pooled and rectified below the top, the top unpooled."""
    h1, w1, _ = d1.shape
    h2, w2, _ = d2.shape
    gx, gy = _grid(w1, h1, 0)
    a = F.pad(d1.permute(2, 0, 1), (0, max(0, 4 * gx - w1), 0, max(0, 4 * gy - h1)))[:, :4 * gy, :4 * gx]
    a = a.reshape(9, gy, 4, gx, 4).permute(1, 3, 0, 2, 4).reshape(gx * gy, 9 * 16)
    b = F.unfold(F.pad(d2.permute(2, 0, 1)[None], (2, 1, 2, 1)), 4)[0]
    step = max(1, int(1.5e8) // (w2 * h2))
    low = [F.max_pool2d((a[i:i + step] @ b / 16).view(-1, 1, h2, w2), 3, 2, 1)[:, 0] for i in range(0, gx * gy, step)]
    maps, ok = torch.cat(low) ** lam, torch.ones(gx * gy, dtype=torch.bool, device=DEV)
    levels, wanted, l = [maps], 0, 0
    while 4 * 2 ** wanted < max(w1, h1):
        wanted += 1
    for l in range(1, wanted + 1):
        c = _children(w1, h1, l)
        here = (c >= 0) & ok[c.clamp_min(0)]
        if not bool(here.any()):
            break
        n, (_, mh, mw) = c.shape[1], maps.shape
        padded = F.pad(torch.cat([maps, maps.new_zeros(1, mh, mw)]), (1, 1, 1, 1))
        s = 0.0
        for i, (ox, oy) in enumerate(((-1, -1), (-1, 1), (1, -1), (1, 1))):
            pick = torch.where(here[i], c[i], torch.full_like(c[i], maps.shape[0]))
            s = s + padded[pick][:, 1 + oy:1 + oy + mh, 1 + ox:1 + ox + mw]
        top = s / here.sum(0).clamp_min(1)[:, None, None]
        ok = here.any(0)
        maps = F.max_pool2d(top[:, None], 3, 2, 1)[:, 0] ** lam
        levels.append(maps)
    # the last level that has a patch is stored unpooled
    levels[-1] = top ** lam
    return levels, ok


def _exact_grad(case, seed):
    d1, d2 = (d.double().requires_grad_() for d in _descriptor_fields(case, seed))
    levels, ok = _pyramid64(d1, d2)
    loss = levels[-1].flatten(1).amax(1)[ok].sum()
    return loss.detach(), *torch.autograd.grad(loss, (d1, d2))


def _flow_sizes(w, h):
    sizes = [(w, h)]
    while True:
        w, h = math.floor(0.95 * w + 0.5), math.floor(0.95 * h + 0.5)
        if min(w, h) < 16:
            return sizes
        sizes.append((w, h))


def _resampled(f, w, h, scale):
    x = (torch.arange(w, device=DEV, dtype=torch.float64) + 0.5) * scale - 0.5
    y = (torch.arange(h, device=DEV, dtype=torch.float64) + 0.5) * scale - 0.5
    return _sample(f, x[None, :].expand(h, w), y[:, None].expand(h, w))


def _exact_flow(case, seed):
    """Coarse-to-fine variational flow with the default parameters, n = 5 fixed-point steps of 25 red-black sweeps."""
    img1, img2, field, gen = _case_images(case, seed)
    m, n = _matches(case, field, gen)
    m = m[:int(n)].double()
    eta, gamma, beta, b, kappa, zeta2, eps2, sigma_m, omega = 0.95, 0.8, 300.0, 0.6, 5.0, 0.01, 1e-6, 50.0, 1.6
    sizes = _flow_sizes(case["w1"], case["h1"])
    P = [[_smooth64(255.0 * i.double()[..., None], 0.5)[..., 0]] for i in (img1, img2)]
    for w, h in sizes[1:]:
        for p in P:
            p.append(_resampled(p[-1], w, h, 1 / eta))
    psi = lambda s: 0.5 / (s + eps2).sqrt()  # noqa: E731
    # weight of each match at full resolution: texture of image 1 and difference of appearance
    I1, I2 = P[0][0], P[1][0]
    gx, gy = _dx(I1), _dy(I1)
    box = lambda f: F.avg_pool2d(F.pad(f[None, None], (1, 1, 1, 1), mode="replicate"), 3, 1)[0, 0] * 9  # noqa: E731
    sa, sb, sc = box(gx * gx), box(gx * gy), box(gy * gy)
    lmin = ((sa + sc) / 2 - (((sa - sc) / 2) ** 2 + sb * sb).sqrt()).clamp_min(0)
    x1, y1, x2, y2 = (m[:, i].long() for i in range(4))
    delta = sum((f[y1, x1] - g[y2, x2]).abs() for f, g in ((I1, I2), (gx, _dx(I2)), (gy, _dy(I2))))
    phi = (10 * lmin[y1, x1]).sqrt() / (sigma_m * math.sqrt(2 * math.pi)) * torch.exp(-delta / (2 * sigma_m))
    order = torch.sort(m[:, 4], descending=False, stable=True).indices   # a higher score is written later
    kmax, u, v = len(sizes) - 1, None, None
    for k in range(kmax, -1, -1):
        w, h = sizes[k]
        I1, I2 = P[0][k], P[1][k]
        u, v = (torch.zeros((h, w), device=DEV, dtype=torch.float64) if f is None else _resampled(f, w, h, eta) / eta for f in (u, v))
        sk = eta ** k
        # float32 rounds these pixel positions; so does this, that both pick the same pixel
        px, py = (((m[:, i].float() + 0.5) * sk - 0.5 + 0.5).floor().long().clamp(0, q - 1) for i, q in ((0, w), (1, h)))
        mc, mu, mv = (torch.zeros((h, w), device=DEV, dtype=torch.float64) for _ in range(3))
        owner = torch.full((h * w,), -1, device=DEV, dtype=torch.long)
        rank = torch.empty_like(order)
        rank[order] = torch.arange(order.numel(), device=DEV)
        owner.scatter_reduce_(0, py * w + px, rank, "amax")
        at = (owner >= 0).nonzero()[:, 0]
        who = order[owner[at]]
        mc.view(-1)[at] = beta * (k / kmax if kmax else 1.0) ** b * phi[who]
        mu.view(-1)[at], mv.view(-1)[at] = (m[who, 2] - m[who, 0]) * sk, (m[who, 3] - m[who, 1]) * sk
        alpha = torch.exp(-kappa * ((_dx(I1) / 255) ** 2 + (_dy(I1) / 255) ** 2).sqrt())
        y, x = torch.meshgrid(torch.arange(h, device=DEV, dtype=torch.float64),
                              torch.arange(w, device=DEV, dtype=torch.float64), indexing="ij")
        I2w = _sample(I2, x + u, y + v)
        Im = 0.5 * (I1 + I2w)
        Ix, Iy = _dx(Im), _dy(Im)
        Ixx, Ixy, Iyy = _dx(Ix), _dy(Ix), _dy(Iy)
        Ixz, Iyz = _dx(I2w) - _dx(I1), _dy(I2w) - _dy(I1)
        thx, thy = 1 / (Ixx ** 2 + Ixy ** 2 + zeta2), 1 / (Ixy ** 2 + Iyy ** 2 + zeta2)
        du, dv = torch.zeros_like(u), torch.zeros_like(u)
        red = ((x + y) % 2) == 0
        for _ in range(5):
            U, V = u + du, v + dv
            s = 0.0
            for f in (U, V):
                s = s + F.pad(f[:, 1:] - f[:, :-1], (0, 1)) ** 2 + F.pad(f[1:] - f[:-1], (0, 0, 0, 1)) ** 2
            ps = alpha * psi(s)
            rx, ry = Ixx * du + Ixy * dv + Ixz, Ixy * du + Iyy * dv + Iyz
            ag = gamma * psi(thx * rx * rx + thy * ry * ry)
            mw = mc * psi((U - mu) ** 2 + (V - mv) ** 2)
            ax, ay = ag * thx, ag * thy
            a11, a12, a22 = ax * Ixx ** 2 + ay * Ixy ** 2 + mw, ax * Ixx * Ixy + ay * Ixy * Iyy, ax * Ixy ** 2 + ay * Iyy ** 2 + mw
            b1, b2 = -(ax * Ixx * Ixz + ay * Ixy * Iyz) - mw * (u - mu), -(ax * Ixy * Ixz + ay * Iyy * Iyz) - mw * (v - mv)
            ex, ey = 0.5 * (ps[:, 1:] + ps[:, :-1]), 0.5 * (ps[1:] + ps[:-1])
            wl, wr, wu, wd = F.pad(ex, (1, 0)), F.pad(ex, (0, 1)), F.pad(ey, (0, 0, 1, 0)), F.pad(ey, (0, 0, 0, 1))
            sw = wl + wr + wu + wd

            def flux(f, g):
                """Sum over the neighbours of their edge weight times (f_p + g_p)."""
                t = F.pad(f + g, (1, 1, 1, 1))
                return wl * t[1:-1, :-2] + wr * t[1:-1, 2:] + wu * t[:-2, 1:-1] + wd * t[2:, 1:-1]

            d1, d2, c1, c2 = omega / (a11 + sw), omega / (a22 + sw), b1 - sw * u, b2 - sw * v
            for _ in range(25):
                for color in (red, ~red):
                    nu = (1 - omega) * du + d1 * (c1 + flux(du, u) - a12 * dv)
                    du = torch.where(color, nu, du)
                    nv = (1 - omega) * dv + d2 * (c2 + flux(dv, v) - a12 * du)
                    dv = torch.where(color, nv, dv)
        u, v = u + du, v + dv
    return u, v


def exact(case, seed):
    kind = case["kind"]
    if kind == "grad":
        return _exact_grad(case, seed)
    if kind == "deepflow":
        return _exact_flow(case, seed)
    if kind == "pyramid":
        img1, img2, _, _ = _case_images(case, seed)
        d1, d2 = _descriptors64(img1), _descriptors64(img2)
        return {"desc": (d1, d2), "vals": _pyramid64(d1, d2)[0], "argmax": None}
    return None
