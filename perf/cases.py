"""The calls that programs make of this package, as measurable cases.

A case is a dict of plain values.  ``prepare`` makes its inputs on the GPU (host
frames for the host-buffer path) from a seed, ``run`` is one pass through the
public entry points, ``work`` the bytes and operations that a pass cannot do
without, and ``exact`` the same outputs in 64 bits by plain torch.

Kinds of case:
  fill      one frame, guide field in hand            Context.fill
  movie     splines and frames, filled in place       Context.guidance_batched + Context.fill_batched
  guidance  splines to guide fields                   Context.guidance_batched
  detect    frames to guide fields                    Context.guidance_auto_batched
  train     forward and backward of the fill layer    autograd.guidefill_fill
  host      frames in pinned host memory, in place    Context.fill_batched_host
"""
import math

import numpy as np
import torch

import paper_1611_05319_gb300 as gf
from paper_1611_05319_gb300.autograd import guidefill_fill

DEV = "cuda:0"
_DEFAULT = dict(kind="fill", n=1, H=128, W=128, hole="bands", frac=0.03, hw0=1.5, hw1=7.5, guide="splines",
                eps=3.0, mu=50.0, c=0.05, ghost=True, smart=True, data=False, byst=False, curves=20)


def _case(name=None, **kw):
    c = dict(_DEFAULT, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: a scratch on a thumbnail, one constant direction
        _case("fill_128", hole="annulus", guide="const", curves=0),
        # a small still of odd size with bystanders, guided regions first (data term)
        _case("fill_961x529_data", H=529, W=961, frac=0.03, byst=True, data=True),
        # one HD film frame: thin cracks along its splines
        _case("fill_1080", H=1080, W=1920, frac=0.03),
        # the widest usual frame: one large blob plus thin cracks, a wider ball
        _case("fill_4k_blob", H=2160, W=3840, hole="blob", frac=0.02, eps=4.0),
        # a wide ball on an SD video frame
        _case("fill_960_wide", H=960, W=1280, frac=0.02, eps=6.0),
        # fill in onion order, nothing guided: a large plain hole crossed by a line
        _case("fill_line_onion", H=500, W=2000, hole="line", guide="zero", smart=False, curves=0),
        # coherence transport (lattice ball) on a still, the method Guidefill is compared with
        _case("fill_still_lattice", H=1125, W=1500, frac=0.05, hw0=2.0, hw1=12.0, eps=5.0, ghost=False),
        # a shot of film: uneven frames, guide fields from the artist's splines, filled in place
        _case("movie_32x1080", kind="movie", n=32, H=1080, W=1920, frac=0.0, hw0=1.0, hw1=20.0),
        # the guide fields alone (splines being edited)
        _case("guidance_16x1080", kind="guidance", n=16, H=1080, W=1920, frac=0.04, hw0=1.0, hw1=20.0),
        # automatic splines on a short shot
        _case("detect_8x1080", kind="detect", n=8, H=1080, W=1920, frac=0.04, hw0=1.0, hw1=20.0),
        # the fill as a layer of a trained model: forward and backward
        _case("train_16x512", kind="train", n=16, H=512, W=512, frac=0.05, hw0=1.5, hw1=4.5, mu=10.0, curves=12),
        # frames owned by a host program, in pinned memory, transfers included
        _case("host_8x1080", kind="host", n=8, H=1080, W=1920, frac=0.0, hw0=1.0, hw1=20.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fill", "fill", "fill", "movie", "guidance", "detect", "train", "host"])
    if kind == "fill":
        H, W = _log_int(rng, 64, 2160), _log_int(rng, 64, 3840)
        eps = rng.choice([1.5, 2.0, 3.0, 3.0, 4.0, 5.0, 6.0])
        if eps > 4.0:
            H, W = min(H, 960), min(W, 1280)
        ghost = rng.random() < 0.75
        smart = rng.random() < 0.75
        return _case(kind=kind, H=H, W=W, hole=rng.choice(["bands", "bands", "blob", "annulus"]),
                     frac=round(rng.uniform(0.005, 0.05), 4), hw1=round(rng.uniform(3.0, 10.0), 2),
                     guide=rng.choice(["splines", "splines", "const", "zero"]), eps=eps,
                     mu=rng.choice([10.0, 50.0, 100.0]), ghost=ghost, smart=smart,
                     data=smart and rng.random() < 0.25, byst=rng.random() < 0.25, curves=rng.randint(1, 20))
    if kind == "train":
        H, W = _log_int(rng, 96, 700), _log_int(rng, 96, 700)
        n = min(16, max(1, 4194304 // (H * W)))
        return _case(kind=kind, n=_log_int(rng, 1, n), H=H, W=W, frac=round(rng.uniform(0.01, 0.06), 4), hw1=4.5,
                     curves=rng.randint(1, 12), eps=rng.choice([2.0, 3.0, 3.0, 4.0]), mu=rng.choice([5.0, 10.0, 20.0]))
    H, W = _log_int(rng, 240, 1440), _log_int(rng, 320, 2560)
    most = {"movie": 32, "guidance": 16, "detect": 8, "host": 8}[kind]
    most = min(most, max(1, most * 1080 * 1920 // (H * W)))
    return _case(kind=kind, n=_log_int(rng, 1, most), H=H, W=W, frac=round(rng.uniform(0.01, 0.06), 4),
                 hw0=1.0, hw1=round(rng.uniform(3.0, 20.0), 2), curves=rng.randint(4, 30), byst=rng.random() < 0.25)


# ------------------------------------------------------------------ inputs
def _polylines(rng, H, W, n, length, n_seg=64):
    """n flattened cubic Beziers of about ``length`` px inside the frame: (offsets, points)."""
    margin = min(40.0, 0.1 * min(H, W))
    lo, hi = np.array([margin, margin]), np.array([W - 1 - margin, H - 1 - margin])
    t = np.linspace(0.0, 1.0, n_seg + 1)[:, None]
    pts = []
    for _ in range(n):
        p = rng.uniform(lo, hi)
        heading = rng.uniform(0, 2 * np.pi)
        ctrl = [p]
        for _ in range(3):
            heading += rng.normal(0.0, 0.6)
            p = np.clip(p + length * rng.uniform(0.6, 1.4) / 3.0 * np.array([np.cos(heading), np.sin(heading)]), lo, hi)
            ctrl.append(p)
        c0, c1, c2, c3 = ctrl
        pts.append((1 - t) ** 3 * c0 + 3 * t * (1 - t) ** 2 * c1 + 3 * t * t * (1 - t) * c2 + t ** 3 * c3)
    off = np.arange(0, (n_seg + 1) * (n + 1), n_seg + 1, dtype=np.int32)
    return off, (np.concatenate(pts) if pts else np.zeros((0, 2))).astype(np.float32)


def _stamp_bands(hole, off, pts, half_widths):
    """Sets the pixels within half_widths[i] of polyline i."""
    H, W = hole.shape
    p = torch.from_numpy(pts).to(DEV)
    for i, hw in enumerate(half_widths):
        q = pts[off[i]:off[i + 1]]
        x0, y0 = np.maximum(np.floor(q.min(0) - hw - 1), 0).astype(int)
        x1, y1 = np.minimum(np.ceil(q.max(0) + hw + 2), [W, H]).astype(int)
        a, b = p[off[i]:off[i + 1] - 1], p[off[i] + 1:off[i + 1]]
        v = b - a
        il = 1.0 / (v * v).sum(1).clamp_min(1e-12)
        ys = torch.arange(y0, y1, device=DEV, dtype=torch.float32)[:, None, None] - a[:, 1]
        xs = torch.arange(x0, x1, device=DEV, dtype=torch.float32)[None, :, None] - a[:, 0]
        t = ((xs * v[:, 0] + ys * v[:, 1]) * il).clamp_(0.0, 1.0)
        d2 = ((xs - t * v[:, 0]) ** 2 + (ys - t * v[:, 1]) ** 2).amin(2)
        hole[y0:y1, x0:x1] |= d2 <= hw * hw


def _image(rng, H, W, n_polys=16):
    """[H, W, 4] float32: convex polygons with colour gradients, noise 0.01, alpha 1."""
    ys = torch.arange(H, device=DEV, dtype=torch.float32)[:, None, None]
    xs = torch.arange(W, device=DEV, dtype=torch.float32)[None, :, None]

    def ramp(c0, gx, gy, X, Y):
        c0, gx, gy = (torch.tensor(np.append(v, z), device=DEV, dtype=torch.float32)
                      for v, z in ((c0, 1.0), (gx, 0.0), (gy, 0.0)))
        return c0 + gx * X + gy * Y

    img = ramp(rng.uniform(0.2, 0.8, 3), rng.uniform(-0.2, 0.2, 3) / W, rng.uniform(-0.2, 0.2, 3) / H, xs, ys)
    s = float(min(H, W))
    for _ in range(n_polys):
        nv = int(rng.integers(3, 8))
        cx, cy, r = rng.uniform(0, W), rng.uniform(0, H), rng.uniform(0.05, 0.3) * s
        ang = np.sort(rng.uniform(0, 2 * np.pi, nv))
        px, py = cx + r * np.cos(ang), cy + r * np.sin(ang)
        x0, x1 = int(max(0, np.floor(px.min()))), int(min(W, np.ceil(px.max()) + 1))
        y0, y1 = int(max(0, np.floor(py.min()))), int(min(H, np.ceil(py.max()) + 1))
        col = rng.uniform(0.0, 1.0, 3), rng.uniform(-0.5, 0.5, 3) / r, rng.uniform(-0.5, 0.5, 3) / r
        if x0 >= x1 or y0 >= y1:
            continue
        X, Y = xs[:, x0:x1], ys[y0:y1]
        inside = torch.ones((y1 - y0, x1 - x0, 1), dtype=torch.bool, device=DEV)
        for i in range(nv):
            ax, ay, bx, by = px[i], py[i], px[(i + 1) % nv], py[(i + 1) % nv]
            inside &= (bx - ax) * (Y - ay) >= (by - ay) * (X - ax)
        sub = img[y0:y1, x0:x1]
        img[y0:y1, x0:x1] = torch.where(inside, ramp(*col, X - cx, Y - cy), sub)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(rng.integers(1 << 62)))
    img[..., :3] += 0.01 * torch.randn((H, W, 3), generator=gen, device=DEV)
    return img.clamp_(0.0, 1.0)


def _frame(case, seed, i):
    """(rgba [H,W,4], labels [H,W], splines) of frame i."""
    H, W = case["H"], case["W"]
    rng = np.random.default_rng([int(seed), i])
    frac = case["frac"] or float(rng.uniform(0.005, 0.08))
    hw = rng.uniform(case["hw0"], case["hw1"], max(case["curves"], 1))
    hw = np.minimum(hw, 0.05 * min(H, W))
    length = float(np.clip(frac * H * W / (2.0 * hw.sum()), 8.0, 2.0 * max(H, W)))
    off, pts = _polylines(rng, H, W, case["curves"], length)
    hole = torch.zeros((H, W), dtype=torch.bool, device=DEV)
    y = torch.arange(H, device=DEV)[:, None]
    x = torch.arange(W, device=DEV)[None, :]
    if case["hole"] in ("bands", "blob") and case["curves"]:
        _stamp_bands(hole, off, pts, hw)
    if case["hole"] == "annulus":  # radii 24 .. 32 in a 128 x 128 frame
        r = min(H, W) / 128.0
        r0, r1 = 24.0 * min(r, 2.0), 32.0 * min(r, 2.0)
        d2 = (x - (W - 1) / 2.0) ** 2 + (y - (H - 1) / 2.0) ** 2
        hole |= (d2 >= r0 * r0) & (d2 <= r1 * r1)
    if case["hole"] == "blob":  # 400 x 400 in a 4K frame
        b = max(8, int(min(H, W) * 400 / 2160))
        x0, y0 = int(rng.integers(2, W - b - 2)), int(rng.integers(2, H - b - 2))
        hole[y0:y0 + b, x0:x0 + b] = True
    rgba = _image(rng, H, W)
    if case["hole"] == "line":  # the line problem: [0, 4] x [0, 1], hole [0.4, 3.96] x [0.2, 0.8]
        u, v = (x + 0.5) * (4.0 / W), (y + 0.5) / H
        hole |= (v >= 0.2) & (v <= 0.8) & (u >= 0.4) & (u <= 3.96)
        a, b = (torch.tensor(np.append(rng.uniform(0.1, 0.9, 3), 1.0), device=DEV, dtype=torch.float32) for _ in "ab")
        rgba = torch.where(((v >= 0.45) & (v <= 0.55)).expand(H, W)[..., None], a, b).contiguous()
    labels = hole.to(torch.uint8)
    if case["byst"]:
        labels[:, int(0.8 * W):] = 2
    return rgba, labels, (off, pts)


def _nearest_field(labels, off, pts, eta=3.0):
    """Guide field of the nearest segment within 3 eta at hole pixels (values in 64 bits)."""
    H, W = labels.shape
    field = torch.zeros((H, W, 2), dtype=torch.float64, device=DEV)
    pix = torch.nonzero(labels == 1)
    first = np.setdiff1d(np.arange(len(pts)), off[1:] - 1)
    if not len(pix) or not len(first):
        return field
    p = torch.from_numpy(pts).to(DEV)
    a, b = p[first], p[first + 1]
    keep = ((b - a) ** 2).sum(1) > 0
    a, b = a[keep], b[keep]
    v = b - a
    il = 1.0 / (v[:, 0] * v[:, 0] + v[:, 1] * v[:, 1])
    a64, v64 = a.double(), b.double() - a.double()
    for part in torch.split(pix, max(1, (1 << 26) // len(a))):
        wx, wy = part[:, 1:].float() - a[:, 0], part[:, :1].float() - a[:, 1]
        t = ((wx * v[:, 0] + wy * v[:, 1]) * il).clamp_(0.0, 1.0)
        qx, qy = wx - t * v[:, 0], wy - t * v[:, 1]
        d2, j = (qx * qx + qy * qy).min(1)  # the choice of the segment is made in 32 bits
        w = part.flip(1).double() - a64[j]
        vj = v64[j]
        t = ((w * vj).sum(1) / (vj * vj).sum(1)).clamp_(0.0, 1.0)
        g = vj / vj.norm(dim=1, keepdim=True)
        g = g * torch.exp(-((w - t[:, None] * vj) ** 2).sum(1, keepdim=True) / (2.0 * eta * eta))
        near = d2 <= torch.tensor(3.0 * eta, device=DEV) ** 2
        field[part[:, 0], part[:, 1]] = torch.where(near[:, None], g, torch.zeros_like(g))
    return field


def _guide(case, rng_seed, labels, splines):
    H, W = labels.shape
    if case["guide"] == "splines":
        return _nearest_field(labels, *splines).float().contiguous()
    g = torch.zeros((H, W, 2), dtype=torch.float32, device=DEV)
    if case["guide"] == "const":
        th = math.radians(float(np.random.default_rng([int(rng_seed), 7]).uniform(0.0, 180.0)))
        g[..., 0], g[..., 1] = math.cos(th), math.sin(th)
    return g


def _inputs(case, seed):
    frames = [_frame(case, seed, i) for i in range(case["n"])]
    return [f[0] for f in frames], [f[1] for f in frames], [f[2] for f in frames]


def _angles(case, seed, splines, labels):
    """The train case's guidance as magnitude and angle, and the gradient from the layers above."""
    field = torch.stack([_nearest_field(lab, *sp) for lab, sp in zip(labels, splines)])
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) + 99)
    up = torch.randn((case["n"], case["H"], case["W"], 4), generator=gen, device=DEV)
    return field.norm(dim=-1).float(), torch.atan2(field[..., 1], field[..., 0]).float(), up


def prepare(case, seed):
    rgba, labels, splines = _inputs(case, seed)
    kind = case["kind"]
    s = dict(case=case, ctx=gf.context(0), fill=dict(eps=case["eps"], mu=case["mu"], c=case["c"], ghost=case["ghost"],
                                                     smart=case["smart"], data_term=case["data"]))
    if kind == "fill":
        return dict(s, rgba=rgba[0], labels=labels[0], guide=_guide(case, seed, labels[0], splines[0]))
    if kind == "train":
        mag, phi, up = _angles(case, seed, splines, labels)
        return dict(s, rgba=torch.stack(rgba).requires_grad_(), labels=torch.stack(labels), mag=mag,
                    phi=phi.requires_grad_(), mu=torch.tensor(case["mu"], device=DEV, requires_grad=True), up=up)
    if kind == "host":
        # frames of a host program in pinned memory, its pointer tables built once
        host = [r.cpu().pin_memory() for r in rgba]
        hlab = [v.cpu().pin_memory() for v in labels]
        hsh = [torch.empty((case["H"], case["W"]), dtype=torch.int32).pin_memory() for _ in rgba]
        np_rgba, np_shell = [h.numpy() for h in host], [h.numpy() for h in hsh]
        batch = gf.HostBatch(np_rgba, [h.numpy() for h in hlab], None, np_rgba, np_shell, splines=splines)
        return dict(s, batch=batch, rgba=np_rgba, shell=np_shell, keep=(host, hlab, hsh))
    dev = [(torch.from_numpy(o).to(DEV), torch.from_numpy(p).to(DEV)) for o, p in splines]
    return dict(s, rgba=rgba, labels=labels, off=[d[0] for d in dev], pts=[d[1] for d in dev],
                guides=[torch.zeros((case["H"], case["W"], 2), device=DEV) for _ in rgba])


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "fill":
        r = ctx.fill(state["rgba"], state["labels"], state["guide"], **state["fill"])
        return {"rgba": r.rgba, "shell": r.shell}
    if kind == "movie":
        ctx.guidance_batched(state["labels"], state["off"], state["pts"], out=state["guides"])
        rs = ctx.fill_batched(state["rgba"], state["labels"], state["guides"], out=["inplace"] * case["n"],
                              **state["fill"])
        return {"rgba": [r.rgba for r in rs], "shell": [r.shell for r in rs]}
    if kind == "guidance":
        return {"guide": ctx.guidance_batched(state["labels"], state["off"], state["pts"])}
    if kind == "detect":
        guides, det = ctx.guidance_auto_batched(state["rgba"], state["labels"])
        return {"guide": guides, "pts": [d.pts for d in det], "weight": [d.weight for d in det],
                "base": [d.base for d in det], "offsets": [d.offsets for d in det], "found": [d.result for d in det]}
    if kind == "host":
        st = ctx.fill_batched_host(state["batch"], **state["fill"])
        return {"rgba": state["rgba"], "shell": state["shell"], "filled": np.array(st["filled"])}
    out = guidefill_fill(state["rgba"], state["labels"], state["mag"], state["phi"], state["mu"], eps=case["eps"],
                         c=case["c"])
    g = torch.autograd.grad(out, [state["rgba"], state["phi"], state["mu"]], grad_outputs=state["up"])
    return {"out": out, "grad_rgba": g[0], "grad_phi": g[1], "grad_mu": g[2]}


def work(case):
    """Bytes: every input read once and every output written once (in-place calls write
    the hole's colours only).  Operations: per hole pixel its ball's samples, four taps
    of four channels each, in a fill; twice that again in its backward."""
    px, n, kind = float(case["H"] * case["W"]), case["n"], case["kind"]
    share = {"annulus": 0.03, "blob": 0.03, "line": 0.53}.get(case["hole"], case["frac"] or 0.0425)
    holes = share * px
    R = int(math.ceil(case["eps"]))
    ball = sum(1 for a in range(-R, R + 1) for b in range(-R, R + 1) if 0 < a * a + b * b <= case["eps"] ** 2)
    fill = holes * ball * 4 * 4 * 2
    near = min(px, 3.0 * holes)
    segs = 64.0 * case["curves"]
    if kind == "fill":
        return {"bytes": px * (16 + 1 + 16 + 4) + holes * 8, "flops": fill}
    if kind == "movie":
        return {"bytes": n * (px * (1 + 4) + near * 16 + holes * (8 + 16)), "flops": n * (fill + holes * 60)}
    if kind == "guidance":
        return {"bytes": n * (px * (1 + 8) + segs * 8), "flops": n * holes * 60}
    if kind == "detect":
        return {"bytes": n * (px * (1 + 8) + near * 16), "flops": n * near * 3 * 2 * (9 + 9)}
    if kind == "host":
        return {"bytes": n * (px * (1 + 4) + near * 16 + holes * 16), "flops": n * (fill + holes * 60)}
    return {"bytes": n * px * ((16 + 1 + 8 + 16 + 4) + (16 + 16 + 16 + 8 + 4 + 4)), "flops": n * 3 * fill}


# ------------------------------------------------------------------ 64 bits
def _fill64(rgba, labels, guide, eps, mu, c, ghost, smart, data_term, phi=None, mu_t=None, most_steps=3000):
    """The shell-by-shell fill of frames [n,H,W,..] in 64 bits, every frame and front pixel
    of a step at once: step k averages each front pixel's readable ball samples
    (bilinear, offsets formed and snapped to the lattice in 32 bits) and fills the
    ready ones.  ``phi`` and ``mu_t``: tensors whose gradients are wanted.
    Returns [n,H,W,4] float64, or None past ``most_steps`` steps."""
    n, H, W = labels.shape
    R = int(math.ceil(eps))
    pad = R + 2
    Hp, Wp = H + 2 * pad, W + 2 * pad

    def padded(v, fill):
        out = torch.full((n, Hp, Wp) + tuple(v.shape[3:]), fill, dtype=v.dtype, device=DEV)
        out[:, pad:pad + H, pad:pad + W] = v
        return out.reshape((n * Hp * Wp,) + tuple(v.shape[3:]))

    if rgba.requires_grad:
        u = torch.nn.functional.pad(rgba.double(), (0, 0, pad, pad, pad, pad)).reshape(-1, 4)
    else:
        u = padded(rgba.double(), 0.0)
    label = padded(labels, 2)
    g32 = padded(guide, 0.0)
    readable = label == 0
    rest = torch.nonzero(label == 1)[:, 0]
    frame_of = torch.div(rest, Hp * Wp, rounding_mode="floor")
    if phi is not None:
        phi = torch.nn.functional.pad(phi.double(), (pad, pad, pad, pad)).reshape(-1)
    square = [(a, b) for b in range(-R, R + 1) for a in range(-R, R + 1)]
    ball = [(a, b) for a, b in square if 0 < a * a + b * b <= float(np.float32(eps)) ** 2]
    sn = torch.tensor([a for a, _ in ball], device=DEV, dtype=torch.float32)
    sm = torch.tensor([b for _, b in ball], device=DEV, dtype=torch.float32)
    dist = (sn.double() ** 2 + sm.double() ** 2).sqrt()
    mu64 = mu_t.double() if mu_t is not None else float(np.float32(mu))
    coef = mu64 * mu64 / (2.0 * float(np.float32(eps)) ** 2)
    c64 = float(np.float32(c))
    tau = torch.tensor(1e-5, device=DEV, dtype=torch.float32)
    phase1 = torch.full((n,), bool(data_term), device=DEV)

    def average(at, unguided):
        """(value, ready without the data term) of pixels ``at`` against the present readable set"""
        gx, gy = g32[at, 0:1], g32[at, 1:2]
        if unguided:
            gx, gy = torch.zeros_like(gx), torch.zeros_like(gy)
        if ghost:
            a = (gx * gx + gy * gy).sqrt()
            ch = torch.where(a > 0, gx / a, torch.ones_like(a))
            sh = torch.where(a > 0, gy / a, torch.zeros_like(a))
            pos = [sn * ch - sm * sh, sn * sh + sm * ch]
            moved = None
            if phi is not None and not unguided:
                cp, sp = phi[at][:, None].cos(), phi[at][:, None].sin()
                moved = [torch.where(a > 0, d - d.detach(), torch.zeros_like(d))
                         for d in (sn * cp - sm * sp, sn * sp + sm * cp)]
            for i in range(2):
                near = pos[i].round()
                pos[i] = torch.where((pos[i] - near).abs() <= tau, near, pos[i])
        else:
            pos, moved = [sn.expand(len(at), -1), sm.expand(len(at), -1)], None
        low = [p.floor() for p in pos]
        fr32 = [p - f for p, f in zip(pos, low)]
        fr = [f.double() for f in fr32]
        if moved is not None:
            fr = [torch.where(f32 > 0, f + d, f) for f32, f, d in zip(fr32, fr, moved)]
        hx, hy = fr32[0] > 0, fr32[1] > 0
        base = at[:, None] + low[1].long() * Wp + low[0].long()
        ok = readable[base] & (~hx | readable[base + 1]) & (~hy | readable[base + Wp])
        ok = ok & (~(hx & hy) | readable[base + Wp + 1])
        gx64, gy64 = gx.double(), gy.double()
        if ghost:
            t = coef * (gx64 * gx64 + gy64 * gy64) * sm.double() ** 2
        else:
            t = coef * (gx64 * sm.double() - gy64 * sn.double()) ** 2
        if smart and not unguided:
            w = torch.exp(-t.detach()) / dist
            ready = (w * ok).sum(1) / w.sum(1) > c64
        else:
            ready = ok.any(1)
        least = torch.where(ok, t, torch.full_like(t, math.inf)).amin(1, keepdim=True).detach()
        w = torch.where(ok, torch.exp(-(t - torch.where(least.isinf(), torch.zeros_like(least), least))) / dist,
                        torch.zeros_like(t))
        w = w / w.sum(1, keepdim=True).clamp_min(1e-300)
        value = 0.0
        for dx, dy, lx in ((0, 0, (1 - fr[0]) * (1 - fr[1])), (1, 0, fr[0] * (1 - fr[1])),
                           (0, 1, (1 - fr[0]) * fr[1]), (1, 1, fr[0] * fr[1])):
            used = ok & (hx if dx else True) & (hy if dy else True)
            tap = torch.where(used, base + dx + dy * Wp, at[:, None])
            value = value + (torch.where(used, w * lx, torch.zeros_like(w))[..., None] * u[tap]).sum(1)
        return value, ready

    def evaluate(at, unguided=False):
        parts = [average(p, unguided) for p in torch.split(at, max(1, (1 << 23) // len(ball)))]
        return torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts])

    neighbours = torch.tensor([dy * Wp + dx for dy in (-1, 0, 1) for dx in (-1, 0, 1) if dx or dy], device=DEV)
    for _ in range(most_steps):
        on_front = torch.zeros(len(rest), dtype=torch.bool, device=DEV)
        for d in neighbours.tolist():
            on_front |= readable[rest + d]
        at, of = rest[on_front], frame_of[on_front]
        if not len(at):
            break
        value, can = evaluate(at)
        guided = (g32[at] != 0).any(1)
        left = torch.zeros(n, dtype=torch.bool, device=DEV)
        left[frame_of[(g32[rest] != 0).any(1)]] = True
        phase1 &= left
        ready = can & (~phase1[of] | guided)
        some = torch.zeros(n, dtype=torch.bool, device=DEV)
        some[of[ready]] = True
        phase1 &= some  # frames that fill nothing under the data term go on without it, at this step
        ready = can & (~phase1[of] | guided)
        some[of[ready]] = True
        stuck = ~some[of]
        if bool(stuck.any()):  # the stall rule: these fronts are filled as if unguided
            v, r = evaluate(at[stuck], True)
            value = value.index_put((torch.nonzero(stuck)[:, 0],), v)
            ready = ready.clone()
            ready[stuck] = r
            some[of[ready]] = True
        u = u.index_put((at[ready],), value[ready])
        readable[at[ready]] = True
        keep = ~readable[rest] & some[frame_of]
        rest, frame_of = rest[keep], frame_of[keep]
        if not len(rest):
            break
    else:
        return None
    return u.reshape(n, Hp, Wp, 4)[:, pad:pad + H, pad:pad + W]


def exact(case, seed):
    kind = case["kind"]
    if kind == "detect":  # a list whose length hangs on thresholds: no value in 64 bits to set beside it
        return None
    rgba, labels, splines = _inputs(case, seed)
    args = dict(eps=case["eps"], mu=case["mu"], c=case["c"], ghost=case["ghost"], smart=case["smart"],
                data_term=case["data"])
    if kind == "guidance":
        return {"guide": [_nearest_field(lab, *sp) for lab, sp in zip(labels, splines)]}
    if kind == "train":
        mag, phi, up = _angles(case, seed, splines, labels)
        lab = torch.stack(labels)
        rgba = torch.stack(rgba).requires_grad_()
        phi64, m = phi.double().requires_grad_(), mag.double()
        mu = torch.tensor(case["mu"], device=DEV, dtype=torch.float64, requires_grad=True)
        guide = torch.stack([m * phi64.cos(), m * phi64.sin()], -1).float().detach()
        out = _fill64(rgba, lab, guide, phi=phi64, mu_t=mu, **args)
        if out is None:
            return None
        g = torch.autograd.grad(out, [rgba, phi64, mu], grad_outputs=up.double())
        return {"out": out.detach(), "grad_rgba": g[0], "grad_phi": g[1], "grad_mu": g[2]}
    lab = torch.stack(labels)
    if kind == "fill":
        guide = _guide(case, seed, labels[0], splines[0])[None]
    else:
        guide = torch.stack([_nearest_field(v, *sp).float() for v, sp in zip(labels, splines)])
    out = _fill64(torch.stack(rgba), lab, guide, **args)
    if out is None:
        return None
    if kind == "fill":
        return {"rgba": out[0], "shell": None}
    if kind == "movie":
        return {"rgba": list(out), "shell": [None] * case["n"]}
    return {"rgba": [o.cpu().numpy() for o in out], "shell": [None] * case["n"], "filled": None}
