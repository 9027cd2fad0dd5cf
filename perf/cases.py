"""What this library is measured on: the calls its users make, with the inputs they make
them on.  `listed()` holds the fixed cases, `draw()` more of the same ranges, `prepare()`
what a caller has in hand, `run()` one pass through the public entry points, `work()` what
a pass cannot do without and `exact()` the same outputs in 64 bits, from plain torch.

Inputs are procedural: a scene of gratings and soft-edged patches (half of them filled
with detail fine enough to alias on the Bayer grid), seen through hand tremor and a small
rotation, one patch moving on its own, sampled as 12-bit RGGB with shot and read noise.
Merges that take a given motion field get the frames' true displacement at the tile
centres with an alignment error of a few hundredths of a pixel.
"""
import math
import random

import numpy as np
import torch
import torch.nn.functional as F

import paper_1905_03277_gb300 as hm

WL = 4095


def listed():
    return [
        # a viewfinder preview, or one thumbnail of a gallery: latency is all of it
        dict(name="preview_256_1x", op="align_merge", n=8, h=256, w=256, num=1, den=1, ref=0, gain=0.5, read=2.0,
             light=1.0, pad=0),
        # the ordinary capture: 12 MP, 8 frames, merged at its own size
        dict(name="photo_12mp_1x", op="align_merge", n=8, h=3024, w=4032, num=1, den=1, ref=0, gain=4.0, read=6.0,
             light=1.0, pad=0),
        # super-resolution at full size: 15 frames to 48 MP
        dict(name="superres_12mp_2x", op="align_merge", n=15, h=3024, w=4032, num=2, den=1, ref=0, gain=1.0, read=3.0,
             light=1.0, pad=0),
        # alignment by itself (stabilisation, frame selection): odd tile counts, padded sensor rows, a base frame
        # from the middle of the burst
        dict(name="align_5mp_padded", op="align", n=10, h=1942, w=2590, num=1, den=1, ref=3, gain=2.0, read=4.0,
             light=1.0, pad=34),
        # a crop zoomed in by 1.5 with motion the caller already has
        dict(name="zoom_3mp_1.5x", op="merge", n=6, h=1538, w=2050, num=3, den=2, ref=2, gain=2.0, read=4.0, light=1.0,
             pad=0),
        # night capture: every parameter and the tile size chosen from the base frame's signal-to-noise ratio
        dict(name="night_3mp_auto", op="auto", n=13, h=1512, w=2016, num=1, den=1, ref=0, gain=1.2, read=3.0, light=0.1,
             pad=0),
        # a long burst merged in bounded memory
        dict(name="long_burst_2mp", op="chunked", n=24, h=1224, w=1632, num=1, den=1, ref=0, gain=3.0, read=5.0,
             light=1.0, pad=0, chunk=4),
        # a capture merged with the simulated noise statistics of its own sensor gain and the rejection of
        # high-frequency artifacts
        dict(name="noise_table_2mp", op="noise", n=8, h=1080, w=1920, num=1, den=1, ref=0, gain=2.0, read=4.0, light=1.0,
             pad=0),
        # one training step of the parameter fit: forward, loss and adjoint
        dict(name="fit_step_1mp_1.5x", op="fit", n=8, h=1024, w=1024, num=3, den=2, ref=0, gain=1.0, read=3.0, light=1.0,
             pad=0),
        # the same on a training crop at 2x, where the small launches count
        dict(name="fit_crop_2x", op="fit", n=4, h=256, w=320, num=2, den=1, ref=1, gain=1.0, read=3.0, light=1.0, pad=0),
        # a ragged batch from a server's queue
        dict(name="batch_ragged", op="batch", gain=2.0, read=4.0, light=1.0,
             bursts="6x1224x1632:1/1:0 9x720x960:2/1:0 4x1538x2050:1/1:1 12x480x640:3/2:0 5x902x1606:3/2:2 8x612x816:1/1:0"),
    ]


def _even(v, lo=64):
    return max(lo, 2 * int(round(v / 2)))


def _size(rng, mp_lo, mp_hi):
    mp = math.exp(rng.uniform(math.log(mp_lo), math.log(mp_hi))) * 1e6
    a, b = rng.choice([(4, 3), (16, 9), (1, 1), (3, 4)])
    unit = math.sqrt(mp / (a * b))
    return _even(unit * b), _even(unit * a)


def draw(rng):
    op = rng.choice(["align_merge"] * 4 + ["align", "merge", "merge", "auto", "chunked", "noise", "fit", "fit", "batch"])
    gain = round(math.exp(rng.uniform(math.log(0.5), math.log(8.0))), 3)
    c = dict(op=op, gain=gain, read=round(2.0 + gain, 3), light=1.0)
    scales = [(1, 1), (3, 2), (2, 1)]
    if op == "batch":
        parts = []
        for _ in range(rng.randint(3, 8)):
            h, w = _size(rng, 0.1, 3.0)
            n = rng.randint(3, 10)
            num, den = rng.choice(scales)
            parts.append("%dx%dx%d:%d/%d:%d" % (n, h, w, num, den, rng.randrange(n)))
        return dict(c, bursts=" ".join(parts))
    top = {"align_merge": 12.2, "align": 12.2, "merge": 8.0, "auto": 6.0, "chunked": 3.0, "noise": 4.0, "fit": 1.0}[op]
    h, w = _size(rng, 0.06, top)
    n = rng.randint(3, 8) if op == "fit" else rng.randint(12, 32) if op == "chunked" else rng.randint(2, 15)
    num, den = rng.choice(scales)
    c.update(n=n, h=h, w=w, num=num, den=den, ref=rng.randrange(n), pad=rng.choice([0, 0, 2, 32]))
    if op == "align":
        c.update(num=1, den=1)
    if op in ("chunked", "fit"):
        c["pad"] = 0
    if op == "chunked":
        c.update(num=1, den=1, chunk=rng.choice([2, 4, 8]))
    if op == "fit" and (num, den) == (2, 1):  # no more output pixels than the listed step
        s = math.sqrt(min(1.0, 0.5e6 / (h * w)))
        c.update(h=_even(h * s), w=_even(w * s))
    if op == "auto":
        c.update(light=rng.choice([0.05, 0.1, 0.2, 1.0]))
    return c


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
class _Scene:
    """Value in [0.05, 0.95] of colour channel ch at base-frame positions."""

    def __init__(self, rng, h, w):
        self.base = [rng.uniform(0.3, 0.7) for _ in range(3)]
        self.low = [self._grating(rng, 40.0, 200.0, 0.08) for _ in range(3)]
        self.patches = []
        for _ in range(max(8, min(48, h * w // 60_000))):
            r = rng.uniform(0.03, 0.14) * min(h, w)
            self.patches.append((rng.uniform(0, w), rng.uniform(0, h), max(r, 6.0), max(r * rng.uniform(0.4, 1.0), 6.0),
                                 [rng.uniform(0.15, 0.85) for _ in range(3)],
                                 self._grating(rng, 1.5, 20.0, 0.25) if rng.random() < 0.5 else None))

    @staticmethod
    def _grating(rng, lo, hi, amp):
        t, per = rng.uniform(0, math.pi), rng.uniform(lo, hi)
        return (math.cos(t) / per, math.sin(t) / per, rng.uniform(0, 2 * math.pi),
                [amp * rng.uniform(0.3, 1.0) for _ in range(3)])

    @staticmethod
    def _colour(v, ch):
        return torch.tensor(v, dtype=torch.float32, device=ch.device)[ch]

    def __call__(self, x, y, ch):
        def wave(g, x, y, ch):
            return self._colour(g[3], ch) * torch.sin(2 * math.pi * (g[0] * x + g[1] * y) + g[2])

        out = self._colour(self.base, ch)
        for g in self.low:
            out = out + wave(g, x, y, ch)
        hh, ww = x.shape
        # plane coordinates of a patch's box: the positions run with the indices
        sx, sy = float(x[0, -1] - x[0, 0]) / max(1, ww - 1), float(y[-1, 0] - y[0, 0]) / max(1, hh - 1)
        ox, oy = float(x[0, 0]), float(y[0, 0])
        for cx, cy, rx, ry, col, g in self.patches:
            m = 24.0 + 0.02 * max(hh, ww)
            a, b = int((cx - rx - m - ox) / sx), int((cx + rx + m - ox) / sx) + 2
            c, d = int((cy - ry - m - oy) / sy), int((cy + ry + m - oy) / sy) + 2
            box = (slice(max(c, 0), max(min(d, hh), 0)), slice(max(a, 0), max(min(b, ww), 0)))
            px, py, pc = x[box], y[box], ch[box]
            if px.numel() == 0:
                continue
            inside = ((1.0 - torch.sqrt(((px - cx) / rx) ** 2 + ((py - cy) / ry) ** 2)) * min(rx, ry) + 0.5).clamp(0, 1)
            v = self._colour(col, pc)
            if g is not None:
                v = v + wave(g, px, py, pc)
            out[box] = out[box] * (1 - inside) + v * inside
        return out.clamp(0.05, 0.95)


def _tremor(rng, n, ref):
    """Per frame (shift x, shift y, rotation) against the base frame."""
    pos, out = [0.0, 0.0], []
    for _ in range(n):
        pos = [min(4.0, max(-4.0, p + rng.gauss(0, 1.2))) for p in pos]
        out.append((pos[0], pos[1], math.radians(rng.uniform(-0.05, 0.05))))
    b = out[ref]
    return [(x - b[0], y - b[1], r - b[2]) for x, y, r in out]


def _displacement(t, x, y, h, w):
    return t[0] - t[2] * (y - (h - 1) / 2), t[1] + t[2] * (x - (w - 1) / 2)


def _burst(rng, seed, n, h, w, ref, gain, read, light, pad, dev):
    """(frames uint16 [n, h, w] on rows of w + pad samples, scene, tremor)."""
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    sc, tr = _Scene(rng, h, w), _tremor(rng, n, ref)
    thing, speed = _Scene(rng, 200, 200), [rng.uniform(-25, 25) for _ in range(2)]
    ox, oy, half = rng.uniform(0.25, 0.7) * w, rng.uniform(0.25, 0.7) * h, 0.08 * min(h, w)
    full = torch.zeros((n, h, w + pad), dtype=torch.uint16, device=dev)
    x = torch.arange(w, device=dev, dtype=torch.float32)[None, :].expand(h, w)
    y = torch.arange(h, device=dev, dtype=torch.float32)[:, None].expand(h, w)
    ch = (torch.arange(w, device=dev) & 1)[None, :] + (torch.arange(h, device=dev) & 1)[:, None]
    for f in range(n):
        dx, dy = _displacement(tr[f], x, y, h, w)
        sx, sy = x - dx, y - dy
        v = sc(sx, sy, ch)
        ax, ay = ox + speed[0] * f / n, oy + speed[1] * f / n  # the moving patch, in the frame
        box = (slice(max(0, int(ay - half)), max(0, int(ay + half))), slice(max(0, int(ax - half)), max(0, int(ax + half))))
        if v[box].numel():
            v[box] = thing((sx[box] - ax + 100).contiguous(), (sy[box] - ay + 100).contiguous(), ch[box])
        v = v * (WL * light)
        v = v + torch.sqrt(gain * v + read * read) * torch.randn(v.shape, generator=gen, device=dev)
        full[f, :, :w] = v.round().clamp(0, WL).to(torch.int32).to(torch.uint16)
    return full[:, :, :w], sc, tr


def _motion(rng, seed, tr, n, h, w, tile, dev):
    """The tiles' true displacements, with the error of an alignment."""
    ty, tx = -(-h // tile), -(-w // tile)
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed + 77)
    cx = (torch.arange(tx, device=dev, dtype=torch.float32) * tile + (tile - 1) / 2)[None, :].expand(ty, tx)
    cy = (torch.arange(ty, device=dev, dtype=torch.float32) * tile + (tile - 1) / 2)[:, None].expand(ty, tx)
    mv = torch.empty((n, ty, tx, 2), device=dev)
    for f in range(n):
        mv[f, :, :, 0], mv[f, :, :, 1] = _displacement(tr[f], cx, cy, h, w)
    return mv + 0.04 * torch.randn(mv.shape, generator=gen, device=dev)


def _parse(case):
    out = []
    for part in case["bursts"].split():
        shape, scale, ref = part.split(":")
        out.append((tuple(int(v) for v in shape.split("x")), tuple(int(v) for v in scale.split("/")), int(ref)))
    return out


def _params(case):
    return hm.MergeParams(noise_a=case["gain"], noise_b=case["read"] ** 2)


def _inputs(case, seed, dev):
    """What the call is given, without anything of the library."""
    rng = random.Random(seed * 1000003 + 17)
    if case["op"] == "batch":
        return [_burst(rng, seed * 64 + k, *shape, ref, case["gain"], case["read"], case["light"], 0, dev)[0]
                for k, (shape, _, ref) in enumerate(_parse(case))]
    n, h, w, ref = case["n"], case["h"], case["w"], case["ref"]
    burst, sc, tr = _burst(rng, seed, n, h, w, ref, case["gain"], case["read"], case["light"], case["pad"], dev)
    motion = _motion(rng, seed, tr, n, h, w, 16, dev)
    motion[ref] = 0
    gt = None
    if case["op"] == "fit":
        ho, wo = h * case["num"] // case["den"], w * case["num"] // case["den"]
        s = case["den"] / case["num"]
        x = ((torch.arange(wo, device=dev, dtype=torch.float32) + 0.5) * s - 0.5)[None, :].expand(ho, wo)
        y = ((torch.arange(ho, device=dev, dtype=torch.float32) + 0.5) * s - 0.5)[:, None].expand(ho, wo)
        gt = torch.stack([sc(x, y, torch.full((ho, wo), k, device=dev, dtype=torch.int64)) for k in range(3)]) * WL
    return burst, motion, gt


def prepare(case, seed):
    dev = torch.device("cuda")
    op = case["op"]
    p = _params(case)
    s = dict(case=case, p=p)
    if op == "batch":
        parts = _parse(case)
        s["bursts"] = _inputs(case, seed, dev)
        s["plan"] = hm.BatchPlan([b[0] for b in parts], p, [b[1] for b in parts], [b[2] for b in parts])
        s["plan"].set_mode(4)  # what the tuner settles on for such batches
        s["rgbs"] = s["plan"].outputs(dev)
        s["motions"] = [torch.empty((n,) + hm.n_tiles(h, w, 16) + (2,), device=dev) for (n, h, w), _, _ in parts]
        return s
    s["burst"], s["motion"], s["gt"] = _inputs(case, seed, dev)
    if op == "fit":
        s["values"] = [getattr(p, k) for k in hm.PARAM_NAMES]
        s["theta"] = torch.tensor(s["values"], dtype=torch.float32, device=dev, requires_grad=True)
        s["motion"].requires_grad_(True)
    return s


# ---------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------
def run(s):
    c = s["case"]
    op, p = c["op"], s["p"]
    if op == "batch":
        s["plan"].run(s["bursts"], s["rgbs"], s["motions"])
        return {"rgb": s["rgbs"], "motion": s["motions"]}
    burst, scale, ref = s["burst"], (c["num"], c["den"]), c["ref"]
    if op == "align_merge":
        rgb, motion = hm.align_merge(burst, p, scale, ref, with_motion=True)
        return {"rgb": rgb, "motion": motion}
    if op == "align":
        motion, vectors = hm.align(burst, ref, with_int=True)
        return {"motion": motion, "vectors": vectors}
    if op == "merge":
        return {"rgb": hm.merge(burst, s["motion"], p, scale, ref)}
    if op == "auto":
        mp, ap, snr = hm.auto_params(burst, c["gain"], c["read"] ** 2, ref)
        rgb, motion = hm.align_merge(burst, mp, scale, ref, ap, with_motion=True)
        return {"rgb": rgb, "motion": motion, "snr": snr}
    if op == "chunked":
        return {"rgb": hm.merge_chunked(burst, s["motion"], p, scale, ref, chunk_frames=c["chunk"])}
    if op == "noise":
        table = hm.noise_table(p.noise_a, p.noise_b, device=burst.device)
        rgb = hm.merge_ex(burst, s["motion"], p, scale, ref, noise_table=table, hf_loss=0.03)
        return {"rgb": rgb, "table": table}
    rgb = hm.MergeFn.apply(s["theta"], s["motion"], burst, p, scale, ref, s["values"])
    loss = ((rgb - s["gt"]) ** 2).mean()
    g_theta, g_motion = torch.autograd.grad(loss, (s["theta"], s["motion"]))
    return {"rgb": rgb.detach(), "loss": loss.detach(), "g_theta": g_theta, "g_motion": g_motion}


def work(case):
    """Bytes: the frames (and a given motion) in, the outputs out.  Operations of the
    method itself: per output pixel and frame 9 window samples' weights and sums and the
    interpolated kernel (about 240), per half-res pixel and frame its kernel, statistics
    and robustness (130), per half-res pixel and frame of an alignment the searches'
    squared differences and three refinements (150), and four times the accumulation for
    its adjoint."""
    if case["op"] == "batch":
        parts = [(n, h, w, num, den) for (n, h, w), (num, den), _ in _parse(case)]
    else:
        parts = [(case["n"], case["h"], case["w"], case["num"], case["den"])]
    op = case["op"]
    nbytes = flops = 0
    for n, h, w, num, den in parts:
        px, half, tiles = (h * num // den) * (w * num // den), h * w // 4, -(-h // 16) * -(-w // 16)
        nbytes += 2 * n * h * w + 8 * n * tiles
        if op == "align":
            nbytes += 8 * n * tiles
            flops += 150 * n * half
            continue
        nbytes += 12 * px
        flops += 240 * px * n + 130 * half * n
        if op in ("align_merge", "auto", "batch"):
            flops += 150 * n * half
        if op == "fit":
            nbytes += 12 * px + 8 * n * tiles
            flops += 960 * px * n
        if op == "noise":
            flops += 129 * 4096 * 54 * 100
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------------------
# the method in 64 bits
# ---------------------------------------------------------------------------------------
def _f32(v):
    return float(np.float32(v))


def _quads(frame):
    r = frame.to(torch.int32)
    return r[0::2, 0::2], r[0::2, 1::2], r[1::2, 0::2], r[1::2, 1::2]


def _edge(t, k=1):
    return F.pad(t[None, None].double(), (k, k, k, k), mode="replicate")[0, 0]


def _box3(t):
    p = _edge(t)
    hh, wh = t.shape
    return sum(p[j:j + hh, i:i + wh] for j in range(3) for i in range(3))


def _omega64(frame, q):
    """Kernel covariance entries (xx, xy, yy) per half-res pixel (Eq. 3-4, supplement S.1)."""
    r, g1, g2, b = _quads(frame)
    p = _edge(r + g1 + g2 + b)
    hh, wh = r.shape
    L = [[p[j:j + hh, i:i + wh] for i in range(3)] for j in range(3)]
    ta = tb = tc = 0
    for j in range(2):
        for i in range(2):
            gx = L[j][i + 1] - L[j][i] + L[j + 1][i + 1] - L[j + 1][i]
            gy = L[j + 1][i] - L[j][i] + L[j + 1][i + 1] - L[j][i + 1]
            ta, tb, tc = ta + gx * gx, tb + gx * gy, tc + gy * gy
    tr, amc, b2 = ta + tc, ta - tc, 2 * tb
    rad = torch.sqrt(amc * amc + b2 * b2)
    tie = rad == 0
    safe = torch.where(tie, 1.0, rad)
    cs, sn = torch.where(tie, 1.0, amc / safe), torch.where(tie, 0.0, b2 / safe)
    A = torch.where(tr == 0, 1.0, 1 + torch.sqrt(rad / torch.where(tr == 0, 1.0, tr)))
    rl = torch.sqrt(0.5 * (tr + rad)) / (16 * WL)
    D = (1 - rl / q["d_tr"] + q["d_th"]).clamp(0, 1)
    kd = q["k_detail"] * q["k_denoise"]
    al = ((1 - D) * q["k_detail"] * q["k_stretch"] * A + D * kd) ** 2
    ac = ((1 - D) * q["k_detail"] / (q["k_shrink"] * A) + D * kd) ** 2
    exx, exy, eyy = 0.5 * (1 + cs), 0.5 * sn, 0.5 * (1 - cs)
    return ac * exx + al * (1 - exx), (ac - al) * exy, ac * eyy + al * (1 - eyy)


def _span(mv, m_th):
    """Per tile: the motion span of its 3x3 tile neighbourhood exceeds m_th (Eq. 7)."""
    v = mv.permute(2, 0, 1)[None]
    hi, lo = F.max_pool2d(v, 3, 1, 1)[0], -F.max_pool2d(-v, 3, 1, 1)[0]
    d = hi - lo
    return torch.sqrt(d[0] * d[0] + d[1] * d[1]) > m_th


def _merge64(burst, motion, q, scale, ref, tile=16, table=None, hf=0.0):
    """Sec. 5 (Eq. 1-9, S.1).  q: the parameters (numbers or 0-d tensors)."""
    dev = burst.device
    n, h, w = burst.shape
    hh, wh = h // 2, w // 2
    num, den = scale
    ho, wo = h * num // den, w * num // den
    ty, tx = motion.shape[1:3]

    def guide(f):
        r, g1, g2, b = _quads(burst[f])
        return [r.double(), 0.5 * (g1 + g2).double(), b.double()]

    gb = guide(ref)
    mus = [_box3(c) / 9 for c in gb]
    sig, dmd = 0, []
    for k, (c, mu) in enumerate(zip(gb, mus)):
        half = 0.5 if k == 1 else 1.0
        ms = (_box3(c * c) / 9 - mu * mu).clamp(min=0)
        x = mu.clamp(0, WL)
        if table is None:
            md = ((q["noise_a"] * x + q["noise_b"]) * half).clamp(min=0)
            dmd.append(md * (2 / 9))
        else:
            t = x * (128 / WL)
            i = t.long().clamp(max=127)
            col = 1 if k == 1 else 0
            lerp = lambda j: table[i, j] + (t - i) * (table[i + 1, j] - table[i, j])  # noqa: E731
            md = lerp(col)
            dmd.append(lerp(2 + col))
        sig = sig + torch.maximum(ms, md)
    sig = sig.clamp(min=1e-12 * WL * WL)
    flag = None
    if hf > 0:
        keep = sum(_box3(m * m) / 9 - (_box3(m) / 9) ** 2 for m in mus)
        have = sum(_box3(c * c) / 9 - m * m for c, m in zip(gb, mus))
        flag = (have > 1e-9) & (keep < hf * have)
    tyh = (torch.arange(hh, device=dev) // (tile // 2)).clamp(max=ty - 1)[:, None]
    txh = (torch.arange(wh, device=dev) // (tile // 2)).clamp(max=tx - 1)[None, :]

    def rhat(f):
        mv = motion[f][tyh, txh] * 0.5
        fl = torch.floor(mv.detach())
        fx, fy = mv[..., 0] - fl[..., 0], mv[..., 1] - fl[..., 1]
        ix = torch.arange(wh, device=dev)[None, :] + fl[..., 0].long()
        iy = torch.arange(hh, device=dev)[:, None] + fl[..., 1].long()
        x0, x1, y0, y1 = ix.clamp(0, wh - 1), (ix + 1).clamp(0, wh - 1), iy.clamp(0, hh - 1), (iy + 1).clamp(0, hh - 1)
        dd = 0
        for c, mu, d2 in zip(guide(f), mus, dmd):
            m = _box3(c) / 9
            al = (1 - fy) * ((1 - fx) * m[y0, x0] + fx * m[y0, x1]) + fy * ((1 - fx) * m[y1, x0] + fx * m[y1, x1])
            e = mu - al
            e2 = e * e
            dd = dd + (e * e2 / (e2 + d2).clamp(min=1e-300)) ** 2
        span = _span(motion[f].detach(), q["m_th"])
        s = torch.where(span, torch.as_tensor(q["s1"], dtype=torch.float64, device=dev),
                        torch.as_tensor(q["s2"], dtype=torch.float64, device=dev))[tyh, txh]
        R = (s * torch.exp(-dd / sig) - q["t"]).clamp(0, 1)
        if flag is not None:
            R = torch.where(flag & span[tyh, txh], 0.0, R)
        return -F.max_pool2d(-R[None, None], 5, 1, 2)[0, 0]

    Q = 2 * num
    Px = (2 * den * torch.arange(wo, device=dev) + den - num)[None, :]
    Py = (2 * den * torch.arange(ho, device=dev) + den - num)[:, None]
    fdiv = lambda a, b: torch.div(a, b, rounding_mode="floor")  # noqa: E731
    tyi, txi = fdiv(Py, Q * tile).clamp(0, ty - 1), fdiv(Px, Q * tile).clamp(0, tx - 1)

    def cell(P, size):  # lower texel and fraction of a half-res sampling position P / 2Q
        c = fdiv(P, 2 * Q)
        return c.clamp(0, size - 1), (c + 1).clamp(0, size - 1), (P - c * 2 * Q).double() / (2 * Q)

    rx0, rx1, rfx = cell(Px - num, wh)
    ry0, ry1, rfy = cell(Py - num, hh)
    nums, dens = [0, 0, 0], [0, 0, 0]
    for f in range(n):
        v = motion[f][tyi, txi] if f != ref else torch.zeros((1, 1, 2), dtype=torch.float64, device=dev)
        rh = 1.0
        if f != ref:
            R = rhat(f)
            rh = (1 - rfy) * ((1 - rfx) * R[ry0, rx0] + rfx * R[ry0, rx1]) + rfy * (
                (1 - rfx) * R[ry1, rx0] + rfx * R[ry1, rx1])
        FX, FY = torch.floor(Q * v[..., 0].detach()).long(), torch.floor(Q * v[..., 1].detach()).long()
        zx, zy = Q * v[..., 0] - FX, Q * v[..., 1] - FY
        kx, ky = fdiv(Px + num + FX, Q), fdiv(Py + num + FY, Q)
        ddx, ddy = ((kx * Q - Px - FX) - zx) / Q, ((ky * Q - Py - FY) - zy) / Q
        ox0, ox1, ax = cell(Px - num + FX, wh)
        oy0, oy1, ay = cell(Py - num + FY, hh)
        ax, ay = ax + zx / (2 * Q), ay + zy / (2 * Q)
        xx, xy, yy = ((1 - ay) * ((1 - ax) * o[oy0, ox0] + ax * o[oy0, ox1]) + ay * ((1 - ax) * o[oy1, ox0] + ax * o[oy1, ox1])
                      for o in _omega64(burst[f], q))
        det = xx * yy - xy * xy
        ixx, ixy, iyy = yy / det, -xy / det, xx / det
        fr = burst[f].to(torch.int32)
        for j in (-1, 0, 1):
            for i in (-1, 0, 1):
                qx, qy = (kx + i).expand(ho, wo), (ky + j).expand(ho, wo)
                ok = (qx >= 0) & (qx < w) & (qy >= 0) & (qy < h)
                ex, ey = ddx + i, ddy + j
                wgt = torch.exp(-0.5 * (ixx * ex * ex + 2 * ixy * ex * ey + iyy * ey * ey)) * rh * ok
                val = fr[qy.clamp(0, h - 1), qx.clamp(0, w - 1)]
                ch = (qx & 1) + (qy & 1)
                for k in range(3):
                    wk = torch.where(ch == k, wgt, 0.0)
                    nums[k], dens[k] = nums[k] + wk * val, dens[k] + wk
    return torch.stack([a / b for a, b in zip(nums, dens)])


def _align64(burst, ref, tile=16, radius=(1, 4, 4, 4), iters=3):
    """Sec. 3.2: (motion in raw px, float64; integer vectors)."""
    dev = burst.device
    n = burst.shape[0]
    T = tile // 2
    levels = [torch.stack([sum(_quads(f)) for f in burst])]
    for fct in (2, 4, 4):
        lh, lw = levels[-1].shape[1] // fct, levels[-1].shape[2] // fct
        if lh < 16 or lw < 16:
            break
        a = levels[-1][:, :lh * fct, :lw * fct].reshape(n, lh, fct, lw, fct)
        levels.append(torch.div(a.sum((2, 4)), fct * fct, rounding_mode="floor").int())

    def spread(t):  # per tile -> per pixel of the (padded) level
        return t.repeat_interleave(T, 0).repeat_interleave(T, 1)

    motion, vecs = [], []
    for f in range(n):
        vec = None
        for l in range(len(levels) - 1, -1, -1):
            img = levels[l]
            lh, lw = img.shape[1:]
            ty, tx = -(-lh // T), -(-lw // T)
            if f == ref:
                continue
            if vec is None:
                vec = torch.zeros((ty, tx, 2), dtype=torch.int64, device=dev)
            else:
                fct = 2 if l == 0 else 4
                pty, ptx = vec.shape[:2]
                at = lambda k, m: ((torch.arange(k, device=dev) * T + T // 2) // fct // T).clamp(max=m - 1)  # noqa: E731
                vec = vec[at(ty, pty)[:, None], at(tx, ptx)[None, :]] * fct
            Y, X = torch.arange(ty * T, device=dev)[:, None], torch.arange(tx * T, device=dev)[None, :]
            base = img[ref][Y.clamp(max=lh - 1), X.clamp(max=lw - 1)]
            px, py = spread(vec[..., 0]), spread(vec[..., 1])
            best = torch.full((ty, tx), 2**62, dtype=torch.int64, device=dev)
            r = radius[l]
            for dy in range(-r, r + 1):
                for dx in range(-r, r + 1):
                    d = (base - img[f][(Y + py + dy).clamp(0, lh - 1), (X + px + dx).clamp(0, lw - 1)]).long()
                    ssd = (d * d).reshape(ty, T, tx, T).sum((1, 3))
                    best = torch.minimum(best, (ssd << 12) + ((abs(dx) + abs(dy)) << 8) + ((dy + 7) << 4) + dx + 7)
            vec = vec + torch.stack([(best & 15) - 7, ((best >> 4) & 15) - 7], -1)
        lh, lw = levels[0].shape[1:]
        ty, tx = -(-lh // T), -(-lw // T)
        if f == ref:
            vecs.append(torch.zeros((ty, tx, 2), dtype=torch.int64, device=dev))
            motion.append(torch.zeros((ty, tx, 2), dtype=torch.float64, device=dev))
            continue
        y, x = torch.arange(ty * T, device=dev).clamp(max=lh - 1)[:, None], torch.arange(tx * T, device=dev).clamp(max=lw - 1)[None, :]
        R, A = levels[0][ref].double(), levels[0][f].double()
        gx = (R[y, (x + 1).clamp(max=lw - 1)] - R[y, (x - 1).clamp(min=0)]) / 8
        gy = (R[(y + 1).clamp(max=lh - 1), x] - R[(y - 1).clamp(min=0), x]) / 8
        tsum = lambda t: t.reshape(ty, T, tx, T).sum((1, 3))  # noqa: E731
        hxx, hxy, hyy = tsum(gx * gx), tsum(gx * gy), tsum(gy * gy)
        det, tr = hxx * hyy - hxy * hxy, hxx + hyy
        skip = (tr == 0) | (1e9 * det <= tr * tr)
        inv = torch.where(skip, 0.0, 1 / torch.where(skip, 1.0, det))
        dx = torch.zeros((ty, tx), dtype=torch.float64, device=dev)
        dy = torch.zeros_like(dx)
        for _ in range(iters):
            fx, fy = torch.floor(dx), torch.floor(dy)
            ax, ay = spread(dx - fx), spread(dy - fy)
            ix, iy = x + spread(vec[..., 0] + fx.long()), y + spread(vec[..., 1] + fy.long())
            x0, x1, y0, y1 = ix.clamp(0, lw - 1), (ix + 1).clamp(0, lw - 1), iy.clamp(0, lh - 1), (iy + 1).clamp(0, lh - 1)
            v = (1 - ay) * ((1 - ax) * A[y0, x0] + ax * A[y0, x1]) + ay * ((1 - ax) * A[y1, x0] + ax * A[y1, x1])
            e = (v - R[y, x]) / 4
            bx, by = tsum(gx * e), tsum(gy * e)
            dx = (dx - (hyy * bx - hxy * by) * inv).clamp(-1, 1)
            dy = (dy - (hxx * by - hxy * bx) * inv).clamp(-1, 1)
        vecs.append(vec)
        motion.append(2 * (vec.double() + torch.stack([dx, dy], -1)))
    return torch.stack(motion), torch.stack(vecs)


def _table64(a, b, dev):
    """The Monte-Carlo noise statistics: 129 levels x 4096 trials of two 3x3 patches, with
    Philox-4x32-10 (Salmon et al. 2011) uniforms."""
    M = 0xFFFFFFFF
    out = []
    trial = torch.arange(4096, device=dev)[:, None]
    j = torch.arange(54, device=dev)[None, :]

    def mul(c, x):  # high and low words of the 32 x 32 bit product
        lo = c * (x & 0xFFFF)
        hi = c * (x >> 16) + (lo >> 16)
        return hi >> 16, ((hi & 0xFFFF) << 16) | (lo & 0xFFFF)

    for level in range(129):
        x = level * WL / 128
        sigma = math.sqrt(_f32(a) * x + _f32(b))
        total = torch.zeros((4096, 54), dtype=torch.int64, device=dev)
        for blk in range(3):
            c0, c1 = (3 * j + blk).expand(4096, 54), trial.expand(4096, 54)
            c2, c3 = torch.full_like(c0, level), torch.zeros_like(c0)
            k0, k1 = 0x19050327, 0x5EED0001
            for r in range(10):
                if r:
                    k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
                h0, l0 = mul(0xD2511F53, c0)
                h1, l1 = mul(0xCD9E8D57, c2)
                c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
            total += c0 + c1 + c2 + c3
        z = (total.double() + 6) / 4294967296.0 - 6
        v = torch.floor(x + sigma * z + 0.5).clamp(0, WL).reshape(4096, 2, 27)
        row = []
        rb, gr = v[:, :, :9], 0.5 * (v[:, :, 9::2] + v[:, :, 10::2])
        for t in (rb, gr):
            row.append(((t[:, 0] - t[:, 0].mean(1, keepdim=True)) ** 2).mean())
        for t in (rb, gr):
            row.append(((t[:, 0].mean(1) - t[:, 1].mean(1)) ** 2).mean())
        out.append(torch.stack(row))
    return torch.stack(out)


def _snr_params(burst, ref, a, b):
    """Supplement, "Noise-dependent Tuning": (parameters, tile, snr)."""
    mean = float(burst[ref].to(torch.int32).double().sum()) / burst[ref].numel()
    snr = mean / math.sqrt(_f32(a) * mean + _f32(b))
    t = min(max((snr - 6) / 24, 0.0), 1.0)
    lerp = lambda lo, hi: _f32((1 - t) * lo + t * hi)  # noqa: E731
    q = _numbers(hm.MergeParams(lerp(0.33, 0.25), lerp(5.0, 3.0), lerp(0.010, 0.001), lerp(0.020, 0.006), 4.0, 2.0, 0.12, 12.0,
                                2.0, 0.8, a, b))
    return q, 64 if snr < 10 else 32 if snr < 14 else 16, snr


def _numbers(p):
    return {k: _f32(v) for k, v in p.__dict__.items() if k != "tile"}


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    op, q = case["op"], _numbers(_params(case))
    got = _inputs(case, seed, dev)
    if op == "batch":
        rgbs, motions = [], []
        for burst, (_, scale, ref) in zip(got, _parse(case)):
            m, _ = _align64(burst, ref)
            motions.append(m)
            rgbs.append(_merge64(burst, m.float().double(), q, scale, ref))
        return {"rgb": rgbs, "motion": motions}
    burst, motion, gt = got
    scale, ref = (case["num"], case["den"]), case["ref"]
    if op == "align_merge":
        m, _ = _align64(burst, ref)
        return {"rgb": _merge64(burst, m.float().double(), q, scale, ref), "motion": m}
    if op == "align":
        m, v = _align64(burst, ref)
        return {"motion": m, "vectors": v.int()}
    if op in ("merge", "chunked"):
        return {"rgb": _merge64(burst, motion.double(), q, scale, ref)}
    if op == "auto":
        q, tile, snr = _snr_params(burst, ref, case["gain"], case["read"] ** 2)
        m, _ = _align64(burst, ref, tile)
        return {"rgb": _merge64(burst, m.float().double(), q, scale, ref, tile), "motion": m, "snr": snr}
    if op == "noise":
        table = _table64(q["noise_a"], q["noise_b"], dev)
        return {"rgb": _merge64(burst, motion.double(), q, scale, ref, 16, table.float().double(), 0.03), "table": table}
    names = hm.PARAM_NAMES
    theta = torch.tensor([q[k] for k in names], dtype=torch.float64, device=dev, requires_grad=True)
    m = motion.double().requires_grad_(True)
    rgb = _merge64(burst, m, dict(q, **dict(zip(names, theta.unbind()))), scale, ref)
    loss = ((rgb - gt.double()) ** 2).mean()
    g_theta, g_motion = torch.autograd.grad(loss, (theta, m))
    return {"rgb": rgb.detach(), "loss": loss.detach(), "g_theta": g_theta, "g_motion": g_motion}
