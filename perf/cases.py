"""Performance cases of the library: the calls a user makes, over the range of sizes, types and options they are made with.

Every case runs public entry points only (`Engine`, `stage_*`, `refine`).  Inputs are seeded synthetic particle images,
rendered on the GPU: uniform particle positions, Gaussian particles, a smooth flow (uniform motion, a shear layer, a
Lamb-Oseen vortex), out-of-plane loss and sensor noise.  `exact` restates each path in 64 bits with plain torch.
"""
import math

import torch
import torch.nn.functional as F

import paper_2504_17987_gb300 as rp
from paper_2504_17987_gb300 import binding

DEV = "cuda"


# ------------------------------------------------------------------ the cases --

def _process(name, width, height, bits, windows, radii, levels, pairs, precision="fp32", deform="b", pred=False,
             host=False):
    return {"name": name, "do": "process", "width": width, "height": height, "bits": bits, "windows": windows,
            "radii": radii, "levels": levels, "pairs": pairs, "precision": precision, "deform": deform, "pred": pred,
            "host": host}


def listed():
    return [
        # one small frame pair, the plain single-pass method: the smallest call, launches and latency
        _process("pair_256_r8", 256, 256, 8, "32", "8", 0, 1),
        # a live camera: one 12-bit 1 MP pair through the whole coarse-to-fine schedule
        _process("pair_1mp", 1024, 1024, 12, "64-32-16", "4-4-4", 2, 1),
        # offline processing of a recording: the same schedule, the largest batch a call takes
        _process("batch_1mp", 1024, 1024, 12, "64-32-16", "4-4-4", 2, 64),
        # the paper's operating point (16 px windows, +-1 around the predictor) on a recording
        _process("batch_1mp_16px", 1024, 1024, 12, "32-16", "4-1", 2, 32),
        # large frames, large displacements: 8 MP, 48 and 24 px windows, +-6
        _process("batch_8mp_r6", 3840, 2160, 8, "48-24", "6-6", 2, 4),
        # the 16-bit correlation on the 1 MP schedule
        _process("batch_1mp_bf16", 1024, 1024, 12, "64-32-16", "4-4-4", 2, 16, precision="bf16"),
        # serving: pinned camera frames, the previous field as the predictor, 16 px windows, 16-bit correlation
        _process("stream_host_bf16", 2048, 2048, 8, "16", "4", 0, 4, precision="bf16", pred=True, host=True),
        # a sensor region of odd size, both frames warped by half the predictor (central differences)
        _process("central_odd", 1391, 1037, 12, "32-16", "4-2", 1, 3, deform="central"),
        # differentiation: the score of a field and its gradient, 32 px windows at 75 % overlap
        {"name": "score_grad_1mp", "do": "grad", "width": 1024, "height": 1024, "bits": 8, "window": 32, "overlap": 0.75},
        # gradient refinement of a field, five steps
        {"name": "refine_1mp", "do": "refine", "width": 1024, "height": 1024, "bits": 8, "window": 32, "overlap": 0.75,
         "steps": 5},
        # pre-processing of a 12-bit pair before the flow estimate: high-pass and CLAHE
        {"name": "preprocess_1mp", "do": "preprocess", "width": 1024, "height": 1024, "bits": 12, "radius": 7, "tiles": 8,
         "clip": 200},
        # a schedule composed from the stage calls on an odd frame: pyramid level, correlation, outlier test,
        # interpolation onto the next grid, smoothing in time, vorticity
        {"name": "stages_odd", "do": "stages", "width": 1237, "height": 909, "bits": 8, "window": 24, "step": 12,
         "radius": 3},
    ]


SCHEDULES = [  # windows, radii, pyramid levels, frame-pair predictor, central warp allowed
    ("32", "8", 0, False), ("64-32-16", "4-4-4", 2, False), ("32-16", "4-1", 2, False), ("48-24", "6-6", 2, False),
    ("16", "4", 0, True), ("32-16", "4-2", 1, False), ("32-16", "4-0", 1, False), ("32", "4", 0, False),
]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same calls at other sizes (odd ones among them), types and options."""
    top = max(work(c)["flops"] for c in listed())
    while True:
        W, H = _log(rng, 256, 3840), _log(rng, 256, 2160)
        if rng.random() < 0.5:
            W, H = W // 16 * 16, H // 16 * 16
        bits = rng.choice([8, 12])
        do = rng.choice(["process"] * 7 + ["grad", "refine", "preprocess", "stages", "stages"])
        if do == "process":
            win, rad, lv, pred = rng.choice(SCHEDULES)
            c = _process("", W, H, bits, win, rad, lv, _log(rng, 1, 64),
                         precision=rng.choice(["fp32", "fp32", "fp32", "bf16", "fp16"]),
                         deform="central" if rng.random() < 0.2 else "b", pred=pred, host=rng.random() < 0.25)
            w0, r0 = int(win.split("-")[0]), int(rad.split("-")[0])
            if min(W, H) >> lv < w0 + 2 * (r0 + 1):
                continue
            if W * H * c["pairs"] > 70e6:
                continue
        elif do in ("grad", "refine"):
            c = {"do": do, "width": W, "height": H, "bits": bits, "window": rng.choice([16, 32]),
                 "overlap": rng.choice([0.5, 0.75])}
            if do == "refine":
                c["steps"] = rng.choice([3, 5])
            if W * H > 2.2e6:
                continue
        elif do == "preprocess":
            c = {"do": do, "width": W, "height": H, "bits": bits, "radius": rng.choice([0, 5, 7, 15]),
                 "tiles": rng.choice([4, 8, 16]), "clip": rng.choice([0, 200, 300])}
        else:
            w = rng.choice([16, 24, 32, 48])
            c = {"do": do, "width": W, "height": H, "bits": bits, "window": w,
                 "step": w // rng.choice([2, 4]), "radius": rng.choice([1, 2, 3, 4, 6, 8])}
        if work(c)["flops"] <= top:
            c.pop("name", None)
            return c


def _ints(text):
    return [int(t) for t in str(text).split("-")]


def _grid(W, H, w, s):
    return (W - w) // s + 1, (H - w) // s + 1


def work(case):
    """Bytes: each frame and field read or written once; flops: one multiply-add per pixel and shift of a search."""
    W, H, bpp = case["width"], case["height"], 1 if case["bits"] == 8 else 2
    px = W * H
    if case["do"] == "process":
        n, ws, rs = case["pairs"], _ints(case["windows"]), _ints(case["radii"])
        nx, ny = _grid(W, H, ws[-1], ws[-1] // 2)
        flops = sum(2 * (2 * r + 1) ** 2 * px for r in rs)
        flops += sum(2 * (2 * rs[0] + 1) ** 2 * (px >> (2 * lv)) for lv in range(1, case["levels"] + 1))
        return {"bytes": n * (2 * px * bpp + nx * ny * (13 + (8 if case["pred"] else 0))), "flops": n * flops}
    if case["do"] in ("grad", "refine"):
        nx, ny = _grid(W, H, case["window"], int(case["window"] * (1 - case["overlap"])))
        # warp 12, moments 6, adjoint 8 operations per pixel and evaluation
        one = {"bytes": 2 * px * bpp + 16 * nx * ny, "flops": 26 * px}
        k = 1 if case["do"] == "grad" else 2 * case["steps"] + 1
        return {"bytes": one["bytes"] * (1 if k == 1 else case["steps"] + 1), "flops": one["flops"] * k}
    if case["do"] == "preprocess":
        return {"bytes": 2 * px * (bpp + 4), "flops": 2 * 20 * px}
    nx, ny = _grid(W, H, case["window"], case["step"])
    dnx, dny = _grid(W, H, 16, 8)
    return {"bytes": 2 * px * bpp + px * bpp + px + nx * ny * (8 + 12 + 8 + 9 + 8) + dnx * dny * (8 + 12 + 4),
            "flops": 2 * (2 * case["radius"] + 1) ** 2 * px + 20 * px}


# -------------------------------------------------------------------- inputs --

def _flow(gen, W, H, large):
    """Parameters of a smooth flow: uniform motion, a shear layer, a Lamb-Oseen vortex."""
    r = torch.rand(8, generator=gen, dtype=torch.float64).tolist()
    return {"U": (12.0 if large else 3.3) * (0.8 + 0.4 * r[0]), "V": -1.7 + 2.0 * r[1],
            "shear": (6.0 if large else 1.0, (0.3 + 0.2 * r[2]) * H, 10.0),
            "vortex": ((0.3 + 0.4 * r[3]) * W, (0.5 + 0.3 * r[4]) * H, 200.0 if r[5] < 0.5 else -200.0, 20.0)}


def _velocity(f, x, y):
    dU, y0, delta = f["shear"]
    xc, yc, gamma, rc = f["vortex"]
    dx, dy = x - xc, y - yc
    r2 = dx * dx + dy * dy + 1e-9
    k = gamma / (2 * math.pi) * -torch.expm1(-r2 / (rc * rc)) / r2
    return f["U"] + 0.5 * dU * torch.tanh((y - y0) / delta) - k * dy, f["V"] + k * dx


def _splat(x, y, dp, amp, W, H):
    """Gaussian particles integrated over each pixel, summed in fixed point (the sum does not depend on its order)."""
    half = 4
    k = torch.arange(-half, half + 1, device=x.device)
    ix, iy = torch.floor(x + 0.5).long(), torch.floor(y + 0.5).long()
    a = (8.0 ** 0.5) / dp[:, None]
    img = torch.zeros(H * W, dtype=torch.int32, device=x.device)

    def side(i, p):
        e = (i[:, None] + k[None, :]).double() - p[:, None]
        return (torch.erf(a * (e + 0.5)) - torch.erf(a * (e - 0.5))) / (2 * a)

    gx, gy = side(ix, x), side(iy, y)
    val = torch.round(256.0 * math.pi * amp[:, None, None] * gy[:, :, None] * gx[:, None, :]).int()
    X, Y = ix[:, None] + k[None, :], iy[:, None] + k[None, :]
    ok = ((Y >= 0) & (Y < H))[:, :, None] & ((X >= 0) & (X < W))[:, None, :]
    at = Y.clamp(0, H - 1)[:, :, None] * W + X.clamp(0, W - 1)[:, None, :]
    img.index_add_(0, at.reshape(-1), torch.where(ok, val, torch.zeros_like(val)).reshape(-1))
    return img.view(H, W)


def _frames(W, H, bits, seed, f):
    """One image pair: uint8, or 12-bit values carried as int16."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    m = 24.0
    n = int((0.05 if bits == 8 else 0.03) * (W + 2 * m) * (H + 2 * m))
    r = torch.rand(n, 6, generator=g, device=DEV, dtype=torch.float64)
    x, y = r[:, 0] * (W + 2 * m) - m, r[:, 1] * (H + 2 * m) - m
    dp = torch.full_like(x, 2.5) if bits == 8 else 2.0 + 2.0 * r[:, 2]
    full = 255.0 if bits == 8 else 4095.0
    amp = (150.0 + 105.0 * r[:, 3]) / 255.0 * full
    u, v = _velocity(f, x, y)
    lost = (r[:, 4] < (0.0 if bits == 8 else 0.1))  # out of plane: elsewhere in the second frame
    x2 = torch.where(lost, r[:, 5] * (W + 2 * m) - m, x + 0.5 * u)
    y2 = torch.where(lost, ((r[:, 5] * 7919.0) % 1.0) * (H + 2 * m) - m, y + 0.5 * v)
    out = []
    for px, py in ((x - 0.5 * u, y - 0.5 * v), (x2, y2)):
        img = _splat(px, py, dp, amp, W, H).double() / 256.0
        img = img + 0.02 * full * torch.randn(H, W, generator=g, device=DEV, dtype=torch.float64)
        img = torch.round(img).clamp_(0, full)
        out.append(img.to(torch.uint8 if bits == 8 else torch.int16))
    return out


def _nodes(W, H, w, s):
    nx, ny = _grid(W, H, w, s)
    x = torch.arange(nx, device=DEV, dtype=torch.float64) * s + 0.5 * (w - 1)
    y = torch.arange(ny, device=DEV, dtype=torch.float64) * s + 0.5 * (w - 1)
    return x[None, :].expand(ny, nx), y[:, None].expand(ny, nx)


def _field(f, W, H, w, s, seed, noise):
    """A measured field: the flow at the nodes with the scatter of a measurement."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    x, y = _nodes(W, H, w, s)
    u, v = _velocity(f, x, y)
    e = noise * torch.randn(2, *u.shape, generator=g, device=DEV, dtype=torch.float64)
    return (u + e[0]).float().contiguous(), (v + e[1]).float().contiguous()


def _inputs(case, seed):
    W, H, bits = case["width"], case["height"], case["bits"]
    gen = torch.Generator().manual_seed(seed)
    if case["do"] == "process":
        large = "6" in case["radii"] or case["levels"] == 2 or case["pred"]
        fs = [_flow(gen, W, H, large) for _ in range(case["pairs"])]
        if case["levels"] == 0 and not case["pred"]:
            for f in fs:  # within reach of the search around zero
                r = min(_ints(case["radii"])) - 1.5
                k = min(1.0, r / 4.5)
                f["U"], f["V"], f["shear"] = k * f["U"], k * f["V"], (0.5 * k,) + f["shear"][1:]
        ab = [_frames(W, H, bits, seed * 1000 + i, f) for i, f in enumerate(fs)]
        preds = None
        if case["pred"]:
            w = _ints(case["windows"])[-1]
            preds = []
            for i, f in enumerate(fs):  # the frame before: the vortex half a pixel back
                before = dict(f, vortex=(f["vortex"][0] - 0.5,) + f["vortex"][1:])
                preds.append(_field(before, W, H, w, w // 2, seed * 1000 + 500 + i, 0.05))
        return [p[0] for p in ab], [p[1] for p in ab], preds
    f = _flow(gen, W, H, False)
    a, b = _frames(W, H, bits, seed * 1000, f)
    if case["do"] == "preprocess":  # uneven illumination under the particles
        full = 255 if bits == 8 else 4095
        ramp = torch.linspace(0.02, 0.12, W, device=DEV, dtype=torch.float64)[None, :] * full
        return tuple((t.double() + ramp).round().clamp(0, full).to(t.dtype) for t in (a, b))
    if case["do"] == "stages":
        return a, b, _field(f, W, H, case["window"], case["step"], seed * 1000 + 1, 0.1)
    s = int(case["window"] * (1 - case["overlap"]))
    return a, b, _field(f, W, H, case["window"], s, seed * 1000 + 1, 0.15)


def prepare(case, seed):
    W, H, bits = case["width"], case["height"], case["bits"]
    st = {"case": case}
    if case["do"] == "process":
        a, b, preds = _inputs(case, seed)
        if case["host"]:
            a, b = [t.cpu().pin_memory() for t in a], [t.cpu().pin_memory() for t in b]
        ws = _ints(case["windows"])
        cfg = rp.Config(W, H, windows=ws, overlaps=[0.5] * len(ws), radii=_ints(case["radii"]), levels=case["levels"],
                        bit_depth=bits, precision=case["precision"], deform=case["deform"], max_batch=case["pairs"],
                        host_frames=case["host"])
        st.update(a=a, b=b, preds=preds, engine=rp.Engine(cfg))
    elif case["do"] in ("grad", "refine"):
        a, b, (u, v) = _inputs(case, seed)
        cfg = rp.Config(W, H, windows=[case["window"]], overlaps=[case["overlap"]], radii=[4], bit_depth=bits)
        st.update(a=a, b=b, u=u, v=v, engine=rp.Engine(cfg))
    elif case["do"] == "preprocess":
        a, b = _inputs(case, seed)
        # a program keeps the scratch of its frame size
        t = (case["tiles"], case["tiles"])
        st.update(a=a, b=b, scratch=torch.empty(binding.preprocess_scratch_bytes(W, H, t), dtype=torch.uint8, device=DEV))
    else:
        a, b, (u, v) = _inputs(case, seed)
        st.update(a=a, b=b, u=u, v=v)
    return st


def run(state):
    c, a, b = state["case"], state["a"], state["b"]
    if c["do"] == "process":
        if c["pairs"] == 1:
            return state["engine"].process_pair(a[0], b[0], pred=state["preds"][0] if state["preds"] else None)
        return state["engine"].process_batch(a, b, preds=state["preds"])
    if c["do"] == "grad":
        return state["engine"].score_and_grad(a, b, state["u"], state["v"])
    if c["do"] == "refine":
        return binding.refine(state["engine"], a, b, state["u"], state["v"], steps=c["steps"])
    if c["do"] == "preprocess":
        kw = dict(vmax=255 if c["bits"] == 8 else 4095, hp=c["radius"], tiles=(c["tiles"], c["tiles"]),
                  clip_pct=c["clip"], scratch=state["scratch"])
        return binding.stage_preprocess(a, **kw), binding.stage_preprocess(b, **kw)
    w, s = c["window"], c["step"]
    half = binding.stage_downsample(a)
    u, v, info = binding.stage_correlate(a, b, w, s, c["radius"], state["u"], state["v"])
    uo, vo, mask = binding.stage_validate(u, v, info)
    nx, ny = _grid(c["width"], c["height"], 16, 8)
    du, dv = binding.stage_interp(uo, vo, w, s, nx, ny, 16, 8)
    smooth = binding.stage_ema(du, torch.full_like(du, 3.0), 0.3)
    return half, u, v, info, uo, vo, mask, du, dv, smooth, binding.stage_vorticity(du, dv, 8)


# ------------------------------------------------------------- 64-bit restatement --

def _axis(pos, n, c0, s):
    if n <= 1:
        z = torch.zeros_like(pos)
        return z.long(), z.long(), z
    f = ((pos - c0) / s).clamp(0, n - 1)
    i = torch.floor(f).long().clamp(max=n - 2)
    return i, i + 1, f - i


def _bilinear_grid(q, xs, ys, w, s):
    """Field q (ny x nx) at positions xs (columns), ys (rows)."""
    ny, nx = q.shape
    i0, i1, tx = _axis(xs, nx, 0.5 * (w - 1), s)
    j0, j1, ty = _axis(ys, ny, 0.5 * (w - 1), s)
    r = q[:, i0] + tx * (q[:, i1] - q[:, i0])
    return r[j0] + ty[:, None] * (r[j1] - r[j0])


def _warp(img, du, dv, x, y):
    """Bilinear, clamp-to-edge samples of img at (x + du, y + dv)."""
    H, W = img.shape
    fx, fy = torch.floor(du.detach()), torch.floor(dv.detach())
    tx, ty = du - fx, dv - fy
    ix, iy = x[None, :].long() + fx.long(), y[:, None].long() + fy.long()
    xa, xb, ya, yb = ix.clamp(0, W - 1), (ix + 1).clamp(0, W - 1), iy.clamp(0, H - 1), (iy + 1).clamp(0, H - 1)
    top = img[ya, xa] + tx * (img[ya, xb] - img[ya, xa])
    bot = img[yb, xa] + tx * (img[yb, xb] - img[yb, xa])
    return top + ty * (bot - top)


def _box(img, w, s, G, nx, ny):
    """Sums over the windows of a grid, from sums over G x G blocks."""
    k, st = w // G, s // G
    nbx, nby = (nx - 1) * st + k, (ny - 1) * st + k
    b = img[:nby * G, :nbx * G].reshape(nby, G, nbx, G).sum(dim=(1, 3))
    return F.avg_pool2d(b[None, None], k, st)[0, 0] * (k * k)


def _fit(cm, c0, cp):
    ok = (cm > 0) & (c0 > 0) & (cp > 0)
    lm, l0, lp = (torch.log(torch.where(ok, c, torch.ones_like(c))) for c in (cm, c0, cp))
    den, pden = 2 * lm - 4 * l0 + 2 * lp, 2 * cm - 4 * c0 + 2 * cp
    log_ok, par_ok = ok & (den < 0), pden < 0
    d = torch.where(par_ok, (cm - cp) / torch.where(par_ok, pden, torch.ones_like(pden)), torch.zeros_like(cm))
    d = torch.where(log_ok, (lm - lp) / torch.where(log_ok, den, torch.ones_like(den)), d)
    return d.clamp(-1, 1)


def _correlate(A, B, w, s, R, pu, pv, central):
    """One pass in 64 bits: the peak of the correlation coefficient around the predictor, Gaussian fit."""
    H, W = A.shape
    nx, ny = _grid(W, H, w, s)
    G, M = math.gcd(w, s), R + 1
    x = torch.arange(-M, W + M, device=DEV, dtype=torch.float64)
    y = torch.arange(-M, H + M, device=DEV, dtype=torch.float64)
    du, dv = _bilinear_grid(pu, x, y, w, s), _bilinear_grid(pv, x, y, w, s)
    if central:
        A = _warp(A, -0.5 * du, -0.5 * dv, x, y)[M:M + H, M:M + W]
        du, dv = 0.5 * du, 0.5 * dv
    Bw = _warp(B, du, dv, x, y)
    del du, dv
    n, tau = float(w * w), 1e-6 * w * w
    muA = _box(A, w, s, G, nx, ny) / n
    EA = _box(A * A, w, s, G, nx, ny) - n * muA * muA
    B2 = Bw * Bw
    ND = 2 * M + 1
    C = torch.empty(ND * ND, ny, nx, device=DEV, dtype=torch.float64)
    for sy in range(ND):
        for sx in range(ND):
            sh = Bw[sy:sy + H, sx:sx + W]
            S1 = _box(sh, w, s, G, nx, ny)
            EB = _box(B2[sy:sy + H, sx:sx + W], w, s, G, nx, ny) - S1 * S1 / n
            num = _box(A * sh, w, s, G, nx, ny) - muA * S1
            ok = EB > tau
            C[sy * ND + sx] = torch.where(ok, num / torch.sqrt(torch.where(ok, EB * EA.clamp(min=tau), torch.ones_like(EB))),
                                          torch.zeros_like(num))
    P = C.view(ND, ND, ny, nx)
    inner = P[1:-1, 1:-1].reshape((2 * R + 1) ** 2, ny, nx)
    at = inner.argmax(0)
    ky, kx = torch.div(at, 2 * R + 1, rounding_mode="floor"), at % (2 * R + 1)

    def take(dy, dx):
        return C.gather(0, ((ky + 1 + dy) * ND + kx + 1 + dx)[None])[0]

    c0 = take(0, 0)
    good = EA > tau
    u = torch.where(good, pu + (kx - R) + _fit(take(0, -1), c0, take(0, 1)), pu)
    v = torch.where(good, pv + (ky - R) + _fit(take(-1, 0), c0, take(1, 0)), pv)
    return u, v, good


def _median(vals, count):
    """Median of the first `count` of the sorted values (missing ones are inf)."""
    v, c = vals.sort(0)[0], count.clamp(min=1)[None]
    return 0.5 * (v.gather(0, (c - 1) // 2)[0] + v.gather(0, c // 2)[0])


def _neighbours(q, there):
    inf = torch.full_like(q, math.inf)
    p = F.pad(torch.where(there, q, inf), (1, 1, 1, 1), value=math.inf)
    ny, nx = q.shape
    return torch.stack([p[j:j + ny, i:i + nx] for j in range(3) for i in range(3) if (i, j) != (1, 1)])


def _validate(u, v, good):
    every = torch.ones_like(good)
    count = torch.isfinite(_neighbours(u, every)).sum(0)
    bad = ~good
    for q in (u, v):
        nb = _neighbours(q, every)
        m = _median(nb, count)
        res = torch.where(torch.isfinite(nb), (nb - m).abs(), nb)
        bad = bad | ((count > 0) & ((q - m).abs() / (_median(res, count) + 0.1) > 2.0))
    left = torch.isfinite(_neighbours(u, ~bad)).sum(0)
    return [torch.where(bad & (left > 0), _median(_neighbours(q, ~bad), left), q) for q in (u, v)]


def _interp(q, w, s, dnx, dny, dw, ds, up):
    f = float(1 << up)
    x = (torch.arange(dnx, device=DEV, dtype=torch.float64) * ds + 0.5 * (dw - 1) + 0.5) / f - 0.5
    y = (torch.arange(dny, device=DEV, dtype=torch.float64) * ds + 0.5 * (dw - 1) + 0.5) / f - 0.5
    return f * _bilinear_grid(q, x, y, w, s)


def _vorticity(u, v, s):
    def d(q, dim):
        if q.shape[dim] < 2:
            return torch.zeros_like(q)
        return torch.gradient(q, spacing=float(s), dim=dim)[0]
    return d(v, 1) - d(u, 0)


def _half(img):
    H, W = img.shape
    return F.avg_pool2d(img[None, None, :H // 2 * 2, :W // 2 * 2], 2)[0, 0]


def _pipeline(case, A, B, pred):
    W, H = case["width"], case["height"]
    ws, rs, L = _ints(case["windows"]), _ints(case["radii"]), case["levels"]
    central = case["deform"] == "central"
    lv = [(A, B)]
    for _ in range(L):
        lv.append((_half(lv[-1][0]), _half(lv[-1][1])))
    stages = [(l, ws[0], rs[0]) for l in range(L, 0, -1)] + [(0, w, r) for w, r in zip(ws, rs)]
    q = None
    for k, (l, w, r) in enumerate(stages):
        a, b = lv[l]
        s = w // 2
        nx, ny = _grid(a.shape[1], a.shape[0], w, s)
        if q is not None:
            q = [_interp(t, *src, nx, ny, w, s, up) for t in q for src, up in [(at, up_l - l)]]
        elif pred is not None:
            q = [_interp(t.double(), ws[-1], ws[-1] // 2, nx, ny, w, s, 0) for t in pred]
        else:
            q = [torch.zeros(ny, nx, device=DEV, dtype=torch.float64)] * 2
        u, v, good = _correlate(a, b, w, s, r, q[0], q[1], central)
        q = _validate(u, v, good)
        at, up_l = (w, s), l
    return q[0], q[1], _vorticity(q[0], q[1], ws[-1] // 2)


def _score(case, A, B, u, v):
    H, W = A.shape
    w = case["window"]
    s = int(w * (1 - case["overlap"]))
    nx, ny = _grid(W, H, w, s)
    G, n, tau = math.gcd(w, s), float(w * w), 1e-6 * w * w
    x = torch.arange(W, device=DEV, dtype=torch.float64)
    y = torch.arange(H, device=DEV, dtype=torch.float64)
    Bw = _warp(B, _bilinear_grid(u, x, y, w, s), _bilinear_grid(v, x, y, w, s), x, y)
    ma, mb = _box(A, w, s, G, nx, ny) / n, _box(Bw, w, s, G, nx, ny) / n
    ea = _box(A * A, w, s, G, nx, ny) - n * ma * ma
    eb = _box(Bw * Bw, w, s, G, nx, ny) - n * mb * mb
    ok = (ea > tau) & (eb > tau)
    num = _box(A * Bw, w, s, G, nx, ny) - n * ma * mb
    return torch.where(ok, num / torch.sqrt(torch.where(ok, ea * eb, torch.ones_like(ea))), torch.zeros_like(num)).sum()


def _score_grad(case, A, B, u, v):
    with torch.enable_grad():
        u, v = u.detach().requires_grad_(), v.detach().requires_grad_()
        S = _score(case, A, B, u, v)
        gu, gv = torch.autograd.grad(S, (u, v))
    return S.detach(), gu, gv


def _preprocessed(img, vmax, hp, tiles, clip):
    H, W = img.shape
    I = img.long()
    n, d = 1, I
    if hp > 0:
        k = 2 * hp + 1
        n = k * k
        S = F.avg_pool2d(F.pad(I.double()[None, None], (hp, hp, hp, hp), mode="replicate"), k, 1)[0, 0] * n
        d = (n * I - torch.round(S).long()).clamp(min=0)
    if clip <= 0:
        return d.double() / n
    tw, th = -(-W // tiles), -(-H // tiles)
    bins = torch.div(d * 256, n * (vmax + 1), rounding_mode="floor").clamp(max=255)
    maps = torch.zeros(tiles, tiles, 256, device=DEV, dtype=torch.float64)
    for j in range(tiles):
        for i in range(tiles):
            t = bins[j * th:min(H, (j + 1) * th), i * tw:min(W, (i + 1) * tw)]
            N = t.numel()
            if not N:
                continue
            h = torch.bincount(t.reshape(-1), minlength=256)
            L = max(1, clip * N // 25600)
            E = int((h - L).clamp(min=0).sum())
            h = h.clamp(max=L) + E // 256
            h[:E % 256] += 1
            maps[j, i] = h.cumsum(0).double() * vmax / N

    def axis(ext, ts):
        p = torch.arange(ext, device=DEV, dtype=torch.float64)
        c = torch.tensor([t * ts + 0.5 * (min(ext, (t + 1) * ts) - t * ts - 1) for t in range(tiles)], device=DEV,
                         dtype=torch.float64)
        c0 = 0.5 * (ts - 1)
        t0 = torch.floor((p - c0) / ts).long().clamp(0, max(tiles - 2, 0))
        t1 = (t0 + 1).clamp(max=tiles - 1)
        wgt = ((p - c[t0]) / torch.where(t1 > t0, c[t1] - c[t0], torch.ones_like(p))).clamp(0, 1)
        return t0, t1, wgt

    i0, i1, wx = axis(W, tw)
    j0, j1, wy = axis(H, th)
    at = [[maps[j[:, None], i[None, :], bins] for i in (i0, i1)] for j in (j0, j1)]
    top, bot = ((1 - wx) * r[0] + wx * r[1] for r in at)
    return (1 - wy)[:, None] * top + wy[:, None] * bot


def exact(case, seed):
    if case["do"] == "process":
        a, b, preds = _inputs(case, seed)
        got = [_pipeline(case, p.double(), q.double(), preds[i] if preds else None) for i, (p, q) in enumerate(zip(a, b))]
        if case["precision"] != "fp32":  # a peak that 16 bits move shows as a spike in the derivative
            got = [t[:2] for t in got]
            none = (None, None)
        else:
            none = (None,)
        if case["pairs"] == 1:
            return got[0] + none
        return tuple(torch.stack(t) for t in zip(*got)) + none
    if case["do"] in ("grad", "refine"):
        a, b, (u, v) = _inputs(case, seed)
        A, B, u, v = a.double(), b.double(), u.double(), v.double()
        S, gu, gv = _score_grad(case, A, B, u, v)
        if case["do"] == "grad":
            return S, gu, gv
        gmax, hist = float(torch.maximum(gu.abs().max(), gv.abs().max())), [float(S)]
        for k in range(case["steps"]):
            eta = 0.25 * 0.5 ** k / gmax
            for _ in range(4):
                cu, cv = u + eta * gu, v + eta * gv
                if float(_score(case, A, B, cu, cv)) > hist[-1]:
                    u, v = cu, cv
                    break
                eta *= 0.5
            S, gu, gv = _score_grad(case, A, B, u, v)
            hist.append(float(S))
        return u, v, hist
    if case["do"] == "preprocess":
        vmax = 255 if case["bits"] == 8 else 4095
        return tuple(_preprocessed(t, vmax, case["radius"], case["tiles"], case["clip"]) for t in _inputs(case, seed))
    a, b, (u, v) = _inputs(case, seed)
    w, s = case["window"], case["step"]
    A = a.double()
    u, v, good = _correlate(A, b.double(), w, s, case["radius"], u.double(), v.double(), False)
    uo, vo = _validate(u, v, good)
    nx, ny = _grid(case["width"], case["height"], 16, 8)
    du, dv = _interp(uo, w, s, nx, ny, 16, 8, 0), _interp(vo, w, s, nx, ny, 16, 8, 0)
    return _half(A), u, v, None, uo, vo, None, du, dv, 0.3 * du + 0.7 * 3.0, _vorticity(du, dv, 8)
