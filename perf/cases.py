"""The work a user of this library has it do, as callable cases.

Every case goes through the public Python binding (`paper_2202_13347_gb300`)
on seeded synthetic inputs made on the GPU: multi-octave texture with
rectangles, a radiometrically mapped and shifted (optionally speckled) copy
as the sensed image, one jittered point per grid cell.  Sizes follow the
paper's experiments (512-1501 px pairs; 400 points, templates of 80 px,
search window 200) and this repository's own workloads (512^2, 2048^2, 10000^2
uint16, the mixed batch).

`listed` gives the cases, `draw` more of the same ranges, `prepare` what a
program holds before the call, `run` one pass, `work` its unavoidable bytes
and operations, `exact` the same outputs in 64 bits by plain torch.
"""
import math
import random

import torch
import torch.nn.functional as F

import paper_2202_13347_gb300 as pkg

B = pkg.load()
DEV = "cuda:0"
Z = 12  # channels of the default descriptor

# ---- the cases ------------------------------------------------------------


def _build(name, H, W, dtype, u16=False):
    return dict(name=name, kind="build", H=H, W=W, dtype=dtype, u16=u16)


def _pair(name, kind, H, W, n, m, R, dtype, maps=False, speckled=False):
    return dict(name=name, kind=kind, H=H, W=W, n=n, m=m, R=R, dtype=dtype, maps=maps, speckled=speckled)


def listed():
    return [
        # the descriptor of one small image (the smallest pairs of the paper's Table 1)
        _build("build_512_f32", 512, 512, "f32"),
        # an ordinary odd-sized image (Table 1's largest), stored as bf16 for the tensor cores
        _build("build_1501x1207_bf16", 1501, 1207, "bf16"),
        # a large 16-bit scene, the biggest single image a user builds
        _build("build_u16_10000_bf16", 10000, 10000, "bf16", True),
        # the whole path for one small pair on the device: launches and latency count
        _pair("register_512_f32", "register", 512, 512, 100, 41, 10, "f32"),
        # matching an optical / SAR-like pair against cubes already built
        _pair("match_2048_m81_r20_f32", "match", 2048, 2048, 1000, 81, 20, "f32", speckled=True),
        # the paper's windows: template 80, search window 200, 400 points, with the NCC maps
        _pair("match_2048_m80_r60_maps_f32", "match", 2048, 2048, 400, 80, 60, "f32", maps=True),
        # dense matching with a large radius on bf16 cubes of a larger scene
        _pair("match_4096x3000_m81_r40_bf16", "match", 4096, 3000, 2000, 81, 40, "bf16"),
        # one pair from pinned host memory to host results, as a service would call it
        _pair("register_host_2048_bf16", "register_host", 2048, 2048, 1000, 81, 20, "bf16"),
        # many pairs of uneven size, points, templates and radii in one batched call
        dict(name="register_batch_20_bf16", kind="batch", pairs=20, side_max=3200, n_max=2400, dtype="bf16", layout=4000),
        # interest points of a sensed image, one per block
        dict(name="fast_2048", kind="fast", H=2048, W=2048, grid=32, margin=61),
        # outlier rejection over one pair's control points
        dict(name="ransac_1000x4096", kind="ransac", n=1000, hyps=4096, projective=True),
        # the sensed image resampled into the reference frame
        dict(name="rectify_2048", kind="rectify", H=2048, W=2048),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges (sizes over their logarithm)."""
    kind = rng.choice(["build", "build", "register", "match", "match", "match", "register_host", "batch", "fast",
                       "ransac", "rectify"])
    dtype = rng.choice(["f32", "bf16"])
    if kind == "build":
        u16 = rng.random() < 0.3
        hi = 5000 if u16 else 3500
        return dict(kind=kind, H=_log_int(rng, 300, hi), W=_log_int(rng, 300, hi), dtype=dtype, u16=u16)
    if kind in ("register", "match", "register_host"):
        f32 = dtype == "f32"
        m = rng.choice([41, 61, 80 if f32 else 81])
        R = rng.randint(8, 60 if f32 else 40)
        side = 2600 if kind == "match" else 2048
        lo = max(500, m + 2 * R + 60)
        return dict(kind=kind, H=_log_int(rng, lo, side), W=_log_int(rng, lo, side), n=_log_int(rng, 50, 700), m=m,
                    R=R, dtype=dtype, maps=f32 and kind == "match" and rng.random() < 0.4,
                    speckled=f32 and m + 2 * R <= 128 and rng.random() < 0.5)
    if kind == "batch":
        few = dtype == "f32"
        return dict(kind=kind, pairs=rng.randint(2, 6 if few else 12), side_max=_log_int(rng, 700, 2400),
                    n_max=_log_int(rng, 250, 500 if few else 1400), dtype=dtype, layout=rng.randint(0, 10 ** 6))
    if kind == "fast":
        return dict(kind=kind, H=_log_int(rng, 400, 4096), W=_log_int(rng, 400, 4096), grid=rng.randint(8, 48),
                    margin=rng.randint(3, 100))
    if kind == "ransac":
        return dict(kind=kind, n=_log_int(rng, 60, 3000), hyps=_log_int(rng, 500, 8000),
                    projective=rng.random() < 0.6)
    return dict(kind=kind, H=_log_int(rng, 400, 4096), W=_log_int(rng, 400, 4096))


# ---- inputs -----------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _scale01(img):
    lo, hi = img.min(), img.max()
    return ((img - lo) / (hi - lo)).contiguous()


def _optical(g, rnd, H, W):
    """Value noise of several octaves plus bright and dark rectangles, in [0, 1]."""
    img = torch.zeros((H, W), device=DEV)
    amp = 0.5
    for cell in (64, 32, 16, 8, 4, 2):
        lat = torch.rand((1, 1, H // cell + 2, W // cell + 2), device=DEV, generator=g)
        up = F.interpolate(lat, scale_factor=cell, mode="bilinear", align_corners=False)
        img += amp * up[0, 0, :H, :W]
        amp *= 0.6
    for _ in range(60):
        h, w = rnd.randint(8, max(9, H // 6)), rnd.randint(8, max(9, W // 6))
        y, x = rnd.randint(0, max(0, H - h - 1)), rnd.randint(0, max(0, W - w - 1))
        img[y:y + h, x:x + w] += rnd.uniform(-1.0, 1.0)
    return _scale01(img)


def _sensed(g, rnd, ref, R, speckled):
    """The reference shifted inside the search radius through one of the radiometric maps."""
    shift = [rnd.choice([-1, 1]) * rnd.randint(max(1, R // 3), max(1, 3 * R // 4)) for _ in range(2)]
    img = torch.roll(ref, shift, (0, 1))
    kind = rnd.choice(["linear", "gamma", "inverted"])
    if kind == "gamma":
        img = img.clamp_min(0).pow(rnd.uniform(0.6, 2.0))
    elif kind == "inverted":
        img = 1.0 - img
    if speckled:  # four looks of unit-mean multiplicative speckle
        u = torch.rand((4,) + tuple(img.shape), device=DEV, generator=g).clamp_min(1e-7)
        img = img * (-u.log()).mean(0)
    return _scale01(img)


def _half(m):
    return (m - 1) // 2 if m % 2 else m // 2


def _points(g, H, W, n, m, R):
    """n points, one jittered in each cell of a grid, inside the margin matching needs."""
    lo = _half(m) + R
    gy = max(1, int(round(math.sqrt(n * H / W))))
    gx = -(-n // gy)
    k = torch.arange(n, device=DEV)
    u = torch.rand((2, n), device=DEV, generator=g)
    y = ((k // gx + u[0]) / gy).clamp(max=0.999999) * (H - m - 2 * R + 1) + lo
    x = ((k % gx + u[1]) / gx).clamp(max=0.999999) * (W - m - 2 * R + 1) + lo
    return torch.stack([x.to(torch.int32).clamp(max=W - m + _half(m) - R),
                        y.to(torch.int32).clamp(max=H - m + _half(m) - R)], 1).contiguous()


def _batch_layout(case):
    """(H, W, n, m, R) of each pair of a batch; part of the case, not of the seed."""
    r = random.Random(case["layout"])
    out = []
    for _ in range(case["pairs"]):
        out.append((_log_int(r, 512, case["side_max"]), _log_int(r, 512, case["side_max"]),
                    _log_int(r, 200, case["n_max"]), r.choice([41, 61, 80 if case["dtype"] == "f32" else 81]),
                    r.randint(10, 40)))
    return out


def _u16(img):
    """The image as 16-bit samples, held in int16 as the binding takes them."""
    v = (img * 65535.0).round().to(torch.int32)
    return torch.where(v >= 32768, v - 65536, v).to(torch.int16).contiguous()


def _images(case, seed):
    g, rnd = _gen(seed), random.Random(seed)
    ref = _optical(g, rnd, case["H"], case["W"])
    if case["kind"] == "build":
        return ref
    sen = _sensed(g, rnd, ref, case["R"], case["speckled"])
    return ref, sen, _points(g, case["H"], case["W"], case["n"], case["m"], case["R"])


def _batch_images(case, seed):
    g, rnd = _gen(seed), random.Random(seed)
    refs, sens, pts = [], [], []
    for H, W, n, m, R in _batch_layout(case):
        refs.append(_optical(g, rnd, H, W))
        sens.append(_sensed(g, rnd, refs[-1], R, False))
        pts.append(_points(g, H, W, n, m, R))
    return refs, sens, pts


def _control_points(case, seed):
    """Source points, their images under a near-identity model, 30 % of them outliers, and the minimal samples."""
    g, rnd = _gen(seed), random.Random(seed)
    u = lambda a: rnd.uniform(-a, a)  # noqa: E731
    p = 2e-5 if case["projective"] else 0.0
    M = torch.tensor([[1 + u(0.02), u(0.02), u(40)], [u(0.02), 1 + u(0.02), u(40)], [u(p), u(p), 1.0]],
                     dtype=torch.float64, device=DEV)
    n, k = case["n"], 4 if case["projective"] else 3
    src = torch.rand((n, 2), device=DEV, generator=g, dtype=torch.float64) * 2000.0
    q = torch.cat([src, torch.ones((n, 1), dtype=torch.float64, device=DEV)], 1) @ M.T
    dst = q[:, :2] / q[:, 2:]
    dst += 0.3 * torch.randn((n, 2), device=DEV, generator=g, dtype=torch.float64)
    out = torch.rand(n, device=DEV, generator=g) < 0.3
    off = torch.rand((n, 2), device=DEV, generator=g, dtype=torch.float64) * 180.0 + 20.0
    dst = torch.where(out[:, None], dst + off, dst).contiguous()
    base = torch.randint(0, n, (case["hyps"], 1), device=DEV, generator=g)
    step = torch.randint(1, max(2, n // k), (case["hyps"], 1), device=DEV, generator=g)
    samples = ((base + step * torch.arange(k, device=DEV)) % n).to(torch.int32).contiguous()
    return src, dst, samples


def _rectify_inputs(case, seed):
    g, rnd = _gen(seed), random.Random(seed)
    img = _optical(g, rnd, case["H"], case["W"])
    u = lambda a: rnd.uniform(-a, a)  # noqa: E731
    M = torch.tensor([[1 + u(0.02), u(0.02), u(40)], [u(0.02), 1 + u(0.02), u(40)], [u(2e-5), u(2e-5), 1.0]],
                     dtype=torch.float64, device=DEV)
    return img, M


# ---- what a program holds, and one pass ---------------------------------------


class _Device:
    """A cube's device memory as torch sees foreign memory; the cube lives as long as this does."""

    def __init__(self, cube, ptr, shape, typestr, strides=None):
        self.cube = cube
        self.__cuda_array_interface__ = dict(data=(ptr, False), shape=shape, typestr=typestr, strides=strides,
                                             version=3)


def _cube_values(cube):
    """The cube's own values as a tensor (sfoc_cube_view), without a copy; it keeps the cube."""
    ptr, z, H, W, pitch, dt = cube.view()
    if dt == B.DTYPE_F32:
        t = torch.as_tensor(_Device(cube, ptr, (z, H, W), "<f4", (4 * pitch * H, 4 * pitch, 4)), device=DEV)
    else:
        t = torch.as_tensor(_Device(cube, ptr, (z // 6, H, W, 8), "<i2"), device=DEV).view(torch.bfloat16)
    t.cube = cube
    return t


def _params(case):
    return B.params(dtype=B.DTYPE_BF16 if case["dtype"] == "bf16" else B.DTYPE_F32)


def _tune(ctx, p, keys):
    """A program's warm-up: the correlation form of each (m, R) is measured on a small pair of other images."""
    for m, R in sorted(set(keys)):
        side = m + 2 * R + 40
        g, rnd = _gen(17), random.Random(17)
        img = _optical(g, rnd, side, side)
        cube = ctx.sfoc_build(img, p=p)
        ctx.fastncc_match(cube, cube, _points(g, side, side, 304, m, R), m, R)
        ctx.sync()
        cube.free()


def _fields(raw):
    f = B.results(raw)
    return {k: f[k] for k in ("dx", "dy", "status", "ncc", "sub_dx", "sub_dy")}


def prepare(case, seed):
    k = case["kind"]
    ctx = B.Context(0)
    s = dict(case=case, ctx=ctx)
    if k == "build":
        img = _images(case, seed)
        s["p"] = _params(case)
        s["img"] = _u16(img) if case["u16"] else img
        s["cube"] = (ctx.sfoc_build_u16 if case["u16"] else ctx.sfoc_build)(s["img"], p=s["p"])
        s["values"] = _cube_values(s["cube"])
    elif k in ("register", "match", "register_host"):
        s["p"] = _params(case)
        _tune(ctx, s["p"], [(case["m"], case["R"])])
        s["ref"], s["sen"], s["pts"] = _images(case, seed)
        if k == "match":
            s["ref"] = ctx.sfoc_build(s["ref"], p=s["p"])
            s["sen"] = ctx.sfoc_build(s["sen"], p=s["p"])
        else:
            s["out"] = torch.empty((case["n"], 6), dtype=torch.int32, device=DEV)
        if k == "register_host":
            for name in ("ref", "sen", "pts", "out"):
                s[name] = s[name].cpu().pin_memory()
    elif k == "batch":
        s["p"] = _params(case)
        lay = _batch_layout(case)
        _tune(ctx, s["p"], [(l[3], l[4]) for l in lay])
        s["refs"], s["sens"], s["pts"] = _batch_images(case, seed)
        s["ms"], s["Rs"] = [l[3] for l in lay], [l[4] for l in lay]
        s["raw"] = torch.empty((sum(l[2] for l in lay), 6), dtype=torch.int32, device=DEV)
        s["outs"] = list(torch.split(s["raw"], [l[2] for l in lay]))
    elif k == "fast":
        s["img"] = _optical(_gen(seed), random.Random(seed), case["H"], case["W"])
    elif k == "ransac":
        s["src"], s["dst"], s["samples"] = _control_points(case, seed)
    else:
        s["img"], s["model"] = _rectify_inputs(case, seed)
        s["out"] = torch.empty((case["H"], case["W"]), dtype=torch.float32, device=DEV)
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    k = case["kind"]
    if k == "build":
        (ctx.sfoc_build_u16 if case["u16"] else ctx.sfoc_build)(s["img"], p=s["p"], out=s["cube"])
        return s["values"]
    if k == "match":
        r = ctx.fastncc_match(s["ref"], s["sen"], s["pts"], case["m"], case["R"], want_maps=case["maps"])
        out = {f: r[f] for f in ("dx", "dy", "status", "ncc", "sub_dx", "sub_dy")}
        if case["maps"]:
            out["maps"] = r["maps"]
        return out
    if k == "register":
        return _fields(ctx.register_pair(s["ref"], s["sen"], s["pts"], case["m"], case["R"], p=s["p"], out=s["out"]))
    if k == "register_host":
        return _fields(ctx.register_pair_host(s["ref"], s["sen"], s["pts"], case["m"], case["R"], p=s["p"],
                                              out=s["out"]))
    if k == "batch":
        ctx.register_batch(s["refs"], s["sens"], s["pts"], s["ms"], s["Rs"], p=s["p"], outs=s["outs"])
        return _fields(s["raw"])
    if k == "fast":
        pts, sc = ctx.fast_blocks(s["img"], grid_y=case["grid"], grid_x=case["grid"], margin=case["margin"])
        return dict(points=pts, scores=sc)
    if k == "ransac":
        return ctx.fastncc_ransac(s["src"], s["dst"], s["samples"],
                                  model=B.MODEL_PROJECTIVE if case["projective"] else B.MODEL_AFFINE,
                                  want_scores=True)
    return ctx.rectify(s["img"], s["model"], out=s["out"])


# ---- unavoidable work -----------------------------------------------------------


def _build_work(H, W, dtype, sample=4):
    """Image in, cube out; multiply-adds of the separable bases, the steering and the dilated smoothing."""
    return H * W * (sample + (4 * Z if dtype == "f32" else 2 * 8 * Z / 6)), H * W * 2.0 * (76 + 66 + 54 + 648)


def _match_work(H, W, n, m, R, dtype):
    """Both cubes read once where the points use them, results out; the operations of the Fourier form (Eq. 13)."""
    L, P = m + 2 * R, 2 * R + 1
    el = 4 * Z if dtype == "f32" else 2 * Z
    touched = min(H * W, n * L * L) + min(H * W, n * m * m)
    flops = n * (5 * L * math.log2(L) * (Z * (L + L) + L / 2 + 1 + P) + 6.0 * Z * L * L)
    return touched * el + 24 * n, min(flops, n * 2.0 * m * m * P * P * Z)


def work(case):
    k = case["kind"]
    if k == "build":
        b, f = _build_work(case["H"], case["W"], case["dtype"], 2 if case["u16"] else 4)
    elif k in ("match", "register", "register_host"):
        b, f = _match_work(case["H"], case["W"], case["n"], case["m"], case["R"], case["dtype"])
        if k != "match":
            b = 8 * case["H"] * case["W"] + 24 * case["n"]
            f += 2 * _build_work(case["H"], case["W"], case["dtype"])[1]
        elif case["maps"]:
            b += 4 * case["n"] * (2 * case["R"] + 1) ** 2
    elif k == "batch":
        b = f = 0
        for H, W, n, m, R in _batch_layout(case):
            b += 8 * H * W + 24 * n
            f += 2 * _build_work(H, W, case["dtype"])[1] + _match_work(H, W, n, m, R, case["dtype"])[1]
    elif k == "fast":
        b, f = 4 * case["H"] * case["W"], 179.0 * case["H"] * case["W"]
    elif k == "ransac":
        b = 32 * case["n"] + 16 * case["hyps"]
        f = 15.0 * case["n"] * case["hyps"]
    else:
        b, f = 8 * case["H"] * case["W"], 24.0 * case["H"] * case["W"]
    return dict(bytes=float(b), flops=float(f))


# ---- the same in 64 bits ----------------------------------------------------------


def _conv(x, taps, axis, step=1):
    """out[p] = sum_q taps[q] x[p + step (q - K)] along an axis, edges clamped (taps indexed 0 .. 2K)."""
    K = (len(taps) - 1) // 2 * step
    idx = torch.arange(-K, x.shape[axis] + K, device=x.device).clamp(0, x.shape[axis] - 1)
    xp = x.index_select(axis, idx)
    out = torch.zeros_like(x)
    for q, w in enumerate(taps):
        out.add_(xp.narrow(axis, q * step, x.shape[axis]), alpha=float(w))
    return out


def _exact_cube(img):
    """The default descriptor of a float64 image: [12][H][W]."""
    th = [k * math.pi / 6 for k in range(6)]
    groups = [[0.0] * 6, [0.0] * 6]
    for s in (0.6, 0.8, 1.0):
        q = list(range(-math.ceil(3 * s - 1e-9), math.ceil(3 * s - 1e-9) + 1))
        e = [math.exp(-v * v / (2 * s * s)) for v in q]
        a = [v / (2 * math.pi * s ** 4) * w for v, w in zip(q, e)]  # correlation taps of the derivative
        gx, gy = _conv(_conv(img, a, 1), e, 0), _conv(_conv(img, e, 1), a, 0)
        for k in range(6):
            groups[0][k] = groups[0][k] + (math.cos(th[k]) * gx + math.sin(th[k]) * gy).abs()
    s = 1.5
    K = math.ceil(3 * s - 1e-9)
    q = list(range(-K, K + 1))
    e = [math.exp(-v * v / (2 * s * s)) for v in q]
    a2 = [-(1 - v * v / (s * s)) * w / (2 * math.pi * s ** 4) for v, w in zip(q, e)]
    mean = sum(a2) / len(a2)
    a2 = [v - mean for v in a2]
    c = [v * w for v, w in zip(q, e)]
    xx, yy = _conv(_conv(img, a2, 1), e, 0), _conv(_conv(img, e, 1), a2, 0)
    xy = _conv(_conv(img, [v / (2 * math.pi * s ** 6) for v in c], 1), c, 0)
    for k in range(6):
        co, si = math.cos(th[k]), math.sin(th[k])
        groups[1][k] = (co * co * xx + si * si * yy - 2 * si * co * xy).abs()
    out = []
    for chans, sd in zip(groups, (1.0, 1.5)):
        K = math.ceil(3 * sd - 1e-9)
        w = [math.exp(-v * v / (2 * sd * sd)) for v in range(-K, K + 1)]
        w = [v / sum(w) for v in w]
        sm = torch.stack([sum(_conv(_conv(f, w, 1, r), w, 0, r) for r in (1, 2, 3)) for f in chans])
        out.append(sm / (sm.square().sum(0, keepdim=True).sqrt() + 1e-3))
    return torch.cat(out)


def _exact_match(ref, sen, pts, m, R, want_maps):
    """NCC over all channels (Eq. 8), its first maximum and the 3-point parabolas, from float64 cubes."""
    n, h, L, P = len(pts), _half(m), m + 2 * R, 2 * R + 1
    mnz = m * m * Z
    prefix = [F.pad(v.cumsum(0).cumsum(1), (1, 0, 1, 0)) for v in (ref.sum(0), ref.square().sum(0))]
    x0, y0 = pts[:, 0].long() - h, pts[:, 1].long() - h
    ar = lambda k: torch.arange(k, device=ref.device)  # noqa: E731
    res, maps = [], []
    for a in range(0, n, 64):
        px, py = x0[a:a + 64, None], y0[a:a + 64, None]
        num = 0.0
        t = torch.stack([sen[c][(py + ar(m))[:, :, None], (px + ar(m))[:, None, :]] for c in range(Z)])
        tm = t.mean((0, 2, 3))
        t = t - tm[None, :, None, None]
        tt = t.square().sum((0, 2, 3))
        for c in range(Z):
            w = ref[c][(py - R + ar(L))[:, :, None], (px - R + ar(L))[:, None, :]]
            num = num + torch.fft.rfft2(w) * torch.fft.rfft2(t[c], s=(L, L)).conj()
        num = torch.fft.irfft2(num, s=(L, L))[:, :P, :P]
        ys, xs = (py - R + ar(P))[:, :, None], (px - R + ar(P))[:, None, :]
        s1, s2 = (q[ys + m, xs + m] - q[ys, xs + m] - q[ys + m, xs] + q[ys, xs] for q in prefix)
        ncc = num / ((s2 - s1 * s1 / mnz).clamp_min(0) * tt[:, None, None]).sqrt()
        maps.append(ncc)
        flat = ncc.flatten(1)
        best = flat.argmax(1)
        by, bx = best // P, best % P
        k = torch.arange(len(best), device=best.device)
        peak = flat[k, best]
        sub = []
        for at, dy, dx in ((bx, 0, 1), (by, 1, 0)):
            edge = (at == 0) | (at == P - 1)
            lo = ncc[k, (by - dy).clamp_min(0), (bx - dx).clamp_min(0)]
            hi = ncc[k, (by + dy).clamp_max(P - 1), (bx + dx).clamp_max(P - 1)]
            curv = lo - 2 * peak + hi
            d = torch.where(edge | (curv >= 0), torch.zeros_like(peak), ((lo - hi) / (2 * curv)).clamp(-0.5, 0.5))
            sub.append(at - R + d)
        res.append((peak, *sub))
    out = dict(dx=None, dy=None, status=None)
    out["ncc"], out["sub_dx"], out["sub_dy"] = (torch.cat([r[i] for r in res]) for i in range(3))
    if want_maps:
        out["maps"] = torch.cat(maps)
    return out


def exact(case, seed):
    k = case["kind"]
    if k == "build":
        if case["H"] * case["W"] > 4e7:
            return None
        img = _images(case, seed)
        if case["u16"]:
            img = (_u16(img).to(torch.int32) & 0xFFFF).double() / 65535.0
        cube = _exact_cube(img.double())
        if case["dtype"] == "f32":
            return cube
        return F.pad(cube.view(2, 6, case["H"], case["W"]).permute(0, 2, 3, 1), (0, 2)).contiguous()
    if k in ("match", "register", "register_host"):
        ref, sen, pts = _images(case, seed)
        ref, sen = _exact_cube(ref.double()), _exact_cube(sen.double())
        return _exact_match(ref, sen, pts, case["m"], case["R"], case["maps"])
    if k == "batch":
        refs, sens, pts = _batch_images(case, seed)
        got = [_exact_match(_exact_cube(r.double()), _exact_cube(t.double()), p, l[3], l[4], False)
               for r, t, p, l in zip(refs, sens, pts, _batch_layout(case))]
        out = {f: torch.cat([g[f] for g in got]) for f in ("ncc", "sub_dx", "sub_dy")}
        out.update(dx=None, dy=None, status=None)
        return out
    if k == "rectify":
        img, M = _rectify_inputs(case, seed)
        img, (H, W) = img.double(), img.shape
        ys, xs = torch.meshgrid(torch.arange(H, device=DEV).double(), torch.arange(W, device=DEV).double(),
                                indexing="ij")
        q = torch.einsum("ij,jyx->iyx", torch.linalg.inv(M), torch.stack([xs, ys, torch.ones_like(xs)]))
        u, v = q[0] / q[2], q[1] / q[2]
        inside = (u >= 0) & (u <= W - 1) & (v >= 0) & (v <= H - 1)
        i, j = v.floor().clamp(0, max(H - 2, 0)).long(), u.floor().clamp(0, max(W - 2, 0)).long()
        fy, fx = v - i, u - j
        i1, j1 = (i + 1).clamp_max(H - 1), (j + 1).clamp_max(W - 1)
        val = (img[i, j] * (1 - fx) + img[i, j1] * fx) * (1 - fy) + (img[i1, j] * (1 - fx) + img[i1, j1] * fx) * fy
        return torch.where(inside, val, torch.zeros_like(val))
    return None
