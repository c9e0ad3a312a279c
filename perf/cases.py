"""Performance cases of the light-field library: what a user's program has it do, through its tensor API.

``listed()`` names the cases, ``draw(rng)`` gives others of the same ranges, ``prepare(case, seed)`` makes what a
program holds before the call, ``run(state)`` is one pass, ``work(case)`` the bytes and operations the pass cannot
do without, and ``exact(case, seed)`` the pass's result in 64 bits by plain torch. A case is a dict of plain values;
``kind`` says which entry point it stands for:

* ``render``: views of a light-field table (``LightField.render``), FP32, FP16 or E4M3 texels;
* ``fit``: the forward and backward of a table fit (``torch_api.render`` under autograd, or with ``search`` the
  backward that searches the neighbours again);
* ``precompute``: the light field of a volume scene (``precompute_table``);
* ``volume``: the direct render of that scene (``render_volume``);
* ``post_filter``: the learned filter of a rendered image (``PostFilter``);
* ``quantize``: the storage form of a table (``quantize_table``).

Views look at the sphere's centre from ``near`` .. ``far`` radii; their sizes and distances follow from the case
(``layout``), their directions, the tables and the scenes from the seed.
"""
from __future__ import annotations

import math
import random
from types import SimpleNamespace

import torch

from paper_1903_03837_gb300 import post_filter as pf
from paper_1903_03837_gb300 import torch_api as api

DEV = "cuda"
TAN_Y = math.tan(math.radians(45.0) / 2)     # vertical field of view 45 degrees
LOBES = 16
FILTER = [("W1", (16, 4, 3, 3)), ("b1", (16,)), ("W2", (16, 16, 3, 3)), ("b2", (16,)), ("W3", (3, 16, 3, 3)), ("b3", (3,))]
GOLDEN = (math.sqrt(5.0) + 1.0) / 2.0
FRAC_HI = int(0.61803398874989484820 * 2**26) / 2**26        # Phi - 1 in two parts: i * FRAC_HI is exact
FRAC_LO = 0.61803398874989484820458683436563811772 - FRAC_HI


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _render(name, M, N, C, dtype, w, h, views=1, near=3.0, far=3.0, k=5, upper=False, half=False, idx=False, stereo=False,
            mixed=False, persistent=False, R=1.0, off=0.0, layout=0):
    c = dict(kind="render", M=M, N=N, C=C, dtype=dtype, w=w, h=h, views=views, near=near, far=far, k=k, upper=upper,
             half=half, idx=idx, stereo=stereo, mixed=mixed, persistent=persistent, R=R, off=off, layout=layout)
    return dict(c, name=name) if name else c


def _fit(name, M, N, C, w, h, views, near=2.0, far=4.0, search=False, layout=0):
    c = dict(kind="fit", M=M, N=N, C=C, dtype="f32", w=w, h=h, views=views, near=near, far=far, k=5, upper=False,
             stereo=False, mixed=False, search=search, R=1.0, off=0.0, layout=layout)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a preview or thumbnail while a user turns the object: the smallest call, where its latency counts
        _render("preview_rgb_f32", 1024, 256, 3, "f32", 256, 256),
        # one ordinary 1080p frame of a half-precision table
        _render("frame_f16", 65536, 1024, 4, "f16", 1920, 1080, near=2.5, far=2.5),
        # a rendering service's batch: 64 views of many clients, stereo headsets and uneven windows, one call
        _render("batch_f16", 16384, 512, 4, "f16", 1440, 1600, views=64, near=1.5, far=4.0, mixed=True, persistent=True,
                layout=7),
        # the largest frame: a 4K stereo pair of the largest table
        _render("orbit_stereo_4k_e4m3", 262144, 4096, 4, "e4m3", 3840, 2160, views=2, stereo=True),
        # the paper's own table shape, upper hemisphere only, a headset's stereo pair in half precision for read-back
        _render("paper_upper_e4m3_half", 12288, 23576, 4, "e4m3", 1280, 720, views=2, near=2.5, far=2.5, upper=True,
                half=True, stereo=True),
        # nearest sampling (the paper's Fig. 2) with the indices kept, odd sizes, a moved and scaled sphere
        _render("nearest_odd_f32", 20011, 997, 4, "f32", 1021, 767, near=2.2, far=2.2, k=1, idx=True, R=2.5, off=0.7),
        # nine neighbours on an odd window of an FP32 table
        _render("nine_odd_f32", 65536, 1024, 4, "f32", 1367, 769, near=2.5, far=2.5, k=9),
        # one step of fitting a table to 32 target views: forward and backward
        _fit("fit_rgb_f32", 16384, 512, 3, 512, 512, 32, layout=3),
        # the light field of a new scene, four jittered samples a texel
        dict(name="precompute_rgba", kind="precompute", M=16384, N=512, rows=16384, C=4, blobs=8, spp=4, steps=64, jitter=True,
             R=1.0),
        # ground-truth images of the scene for the filter's training and for checks
        dict(name="volume_views", kind="volume", w=512, h=512, views=8, near=2.0, far=4.0, C=4, blobs=8, steps=64, R=1.0,
             off=0.0, stereo=False, mixed=False, layout=5),
        # the learned filter on a 1080p frame
        dict(name="post_filter_1080p", kind="post_filter", w=1920, h=1080, views=1, near=2.5, far=2.5, C=4, R=1.0, off=0.0,
             stereo=False, mixed=False, layout=0),
        # a finished table stored as E4M3
        dict(name="quantize_e4m3", kind="quantize", M=65536, N=1024, C=4, dtype="e4m3"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _table_size(rng, most_bytes, texel_bytes, lo_m=200, hi_m=262144, lo_n=100, hi_n=23576):
    while True:
        M, N = _log_int(rng, lo_m, hi_m), _log_int(rng, lo_n, hi_n)
        if M * N * texel_bytes <= most_bytes:
            return M, N


def draw(rng):
    kind = rng.choice(["render"] * 6 + ["fit"] * 2 + ["precompute", "volume", "post_filter", "quantize"])
    layout = rng.randrange(1 << 16)
    R, off = (1.0, 0.0) if rng.random() < 0.6 else (round(rng.uniform(0.3, 5.0), 3), round(rng.uniform(0.1, 2.0), 3))
    if kind == "render":
        dtype = rng.choice(["f32", "f16", "e4m3"])
        k = rng.choice([5, 5, 5, 5, 1, 9])
        C = rng.choice([3, 4]) if dtype == "f32" else 4
        M, N = _table_size(rng, 4 << 30, C * {"f32": 4, "f16": 2, "e4m3": 1}[dtype])
        w, h = _log_int(rng, 31, 3840), _log_int(rng, 31, 2160)
        views = rng.choice([1, 1, 1, 2, 2, _log_int(rng, 3, 70)])
        views = max(1, min(views, (6_000_000 if k == 9 else 30_000_000) // (w * h)))
        near = round(rng.uniform(1.5, 4.0), 3)
        return _render(None, M, N, C, dtype, w, h, views=views, near=near, far=round(rng.uniform(near, 4.0), 3), k=k,
                       upper=rng.random() < 0.2, half=k != 9 and rng.random() < 0.25, idx=rng.random() < 0.25,
                       stereo=views == 2, mixed=views > 4 and rng.random() < 0.5, persistent=rng.random() < 0.25,
                       R=R, off=off, layout=layout)
    if kind == "fit":
        C = rng.choice([3, 3, 4])
        M, N = _table_size(rng, 256 << 20, 4 * C, hi_m=65536, hi_n=4096)
        w, h = _log_int(rng, 31, 1024), _log_int(rng, 31, 1024)
        views = max(1, min(_log_int(rng, 1, 40), 8_000_000 // (w * h)))
        return _fit(None, M, N, C, w, h, views, search=rng.random() < 0.3, layout=layout)
    if kind == "precompute":
        blobs, spp, steps = rng.randint(1, 16), rng.randint(1, 8), _log_int(rng, 8, 128)
        while True:
            M, N = _log_int(rng, 200, 65536), _log_int(rng, 100, 4096)
            if M * N * spp * steps * (blobs + 2) <= 16384 * 512 * 4 * 64 * 9:
                break
        return dict(kind=kind, M=M, N=N, rows=M if rng.random() < 0.7 else M // 2, C=rng.choice([3, 4]), blobs=blobs,
                    spp=spp, steps=steps, jitter=rng.random() < 0.8, R=R)
    if kind == "volume":
        w, h = _log_int(rng, 31, 1920), _log_int(rng, 31, 1080)
        views = max(1, min(_log_int(rng, 1, 16), 4_000_000 // (w * h)))
        near = round(rng.uniform(1.5, 4.0), 3)
        return dict(kind=kind, w=w, h=h, views=views, near=near, far=round(rng.uniform(near, 4.0), 3), C=rng.choice([3, 4]),
                    blobs=rng.randint(1, 16), steps=_log_int(rng, 8, 128), R=R, off=off, stereo=False, mixed=False,
                    layout=layout)
    if kind == "post_filter":
        w, h = _log_int(rng, 31, 3840), _log_int(rng, 31, 2160)
        views = max(1, min(_log_int(rng, 1, 40), 12_000_000 // (w * h)))
        near = round(rng.uniform(1.5, 4.0), 3)
        return dict(kind=kind, w=w, h=h, views=views, near=near, far=round(rng.uniform(near, 4.0), 3), C=rng.choice([3, 4]),
                    R=R, off=off, stereo=False, mixed=views > 4 and rng.random() < 0.5, layout=layout)
    C = rng.choice([3, 4])
    M, N = _table_size(rng, 2 << 30, 4 * C)
    return dict(kind=kind, M=M, N=N, C=C, dtype=rng.choice(["f16", "e4m3"]))


# ---------------------------------------------------------------------------
# cameras
# ---------------------------------------------------------------------------
def _layout(case):
    """[(width, height, distance in radii)] of the case's views."""
    r = random.Random(case["layout"])
    n, out = case["views"], []
    for v in range(n):
        w, h = case["w"], case["h"]
        if case["mixed"] and v >= n // 2:                  # the second half: windows of uneven size
            w, h = r.randint(max(16, w // 6), w), r.randint(max(16, h // 6), h)
        d = r.uniform(case["near"], case["far"])
        if (case["stereo"] or (case["mixed"] and v < n // 2)) and v % 2 == 1:
            d = out[-1][2]                                 # the right eye of a pair
        out.append((w, h, d))
    return out


def _f32(v):
    return tuple(float(x) for x in torch.tensor(list(v), dtype=torch.float64).to(torch.float32))


def _unit(v):
    n = math.sqrt(sum(x * x for x in v))
    return [x / n for x in v]


def _cross(a, b):
    return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]


def _centre(case):
    off = case.get("off", 0.0)
    return (off, -1.5 * off, 0.25 * off)


def _views(case, seed):
    """The case's cameras, looking at the centre from random directions; pairs share one, their eyes 0.064 R apart."""
    r = random.Random(seed * 7919 + 17)
    R, O = case["R"], _centre(case)
    out, offset, pair = [], 0, None
    for v, (w, h, dist) in enumerate(_layout(case)):
        paired = case["stereo"] or (case["mixed"] and v < case["views"] // 2)
        if not (paired and v % 2 == 1):
            pair = _unit([r.gauss(0, 1), r.gauss(0, 1), abs(r.gauss(0, 1)) if case.get("upper") else r.gauss(0, 1)])
        fwd = [-x for x in pair]
        right = _unit(_cross(fwd, [0.0, 0.0, 1.0] if abs(fwd[2]) <= 0.999 else [0.0, 1.0, 0.0]))
        side = 0.0 if not paired else (-0.032 * R if v % 2 == 0 else 0.032 * R)
        eye = [O[k] + R * dist * pair[k] + side * right[k] for k in range(3)]
        tx, ty = _f32((TAN_Y * w / h, TAN_Y))
        out.append(SimpleNamespace(eye=_f32(eye), right=_f32(right), up=_f32(_cross(right, fwd)), forward=_f32(fwd),
                                   tan_half_x=tx, tan_half_y=ty, width=w, height=h, out_offset=offset))
        offset += w * h
    return out


def _pixels(views):
    return sum(v.width * v.height for v in views)


# ---------------------------------------------------------------------------
# tables and scenes
# ---------------------------------------------------------------------------
def _points(n):
    """Spherical-Fibonacci points [n, 3] in 64 bits."""
    i = torch.arange(n, dtype=torch.float64, device=DEV)
    turn = torch.frac(torch.frac(i * FRAC_HI) + i * FRAC_LO)
    z = 1.0 - (2.0 * i + 1.0) / n
    s = torch.sqrt((1.0 - z) * (1.0 + z))
    return torch.stack([torch.cos(2 * math.pi * turn) * s, torch.sin(2 * math.pi * turn) * s, z], 1)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 6007 + 29)
    return g


def _table_rows(M, N, C, rows, seed):
    """FP32 blocks of rows of a smooth non-negative radiance field with a little noise: lobes over the origin and the
    exit point, as light from a few sources over a glossy object has it."""
    g = _gen(seed)
    axes = torch.nn.functional.normalize(torch.randn(2, LOBES, 3, generator=g, device=DEV, dtype=torch.float64), dim=2)
    sharp = 2.0 + 18.0 * torch.rand(2, LOBES, generator=g, device=DEV, dtype=torch.float64)
    col = torch.rand(LOBES, C, generator=g, device=DEV)
    a = torch.exp(sharp[0] * (_points(M)[:rows] @ axes[0].T - 1.0)).float()                     # [rows, L]
    b = torch.exp(sharp[1] * (_points(N) @ axes[1].T - 1.0)).float()                            # [N, L]
    b = (b[:, None, :] * col.T[None]).reshape(N * C, LOBES).T.contiguous()                      # [L, N C]
    step = max(1, (1 << 26) // (N * C))
    for r0 in range(0, rows, step):
        t = a[r0:r0 + step] @ b
        yield r0, t + 0.01 * torch.rand(t.shape, generator=g, device=DEV)


def _table(M, N, C, dtype, rows, seed):
    """(texels, scales): the FP32 table, or its row-scaled codes as the storage forms define them."""
    if dtype == "f32":
        T, scales = torch.empty((rows, N, C), device=DEV), None
        for r0, t in _table_rows(M, N, C, rows, seed):
            T[r0:r0 + len(t)] = t.view(-1, N, C)
        return T, scales
    codes = torch.empty((rows, N, C), dtype=torch.int16 if dtype == "f16" else torch.uint8, device=DEV)
    scales = torch.empty(rows, device=DEV)
    for r0, t in _table_rows(M, N, C, rows, seed):
        s = t.amax(1) / (448.0 if dtype == "e4m3" else 1.0)
        q = (t / s[:, None]).to(torch.float8_e4m3fn if dtype == "e4m3" else torch.float16)
        codes[r0:r0 + len(t)] = q.view(codes.dtype).view(-1, N, C)
        scales[r0:r0 + len(t)] = s
    return codes, scales


def _scene(case, seed):
    r = random.Random(seed * 131 + 5)
    B, R, O = case["blobs"], case["R"], _centre(case)
    mu, width, dens, emit = [], [], [], []
    for _ in range(B):
        u, rad = _unit([r.gauss(0, 1) for _ in range(3)]), 0.6 * R * r.random() ** (1 / 3)
        mu.append(_f32([O[k] + rad * u[k] for k in range(3)]))
        width.append(_f32([R * r.uniform(0.08, 0.25)])[0])
        dens.append(_f32([r.uniform(2.0, 12.0) / R])[0])
        emit.append(_f32([r.random() for _ in range(3)]))
    return SimpleNamespace(mu=mu, width=width, dens=dens, emit=emit, bg0=(0.125, 0.125, 0.1875), bg1=(0.25, 0.375, 0.5),
                           spp=case.get("spp", 1), steps=case["steps"], jitter=int(case.get("jitter", False)), seed=seed,
                           R=R, O=O)


def _image(case, views, seed):
    """[P, C] FP32 image as a render leaves it: smooth colours on hit pixels, 0 elsewhere; channel 3 an opacity."""
    g = _gen(seed)
    C, out = case["C"], []
    wave = 4.0 + 60.0 * torch.rand(C, 2, generator=g, device=DEV)
    phase = 6.28 * torch.rand(C, generator=g, device=DEV)
    for v in views:
        hit = _hits(case, v)[2].view(v.height, v.width)
        y = torch.linspace(0, 1, v.height, device=DEV)[:, None, None]
        x = torch.linspace(0, 1, v.width, device=DEV)[None, :, None]
        t = 0.5 + 0.4 * torch.sin(wave[:, 0] * x + wave[:, 1] * y + phase)
        t = t + 0.02 * torch.rand(t.shape, generator=g, device=DEV)
        out.append((t * hit[..., None]).view(-1, C))
    return torch.cat(out)


def _filter_weights(seed):
    """Weights of a trained filter's size: He-scaled hidden layers, a small correction in the last."""
    g = torch.Generator().manual_seed(seed + 41)
    parts = [torch.randn(s, generator=g) * (0.05 if name.startswith("b") else
             math.sqrt(2.0 / (s[1] * 9)) if name != "W3" else 0.02) for name, s in FILTER]
    return torch.cat([p.reshape(-1) for p in parts])


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
def prepare(case, seed):
    s = SimpleNamespace(case=case, kind=case["kind"])
    if s.kind in ("render", "fit"):
        rows = case["M"] // 2 if case["upper"] else case["M"]
        table, scales = _table(case["M"], case["N"], case["C"], case["dtype"], rows, seed)
        s.views = _views(case, seed)
        s.lf = api.LightField(table, case["dtype"], scales=scales, R=case["R"], O=_centre(case), borrow=True,
                              n_origins=case["M"], upper=case["upper"], k_nearest=case["k"])
        if case.get("persistent"):
            s.lf.set_launch(order=1, persistent=1)
        if s.kind == "fit":
            s.table = table.requires_grad_(True)
            s.grad = 1e-3 * torch.randn((_pixels(s.views), case["C"]), generator=_gen(seed + 1), device=DEV)
    elif s.kind in ("precompute", "volume"):
        s.scene = _scene(case, seed)
        s.views = _views(case, seed) if s.kind == "volume" else None
    elif s.kind == "post_filter":
        s.views = _views(case, seed)
        s.image = _image(case, s.views, seed)
        s.filter = pf.PostFilter(_filter_weights(seed))
    else:
        s.table = _table(case["M"], case["N"], case["C"], "f32", case["M"], seed)[0]
    return s


def run(s):
    c = s.case
    if s.kind == "render":
        image, idx = s.lf.render(s.views, with_idx=c["idx"], half=c["half"])
        return {"image": image, "idx": idx}
    if s.kind == "fit":
        if c["search"]:
            image, _ = s.lf.render(s.views)
            return {"image": image, "grad": s.lf.render_backward(s.views, s.grad)}
        image = api.render(s.table, s.lf, s.views)
        return {"image": image, "grad": torch.autograd.grad(image, s.table, grad_outputs=s.grad)[0]}
    if s.kind == "precompute":
        return {"table": api.precompute_table(s.scene, c["M"], c["N"], c["C"], rows=c["rows"])}
    if s.kind == "volume":
        return {"image": api.render_volume(s.scene, s.views, c["C"])}
    if s.kind == "post_filter":
        return {"image": s.filter(s.views, s.image, R=c["R"], O=_centre(c))}
    codes, scales = api.quantize_table(s.table, c["dtype"])
    return {"codes": codes, "scales": scales}


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _disc_share(w, h, dist):
    """Share of a view's pixels whose ray meets the sphere seen from `dist` radii (the disc may exceed the view)."""
    r2, tx, n = 1.0 / (dist * dist - 1.0), TAN_Y * w / h, 96
    inside = 0.0
    for j in range(n):
        y = TAN_Y * (2 * j + 1 - n) / n
        inside += min(tx, math.sqrt(max(0.0, r2 - y * y))) / tx
    return inside / n


def work(case):
    kind, C = case["kind"], case.get("C", 4)
    rays = hits = caps = 0.0
    if kind not in ("precompute", "quantize"):
        for w, h, d in _layout(case):
            rays += w * h
            hits += w * h * _disc_share(w, h, d)
            caps = max(caps, 0.5 * (1.0 - 1.0 / d))              # share of the sphere that faces the eye
    if kind in ("render", "fit"):
        texel = case["C"] * {"f32": 4, "f16": 2, "e4m3": 1}[case["dtype"]]
        K = case["k"]
        # taps inside both kernel radii: pi of each set's neighbours on average (all of them for nearest sampling)
        taps = 1.0 if K == 1 else min(math.pi, K) ** 2
        # distinct texels: no more than the taps, the table, or the facing origins times a kernel's directions and
        # the directions that fall into one origin's cell
        per_origin = taps + 9.0 * case["N"] / case["M"]
        texels = min(hits * taps, case["M"] * case["N"], len(_layout(case)) * caps * case["M"] * per_origin)
        out = rays * C * (2 if case.get("half") else 4) + (rays * 8 * K if case.get("idx") else 0)
        flops = 40.0 * rays + hits * (2 * (8 * (K + 1) + 6 * K) + 2 * taps * C)
        if kind == "render":
            return {"bytes": out + texels * texel, "flops": flops}
        # forward, then the image gradient read and the whole gradient table written
        return {"bytes": out + texels * texel + rays * C * 4 + case["M"] * case["N"] * C * 4,
                "flops": flops + hits * (60 + 2 * taps * C)}
    if kind == "precompute":
        n = case["rows"] * case["N"]
        return {"bytes": n * C * 4.0, "flops": float(n) * case["spp"] * case["steps"] * (5 * case["blobs"] + 8)}
    if kind == "volume":
        return {"bytes": rays * C * 4, "flops": 40 * rays + hits * case["steps"] * (5 * case["blobs"] + 8)}
    if kind == "post_filter":
        return {"bytes": 2.0 * rays * C * 4, "flops": 2.0 * rays * 9 * (4 * 16 + 16 * 16 + 16 * 3)}
    n = case["M"] * case["N"]
    return {"bytes": n * C * 4.0 + n * 4.0 * (2 if case["dtype"] == "f16" else 1) + case["M"] * 4, "flops": 2.0 * n * C}


# ---------------------------------------------------------------------------
# exact: the definitions in 64 bits (the camera ray and its hits are FP32 by definition, one operation at a time)
# ---------------------------------------------------------------------------
def _hits(case, v):
    """FP32 unit directions, front hits, hit mask and back hits of a view's pixels, in raster order."""
    R, O = _f32([case["R"]])[0], _f32(_centre(case))
    sw, sh = _f32((2.0 / v.width, 2.0 / v.height))
    x = torch.arange(v.width, device=DEV, dtype=torch.float32) + 0.5
    y = torch.arange(v.height, device=DEV, dtype=torch.float32) + 0.5
    nx = ((x * sw - 1.0) * v.tan_half_x)[None, :]
    ny = ((1.0 - y * sh) * v.tan_half_y)[:, None]
    d = [((nx * v.right[k] + v.forward[k]) + ny * v.up[k]).reshape(-1) for k in range(3)]
    il = 1.0 / torch.sqrt((d[0] * d[0] + d[1] * d[1]) + d[2] * d[2])
    d = [x * il for x in d]
    e = torch.tensor(v.eye, device=DEV)
    f = e - torch.tensor(O, device=DEV)
    b = (f[0] * d[0] + f[1] * d[1]) + f[2] * d[2]
    r = torch.tensor(R, device=DEV)
    c = ((f[0] * f[0] + f[1] * f[1]) + f[2] * f[2]) - r * r
    disc = b * b - c
    sq = torch.sqrt(disc.clamp_min(0.0))
    near, far = -b - sq, -b + sq
    hit = (disc > 0) & (near > 0)
    ho = torch.stack([near * d[k] + v.eye[k] for k in range(3)], 1)
    hd = torch.stack([far * d[k] + v.eye[k] for k in range(3)], 1)
    return torch.stack(d, 1), ho, hit, hd


def _smallest(d2, cand, K):
    """The K smallest of each row in order (indices from `cand`)."""
    ids, ds = [], []
    for _ in range(K):
        m, a = d2.min(1)
        ids.append(cand.gather(1, a[:, None])[:, 0])
        ds.append(m)
        d2.scatter_(1, a[:, None], math.inf)
    return torch.stack(ids, 1), torch.stack(ds, 1)


def _nearest(q, pts, K):
    """Indices and squared chords of the K nearest points to unit vectors q (fewer points: index -1, distance inf)."""
    n = len(pts)
    if n <= 512:
        d2 = sum((q[:, k:k + 1] - pts[None, :, k]) ** 2 for k in range(3))
        if n < K:
            d2 = torch.nn.functional.pad(d2, (0, K - n), value=math.inf)
        cand = torch.arange(d2.shape[1], device=DEV).expand(len(q), -1)
        ids, ds = _smallest(d2, cand, K)
        return torch.where(torch.isinf(ds), -1, ids), ds
    # corners of the local Fibonacci lattice around q; next to a pole the points nearest the pole
    z = q[:, 2]
    zone = torch.log(math.sqrt(5.0) * math.pi * n * (1 - z * z).clamp_min(1e-12)) / math.log(GOLDEN ** 2)
    zone = zone.floor().clamp(2, 36).long()
    fib = [0, 1]
    while len(fib) < 40:
        fib.append(fib[-1] + fib[-2])
    F = torch.tensor(fib, device=DEV)
    E = torch.tensor([-(-1.0 / GOLDEN) ** k for k in range(40)], device=DEV, dtype=torch.float64)
    F0, F1, e0, e1 = F[zone], F[zone + 1], E[zone], E[zone + 1]
    turn = torch.atan2(q[:, 1], q[:, 0]) / (2 * math.pi)
    at = (n * (1 - z) - 1) / 2
    det = e0 * F1 - e1 * F0
    u = torch.round((F1 * turn - e1 * at) / det).long()
    w = torch.round((e0 * at - F0 * turn) / det).long()
    ids, ds = [], []
    du = torch.arange(-3, 4, device=DEV)
    cand = ((u[:, None, None] + du[None, :, None]) * F0[:, None, None]
            + (w[:, None, None] + du[None, None, :]) * F1[:, None, None]).reshape(len(q), 49)
    pole = (at < 24) | (at > n - 25)
    bad = (cand < 0) | (cand >= n)
    c = cand.clamp(0, n - 1)
    d2 = sum((q[:, k:k + 1] - pts[:, k][c]) ** 2 for k in range(3)).masked_fill_(bad, math.inf)
    ids, ds = _smallest(d2, c, K)
    for top in (True, False):
        sel = (pole & ((z > 0) == top)).nonzero()[:, 0]
        if len(sel):
            cp = torch.arange(128, device=DEV) + (0 if top else n - 128)
            d2 = sum((q[sel, k:k + 1] - pts[cp, k][None]) ** 2 for k in range(3))
            ids[sel], ds[sel] = _smallest(d2, cp.expand(len(sel), -1), K)
    return ids, ds


def _weights(ids, d2, n, keep):
    """Tent weights of the kernel radius sqrt(4 pi / n), normalised over the kept neighbours; the nearest kept one
    where all are outside."""
    w = (1.0 - d2.sqrt() / math.sqrt(4 * math.pi / n)).clamp_min(0.0)
    ok = (ids >= 0) & (ids < keep)
    w = torch.where(ok, w, 0.0)
    s = w.sum(1, keepdim=True)
    first = torch.zeros_like(w).scatter_(1, ok.int().argmax(1, keepdim=True), 1.0)
    return torch.where(s > 0, w / s.clamp_min(1e-300), first), ok.any(1)


def _exact_light_field(case, seed, grad=None):
    M, N, C, K = case["M"], case["N"], case["C"], case["k"]
    rows = M // 2 if case["upper"] else M
    table, scales = _table(M, N, C, case["dtype"], rows, seed)
    flat = table.view(rows * N, C)
    po, pd = _points(M), _points(N)
    O = torch.tensor(_centre(case), device=DEV, dtype=torch.float64)
    views = _views(case, seed)
    image = torch.zeros((_pixels(views), C), device=DEV, dtype=torch.float64)
    total = torch.zeros((rows * N, C), device=DEV, dtype=torch.float64) if grad is not None else None
    for v in views:
        _, ho, hit, hd = _hits(case, v)
        at = hit.nonzero()[:, 0]
        for p in at.split(1 << 18):
            sets = []
            for h, pts, keep in ((ho, po, rows), (hd, pd, N)):
                q = h[p].double() - O
                ids, d2 = _nearest(torch.nn.functional.normalize(q, dim=1), pts, K)
                if K == 1:
                    wgt, ok = torch.ones_like(d2), ids[:, 0] < keep
                else:
                    wgt, ok = _weights(ids, d2, len(pts), keep)
                sets.append((ids, wgt, ok))
            (i, wo, seen), (j, wd, _) = sets
            i, j = torch.where(wo > 0, i, 0).clamp(0, rows - 1), j.clamp_min(0)
            W = (wo[:, :, None] * wd[:, None, :] * seen[:, None, None]).reshape(len(p), -1)
            tap = (i[:, :, None] * N + j[:, None, :]).reshape(len(p), -1)
            t = flat[tap]
            if case["dtype"] == "e4m3":
                t = t.view(torch.float8_e4m3fn).float()
            elif case["dtype"] == "f16":
                t = t.view(torch.float16)
            t = t.double()
            if scales is not None:
                t = t * scales[i].double()[:, :, None].expand(-1, -1, K).reshape(len(p), -1, 1)
            image[v.out_offset + p] = (W[:, :, None] * t).sum(1)
            if grad is not None:
                total.index_add_(0, tap.view(-1), (W[:, :, None] * grad[v.out_offset + p].double()[:, None]).view(-1, C))
    return image, None if total is None else total.view(rows, N, C)


def _march(scene, o, d, length):
    """Radiance and opacity along o + t d, t in [0, length], by the midpoint rule, in 64 bits."""
    def const(v):
        return torch.tensor(v, device=DEV, dtype=torch.float64)
    mu, width, dens, emit = const(scene.mu), const(scene.width), const(scene.dens), const(scene.emit)
    dt = length / scene.steps
    f = o[:, None, :] - mu
    along = (f * d[:, None, :]).sum(2)
    perp = torch.linalg.cross(f, d[:, None, :].expand_as(f)).square().sum(2)
    T, sums = torch.ones_like(length), torch.zeros_like(along)
    for k in range(scene.steps):
        t = (k + 0.5) * dt
        g = dens * torch.exp(-(perp + (along + t[:, None]).square()) / (2 * width * width))
        x = g.sum(1) * dt
        step = torch.where(x > 0, -torch.expm1(-x) / x.clamp_min(1e-300), 1.0) * dt
        sums += g * (T * step)[:, None]
        T = T * torch.exp(-x)
    bg = const(scene.bg0) + const(scene.bg1) * (0.5 * (1 + d[:, 2:]))
    return torch.cat([sums @ emit + T[:, None] * bg, 1 - T[:, None]], 1)


def _splitmix(seed, ctr):
    """Outputs `ctr` + 1 of the SplitMix64 stream, as the top 24 bits times 2^-24."""
    def signed(x):
        return x - (1 << 64) if x >= 1 << 63 else x

    def shift(x, k):
        return (x >> k) & ((1 << (64 - k)) - 1)
    z = seed + (ctr + 1) * signed(0x9E3779B97F4A7C15)
    z = (z ^ shift(z, 30)) * signed(0xBF58476D1CE4E5B9)
    z = (z ^ shift(z, 27)) * signed(0x94D049BB133111EB)
    return shift(z ^ shift(z, 31), 40).double() * 2.0 ** -24


def _exact_precompute(case, seed):
    M, N, rows, R = case["M"], case["N"], case["rows"], case["R"]
    scene = _scene(case, seed)
    O = torch.tensor(scene.O, device=DEV, dtype=torch.float64)
    po, pd = _points(M), _points(N)
    out = torch.empty((rows * N, case["C"]), device=DEV, dtype=torch.float64)
    for t in torch.arange(rows * N, device=DEV).split(1 << 20):
        i, j = t // N, t % N
        p = po[i]
        d = pd[j] - p
        l2 = d.square().sum(1, keepdim=True)
        d = torch.where(l2 < 1e-24, -p, d / l2.clamp_min(1e-300).sqrt())
        rho = p[:, :2].norm(dim=1)
        e_phi = torch.stack([-p[:, 1], p[:, 0], torch.zeros_like(rho)], 1) / rho[:, None]
        e_theta = torch.stack([p[:, 0] * p[:, 2], p[:, 1] * p[:, 2], -rho * rho], 1) / rho[:, None]
        acc = 0.0
        for s in range(case["spp"]):
            offset = torch.zeros_like(p)
            if case["jitter"]:
                ctr = 2 * (t * case["spp"] + s)
                r = (2 * R / math.sqrt(M)) * _splitmix(seed, ctr).sqrt()
                a = 2 * math.pi * _splitmix(seed, ctr + 1)
                offset = r[:, None] * (torch.cos(a)[:, None] * e_phi + torch.sin(a)[:, None] * e_theta)
            f = R * p + offset
            b = (f * d).sum(1)
            disc = b * b - offset.square().sum(1)
            length = torch.where(disc > 0, (disc.clamp_min(0.0).sqrt() - b).clamp_min(0.0), 0.0)
            acc = acc + _march(scene, O + f, d, length)
        out[t] = (acc / case["spp"])[:, :case["C"]]
    return out.view(rows, N, case["C"])


def _exact_volume(case, seed):
    scene, views = _scene(case, seed), _views(case, seed)
    O = torch.tensor(scene.O, device=DEV, dtype=torch.float64)
    out = torch.zeros((_pixels(views), case["C"]), device=DEV, dtype=torch.float64)
    for v in views:
        d, ho, hit, _ = _hits(case, v)
        at = hit.nonzero()[:, 0]
        o, d = ho[at].double(), d[at].double()
        f = o - O
        b = (f * d).sum(1)
        disc = b * b - (f.square().sum(1) - case["R"] ** 2)
        length = torch.where(disc > 0, disc.clamp_min(0.0).sqrt() - b, 0.0).clamp_min(0.0)
        out[v.out_offset + at] = _march(scene, o, d, length)[:, :case["C"]]
    return out


def _conv3(x, w, b):
    """Zero-padded 3 x 3 cross-correlation of [c, H, W] as nine products of channels."""
    _, H, W = x.shape
    p = torch.nn.functional.pad(x, (1, 1, 1, 1))
    y = b[:, None].expand(-1, H * W).clone()
    for dy in range(3):
        for dx in range(3):
            y += w[:, :, dy, dx] @ p[:, dy:dy + H, dx:dx + W].reshape(x.shape[0], -1)
    return y.view(-1, H, W)


def _exact_filter(case, seed):
    views = _views(case, seed)
    image = _image(case, views, seed).double()
    flat = _filter_weights(seed).to(DEV).double()
    w = [t.view(shape) for t, (_, shape) in zip(flat.split([math.prod(shape) for _, shape in FILTER]), FILTER)]
    out = image.clone()
    for v in views:
        n = slice(v.out_offset, v.out_offset + v.width * v.height)
        hit = _hits(case, v)[2].view(1, v.height, v.width).double()
        rgb = image[n, :3].T.reshape(3, v.height, v.width)
        h = _conv3(torch.cat([rgb, hit]), w[0], w[1]).clamp_min(0.0)
        h = _conv3(h, w[2], w[3]).clamp_min(0.0)
        out[n, :3] = ((rgb + _conv3(h, w[4], w[5])) * hit).reshape(3, -1).T
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "render":
        return {"image": _exact_light_field(case, seed)[0], "idx": None}
    if kind == "fit":
        n = _pixels(_views(case, seed))
        g = 1e-3 * torch.randn((n, case["C"]), generator=_gen(seed + 1), device=DEV)
        image, grad = _exact_light_field(case, seed, g)
        return {"image": image, "grad": grad}
    if kind == "precompute":
        return {"table": _exact_precompute(case, seed)}
    if kind == "volume":
        return {"image": _exact_volume(case, seed)}
    if kind == "post_filter":
        return {"image": _exact_filter(case, seed)}
    table = _table(case["M"], case["N"], case["C"], "f32", case["M"], seed)[0]
    amax = table.abs().amax((1, 2)).double()
    return {"codes": None, "scales": torch.where(amax > 0, amax / (448.0 if case["dtype"] == "e4m3" else 1.0), 1.0)}
