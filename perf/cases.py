"""What is measured: the framework's work as a program calls it, through the
Python entry points of the package.

Kinds of case
  pair     FlowContext.stitch_pair, or flow_pair + blend_pair with a Blend array
  static   flow_pair_static (the allocation-free flow)
  rig      Rig.run: every overlap pair of a 360-degree rig onto one canvas
  coeff    blend_coeff: Eq. (1) on a labelled canvas
  canvas   FlowContext.stitch_canvas: Eq. (1), the flows of the overlap crop, Code 1
  energy   refine.pyramid_energy, forward and backward: one step of the differentiable refinement

Inputs are seeded band-limited textures and copies of them displaced by known
fields (smooth, or piecewise planar with steps as in a scene with several
depths), with sensor noise and the small gains that chromaticity correction
leaves.  `exact` restates the whole path in 64-bit torch.
"""
import math

import torch
import torch.nn.functional as F

from paper_2006_01201_gb300 import binding, refine

DEV = "cuda"
SIGMAS = (1.0, 2.0, 4.0, 8.0)
MIX = ((0.60, 0.25, 0.15), (0.20, 0.60, 0.20), (0.15, 0.25, 0.60))
RIG_WIDTHS = "800,950,1100,1250,1400,1600,1800,2000"
PYR = {"f32": binding.PANO_F32, "bf16": binding.PANO_BF16, "f16": binding.PANO_F16}


def _pair(name, h, w, c, dtype, levels, iters=5, radius=2, pyr="f32", ramp=True, field="parallax"):
    return {"name": name, "kind": "pair", "h": h, "w": w, "c": c, "dtype": dtype, "levels": levels, "iters": iters,
            "radius": radius, "pyr": pyr, "ramp": ramp, "field": field}


def listed():
    return [
        # a preview thumbnail: every level is tiny, launches and latency are the time
        _pair("pair_120x85_rgb_u8", 120, 85, 3, "u8", 3),
        # one camera pair at video-preview size, float input (the small benchmark pair)
        _pair("pair_256x512_gray_f32", 256, 512, 1, "f32", 4, field="smooth"),
        # odd sizes, a float RGB pipeline with its own Blend array, wider window and fewer steps
        _pair("pair_1531x677_rgb_f32_r3", 1531, 677, 3, "f32", 5, iters=3, radius=3, ramp=False),
        # one full-resolution overlap of a panorama (the headline benchmark pair)
        _pair("pair_4000x1500_rgb_u8", 4000, 1500, 3, "u8", 6),
        # a survey-camera overlap far beyond the panorama's, one channel, 16-bit pyramids
        _pair("pair_8000x6000_gray_u8_f16", 8000, 6000, 1, "u8", 7, pyr="f16"),
        # flow inside a frame loop that may not allocate: one-megapixel class strips
        {"name": "static_960x1000_gray_u8", "kind": "static", "h": 960, "w": 1000, "c": 1, "dtype": "u8", "levels": 5,
         "iters": 5, "radius": 2, "field": "smooth"},
        # all pairs of a 360-degree rig per frame, from a CUDA graph
        {"name": "rig_8x4000_rgb_u8", "kind": "rig", "h": 4000, "widths": RIG_WIDTHS, "c": 3, "dtype": "u8", "levels": 6,
         "pyr": "f32", "graph": True, "canvas_h": 4000, "canvas_w": 9000},
        # a small rig at live-preview size, bfloat16 pyramids, enqueued directly
        {"name": "rig_4x731_rgb_u8_bf16", "kind": "rig", "h": 731, "widths": "150,187,233,310", "c": 3, "dtype": "u8",
         "levels": 5, "pyr": "bf16", "graph": False, "canvas_h": 750, "canvas_w": 1700},
        # Eq. (1) of a whole panorama, once per rig geometry
        {"name": "coeff_4000x9000", "kind": "coeff", "h": 4000, "w": 9000},
        # the stitch of one pair onto its canvas, every step of Section III-C
        {"name": "canvas_2000x2900_rgb_u8", "kind": "canvas", "h": 2000, "w": 2900, "x0": 950, "cw": 1000, "c": 3,
         "dtype": "u8", "levels": 6},
        # refinement by gradient steps: energy and all gradients at full resolution
        {"name": "energy_1024x1024_l0", "kind": "energy", "h": 1024, "w": 1024, "level": 0},
        # the same step at a coarser level of an odd-sized pair: REDUCE and its transpose on the way
        {"name": "energy_1777x1210_l2", "kind": "energy", "h": 1777, "w": 1210, "level": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _levels(h, w, rng):
    top = max(1, min(7, int(math.log2(max(2, min(h, w)) / 10.0)) + 1))
    return rng.randint(max(1, top - 1), top)


def draw(rng):
    kind = rng.choice(["pair", "pair", "pair", "static", "rig", "coeff", "canvas", "energy"])
    if kind == "pair":
        h, w = _log(rng, 48, 8000), _log(rng, 48, 5000)
        c, dtype = rng.choice([1, 3]), rng.choice(["u8", "f32"])
        iters = rng.choice([2, 3, 4, 5, 5, 5, 8] if h * w <= 1000000 else [2, 3, 4, 5, 5, 5])
        case = _pair("", h, w, c, dtype, _levels(h, w, rng), iters, rng.choice([1, 2, 2, 2, 3]),
                     rng.choice(["f32", "f32", "bf16", "f16"]), rng.random() < 0.7, rng.choice(["parallax", "smooth"]))
        del case["name"]
        return case
    if kind == "static":
        h, w = _log(rng, 48, 1000), _log(rng, 48, 1000)
        return {"kind": "static", "h": h, "w": w, "c": rng.choice([1, 3]), "dtype": rng.choice(["u8", "f32"]),
                "levels": _levels(h, w, rng), "iters": rng.choice([3, 5]), "radius": 2, "field": rng.choice(["parallax", "smooth"])}
    if kind == "rig":
        h, n = _log(rng, 200, 4000), rng.randint(2, 8)
        widths = [_log(rng, 60, max(80, h // 2)) for _ in range(n)]
        return {"kind": "rig", "h": h, "widths": ",".join(map(str, widths)), "c": 3, "dtype": rng.choice(["u8", "u8", "f32"]),
                "levels": _levels(h, min(widths), rng), "pyr": rng.choice(["f32", "f32", "f16"]), "graph": rng.random() < 0.5,
                "canvas_h": h + rng.randint(0, 40), "canvas_w": int(1.2 * sum(widths)) + rng.randint(0, 9)}
    if kind == "coeff":
        return {"kind": "coeff", "h": _log(rng, 60, 4000), "w": _log(rng, 90, 9000)}
    if kind == "canvas":
        h, w = _log(rng, 100, 3000), _log(rng, 160, 4000)
        x0, cw = w // 3 + rng.randint(0, 7), w // 3 - rng.randint(0, 9)
        return {"kind": "canvas", "h": h, "w": w, "x0": x0, "cw": cw, "c": rng.choice([1, 3]), "dtype": rng.choice(["u8", "f32"]),
                "levels": _levels(h, cw, rng)}
    return {"kind": "energy", "h": _log(rng, 64, 2000), "w": _log(rng, 64, 2000), "level": rng.randint(0, 3)}


# --------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _blur(a, sigma):
    """Separable Gaussian, truncated at 3.5 sigma, reflecting border."""
    n = int(3.5 * sigma + 0.5)
    k = [math.exp(-0.5 * (i / sigma) ** 2) for i in range(-n, n + 1)]
    s = sum(k)
    for _ in range(2):
        p = F.pad(a[None, None], (n, n, 0, 0), mode="reflect")[0, 0]
        acc = torch.zeros_like(a)
        for i, v in enumerate(k):
            acc.add_(p[:, i:i + a.shape[1]], alpha=v / s)
        a = acc.t().contiguous()
    return a


def _texture(g, h, w):
    acc = torch.zeros((h, w), device=DEV)
    for s in SIGMAS:
        f = _blur(torch.randn((h, w), generator=g, device=DEV), s)
        acc += f / f.std()
    acc -= acc.min()
    return acc / acc.max()


def _field(g, h, w, kind, dmax):
    """(dx, dy) of the right strip against the left one."""
    ys = torch.arange(h, device=DEV, dtype=torch.float32)[:, None]
    xs = torch.arange(w, device=DEV, dtype=torch.float32)[None, :]
    if kind == "smooth":
        a = dmax / 4.0
        return (a * torch.sin(2 * math.pi * ys / max(128.0, h / 4)) + 0 * xs,
                0.5 * a * torch.cos(2 * math.pi * xs / max(256.0, w / 4)) + 0 * ys)
    r = torch.rand((4, 3), generator=g, device=DEV)
    k = sum((ys > h * j / 4.0 + 0.1 * xs).long() for j in (1, 2, 3))
    base, sx, sy = 0.25 * dmax + 0.5 * dmax * r[:, 0], 0.2 * dmax * (r[:, 1] - 0.5), 0.2 * dmax * (r[:, 2] - 0.5)
    dx = base[k] + sx[k] * xs / w + sy[k] * ys / h + 0.075 * dmax * torch.sin(2 * math.pi * ys / max(200.0, h / 4.5))
    dx = dx.clamp(0, dmax)
    return dx, 0.1 * dx


def _strips(seed, h, w, c, dtype, kind, levels):
    """Two strips: R(p) = L(p + d(p)), times a gain, plus noise."""
    g = _gen(seed)
    dmax = min(8.0, 0.8 * 2 ** (levels - 1), 0.04 * min(h, w) + 1.0)
    pad = 32
    base = [_texture(g, h + 2 * pad, w + 2 * pad) for _ in range(c)]
    planes = base if c == 1 else [sum(MIX[i][k] * base[k] for k in range(3)) for i in range(3)]
    dx, dy = _field(g, h, w, kind, dmax)
    gx = (torch.arange(w, device=DEV)[None, :] + pad + dx) * (2.0 / (w + 2 * pad - 1)) - 1
    gy = (torch.arange(h, device=DEV)[:, None] + pad + dy) * (2.0 / (h + 2 * pad - 1)) - 1
    grid = torch.stack([gx, gy], -1)[None]
    L, R = [], []
    for p in planes:
        q = F.grid_sample(p[None, None], grid, mode="bicubic", padding_mode="reflection", align_corners=True)[0, 0]
        gain = 0.98 + 0.04 * torch.rand((), generator=g, device=DEV)
        q = q * gain + (2.0 / 255) * torch.randn((h, w), generator=g, device=DEV)
        L.append(p[pad:pad + h, pad:pad + w].clamp(0, 1))
        R.append(q.clamp(0, 1))
    L, R = (torch.stack(v, -1) if c == 3 else v[0] for v in (L, R))
    if dtype == "u8":
        L, R = (torch.round(v * 255).to(torch.uint8) for v in (L, R))
    return L.contiguous(), R.contiguous()


def _labels(seed, h, w, x0=None, x1=None):
    """Area1 | Area3 | Area2 with wavy seams, small holes and, on a whole
    panorama (x0 None), several overlaps; bands of no area above and below."""
    r = torch.rand((8,), generator=_gen(seed + 77), device=DEV).tolist()
    ys = torch.arange(h, device=DEV, dtype=torch.float32)[:, None]
    xs = torch.arange(w, device=DEV, dtype=torch.float32)[None, :]
    lab = torch.zeros((h, w), dtype=torch.uint8, device=DEV)
    if x0 is None:
        n = 1 if w < 1500 else 4 if w > 6000 else 2
        step = w / n
        for k in range(n):
            c = (k + 0.5) * step + 0.03 * step * (r[k % 8] - 0.5)
            half = 0.2 * step
            lo = c - half + 0.04 * step * torch.sin(2 * math.pi * (ys / (0.6 * h) + r[(k + 1) % 8]))
            hi = c + half + 0.04 * step * torch.sin(2 * math.pi * (ys / (0.45 * h) + r[(k + 2) % 8]))
            inside = (xs >= k * step) & (xs < (k + 1) * step)
            a, b = (1, 2) if k % 2 == 0 else (2, 1)
            lab[inside & (xs < lo)] = a
            lab[inside & (xs >= lo) & (xs < hi)] = 3
            lab[inside & (xs >= hi)] = b
        top = (0.03 * h * (1 + torch.sin(2 * math.pi * (xs / (0.7 * w) + r[7])))).floor()
        lab[(ys < top) | (ys >= h - top)] = 0
    else:
        wob = 0.1 * (x1 - x0)
        lo = x0 + wob * 0.5 * (1 + torch.sin(2 * math.pi * (ys / (0.6 * h) + r[0])))
        hi = x1 - wob * 0.5 * (1 + torch.sin(2 * math.pi * (ys / (0.45 * h) + r[1])))
        lab[xs.expand(h, w) < lo] = 1
        lab[(xs >= lo) & (xs < hi)] = 3
        lab[xs.expand(h, w) >= hi] = 2
    for k in range(3):  # a sensor defect: a small hole that no camera covers
        cy, cx = int(h * r[k + 3]), int(w * r[(k + 5) % 8])
        lab[cy:cy + max(1, h // 100), cx:cx + max(1, w // 100)] = 0
    return lab


def _params(case):
    return binding.Params(levels=case["levels"], iters=case.get("iters", 5), radius=case.get("radius", 2),
                          pyr_dtype=PYR[case.get("pyr", "f32")])


def _rig_layout(case):
    widths = [int(v) for v in case["widths"].split(",")]
    return widths, [(k * case["canvas_w"]) // len(widths) for k in range(len(widths))], (case["canvas_h"] - case["h"]) // 2


def _canvas_images(case, seed):
    L, R = _strips(seed, case["h"], case["w"], case["c"], case["dtype"], "parallax", case["levels"])
    return L, R, _labels(seed, case["h"], case["w"], case["x0"], case["x0"] + case["cw"])


def _energy_inputs(case, seed):
    T, J = _strips(seed, case["h"], case["w"], 1, "f32", "smooth", 4)
    h, w = case["h"], case["w"]
    for _ in range(case["level"]):
        h, w = (h + 1) // 2, (w + 1) // 2
    # the flow of a refinement under way: some way off the true field
    g = _gen(seed + 5)
    dx, dy = _field(g, h, w, "smooth", 4.8)
    u = torch.stack([dx, dy], -1) + 0.3 * torch.randn((h, w, 2), generator=g, device=DEV)
    return T, J, u


def prepare(case, seed):
    kind = case["kind"]
    if kind == "pair":
        L, R = _strips(seed, case["h"], case["w"], case["c"], case["dtype"], case["field"], case["levels"])
        blend = None if case["ramp"] else _blend_map(case, seed)
        return {"case": case, "ctx": binding.FlowContext(_params(case), case["h"], case["w"], case["c"]), "L": L, "R": R,
                "blend": blend}
    if kind == "static":
        L, R = _strips(seed, case["h"], case["w"], case["c"], case["dtype"], case["field"], case["levels"])
        out = tuple(torch.empty((case["h"], case["w"], 2), device=DEV) for _ in range(2))
        return {"case": case, "params": _params(case), "L": L, "R": R, "out": out}
    if kind == "rig":
        widths, x0, y0 = _rig_layout(case)
        pairs = [_strips(seed * 16 + k, case["h"], w, case["c"], case["dtype"], "parallax", case["levels"])
                 for k, w in enumerate(widths)]
        rig = binding.Rig(_params(case), case["h"], widths, c=case["c"],
                          dtype=torch.uint8 if case["dtype"] == "u8" else torch.float32,
                          canvas_hw=(case["canvas_h"], case["canvas_w"]), canvas_x0=x0, canvas_y0=y0)
        flows = [tuple(torch.empty((case["h"], w, 2), device=DEV) for _ in range(2)) for w in widths]
        return {"case": case, "rig": rig, "L": [p[0] for p in pairs], "R": [p[1] for p in pairs], "flows": flows,
                "canvas": rig.new_canvas()}
    if kind == "coeff":
        n = int(binding.load_library().pano_blend_coeff_scratch_bytes(case["h"], case["w"]))
        return {"case": case, "label": _labels(seed, case["h"], case["w"]),
                "scratch": torch.empty(n, dtype=torch.uint8, device=DEV)}
    if kind == "canvas":
        L, R, lab = _canvas_images(case, seed)
        return {"case": case, "ctx": binding.FlowContext(_params(case), case["h"], case["cw"], case["c"]), "L": L, "R": R,
                "label": lab}
    T, J, u = _energy_inputs(case, seed)
    return {"case": case, "T": T.requires_grad_(True), "J": J.requires_grad_(True), "u": u.requires_grad_(True)}


def _blend_map(case, seed):
    """A Blend array with a slanted, wavy seam instead of the plain ramp."""
    h, w = case["h"], case["w"]
    ys = torch.arange(h, device=DEV, dtype=torch.float32)[:, None]
    xs = torch.arange(w, device=DEV, dtype=torch.float32)[None, :]
    ph = float(torch.rand((), generator=_gen(seed + 9), device=DEV))
    return ((xs + 1) / (w + 1) + 0.15 * torch.sin(2 * math.pi * (ys / h + ph))).clamp(0, 1).contiguous()


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "pair":
        if s["blend"] is None:
            lr, rl, out = s["ctx"].stitch_pair(s["L"], s["R"])
        else:
            lr, rl = s["ctx"].flow_pair(s["L"], s["R"])
            out = s["ctx"].blend_pair(s["L"], s["R"], lr, rl, blend=s["blend"])
        return {"lr": lr, "rl": rl, "F": out}
    if kind == "static":
        lr, rl = binding.flow_pair_static(s["params"], s["L"], s["R"], out=s["out"])
        return {"lr": lr, "rl": rl}
    if kind == "rig":
        s["rig"].run(s["L"], s["R"], flows=s["flows"], canvas=s["canvas"], use_graph=case["graph"])
        return {"flows": [list(f) for f in s["flows"]], "canvas": s["canvas"]}
    if kind == "coeff":
        return {"blend": binding.blend_coeff(s["label"], scratch=s["scratch"])}
    if kind == "canvas":
        lr, rl, blend, out = s["ctx"].stitch_canvas(s["L"], s["R"], s["label"], (0, case["x0"], case["h"], case["cw"]))
        return {"lr": lr, "rl": rl, "blend": blend, "F": out}
    for k in ("T", "J", "u"):
        s[k].grad = None
    E = refine.pyramid_energy(s["T"], s["J"], s["u"], case["level"], 0.05)
    E.backward()
    return {"E": E.detach(), "T": s["T"].grad, "J": s["J"].grad, "u": s["u"].grad}


# ---------------------------------------------------------------- work

def _lk_flops(h, w, levels, iters, radius):
    """Per pixel and step: sample (14), residual (6), two window sums of two
    components (8 radius adds each way), solve (10); per level: gradient, G."""
    total = 0
    for _ in range(levels):
        total += 2 * h * w * (iters * (30 + 8 * radius) + 20 + 12 * radius)
        h, w = (h + 1) // 2, (w + 1) // 2
    return total


def work(case):
    kind, h = case["kind"], case["h"]
    e = 1 if case.get("dtype") == "u8" else 4
    if kind in ("pair", "static"):
        n = h * case["w"]
        b = n * (2 * case["c"] * e + 16)
        f = _lk_flops(h, case["w"], case["levels"], case["iters"], case["radius"])
        if kind == "pair":
            b += n * (case["c"] * e + (0 if case["ramp"] else 4))
            f += n * 60
        return {"bytes": b, "flops": f}
    if kind == "rig":
        n = sum(int(v) for v in case["widths"].split(","))
        f = sum(_lk_flops(h, int(v), case["levels"], 5, 2) for v in case["widths"].split(","))
        return {"bytes": h * n * (3 * case["c"] * e + 16), "flops": f + 60 * h * n}
    if kind == "coeff":
        return {"bytes": 5 * h * case["w"], "flops": 20 * h * case["w"]}
    if kind == "canvas":
        n, m = h * case["w"], h * case["cw"]
        return {"bytes": n * (5 + case["c"] * e) + (n - m) * case["c"] * e + m * (2 * case["c"] * e + 16),
                "flops": _lk_flops(h, case["cw"], case["levels"], 5, 2) + 60 * m}
    n = h * case["w"]
    m = n >> (2 * case["level"])
    return {"bytes": 16 * n + 16 * m, "flops": 60 * m + (20 * n if case["level"] else 0)}


def tolerance(case):
    """About four times what float32 shows against `exact` over the ranges of
    `draw`. Flows sit at the end of up to 35 warped steps, so single pixels at
    depth steps magnify a rounding: hence the "max". Whole values: F is rounded
    to bytes, and a value next to a half goes either way."""
    kind = case["kind"]
    if kind == "coeff":
        return {"rel": 1e-7, "max": 6e-7}
    if kind == "energy":
        return {"rel": 3e-6, "max": 4e-5}
    if case.get("pyr", "f32") != "f32":
        # levels stored in 16 bits: one within a rounding of a tie may be stored one ulp apart
        return {"rel": 1e-3, "max": 0.1, "differ": 1e-3}
    return {"rel": 4e-6, "max": 1e-3, "differ": 6e-5}


# --------------------------------------------------- the path in 64 bits

def _unit(img):
    return img.double() / 255 if img.dtype == torch.uint8 else img.double()


def _luma(img):
    v = _unit(img)
    return v if v.dim() == 2 else 0.299 * v[..., 0] + 0.587 * v[..., 1] + 0.114 * v[..., 2]


def _reduce(a):
    """[1 4 6 4 1]/16 along y then x, replicate border, even rows and columns."""
    for _ in range(2):
        n = a.shape[0]
        i = torch.arange(0, n, 2, device=a.device)
        a = sum(k / 16.0 * a[(i + t).clamp(0, n - 1)] for t, k in zip(range(-2, 3), (1, 4, 6, 4, 1)))
        a = a.t()
    return a.contiguous()


def _sample(img, px, py):
    """Bilinear, clamp-to-edge; img (h, w) or (h, w, c)."""
    h, w = img.shape[:2]
    fx, fy = px.floor(), py.floor()
    ax, ay = px - fx, py - fy
    x0, x1 = (v.clamp(0, w - 1).long() for v in (fx, fx + 1))
    y0, y1 = (v.clamp(0, h - 1).long() for v in (fy, fy + 1))
    if img.dim() == 3:
        ax, ay = ax[..., None], ay[..., None]
    top = img[y0, x0] * (1 - ax) + img[y0, x1] * ax
    bot = img[y1, x0] * (1 - ax) + img[y1, x1] * ax
    return top * (1 - ay) + bot * ay


def _box(a, r):
    """Sum over the (2r + 1)^2 window clipped to the image."""
    for _ in range(2):
        n = a.shape[0]
        p = F.pad(a, (0, 0, r, r))
        a = sum(p[d:d + n] for d in range(2 * r + 1)).t()
    return a


def _grid(h, w):
    return (torch.arange(h, device=DEV, dtype=torch.float64)[:, None].expand(h, w),
            torch.arange(w, device=DEV, dtype=torch.float64)[None, :].expand(h, w))


def _grad(T):
    def d(a):
        n = a.shape[0]
        i = torch.arange(n, device=a.device)
        return 0.5 * (a[(i + 1).clamp(max=n - 1)] - a[(i - 1).clamp(min=0)])
    return d(T.t()).t(), d(T)


def _flow(T, J, params):
    """Flow from T to J, coarse to fine, in 64 bits."""
    pt, pj = [T], [J]
    for _ in range(params.levels - 1):
        pt.append(_reduce(pt[-1]))
        pj.append(_reduce(pj[-1]))
    lam, r = float(torch.tensor(params.lam, dtype=torch.float32)), params.radius
    u = None
    for l in range(params.levels - 1, -1, -1):
        t, j = pt[l], pj[l]
        h, w = t.shape
        ys, xs = _grid(h, w)
        if u is None:
            ux, uy = torch.zeros_like(t), torch.zeros_like(t)
        else:
            ux, uy = (2 * _sample(v, xs / 2, ys / 2) for v in u)
        gx, gy = _grad(t)
        g11, g12, g22 = _box(gx * gx, r) + lam, _box(gx * gy, r), _box(gy * gy, r) + lam
        det = g11 * g22 - g12 * g12
        for _ in range(params.iters):
            s = gx * ux + gy * uy - (_sample(j, xs + ux, ys + uy) - t)
            r1, r2 = _box(gx * s, r) + lam * ux, _box(gy * s, r) + lam * uy
            ux, uy = (g22 * r1 - g12 * r2) / det, (g11 * r2 - g12 * r1) / det
        u = (ux, uy)
    return torch.stack(u, -1)


def _flows(L, R, params):
    a, b = _luma(L), _luma(R)
    return _flow(a, b, params), _flow(b, a, params)


def _code1(L, R, blend, lr, rl, width, params, y0=0, x0=0):
    """Code 1 on the rectangle of the flows, whose origin on the images is (y0, x0)."""
    h, w = lr.shape[:2]
    ys, xs = _grid(h, w)
    ys, xs = ys + y0, xs + x0
    cl = _sample(L, xs + blend * rl[..., 0], ys + blend * rl[..., 1])
    cr = _sample(R, xs + (1 - blend) * lr[..., 0], ys + (1 - blend) * lr[..., 1])
    fl = 1 + params.flow_mag_coef * rl.norm(dim=-1) / width
    fr = 1 + params.flow_mag_coef * lr.norm(dim=-1) / width
    k = params.soft_sharpness
    wl = torch.sigmoid(k * (1 - blend) * fl - k * blend * fr)
    if cl.dim() == 3:
        wl = wl[..., None]
    return cl * wl + cr * (1 - wl)


def _stored(v, dtype):
    return torch.round(v * 255).clamp(0, 255).to(torch.uint8) if dtype == "u8" else v


def _ramp(h, w):
    return ((_grid(h, w)[1] + 1) / (w + 1))


def _eq1(label):
    """Eq. (1) by an exact distance transform: nearest feature per column,
    then the least squared distance over each row's columns."""
    h, w = label.shape
    xs = torch.arange(w, device=DEV)
    ys = torch.arange(h, device=DEV)[:, None]
    cols3 = (label == 3).any(0).nonzero()[:, 0]
    far = 1 << 20
    dist = []
    for area in (1, 2):
        m = label == area
        up = torch.where(m, ys, -far).cummax(0).values
        dn = torch.where(m, ys, 2 * far).flip(0).cummin(0).values.flip(0)
        g = torch.minimum(ys - up, dn - ys).clamp(max=far).double()
        g2 = g * g
        D = (cols3[:, None] - xs[None, :]).double() ** 2
        d2 = torch.full((h, w), float("inf"), dtype=torch.float64, device=DEV)
        for y in range(h):
            if cols3.numel():
                d2[y, cols3] = (D + g2[y]).amin(1)
        dist.append(d2.sqrt() if bool(m.any()) else torch.full_like(d2, float("inf")))
    has1, has2 = bool((label == 1).any()), bool((label == 2).any())
    b3 = dist[0] / (dist[0] + dist[1]) if has1 and has2 else torch.full_like(dist[0], 1.0 if has2 else 0.0 if has1 else 0.5)
    blend = torch.full((h, w), 0.5, dtype=torch.float64, device=DEV)
    blend[label == 1], blend[label == 2] = 0.0, 1.0
    return torch.where(label == 3, b3, blend)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("pair", "static"):
        p = _params(case)
        L, R = _strips(seed, case["h"], case["w"], case["c"], case["dtype"], case["field"], case["levels"])
        lr, rl = _flows(L, R, p)
        if kind == "static":
            return {"lr": lr, "rl": rl}
        blend = _ramp(case["h"], case["w"]) if case["ramp"] else _blend_map(case, seed).double()
        out = _code1(_unit(L), _unit(R), blend, lr, rl, case["w"], p)
        return {"lr": lr, "rl": rl, "F": _stored(out, case["dtype"])}
    if kind == "rig":
        p = _params(case)
        widths, x0, y0 = _rig_layout(case)
        W, h = case["canvas_w"], case["h"]
        shape = (case["canvas_h"], W, case["c"]) if case["c"] > 1 else (case["canvas_h"], W)
        canvas = torch.zeros(shape, dtype=torch.uint8 if case["dtype"] == "u8" else torch.float64, device=DEV)
        flows = []
        for k, w in enumerate(widths):
            L, R = _strips(seed * 16 + k, h, w, case["c"], case["dtype"], "parallax", case["levels"])
            lr, rl = _flows(L, R, p)
            out = _stored(_code1(_unit(L), _unit(R), _ramp(h, w), lr, rl, w, p), case["dtype"])
            canvas[y0:y0 + h, (torch.arange(w, device=DEV) + x0[k]) % W] = out
            flows.append([lr, rl])
        return {"flows": flows, "canvas": canvas}
    if kind == "coeff":
        return {"blend": _eq1(_labels(seed, case["h"], case["w"]))}
    if kind == "canvas":
        p = _params(case)
        L, R, lab = _canvas_images(case, seed)
        x0, x1 = case["x0"], case["x0"] + case["cw"]
        blend = _eq1(lab)
        lr, rl = _flows(L[:, x0:x1], R[:, x0:x1], p)
        l64, r64 = _unit(L), _unit(R)
        area = lab if case["c"] == 1 else lab[..., None]
        out = torch.where(area == 1, l64, torch.where(area == 2, r64, torch.zeros_like(l64)))
        mid = _code1(l64, r64, blend[:, x0:x1], lr, rl, case["cw"], p, 0, x0)
        out[:, x0:x1] = torch.where(area[:, x0:x1] == 3, mid, out[:, x0:x1])
        return {"lr": lr, "rl": rl, "blend": blend, "F": _stored(out, case["dtype"])}
    T, J, u = (v.detach().double().requires_grad_(True) for v in _energy_inputs(case, seed))
    t, j = T, J
    for _ in range(case["level"]):
        t, j = _reduce(t), _reduce(j)
    ys, xs = _grid(*t.shape)
    E = ((_sample(j, xs + u[..., 0], ys + u[..., 1]) - t) ** 2).sum()
    E = E + 0.05 * (((u[:, 1:] - u[:, :-1]) ** 2).sum() + ((u[1:] - u[:-1]) ** 2).sum())
    E.backward()
    return {"E": E.detach(), "T": T.grad, "J": J.grad, "u": u.grad}
