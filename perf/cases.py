"""Timing cases: what a program that uses this library has it do, through the entry points it calls.

Each case names a kind of call and its sizes (see `listed`); `draw` gives other sizes of the same
kinds.  `prepare` makes what the program holds before the call (device inputs, the uploaded SOCS
kernel set, output and workspace buffers), `run` is one pass, `work` the bytes and operations the
pass cannot do without, `exact` the same outputs in 64-bit arithmetic from torch alone.

Kernel sets are computed here (TCC eigen-kernels from the source points' Gram matrix) and uploaded,
so that the 64-bit values start from the same lambda and Phi as the library.
"""
import functools
import math

import numpy as np
import torch

import paper_2602_15036_gb300 as P
from paper_2602_15036_gb300 import litho as L

# wavelength nm, NA, immersion index, source kind, source grid, pixel nm: the DUV settings of the
# aerial, AI and contour benchmarks (quadrupole) and of the ILT benchmark (annular), and the EUV
# setting of the serving benchmark.
OPTICS = {"duv-quad": (193.0, 1.35, 1.44, "quadrupole", 41, 8.0),
          "duv-annular": (193.0, 1.35, 1.44, "annular", 21, 8.0),
          "euv-annular": (13.5, 0.33, 1.0, "annular", 21, 1.0)}
THRESHOLD, RESIST_SIGMA_NM, ROUND_SIGMA_NM = 0.3, 10.0, 20.0
ROUND_TAU, MASK_STEEP, RESIST_STEEP = 0.5, 4.0, 25.0
SUB = 4  # rectangle corners lie on a layout grid of a quarter pixel (2 nm at 8 nm pixels)


def listed():
    return [
        # a correctness-sized clip imaged at nominal focus by itself: all launches and latency
        {"name": "image 1x256", "kind": "image", "n": 256, "b": 1, "k": 8, "optics": "duv-annular", "focus": "0",
         "precision": "fft32/coarse"},
        # one large clip at nominal focus: a serving request, an interactive simulation
        {"name": "image 1x2048", "kind": "image", "n": 2048, "b": 1, "k": 24, "optics": "duv-annular", "focus": "0",
         "precision": "fft32/coarse"},
        # the aerial benchmark's batch through focus with its blurred resist images, which the contour
        # and edge-placement steps take
        {"name": "resist image 64x2048", "kind": "resist_image", "n": 2048, "b": 64, "k": 24, "optics": "duv-quad",
         "focus": "-50,0,50", "precision": "fft32/coarse"},
        # the same on the full grid (the plain path), a small batch
        {"name": "resist image full grid 8x2048", "kind": "resist_image", "n": 2048, "b": 8, "k": 24,
         "optics": "duv-quad", "focus": "-50,0,50", "precision": "fft32"},
        # the same imaging on the tensor cores, at the precision that holds the FP32 error bound
        {"name": "image tensor 8x2048", "kind": "image", "n": 2048, "b": 8, "k": 24, "optics": "duv-quad",
         "focus": "-50,0,50", "precision": "fp16x3/coarse"},
        # the ILT benchmark's gradient step
        {"name": "ilt 16x1024", "kind": "ilt", "n": 1024, "b": 16, "k": 16, "optics": "duv-annular",
         "focus": "-60,-30,0,30,60", "precision": "fft32/coarse"},
        # one gradient step of one small clip, the inner loop of a single-clip optimisation
        {"name": "ilt 1x512", "kind": "ilt", "n": 512, "b": 1, "k": 8, "optics": "duv-annular", "focus": "-40,0,40",
         "precision": "fft32/coarse"},
        # the backward pass of imaging alone, for a loss that the caller computes: one-sided focus range
        {"name": "vjp 4x1024", "kind": "vjp", "n": 1024, "b": 4, "k": 16, "optics": "duv-annular", "focus": "0,40,80",
         "precision": "fft32/coarse"},
        # the AI initialiser's input channels for a training batch
        {"name": "ai inputs 16x2048", "kind": "ai", "n": 2048, "b": 16, "k": 24, "optics": "duv-quad", "focus": "0",
         "precision": "fft32/coarse"},
        # the AI initialiser's print-consistency images and loss
        {"name": "print images 16x2048", "kind": "print", "n": 2048, "b": 16},
        # contours and edge placement of through-focus resist images
        {"name": "contours 16x3x2048", "kind": "contour", "n": 2048, "b": 16, "planes": 3},
        # layout rectangles to grey masks
        {"name": "rasterize 64x2048", "kind": "raster", "n": 2048, "b": 64, "density": 0.35},
    ]


def draw(rng):
    base = dict(rng.choice(listed()))
    cap = _cost(base) if base["name"] != "image 1x256" else _cost(listed()[1])
    base.pop("name")
    kind = base["kind"]
    tensor = not base.get("precision", "fft32").startswith("fft32")

    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        c = dict(base)
        if kind == "contour":
            c.update(n=spread(60, 2048), planes=rng.randint(1, 5))
        elif kind == "raster":
            c.update(n=16 * spread(4, 128), density=round(rng.uniform(0.05, 0.5), 3))
        elif kind == "print":
            c.update(n=32 * spread(4, 64))
        else:
            c.update(n=rng.choice([512, 1024, 2048] if tensor else [128, 256, 512, 1024, 2048]),
                     k=rng.randint(3, 24), optics=rng.choice(sorted(OPTICS)),
                     focus="0" if kind == "ai" else rng.choice(["0", "35", "-50,0,50", "0,45", "-60,-30,0,30,60",
                                                                "0,30,75", "-20,10,40,55"]))
            if kind in ("image", "resist_image", "ilt", "vjp") and not tensor:
                c["precision"] = rng.choice([base["precision"], "fft32/coarse", "fft32"])
        c["b"] = spread(1, 64)
        if _cost(c) <= cap:
            return c


def _cost(case):
    w = work(case)
    return w["flops"] + 10.0 * w["bytes"]


# ---- kernel sets ------------------------------------------------------------------------------------


def _source(kind, grid):
    h = (grid - 1) // 2
    j, i = np.mgrid[-h:h + 1, -h:h + 1]
    r2 = (i * i + j * j).astype(np.float64)
    if kind == "annular":
        keep = (r2 >= (0.6 * h) ** 2 * (1 - 1e-12)) & (r2 <= (0.9 * h) ** 2 * (1 + 1e-12))
    else:
        c, r = 0.8 * h, (0.1 * h) ** 2 * (1 + 1e-12)
        keep = sum((i - x) ** 2 + (j - y) ** 2 <= r for x, y in ((c, 0), (-c, 0), (0, c), (0, -c))) > 0
    return i[keep] / h, j[keep] / h


def _crop(optics, n):
    """Side of the band crop: the multiple of 32 above twice the band radius, at most n."""
    wl, na, _, kind, grid, pixel = OPTICS[optics]
    sx, sy = _source(kind, grid)
    rb = math.floor((1.0 + math.sqrt((sx * sx + sy * sy).max())) * na / wl * n * pixel)
    return min(n, (2 * rb + 2 + 31) // 32 * 32)


def _focus(case):
    scale = 1.0 if case["optics"].startswith("duv") else 0.5  # the EUV depth of focus is shorter
    return [scale * float(z) for z in case["focus"].split(",")]


@functools.lru_cache(maxsize=2)
def _socs(optics, n, k, focus):
    """lambda [F][K] and Phi [F][K][C][C] of the TCC's leading eigen-kernels, 64-bit, on the host."""
    wl, na, index, kind, grid, pixel = OPTICS[optics]
    sx, sy = _source(kind, grid)
    c = _crop(optics, n)
    u = (np.arange(c) - c // 2) / (n * pixel)
    dev = torch.device("cuda")
    fx = torch.tensor(u, device=dev)[None, :, None] + torch.tensor(sx * na / wl, device=dev)
    fy = torch.tensor(u, device=dev)[:, None, None] + torch.tensor(sy * na / wl, device=dev)
    f2 = (fx * fx + fy * fy).reshape(c * c, len(sx))
    kz = torch.sqrt(torch.clamp((index / wl) ** 2 - f2, min=0.0)) - index / wl
    lam, phi = np.zeros((len(focus), k)), np.zeros((len(focus), k, c, c), dtype=np.complex128)
    for f, z in enumerate(focus):
        a = torch.where(f2 <= (na / wl) ** 2, torch.exp(2j * math.pi * z * kz), torch.zeros_like(kz) + 0j)
        a = a / math.sqrt(len(sx))
        w, v = np.linalg.eigh((a.conj().T @ a).cpu().numpy())
        w, v = w[::-1][:k], np.ascontiguousarray(v[:, ::-1][:, :k])
        keep = w > 1e-12 * w[0]
        lam[f, :len(w)][keep] = w[keep]
        vv = torch.tensor(v[:, keep] / np.sqrt(w[keep]), device=dev)
        phi[f, :len(w)][keep] = (a @ vv).T.reshape(-1, c, c).cpu().numpy()
    return lam, phi


@functools.lru_cache(maxsize=16)
def _kernels(optics, n, k, focus):
    lam, phi = _socs(optics, n, k, focus)
    return P.litho_upload_kernels(n, OPTICS[optics][5], lam, phi)


def _key(case):
    return case["optics"], case["n"], case["k"], tuple(_focus(case))


# ---- inputs -----------------------------------------------------------------------------------------


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _rect_cover(n, x0, y0, w, h):
    """Union of rectangles on an n x n cell grid, periodic: 1 in every covered cell (uint8)."""
    pad = int(max(int(w.max()), int(h.max()), 1))
    m = n + pad + 1
    d = torch.zeros(m * m, dtype=torch.int32, device=x0.device)
    one = torch.ones_like(x0, dtype=torch.int32)
    for xx, yy, s in ((x0, y0, 1), (x0 + w, y0, -1), (x0, y0 + h, -1), (x0 + w, y0 + h, 1)):
        d.index_add_(0, yy * m + xx, s * one)
    c = (d.view(m, m).cumsum(0, dtype=torch.int32).cumsum(1, dtype=torch.int32) > 0).to(torch.uint8)
    c[:, :m - n] |= c[:, n:].clone()
    c[:m - n] |= c[n:].clone()
    return c[:n, :n].contiguous()


def _rect_count(n, density):
    return max(1, int(-math.log(1.0 - density) * n * n / 100.0))


def _rects(n, count, gen, cells=1):
    """Corners U over the grid, sides U{5..15} pixels, in units of 1/cells pixel."""
    def ri(lo, hi):
        return torch.randint(lo, hi, (count,), generator=gen, device="cuda")
    return ri(0, n * cells), ri(0, n * cells), ri(5 * cells, 15 * cells + 1), ri(5 * cells, 15 * cells + 1)


def _masks(b, n, gen):
    """Manhattan masks at 35 % coverage, f32 0/1."""
    return torch.stack([_rect_cover(n, *_rects(n, _rect_count(n, 0.35), gen)) for _ in range(b)]).to(torch.float32)


def _blobs(b, n, gen):
    """Smooth curvilinear fields B in [0, 1]: 60 periodic Gaussian blobs of 4 to 10 pixels per 1024^2."""
    out = torch.empty((b, n, n), device="cuda")
    count = max(8, 60 * n * n // (1 << 20))
    x = torch.arange(n, device="cuda", dtype=torch.float32)
    for i in range(b):
        c = torch.rand((2, count, 1), generator=gen, device="cuda") * n
        s = (4 + 6 * torch.rand((count, 1), generator=gen, device="cuda")) * math.sqrt(n / 256)
        g = [torch.exp(-(((x - cc + n / 2) % n - n / 2) / s) ** 2 / 2) for cc in c]
        f = g[0].T @ g[1]
        out[i] = (f - f.min()) / (f.max() - f.min())
    return out


def _blur_spectral(x, sigma_px):
    n = x.shape[-1]
    f = torch.fft.fftfreq(n, device=x.device)
    g = torch.exp(-2 * (math.pi * sigma_px * f) ** 2)
    return torch.fft.irfft2(torch.fft.rfft2(x) * g[:, None] * g[:n // 2 + 1], s=(n, n))


def _edge_points(mask):
    """Midpoints of the pixel boundaries where a mask changes, (x, y) in pixels."""
    y, x = torch.nonzero(mask != torch.roll(mask, -1, 1), as_tuple=True)
    v, u = torch.nonzero(mask != torch.roll(mask, -1, 0), as_tuple=True)
    return torch.stack([torch.cat([x + 0.5, u.float()]), torch.cat([y.float(), v + 0.5])], 1).float()


def _site_count(n):
    """Control points of a clip: about nine in ten of its mask's boundary sites."""
    return max(1, n * n // 10)


def _inputs(case, seed):
    """The device inputs of a case, from the seed alone."""
    gen, n, b = _gen(seed), case["n"], case["b"]
    kind = case["kind"]
    if kind in ("image", "resist_image"):
        return {"mask": _masks(b, n, gen)}
    if kind == "ilt":
        f = _blobs(b, n, gen)
        return {"theta": 2.0 * (f - 0.5), "target": (f >= 0.5).float()}
    if kind == "vjp":
        mask = torch.sigmoid(8.0 * (_blobs(b, n, gen) - 0.5))
        planes = len(_focus(case))
        up = torch.empty((b, planes, n, n), device="cuda")
        for i in range(b):  # a loss's gradient: signed, smooth on the scale of the image
            up[i] = _blur_spectral(torch.randn((planes, n, n), generator=gen, device="cuda"), 2.0)
        return {"mask": mask, "upstream": up}
    if kind == "ai":
        return {"target": _masks(b, n, gen)}
    if kind == "print":
        t = _masks(b, n, gen)
        img = torch.stack([_blur_spectral(m, 2.5) for m in t])
        return {"target": t, "image": img + 0.02 * torch.rand((b, n, n), generator=gen, device="cuda")}
    if kind == "contour":
        t = _masks(b, n, gen)
        sig = [2.0 + 0.3 * abs(p - (case["planes"] - 1) / 2) for p in range(case["planes"])]
        ib = torch.stack([torch.stack([_blur_spectral(m, s) for s in sig]) for m in t])
        m = _site_count(n)
        pts = [p[torch.arange(m, device="cuda") * len(p) // m] for p in map(_edge_points, t)]
        return {"iblur": ib.contiguous(), "points": torch.cat(pts).contiguous(),
                "start": torch.arange(b + 1, device="cuda") * m}
    count = _rect_count(n, case["density"])
    rects = torch.empty((b, count, 4), device="cuda")
    for i in range(b):
        x0, y0, w, h = (v.float() / SUB for v in _rects(n, count, gen, SUB))
        rects[i] = torch.stack([x0, y0, x0 + w, y0 + h], 1)
    return {"rects": rects.view(-1, 4), "start": torch.arange(b + 1, device="cuda") * count, "count": count}


def prepare(case, seed):
    s = dict(_inputs(case, seed), case=case)
    n, b, kind = case["n"], case["b"], case["kind"]

    def empty(*shape, dtype=torch.float32):
        return torch.empty(shape, dtype=dtype, device="cuda")

    def bytes_(count):
        return empty(count, dtype=torch.uint8)

    if "optics" in case:
        s["kern"] = kern = _kernels(*_key(case))
        planes = kern.n_focus
    if kind in ("image", "resist_image"):
        s["out"] = empty(b, planes, n, n)
        if kind == "resist_image":
            s["iblur"] = empty(b, planes, n, n)
        s["ws"] = bytes_(L.litho_aerial_workspace_size(kern, b, case["precision"]))
    elif kind == "ilt":
        s["grad"] = empty(b, n, n)
        s["ws"] = bytes_(P.litho_ilt_workspace_size(kern, b)[0])
    elif kind == "ai":
        s["x"] = empty(b, 3, n, n)
        s["ws"] = bytes_(L.litho_ai_inputs_workspace_size(kern, b))
    elif kind == "contour":
        m, planes = len(s["points"]), case["planes"]
        count = b * planes * (n * n // 8 + n)  # room for every segment (about 8 % of the cells hold one)
        s["seg"] = torch.zeros((count, 4), device="cuda")
        s["cell"] = torch.zeros(count, dtype=torch.int32, device="cuda")
        s["starts"] = empty(b * planes + 1, dtype=torch.int64)
        s["epe"], s["avg"], s["eff"] = empty(planes, m), empty(m), empty(m)
        s["ws"] = bytes_(L.contours_workspace_size(b * planes, n))
    elif kind == "raster":
        s["mask"] = empty(b, n, n)
        s["ws"] = bytes_(L.rasterize_workspace_size(b, n, s["count"], 16))
    return s


def run(s):
    case = s["case"]
    n, b, kind = case["n"], case["b"], case["kind"]
    if kind == "image":
        return P.litho_aerial(s["kern"], s["mask"], precision=case["precision"], out=s["out"], workspace=s["ws"])
    if kind == "resist_image":
        return P.litho_aerial_resist(s["kern"], s["mask"], precision=case["precision"], sigma_nm=RESIST_SIGMA_NM,
                                     threshold=THRESHOLD, out=s["out"], iblur=s["iblur"], want_printed=False,
                                     workspace=s["ws"])[:2]
    if kind == "ilt":
        grad, loss = P.litho_ilt_grad(s["kern"], s["theta"], s["target"], mask_steep=MASK_STEEP,
                                      resist_steep=RESIST_STEEP, threshold=THRESHOLD, sigma_nm=RESIST_SIGMA_NM,
                                      precision=case["precision"], grad=s["grad"], workspace=s["ws"])
        return grad, loss.astype(np.float32)  # the loss record of an FP32 optimisation
    if kind == "vjp":
        return L.litho_intensity_vjp(s["kern"], s["mask"], upstream=s["upstream"], precision=case["precision"])
    if kind == "ai":
        return P.litho_ai_inputs(s["kern"], s["target"], focus=0, precision=case["precision"], out=s["x"],
                                 workspace=s["ws"])
    if kind == "print":
        return P.litho_print_images(s["target"], s["image"], 8.0, ROUND_SIGMA_NM, ROUND_TAU, THRESHOLD)
    if kind == "contour":
        planes = case["planes"]
        L.contours_into(s["iblur"], b * planes, n, THRESHOLD, s["seg"], s["cell"], len(s["cell"]), s["starts"], s["ws"])
        P.litho_epe_batch(s["iblur"], s["points"], s["start"], 8.0, THRESHOLD, out=s["epe"])
        L.epe_through_focus_into(s["epe"], planes // 2, planes - 1, 0, -1.0, 1.0, s["avg"], s["eff"])
        return s["seg"], s["cell"], s["starts"], s["epe"], s["avg"], s["eff"]
    L.rasterize_into(s["rects"], s["start"], b, s["count"], 16, n, s["mask"], s["ws"])
    return s["mask"]


# ---- work -------------------------------------------------------------------------------------------


def _grid(c, n):
    """The smallest power of two that samples an image of band 2c, at most n."""
    g = 32
    while g < 2 * c:
        g *= 2
    return min(g, n)


def work(case):
    n, b, kind = case["n"], case["b"], case["kind"]
    px = float(b) * n * n
    if kind == "print":  # target and image in; two byte images and the blur out; the separable blur
        return {"bytes": px * 14, "flops": px * 4 * (2 * math.ceil(4 * ROUND_SIGMA_NM / 8.0) + 1)}
    if kind == "contour":  # the planes once; a segment and its cell in about 8 % of the cells; the control points
        planes, pts = case["planes"], b * _site_count(n)
        return {"bytes": px * planes * (4 + 0.08 * 20) + pts * (16 + 4 * planes),
                "flops": px * planes * 2 + pts * planes * 60}
    if kind == "raster":
        return {"bytes": px * 4 + b * _rect_count(n, case["density"]) * 16.0, "flops": px * 8}
    c, f, k = _crop(case["optics"], n), len(_focus(case)), case["k"]
    g = _grid(c, n)

    def fft(m):
        return 5.0 * m * math.log2(m)

    # one banded 2-D transform of each field and its |E|^2; the mask's spectrum; the image's resampling to n
    fields = b * f * k * ((c + g) * fft(g) + 4.0 * g * g)
    spectrum = b * (n / 2 + c / 2) * fft(n)
    resample = b * f * ((g / 2 + c) * fft(g) + (c + n / 2) * fft(n)) if g < n else 0.0
    phi = 8.0 * f * k * c * c
    if kind in ("image", "resist_image"):
        outs = f * (2 if kind == "resist_image" else 1)
        return {"bytes": px * 4 * (1 + outs) + phi, "flops": fields + spectrum + resample}
    if kind == "ai":
        return {"bytes": px * 16 + phi, "flops": fields + 2 * spectrum + resample}
    if kind == "ilt":  # theta and target in, gradient out; the forward image, then each field's way back
        return {"bytes": px * 12 + phi, "flops": 3 * fields + 2 * spectrum + 2 * resample}
    return {"bytes": px * (8 + 4 * f) + phi, "flops": 3 * fields + 2 * spectrum + resample}


# ---- 64-bit values ------------------------------------------------------------------------------------


def _embed(spec, g):
    """Crop spectra [..., C, C] (centred) in FFT order on a g x g grid."""
    c = spec.shape[-1]
    out = torch.zeros(spec.shape[:-2] + (g, g), dtype=spec.dtype, device=spec.device)
    i = (torch.arange(c, device=spec.device) - c // 2) % g
    out[..., i[:, None], i] = spec
    return out


def _cropped(spec, c):
    i = (torch.arange(c, device=spec.device) - c // 2) % spec.shape[-1]
    return spec[..., i[:, None], i]


def _inverse(spec, g):
    return torch.fft.ifft2(_embed(spec, g), norm="forward")


def _mask_spectrum(m, c):
    return _cropped(torch.fft.fft2(m.double(), norm="forward"), c)


def _image64(mhat, lam, phi, n):
    """Image of one mask spectrum at one focus plane on n x n, through the smallest grid that holds its band."""
    c = phi.shape[-1]
    g = _grid(c, n)
    img = sum(w * _inverse(mhat * p, g).abs().square() for w, p in zip(lam, phi) if w > 0)
    if g == n:
        return img
    return _inverse(_cropped(torch.fft.fft2(img, norm="forward"), 2 * c - 1), n).real


def _gain64(n, sigma_nm, pixel, device):
    r = math.ceil(4 * sigma_nm / pixel)
    j = torch.arange(-r, r + 1, dtype=torch.float64, device=device)
    t = torch.exp(-(j * pixel) ** 2 / (2 * sigma_nm ** 2))
    f = torch.fft.fftfreq(n, dtype=torch.float64, device=device)
    gain = (t / t.sum() * torch.cos(2 * math.pi * f[:, None] * j)).sum(1)
    return gain[:, None] * gain


def _blur64(x, gain):
    return torch.fft.ifft2(torch.fft.fft2(x) * gain).real


def _adjoint64(mhat, lam, phi, up, n):
    """dm of one plane: 2 N^-2 Re IDFT sum_k lam conj(Phi) DFT(up E), E on the full grid."""
    c = phi.shape[-1]
    s = sum(w * p.conj() * _cropped(torch.fft.fft2(up * _inverse(mhat * p, n)), c)
            for w, p in zip(lam, phi) if w > 0)
    return 2.0 / (n * n) * _inverse(s, n).real


def exact(case, seed):
    x = _inputs(case, seed)
    n, b, kind = case["n"], case["b"], case["kind"]
    if kind == "print":
        g = _gain64(n, ROUND_SIGMA_NM, 8.0, "cuda")
        return [None, None, None, torch.stack([_blur64(t.double(), g) for t in x["target"]])]
    if kind == "contour":
        return [None, None, None] + _epe64(case, x) + [None]
    if kind == "raster":  # corners on quarter pixels: coverage is a count of quarter cells
        out = torch.empty((b, n, n), dtype=torch.float64, device="cuda")
        for i, r in enumerate((x["rects"].view(b, -1, 4) * SUB).round().long()):
            cells = _rect_cover(n * SUB, r[:, 0], r[:, 1], r[:, 2] - r[:, 0], r[:, 3] - r[:, 1])
            out[i] = cells.view(n, SUB, n, SUB).sum((1, 3), dtype=torch.float64) / SUB ** 2
        return out
    pixel = OPTICS[case["optics"]][5]
    lam, phi = _socs(*_key(case))
    phi = torch.tensor(phi, device="cuda")
    planes, c = phi.shape[0], phi.shape[-1]
    empty = functools.partial(torch.empty, dtype=torch.float64, device="cuda")
    blur = _gain64(n, RESIST_SIGMA_NM, pixel, "cuda")
    if kind in ("image", "resist_image"):
        img, ib = empty((b, planes, n, n)), empty((b, planes, n, n) if kind == "resist_image" else 0)
        for i in range(b):
            mhat = _mask_spectrum(x["mask"][i], c)
            for f in range(planes):
                img[i, f] = _image64(mhat, lam[f], phi[f], n)
                if kind == "resist_image":
                    ib[i, f] = _blur64(img[i, f], blur)
        return (img, ib) if kind == "resist_image" else img
    if kind == "ai":
        out = empty((b, 3, n, n))
        for i in range(b):
            mhat = _mask_spectrum(x["target"][i], c)
            out[i, 0] = x["target"][i]
            out[i, 1] = _image64(mhat, lam[0], phi[0], n)
            s = sum(w * p.abs().square() for w, p in zip(lam[0], phi[0])) * mhat
            out[i, 2] = 2.0 * _inverse(s, n).real
        out[:, 1] /= out[:, 1].max()
        lo, hi = out[:, 2].min(), out[:, 2].max()
        out[:, 2] = (out[:, 2] - lo) / (hi - lo)
        return out
    if kind == "vjp":
        dm = empty((b, n, n))
        for i in range(b):
            mhat = _mask_spectrum(x["mask"][i], c)
            dm[i] = sum(_adjoint64(mhat, lam[f], phi[f], x["upstream"][i, f].double(), n) for f in range(planes))
        return dm
    grad, loss = empty((b, n, n)), empty(b)
    for i in range(b):
        m = torch.sigmoid(MASK_STEEP * x["theta"][i].double())
        mhat = _mask_spectrum(m, c)
        dm, total = 0.0, 0.0
        for f in range(planes):
            z = torch.sigmoid(RESIST_STEEP * (_blur64(_image64(mhat, lam[f], phi[f], n), blur) - THRESHOLD))
            d = z - x["target"][i]
            total = total + d.square().sum()
            q = 2.0 * d * RESIST_STEEP * z * (1.0 - z)
            dm = dm + _adjoint64(mhat, lam[f], phi[f], _blur64(q, blur), n)
        grad[i], loss[i] = dm * MASK_STEEP * m * (1.0 - m), total
    return grad, loss


def _epe64(case, x):
    """EPE of every plane at every point, and its mean over the on-focus and the two outer planes."""
    n, planes = case["n"], case["planes"]
    start = x["start"].tolist()
    epe = torch.empty((planes, len(x["points"])), dtype=torch.float64, device="cuda")
    for i, clip in enumerate(x["iblur"].double()):
        p = x["points"][start[i]:start[i + 1]].double()
        j, t = torch.floor(p).long(), p - torch.floor(p)
        for f, a in enumerate(clip):
            def at(v):
                x0, y0, x1, y1 = j[:, 0] % n, j[:, 1] % n, (j[:, 0] + 1) % n, (j[:, 1] + 1) % n
                u, w = t[:, 0], t[:, 1]
                return (v[y0, x0] * (1 - u) + v[y0, x1] * u) * (1 - w) + (v[y1, x0] * (1 - u) + v[y1, x1] * u) * w
            gx = (torch.roll(a, -1, 1) - torch.roll(a, 1, 1)) / 16.0
            gy = (torch.roll(a, -1, 0) - torch.roll(a, 1, 0)) / 16.0
            epe[f, start[i]:start[i + 1]] = -(at(a) - float(np.float32(THRESHOLD))) / torch.hypot(at(gx), at(gy))
    avg = (epe[planes // 2] + epe[planes - 1] + epe[0]) / 3.0
    return [epe, avg]
