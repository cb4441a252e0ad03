"""Tile edges and remainders of the blur, print, raster and contour kernels against the oracle.

Bounds: the blur is a sum of (2R + 1)^2 products of FP32 weights that sum to 1 over values in [0, 1],
so 1e-6; its print is the threshold of the value returned, to the bit; coverage 2e-6 (a few FP32
roundings of areas of at most 1); contour cells and order are integer decisions, equal to the bit."""
import numpy as np
import pytest

import synth
from oracle import contour as OC
from oracle import raster as ORA
from oracle import resist as OR

pytestmark = pytest.mark.gpu


# radius 1, 5, 10, 12 (register windows) and 13, 15, 30, 45, 64 (loop); 128-, 64- and 32-wide tiles, few and many planes
@pytest.mark.parametrize("n,planes", [(32, 3), (96, 2), (64, 5), (128, 1), (256, 40), (192, 3)])
@pytest.mark.parametrize("radius", [1, 5, 10, 12, 13, 15, 30, 45, 64])
def test_blur_tiles(litho_lib, cuda, n, planes, radius):
    import torch
    if 2 * radius >= n:
        pytest.skip("the radius must be below n/2")
    pixel, sigma = 8.0, 8.0 * (radius - 0.5) / 4.0  # ceil(4 sigma / pixel) = radius
    img = synth.random_field((planes, n, n), seed=n + radius, lo=0.0, hi=1.0).astype(np.float32)
    room = torch.zeros(planes * n * n + 1, device=cuda)
    for shift in (0, 1):  # 16-byte aligned, and not
        src = room[shift:shift + planes * n * n].view(planes, n, n)
        src.copy_(torch.from_numpy(img))
        blur = torch.full((planes * n * n + 1,), -1.0, device=cuda)[shift:shift + planes * n * n].view(planes, n, n)
        ib, pr = litho_lib.litho_resist(src, pixel, sigma, 0.5, iblur=blur)
        got = ib.cpu().numpy()
        if shift == 0:
            first = got
        assert np.array_equal(got, first)
        assert np.array_equal(pr.cpu().numpy(), (got >= np.float32(0.5)).astype(np.uint8))
    for p in (0, planes - 1):
        assert np.abs(first[p] - OR.blur(img[p], sigma, pixel)).max() <= 1e-6


# the last radius of two tiles per SM and the first of one, the last and the first that the wide tile does not
# hold; planes enough for the wide tile, and not
@pytest.mark.parametrize("n,planes", [(256, 20), (128, 1)])
@pytest.mark.parametrize("radius", [37, 38, 56, 57])
def test_blur_tile_widths(litho_lib, cuda, n, planes, radius):
    import torch
    pixel, sigma = 8.0, 8.0 * (radius - 0.5) / 4.0
    img = synth.random_field((planes, n, n), seed=radius, lo=0.0, hi=1.0).astype(np.float32)
    ib, pr = litho_lib.litho_resist(torch.from_numpy(img).to(cuda), pixel, sigma, 0.5)
    ib = ib.cpu().numpy()
    assert np.array_equal(pr.cpu().numpy(), (ib >= np.float32(0.5)).astype(np.uint8))
    for p in (0, planes - 1):
        assert np.abs(ib[p] - OR.blur(img[p], sigma, pixel)).max() <= 1e-6


@pytest.mark.parametrize("n,b", [(32, 3), (96, 1), (256, 2)])
def test_print_counts(litho_lib, cuda, n, b):
    import torch
    t = np.stack([synth.random_rect_mask(n, seed=5 + i, count=12) for i in range(b)])
    img = synth.random_field((b, n, n), seed=3, lo=0.0, hi=0.6).astype(np.float32)
    room = torch.zeros(b * n * n + 1, device=cuda)
    for shift in (0, 1):
        d = room[shift:shift + b * n * n].view(b, n, n)
        d.copy_(torch.from_numpy(img))
        zr, zp, loss, blur = litho_lib.litho_print_images(torch.from_numpy(t).to(cuda), d, 8.0, 20.0, 0.5, 0.3)
        zr, zp, blur = zr.cpu().numpy(), zp.cpu().numpy(), blur.cpu().numpy()
        assert np.array_equal(zp, (img >= np.float32(0.3)).astype(np.uint8))
        assert np.array_equal(zr, (blur >= np.float32(0.5)).astype(np.uint8))
        assert np.array_equal(loss.cpu().numpy(), (zr != zp).reshape(b, -1).sum(1))


# one tile, a last CTA of one tile, more pieces in a tile than the cache holds
@pytest.mark.parametrize("n,count,lo,hi", [(16, 5, 2.0, 9.0), (16, 150, 0.2, 3.0), (48, 60, 1.0, 12.0), (80, 900, 0.5, 8.0)])
def test_raster_tiles(litho_lib, cuda, n, count, lo, hi):
    import torch
    st = synth.Stream(count)
    clips = []
    for _ in range(2):
        w, h = (lo + (hi - lo) * st.uniform(count) for _ in range(2))
        x0, y0 = (n * st.uniform(count) for _ in range(2))
        clips.append(np.stack([x0, y0, x0 + w, y0 + h], axis=1).astype(np.float32))
    room = torch.full((2 * n * n + 1,), -1.0, device=cuda)
    for shift in (0, 1):
        out = room[shift:shift + 2 * n * n].view(2, n, n)
        got = litho_lib.litho_rasterize(clips, n, 16, out=out).cpu().numpy()
        for c, r in enumerate(clips):
            assert np.abs(got[c] - ORA.coverage(n, r.astype(np.float64))).max() <= 2e-6


# every cell crossed (two segments in most: the queue at its fullest), and rows without a crossing
@pytest.mark.parametrize("n", [128, 384])
def test_contour_rows(litho_lib, cuda, n):
    import torch
    y, x = np.mgrid[0:n, 0:n]
    checker = np.where((x + y) % 2, 0.9, 0.1).astype(np.float32)
    noise = synth.random_field((n, n), seed=n, lo=0.0, hi=1.0).astype(np.float32)
    band = np.where((y > 40) & (y < 60), noise, 0.0).astype(np.float32)
    planes = np.stack([checker, band, np.zeros((n, n), np.float32), noise])
    seg, cell, start = litho_lib.litho_contours(torch.from_numpy(planes).to(cuda), 0.45)
    seg, cell = seg.cpu().numpy().astype(np.float64), cell.cpu().numpy()
    for p in range(len(planes)):
        ref = OC.marching_squares(planes[p], 0.45)
        assert np.array_equal(cell[start[p]:start[p + 1]], np.array([r[0] for r in ref], dtype=np.int32))
        want = np.array([r[1:5] for r in ref], dtype=np.float64).reshape(-1, 4)
        assert np.all(np.abs(seg[start[p]:start[p + 1]] - want) <= 1e-5 + 2.5e-7 * np.abs(want))


# rows of whole 16-byte pieces, and not
@pytest.mark.parametrize("n", [96, 90])
def test_epe_wraps_outside_the_grid(litho_lib, cuda, n):
    import torch
    img = (0.5 + 0.4 * np.sin(2 * np.pi * np.mgrid[0:n, 0:n][1] * 3 / n) * np.cos(2 * np.pi * np.mgrid[0:n, 0:n][0] * 2 / n))
    img = img.astype(np.float32)
    st = synth.Stream(2)
    pts = np.stack([st.uniform(200) * 4 * n - 2 * n, st.uniform(200) * 4 * n - 2 * n], 1).astype(np.float32)
    got = litho_lib.litho_epe(torch.from_numpy(img[None]).to(cuda), torch.from_numpy(pts).to(cuda), 8.0, 0.5)[0]
    want = OC.epe(img.astype(np.float64), pts.astype(np.float64), 0.5, 8.0)
    assert np.all(np.abs(got.cpu().numpy() - want) <= 1e-3 + 1e-4 * np.abs(want))
