"""The reduced kernel sets the device images with (kernelset.cu) against the FP64 oracle with the
kernels as given: planes that reduce (in focus), planes that share a set (+z and -z), planes that do
neither, and kernels without any symmetry, on every path that reads a set.  Bounds as in the parity
tests of each path: image 1e-5, gradient 1e-4 relative."""
import numpy as np
import pytest

import synth
from oracle import ai as OA
from oracle import ilt as OL
from oracle import imaging as OI
from tests.gpu_util import DUV_ANNULAR, DUV_QUAD21, oracle_kernel_set

pytestmark = pytest.mark.gpu
PIXEL = 8.0


def _random_set(n, c, planes, k, edge):
    """Complex kernels with no symmetry, decaying from DC, |E|^2 of order 1; `edge`: nonzero at u = -C/2."""
    rng = np.random.default_rng(7)
    u = np.arange(c) - c // 2
    r2 = u[:, None] ** 2 + u ** 2
    phi = (rng.standard_normal((planes, k, c, c)) + 1j * rng.standard_normal((planes, k, c, c))) * np.exp(-r2 / (c * c / 18))
    if not edge:
        phi[..., 0, :] = 0
        phi[..., :, 0] = 0
    else:
        phi[..., 0, :] += 0.1j
    lam = np.sort(rng.uniform(0.05, 0.2, (planes, k)))[:, ::-1].copy()
    lam[-1, -2:] = 0.0
    return lam, phi


def _set(name, n):
    if name == "random":
        return _random_set(n, 32, 2, 4, False)
    if name == "edge":
        return _random_set(n, 32, 1, 3, True)
    if name == "full width":  # crop = n: u = -n/2 is its own mirror
        return _random_set(n, n, 1, 3, True)
    if name == "dark plane":
        lam, phi = oracle_kernel_set(DUV_QUAD21, n, PIXEL, [0.0, 30.0], 5)
        lam[0] = 0.0
        return lam, phi
    focus, k, optics = {"nominal": ([0.0], 7, DUV_QUAD21), "one kernel": ([0.0], 1, DUV_ANNULAR),
                        "through focus": ([-40.0, 0.0, 40.0], 8, DUV_ANNULAR),
                        "reordered": ([30.0, -60.0, 60.0, 0.0, -30.0], 5, DUV_ANNULAR),
                        "repeated": ([20.0, 20.0, 0.0, 0.0], 6, DUV_QUAD21)}[name]
    lam, phi = oracle_kernel_set(optics, n, PIXEL, focus, k)
    return lam, phi * np.exp(1j * np.arange(k))[:, None, None]  # eigenvectors have no phase of their own


SETS = ["nominal", "one kernel", "through focus", "reordered", "repeated", "dark plane", "random", "edge"]


@pytest.mark.parametrize("precision", ["fft32", "fft32/coarse", "fp16x3", "fp16x3/coarse"])
@pytest.mark.parametrize("name", SETS + ["full width"])
def test_images_match_the_given_kernels(litho_lib, cuda, name, precision):
    import torch
    n = 32 if name == "full width" else 256
    if name == "full width" and precision.startswith("fp16"):
        pytest.skip("the tensor-core path needs a grid of 128 points")
    if precision == "fp16x3/coarse" and name in ("random", "edge"):
        pytest.skip("a coarse grid of 64 points")
    lam, phi = _set(name, n)
    kern = litho_lib.litho_upload_kernels(n, PIXEL, lam, phi)
    masks = np.stack([synth.random_rect_mask(n, seed=3 + i, count=6 if n == 32 else 40) for i in range(3)])
    img = litho_lib.litho_aerial(kern, torch.from_numpy(masks).to(cuda), precision=precision).cpu().numpy()
    for i, m in enumerate(masks):
        for f in range(len(lam)):
            ref = OI.socs_image(m.astype(np.float64), lam[f], phi[f])
            assert np.abs(img[i, f] - ref).max() <= 1e-5 * max(1.0, ref.max())


@pytest.mark.parametrize("precision", ["fft32", "fft32/coarse"])
@pytest.mark.parametrize("name", SETS)
def test_gradients_match_the_given_kernels(litho_lib, cuda, name, precision):
    import torch
    n, b = 128, 2
    lam, phi = _set(name, n)
    planes = len(lam)
    kern = litho_lib.litho_upload_kernels(n, PIXEL, lam, phi)
    pairs = [(lam[f], phi[f]) for f in range(planes)]
    clips = [synth.ilt_clip(n, PIXEL, seed=40 + i) for i in range(b)]
    theta = torch.from_numpy(np.stack([c[0] for c in clips])).to(cuda)
    target = torch.from_numpy(np.stack([c[1] for c in clips])).to(cuda)
    full, small = litho_lib.litho_ilt_workspace_size(kern, b)
    for size in (full, small):
        ws = torch.empty(size, dtype=torch.uint8, device=cuda)
        grad, loss = litho_lib.litho_ilt_grad(kern, theta, target, precision=precision, workspace=ws)
        for i in range(b):
            ref_loss, ref = OL.loss_and_grad(clips[i][0].astype(np.float64), clips[i][1].astype(np.float64), pairs)
            assert abs(loss[i] - ref_loss) <= 1e-5 * ref_loss
            assert np.linalg.norm(grad[i].cpu().numpy() - ref) <= 1e-4 * np.linalg.norm(ref)
    rng = np.random.default_rng(1)
    up = rng.standard_normal((b, planes, n, n)).astype(np.float32)
    masks = torch.sigmoid(4 * theta)
    m64 = masks.cpu().numpy().astype(np.float64)
    for f0, count in {(0, planes), (planes // 2, planes - planes // 2), (planes - 1, 1)}:
        for given in (up, None):
            dm = litho_lib.litho_intensity_vjp(kern, masks, None if given is None else torch.from_numpy(up).to(cuda),
                                               f_first=f0, f_count=count, precision=precision).cpu().numpy()
            for i in range(b):
                g = [up[i, f] if given is not None else np.ones((n, n)) for f in range(f0, f0 + count)]
                ref = OL.intensity_vjp(m64[i], pairs[f0:f0 + count], g)
                assert np.linalg.norm(dm[i] - ref) <= 1e-4 * np.linalg.norm(ref)


@pytest.mark.parametrize("precision", ["fft32", "fft32/coarse"])
@pytest.mark.parametrize("name", ["through focus", "random", "edge"])
def test_ai_inputs_match_the_given_kernels(litho_lib, cuda, name, precision):
    """Extremes found by the band-row kernel, or (full grid, edge kernels) by a pass over the channel."""
    import torch
    n, b = 128, 5
    lam, phi = _set(name, n)
    kern = litho_lib.litho_upload_kernels(n, PIXEL, lam, phi)
    targets = np.stack([synth.random_rect_mask(n, seed=70 + i, count=15) for i in range(b)]).astype(np.float32)
    x = litho_lib.litho_ai_inputs(kern, torch.from_numpy(targets).to(cuda), focus=0, precision=precision).cpu().numpy()
    ref, _, _ = OA.ai_channels(targets, lam[0], phi[0])
    assert np.array_equal(x[:, 0], targets)
    assert np.abs(x[:, 1] - ref[:, 1]).max() <= 1e-5
    assert np.abs(x[:, 2] - ref[:, 2]).max() <= 1e-4


@pytest.mark.parametrize("n", [128, 256])
@pytest.mark.parametrize("k,rows", [(9, 512), (9, 1024), (8, 2816), (9, 3328), (7, 1024)])
def test_rows_shared_by_warps(litho_lib, cuda, n, k, rows):
    """Short rows: one warp a row, or two that share the kernels (odd and even numbers of them)."""
    import torch
    b = rows // n
    lam, phi = _random_set(n, 32, 1, k, False)
    lam[0, -2:] = lam[0, -3]
    kern = litho_lib.litho_upload_kernels(n, PIXEL, lam, phi)
    masks = np.stack([synth.random_rect_mask(n, seed=90 + i, count=12) for i in range(b)])
    img = litho_lib.litho_aerial(kern, torch.from_numpy(masks).to(cuda), precision="fft32").cpu().numpy()
    for i in (0, b - 1):
        ref = OI.socs_image(masks[i].astype(np.float64), lam[0], phi[0])
        assert np.abs(img[i, 0] - ref).max() <= 1e-5 * max(1.0, ref.max())


# grids whose rows one or two warps take by the number of rows of the launch, and whose row kernels have
# several shapes by the number of planes; 12 and 24 fields of one and three planes
@pytest.mark.parametrize("n,k,focus,counts", [(256, 24, [0.0], (1, 4, 16)), (128, 24, [0.0], (1, 8, 30)),
                                              (512, 16, [-40.0, 0.0, 40.0], (1, 2, 5)),
                                              (1024, 12, [0.0, 30.0], (1, 5))])
@pytest.mark.parametrize("precision", ["fft32", "fft32/coarse"])
def test_images_do_not_depend_on_the_number_of_clips(litho_lib, cuda, n, k, focus, counts, precision):
    import torch
    lam, phi = oracle_kernel_set(DUV_ANNULAR, n, PIXEL, focus, k)
    kern = litho_lib.litho_upload_kernels(n, PIXEL, lam, phi)
    masks = np.stack([synth.random_rect_mask(n, seed=30 + i, count=n // 6) for i in range(max(counts))])
    m = torch.from_numpy(masks).to(cuda)
    alone = [litho_lib.litho_aerial_resist(kern, m[i:i + 1].contiguous(), precision=precision) for i in range(len(m))]
    for b in counts[1:]:
        img, blur, printed = litho_lib.litho_aerial_resist(kern, m[:b].contiguous(), precision=precision)
        for i in range(b):
            assert torch.equal(img[i], alone[i][0][0]), (b, i)
            assert torch.equal(blur[i], alone[i][1][0]) and torch.equal(printed[i], alone[i][2][0]), (b, i)


@pytest.mark.parametrize("n,k,focus,counts", [(512, 16, [-40.0, 0.0, 40.0], (1, 2)), (256, 24, [0.0], (1, 5)),
                                              (128, 16, [-30.0, 0.0, 30.0], (1, 9))])
@pytest.mark.parametrize("precision", ["fft32", "fft32/coarse"])
def test_ilt_does_not_depend_on_the_number_of_clips(litho_lib, cuda, n, k, focus, counts, precision):
    import torch
    lam, phi = oracle_kernel_set(DUV_ANNULAR, n, PIXEL, focus, k)
    kern = litho_lib.litho_upload_kernels(n, PIXEL, lam, phi)
    clips = [synth.ilt_clip(n, PIXEL, seed=60 + i) for i in range(counts[-1])]
    theta = torch.from_numpy(np.stack([c[0] for c in clips])).to(cuda)
    target = torch.from_numpy(np.stack([c[1] for c in clips])).to(cuda)
    grad, loss = litho_lib.litho_ilt_grad(kern, theta, target, precision=precision)
    for i in range(counts[-1]):
        g, lo = litho_lib.litho_ilt_grad(kern, theta[i:i + 1].contiguous(), target[i:i + 1].contiguous(),
                                         precision=precision)
        assert torch.equal(grad[i], g[0]) and loss[i] == lo[0], i


@pytest.mark.parametrize("name,fields", [("nominal", 4), ("one kernel", 1), ("through focus", 8 + 4),
                                         ("reordered", 5 + 5 + 3), ("repeated", 6 + 3), ("dark plane", 5),
                                         ("random", 4 + 2), ("edge", 1)])
def test_planes_reduce_and_share(litho_lib, cuda, name, fields):
    """In focus K kernels of one phase are K real fields, ceil(K/2) complex ones; +z and -z share a set."""
    lam, phi = _set(name, 256)
    assert litho_lib.litho_upload_kernels(256, PIXEL, lam, phi).fields() == fields


def test_planes_of_a_large_crop_share(litho_lib, cuda):
    opt = litho_lib.make_optics(kind="quadrupole", src_grid=41, pole_sigma=0.8, pole_radius=0.1)
    assert litho_lib.litho_make_kernels(opt, 2048, PIXEL, [-50.0, 0.0, 50.0], 24).fields() == 24 + 12


@pytest.mark.parametrize("precision", ["fft32", "fft32/coarse"])
@pytest.mark.parametrize("lams", [[[1.0, 1e-13]], [[1.0, 0.0], [1.0, 1e-9]], [[1.0, 1e-9], [1.0, 0.0]],
                                  [[1.0, 1e-9], [1.0, 1.001e-9]]])
def test_a_weak_kernel_that_images_alone(litho_lib, cuda, lams, precision):
    """A clear mask passes the weak kernel (zero frequency) alone: each plane's image is that kernel's lambda,
    exactly but for the rounding of a few products (1e-6), however little it adds to the plane's Gram matrix."""
    import torch
    n, c = 64, 32
    lam = np.array(lams)
    rng = np.random.default_rng(1)
    phi = np.zeros(lam.shape + (c, c), dtype=np.complex128)
    strong = rng.standard_normal((c, c)) + 1j * rng.standard_normal((c, c))
    strong[0, :] = strong[:, 0] = strong[c // 2, c // 2] = 0.0
    phi[:, 0] = strong / np.linalg.norm(strong)
    phi[:, 1, c // 2, c // 2] = 1.0
    kern = litho_lib.litho_upload_kernels(n, PIXEL, lam, phi)
    img = litho_lib.litho_aerial(kern, torch.ones(1, n, n, device=cuda), precision=precision)[0].cpu().numpy()
    for f in range(len(lam)):
        assert np.abs(img[f] - lam[f, 1]).max() <= 1e-6 * lam[f, 1]


def test_adjoint_of_thousands_of_clips(litho_lib, cuda):
    """4500 clips of 16 fields in one group: 72000 runs of fields in the adjoint's columns."""
    import torch
    n, b = 32, 4500
    lam, phi = _random_set(n, 32, 1, 16, False)
    lam[0, -2:] = lam[0, -3]
    kern = litho_lib.litho_upload_kernels(n, PIXEL, lam, phi)
    gen = torch.Generator(device=cuda).manual_seed(4)
    theta = torch.rand((b, n, n), device=cuda, generator=gen) - 0.5
    target = (torch.rand((b, n, n), device=cuda, generator=gen) > 0.5).float()
    grad, loss = litho_lib.litho_ilt_grad(kern, theta, target, sigma_nm=6.0)
    up = torch.rand((b, 1, n, n), device=cuda, generator=gen)
    dm = litho_lib.litho_intensity_vjp(kern, target, up)
    for i in (0, 4095, b - 1):
        g, lo = litho_lib.litho_ilt_grad(kern, theta[i:i + 1].contiguous(), target[i:i + 1].contiguous(), sigma_nm=6.0)
        assert torch.equal(grad[i], g[0]) and loss[i] == lo[0]
        d = litho_lib.litho_intensity_vjp(kern, target[i:i + 1].contiguous(), up[i:i + 1].contiguous())
        assert torch.equal(dm[i], d[0])


def test_upload_beside_a_nearly_full_device(litho_lib, cuda):
    """Room for the set (134 MB of FP32 kernels) but not for its FP64 kernels (268 MB) beside it: uploaded as given."""
    import torch
    n, c, k, room = 1024, 512, 64, 240 << 20
    rng = np.random.default_rng(3)
    phi = (rng.standard_normal((1, k, c, c)) + 1j * rng.standard_normal((1, k, c, c))) / c
    phi[..., 0, :] = phi[..., :, 0] = 0.0
    lam = np.full((1, k), 1.0 / k)
    mask = torch.from_numpy(synth.random_rect_mask(n, seed=2, count=200)[None]).to(cuda)
    want = litho_lib.litho_aerial(litho_lib.litho_upload_kernels(n, PIXEL, lam, phi), mask)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    full = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device=cuda)
    assert (150 << 20) < torch.cuda.mem_get_info()[0] < (260 << 20)
    try:
        kern = litho_lib.litho_upload_kernels(n, PIXEL, lam, phi)
    finally:
        del full
        torch.cuda.empty_cache()
    assert kern.fields() == k
    assert torch.equal(litho_lib.litho_aerial(kern, mask), want)


def test_upload_does_not_wait_for_running_work(litho_lib, cuda):
    """A set of two planes, one reduced, is built while another stream is busy for a second or so."""
    import torch
    lam, phi = oracle_kernel_set(DUV_ANNULAR, 256, PIXEL, [0.0, 30.0, -30.0], 12)
    keep = [litho_lib.litho_upload_kernels(256, PIXEL, lam, phi)]  # its kernels are loaded
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(2_000_000_000)
        done = torch.cuda.Event()
        done.record()
    keep.append(litho_lib.litho_upload_kernels(256, PIXEL, lam, phi))
    assert not done.query()
    side.synchronize()
    assert keep[1].fields() == 6 + 12
