"""Every call that takes a stream can be captured into a CUDA graph: its launches, the programmatic ones among
them, replay to the bits of the call itself, also for new inputs in the captured buffers."""
import numpy as np
import pytest

import synth
from tests.gpu_util import DUV_ANNULAR, oracle_kernel_set

pytestmark = pytest.mark.gpu

N, B, PIXEL = 256, 3, 8.0

CALLS = {
    "aerial": lambda L, k, d: L.litho_aerial(k, d["mask"], precision="fft32"),
    "aerial coarse": lambda L, k, d: L.litho_aerial(k, d["mask"], precision="fft32/coarse"),
    "aerial tensor": lambda L, k, d: L.litho_aerial(k, d["mask"], precision="fp16x3"),
    "aerial noalloc": lambda L, k, d: L.litho_aerial_noalloc(k, d["mask"], d["out"]),
    "resist": lambda L, k, d: L.litho_aerial_resist(k, d["mask"], precision="fft32/coarse")[1],
    "ilt": lambda L, k, d: L.litho_ilt_grad(k, d["theta"], d["target"], want_loss=False)[0],
    "ilt coarse": lambda L, k, d: L.litho_ilt_grad(k, d["theta"], d["target"], precision="fft32/coarse",
                                                   want_loss=False)[0],
    "vjp": lambda L, k, d: L.litho_intensity_vjp(k, d["mask"], d["up"], precision="fft32/coarse"),
    "vjp of ones": lambda L, k, d: L.litho_intensity_vjp(k, d["mask"]),
    "ai inputs": lambda L, k, d: L.litho_ai_inputs(k, d["target"]),
    "print images": lambda L, k, d: L.litho_print_images(d["target"], d["mask"], PIXEL, 20.0, 0.5, 0.3)[2],
}


@pytest.mark.parametrize("name", sorted(CALLS))
def test_calls_replay_from_a_graph(litho_lib, cuda, name):
    import torch
    lam, phi = oracle_kernel_set(DUV_ANNULAR, N, PIXEL, [-40.0, 0.0, 40.0], 8)
    kern = litho_lib.litho_upload_kernels(N, PIXEL, lam, phi)
    clips = [synth.ilt_clip(N, PIXEL, seed=40 + i) for i in range(B)]
    data = {"mask": np.stack([synth.random_rect_mask(N, seed=i) for i in range(B)]),
            "theta": np.stack([c[0] for c in clips]), "target": np.stack([c[1] for c in clips]),
            "up": np.random.default_rng(2).random((B, 3, N, N))}
    d = {key: torch.from_numpy(np.ascontiguousarray(v, dtype=np.float32)).to(cuda) for key, v in data.items()}
    d["out"] = torch.empty((B, 3, N, N), device=cuda)
    call = CALLS[name]
    want = call(litho_lib, kern, d).clone()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = call(litho_lib, kern, d)
    for _ in range(2):
        out.fill_(-1 if out.dtype.is_floating_point else 7)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
        for key in ("mask", "theta", "target", "up"):  # the clips in another order, in the same buffers
            d[key].copy_(d[key].roll(1, 0))
        got = out.clone()
        want = call(litho_lib, kern, d).clone()
        torch.cuda.synchronize()
        assert not torch.equal(got, want)
