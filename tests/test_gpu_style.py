"""Colour groups and drawing at the sizes where their kernels change shape."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import gpu_pipeline as G  # noqa: E402

B = G.B


# around a tile of 4,096 sorted sizes; the half inside the first, a middle or the last tile; every size 0
@pytest.mark.parametrize("K,kind", [(4095, "flat"), (4096, "hub"), (4097, "skew"), (12_289, "flat"), (70_001, "hub"),
                                    (70_001, "skew"), (5000, "zero")])
@pytest.mark.parametrize("shift", [0, 1])
def test_colour_groups_around_the_tiles(K, kind, shift):
    rng = np.random.default_rng(K)
    sizes = {"flat": np.full(K, 3), "hub": np.ones(K), "skew": rng.lognormal(2, 2, K) + 1, "zero": np.zeros(K)}[kind]
    sizes = sizes.astype(np.uint32)
    if kind == "hub":
        sizes[K // 2] = 4_000_000_000
    n = 2 * K + 3
    node_map = rng.integers(-1, K + 1, n + shift).astype(np.int32)  # ids outside [0, K) are drawn as group 0
    nm = G.dev(node_map)[shift:]  # shift 1: not on a 16-byte boundary
    group = torch.zeros(K, dtype=torch.uint8, device="cuda")
    colour = torch.zeros(n + shift, dtype=torch.uint8, device="cuda")[shift:]
    B.bgv_colour_groups(K, G.dev(sizes), group, B.alloc_ws(B.bgv_colour_groups_ws_size(K)), n=n, node_map=nm,
                        node_colour=colour)
    ref = oracle.colour_groups(sizes)
    assert np.array_equal(group.cpu().numpy(), ref)
    k = node_map[shift:]
    assert np.array_equal(colour.cpu().numpy(), np.where((k >= 0) & (k < K), ref[np.clip(k, 0, K - 1)], 0))


# one disc per warp, a few, and 32, each with discs of a pixel and discs across the image
@pytest.mark.parametrize("K", [9_001, 30_011, 700_001])
def test_render_discs_per_warp(K):
    rng = np.random.default_rng(K)
    xy = (rng.normal(size=(K, 2)) * 100).astype(np.float32)
    radius = np.sqrt(rng.integers(1, 60, K)).astype(np.float32) * np.float32(0.02)
    radius[:: K // 40] *= 200
    group = rng.integers(0, 11, K).astype(np.uint8)
    W, H = 211, 150
    img = torch.zeros((H, W, 4), dtype=torch.uint8, device="cuda")
    B.bgv_render(K, G.dev(xy), G.dev(radius), torch.from_numpy(group).cuda(), W, H, img,
                 B.alloc_ws(B.bgv_render_ws_size(W, H)))
    assert np.array_equal(img.cpu().numpy(), oracle.render(xy, radius, group, W, H))
