"""Colour groups and image frames of few communities, which one block makes (up to
8,192): around the threads' shares and the line, with sizes of 0, all equal, and one that
outweighs the rest, against NumPy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import gpu_pipeline as G  # noqa: E402

B = G.B


def _groups(size):
    K = size.shape[0]
    order = np.lexsort((np.arange(K), size))
    cum = np.cumsum(size[order].astype(np.uint64))
    half = int((2 * cum <= cum[-1]).sum())
    g = np.zeros(K, np.uint8)
    rest = np.arange(K - half)
    g[order[half:]] = 1 + (10 * rest) // max(1, K - half)
    return g


@pytest.mark.parametrize("K", [1, 2, 31, 1023, 1024, 1025, 2049, 4096, 4097, 8191, 8192, 8193])
@pytest.mark.parametrize("kind", ["spread", "equal", "zero", "one"])
def test_groups(K, kind):
    rng = np.random.default_rng(K)
    size = {"spread": np.exp(rng.normal(size=K) * 2).astype(np.uint32), "equal": np.full(K, 7, np.uint32),
            "zero": np.zeros(K, np.uint32), "one": np.ones(K, np.uint32)}[kind]
    if kind == "one":
        size[K // 2] = 4_000_000_000
    grp = torch.full((K,), 77, dtype=torch.uint8, device="cuda")
    ws = B.alloc_ws(B.bgv_colour_groups_ws_size(K))
    B.bgv_colour_groups(K, G.dev(size), grp, ws)
    assert B.bgv_status(ws) == 0 and np.array_equal(grp.cpu().numpy(), _groups(size))


@pytest.mark.parametrize("K", [1, 33, 1024, 1025, 8192, 8193])
def test_frames(K):
    # the far corners' discs are drawn where one block or many find the frame
    rng = np.random.default_rng(K)
    xy = (rng.random((K, 2)) * 100).astype(np.float32)
    rad = np.full(K, 0.5, np.float32)
    W = H = 500
    rgba = torch.zeros((H, W, 4), dtype=torch.uint8, device="cuda")
    ws = B.alloc_ws(B.bgv_render_ws_size(W, H))
    grp = torch.zeros(K, dtype=torch.uint8, device="cuda")
    B.bgv_render(K, G.dev(xy), G.dev(rad), grp, W, H, rgba, ws)
    img = rgba.cpu().numpy()
    lo, hi = (xy - rad[:, None]).min(0), (xy + rad[:, None]).max(0)
    s = np.float32(W) / max(hi - lo)
    c = ((xy - lo) * s).astype(int)
    inside = (c >= 0).all(1) & (c < W).all(1)
    assert inside.all() and (img[c[:, 1], c[:, 0], :3] == (177, 89, 40)).all()
