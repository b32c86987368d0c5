"""The degree sketch around the sizes where endpoints are sorted out by node range: as
many edges as nodes, and half as many again from 8,388,609 nodes on.  Sketches add up, so
the whole list's is compared with its halves', which lie below the lines.  The workspace
query goes by the call's rule: the queried size serves, a smaller one is refused."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import gpu_pipeline as G  # noqa: E402

B = G.B
HALF, MOST, WIDTH = 1 << 23, 1 << 24, 1 << 20


def _sketch(e, n):
    m = e.shape[0]
    S, d = (torch.zeros(k, dtype=torch.int32, device="cuda") for k in (WIDTH, n))
    need = B.bgv_sketch_degrees_ws_size(m, n, 1, WIDTH)
    ws = B.alloc_ws(need)
    B.bgv_sketch_degrees(e, m, n, 1, WIDTH, 1, S, d, ws)
    assert B.bgv_status(ws) == 0
    with pytest.raises(B.BgvError):
        B.bgv_sketch_degrees(e, m, n, 1, WIDTH, 1, S, d, B.alloc_ws(need - 256))
    return S.long(), d.long()


@pytest.mark.parametrize("n,m", [(5_000_000, 4_999_998), (5_000_000, 5_000_000), (HALF, HALF), (HALF + 1, HALF + 2),
                                 (HALF + 1, HALF * 3 // 2), (HALF + 1, HALF * 3 // 2 + 2), (MOST, 2 * MOST - 4),
                                 (MOST + 1, 2 * MOST)])
def test_degrees_around_the_lines(n, m):
    g = torch.Generator(device="cuda").manual_seed(n + m)
    e = torch.randint(n, (m, 2), generator=g, device="cuda", dtype=torch.int32)
    S, d = _sketch(e, n)
    S1, _ = _sketch(e[:m // 2], n)
    S2, _ = _sketch(e[m // 2:].clone(), n)
    assert torch.equal(S, S1 + S2) and int(S.sum()) == 2 * m
    assert bool((d >= torch.bincount(e.view(-1), minlength=n)).all())
