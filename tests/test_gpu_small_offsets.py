"""CSR offsets that fall somewhere, so that rows lie outside the range that a block's
first and last offsets span: a graph of up to 2,048 bodies takes them as the general
path does (each row is its own [off[r], off[r + 1]), empty when that falls)."""
import numpy as np
import pytest

import oracle
from oracle import FA2Params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import gpu_pipeline as G  # noqa: E402

B = G.B


@pytest.mark.parametrize("K,nnz", [(100, 700), (300, 2000), (1500, 9000), (2048, 60_000)])
@pytest.mark.parametrize("kind", ["one", "many", "reversed"])
def test_rows_outside_the_span(K, nnz, kind):
    rng = np.random.default_rng(K)
    off = np.sort(rng.integers(0, nnz + 1, K + 1))
    if kind == "one":
        off[K // 3] = nnz
    elif kind == "many":
        off[rng.permutation(K - 1)[: K // 10] + 1] = rng.integers(0, nnz + 1, K // 10)
    else:
        off = off[::-1].copy()
    if kind == "many":  # no row longer than a few hundred entries
        far = np.nonzero(np.diff(off) > 300)[0]
        off[far + 1] = off[far] + 300
        off = np.minimum(off, nnz)
    off[-1] = nnz if kind != "reversed" else off[-1]
    adj = rng.integers(0, K, nnz).astype(np.int32)
    w = rng.integers(1, 5, nnz).astype(np.uint32)
    args = (oracle.fa2_init(K, 2), rng.integers(1, 9, K).astype(np.uint32), off.astype(np.int32), adj, w, FA2Params())
    small, general = G.Fa2Device(*args), G.Fa2Device(*args)
    small.nnz = general.nnz = nnz
    for dv in (small, general):
        dv.ws = B.alloc_ws(B.bgv_fa2_ws_size(K, nnz))
    small.run(3, False)
    B.bgv_fa2_run_timed(K, nnz, general.off, general.adj, general.w, general.mass, general.params, 3, general.pos,
                        general.F, general.Fprev, general.speed, general.ws)
    assert small.stats().status == 0 and general.stats().status == 0
    for x, y in zip(small.state(), general.state()):
        assert np.array_equal(x, y)
