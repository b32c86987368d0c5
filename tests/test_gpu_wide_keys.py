"""Buckets of the hinted sort whose keys leave no room for the ids in one word
(a batch's graph ids and Morton bits): equal keys must still come out by id.
The order is NumPy's lexsort on (key, id), bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import gpu_pipeline as G  # noqa: E402

B = G.B


@pytest.mark.parametrize("K", [3, 900, 1025, 2048, 70_000])
@pytest.mark.parametrize("bits", [40, 46, 51, 53, 60])
@pytest.mark.parametrize("kind", ["distinct", "repeated", "crowded"])
def test_equal_keys_by_id(K, bits, kind):
    rng = np.random.default_rng(K + bits)
    keys = rng.integers(0, 1 << bits, K, dtype=np.uint64)
    if kind == "repeated":  # runs of a few equal keys, none longer than a bin holds
        keys = keys[rng.integers(0, max(1, K // 3), K)]
    if kind == "crowded":  # most keys in one bin of their bucket
        keys[: K - K // 8] &= np.uint64(63)
    ids = np.arange(K, dtype=np.uint32)
    order = np.lexsort((ids, keys))
    for hint in (ids, order.astype(np.uint32)):
        ok, oi = G.empty(K, np.uint64), G.empty(K, np.uint32)
        ws = B.alloc_ws(B.bgv_sort_hinted_ws_size(K))
        B.bgv_sort_hinted(G.dev(keys), G.dev(hint), K, ok, oi, ws)
        assert np.array_equal(G.host(oi, np.uint32, K), ids[order])
        assert np.array_equal(G.host(ok, np.uint64, K), keys[order])
