"""Sorts between sampled splitters in few buckets: with an odd number of them (3 to
15) some of the blocks that rank the samples have none.  Every call finds its
workspace past the header full of other words, so splitters that were not written
show as another order."""
import numpy as np
import pytest

from oracle import FA2Params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import gpu_pipeline as G  # noqa: E402

B = G.B


def _stale(ws, seed):
    """Falling 64-bit words after the header: no order of splitters that any sort leaves."""
    body = ws[256:256 + (ws.numel() - 256) // 8 * 8].view(torch.int64)
    g = torch.Generator(device="cuda").manual_seed(seed)
    words = torch.randint(0, 1 << 62, body.shape, generator=g, device="cuda", dtype=torch.int64)
    body.copy_(torch.sort(words, descending=True).values)


# odd counts of the 512-body buckets of a first step, 3 to 15
@pytest.mark.parametrize("K", [1025, 2300, 3300, 4500, 5500, 6500, 7500])
def test_first_steps(K):
    rng = np.random.default_rng(K)
    pos = (rng.random((K, 2)) * 1000).astype(np.float32)
    mass = rng.integers(1, 9, K).astype(np.uint32)

    def first(order, seed):
        prev = B.bgv_set_fa2_order(order)
        try:
            dv = G.Fa2Device(pos, mass, np.zeros(K + 1, np.int32), np.zeros(0, np.int32), np.zeros(0, np.uint32),
                             FA2Params())
            _stale(dv.ws, seed)
            B.bgv_fa2_run_timed(K, 0, dv.off, dv.adj, dv.w, dv.mass, dv.params, 1, dv.pos, dv.F, dv.Fprev, dv.speed,
                                dv.ws)
            return dv.state(), dv.stats()
        finally:
            B.bgv_set_fa2_order(prev)

    want, ws = first(0, 0)
    for seed in range(1, 6):
        got, st = first(1, seed)
        assert st.status == 0 and (st.interactions, st.tree_nodes) == (ws.interactions, ws.tree_nodes)
        for x, y in zip(got, want):
            assert np.array_equal(x, y)


# odd counts of the 1,024-key buckets, 3 to 15
@pytest.mark.parametrize("K", [2500, 4500, 6500, 8600, 10_700, 12_700, 14_800])
def test_hinted_sorts(K):
    rng = np.random.default_rng(K)
    keys = rng.integers(0, 1 << 48, K, dtype=np.uint64)
    order = np.lexsort((np.arange(K), keys)).astype(np.uint32)
    ok, oi, ws = G.empty(K, np.uint64), G.empty(K, np.uint32), B.alloc_ws(B.bgv_sort_hinted_ws_size(K))
    dk, dh = G.dev(keys), G.dev(rng.permutation(K).astype(np.uint32))
    for seed in range(5):
        _stale(ws, seed)
        B.bgv_sort_hinted(dk, dh, K, ok, oi, ws)
        assert np.array_equal(G.host(oi, np.uint32, K), order)
        assert np.array_equal(G.host(ok, np.uint64, K), keys[order])
