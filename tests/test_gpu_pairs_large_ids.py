"""26-bit ids: a hub's piece that both splits leave too long spans more key values
than are counted out, so a split sets the guard beside the sorting of the other
buckets, and the LSD sort gives the keys."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import gpu_pipeline as G  # noqa: E402


def test_guard_set_by_a_split():
    n = (1 << 25) + 5
    rng = np.random.default_rng(3)
    hubs = [np.stack([np.full(40_000, h), h + 1 + rng.permutation(1 << 21)[:40_000]], 1) for h in (3, 9_000_000, 31_000_000)]
    e = np.concatenate(hubs + [rng.integers(0, n, ((1 << 20) + 3, 2))])
    e = np.ascontiguousarray(np.minimum(e[rng.permutation(e.shape[0])], n - 1), np.int32)
    lab, dh = np.arange(n, dtype=np.int32), np.ones(n, np.uint32)
    sg, sg0 = (f(e, n, lab, dh, 1, 64, 5) for f in (G.supergraph, oracle.supergraph))
    assert sg["status"] == 0 and sg["K"] == sg0["K"] and sg["Es"] == sg0["Es"]
    for k in ("src", "dst", "w", "csr_off", "csr_adj", "csr_w"):
        assert np.array_equal(np.asarray(sg[k]).astype(np.int64), np.asarray(sg0[k]).astype(np.int64)), k
