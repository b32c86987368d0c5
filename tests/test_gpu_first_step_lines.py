"""Around the sizes where a step changes its sort (65,536 bodies in a first step) and
its launches (131,072 in later steps, 262,144 in a first one): equal to steps with the
radix sort bit for bit, launched one by one, from a run, and replayed."""
import numpy as np
import pytest

import graphgen
from oracle import FA2Params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import gpu_pipeline as G  # noqa: E402

B = G.B


def _run(args, order, replay):
    prev = B.bgv_set_fa2_order(order)
    try:
        dv, st = G.Fa2Device(*args), torch.cuda.Stream()
        dv.run(4, replay, stream=st)
        torch.cuda.synchronize()
        dv.step()
        return dv.state(), dv.stats()
    finally:
        B.bgv_set_fa2_order(prev)


@pytest.mark.parametrize("K", [65_536, 65_537, 131_072, 131_073, 262_144, 262_145])
@pytest.mark.parametrize("kind", ["uniform", "clusters"])
def test_steps_agree(K, kind):
    rng = np.random.default_rng(K)
    pos = rng.random((K, 2)) * 1000
    if kind == "clusters":  # buckets that span far-apart clusters
        pos = rng.random((97, 2))[rng.integers(0, 97, K)] * 1e5 + rng.normal(size=(K, 2))
    off, adj, w = G.csr_from_edges(graphgen.random_graph(K, 2 * K, seed=3), K)
    args = (pos.astype(np.float32), rng.integers(1, 9, K).astype(np.uint32), off, adj, w, FA2Params())
    want, sw = _run(args, 0, False)
    for replay in (False, True):
        got, sg = _run(args, 1, replay)
        assert sg.status == 0 and (sg.interactions, sg.tree_nodes) == (sw.interactions, sw.tree_nodes)
        for x, y in zip(got, want):
            assert np.array_equal(x, y)
