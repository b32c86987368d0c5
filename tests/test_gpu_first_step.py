"""The Morton order of a first or single step: from id order with sampled
splitters up to 262,144 bodies, by the radix sort above.  Both orders are (key,
id), so steps with either sort are equal bit for bit."""
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


def _step(pos, mass, order):
    K = pos.shape[0]
    prev = B.bgv_set_fa2_order(order)
    try:
        dv = G.Fa2Device(pos, mass, np.zeros(K + 1, np.int32), np.zeros(0, np.int32), np.zeros(0, np.uint32),
                         FA2Params())
        # launched one by one: the general path at every size, its first step from no order and its second from the first's
        B.bgv_fa2_run_timed(K, 0, dv.off, dv.adj, dv.w, dv.mass, dv.params, 2, dv.pos, dv.F, dv.Fprev, dv.speed, dv.ws)
        return dv.state(), dv.stats()
    finally:
        B.bgv_set_fa2_order(prev)


@pytest.mark.parametrize("K", [1, 2, 511, 512, 513, 1024, 1025, 5000, 60_013, 262_144, 262_145])
@pytest.mark.parametrize("kind", ["uniform", "clump", "equal"])
def test_first_step_sorts_agree(K, kind):
    rng = np.random.default_rng(K)
    pos = rng.random((K, 2)) * 1000
    if kind == "clump":  # nine in ten in a corner: full buckets, crowded bins
        pos[: K * 9 // 10] *= 1e-4
    elif kind == "equal":  # coincident bodies, in order by id
        pos[:] = pos[rng.integers(0, max(1, K // 300), K)]
    pos = pos.astype(np.float32)
    if kind == "equal" and K > 60_013:
        pytest.skip("hundreds of coincident bodies per leaf: slow")
    mass = rng.integers(1, 9, K).astype(np.uint32)
    (a, sa), (b, sb) = _step(pos, mass, 1), _step(pos, mass, 0)
    assert sa.status == 0 and sb.status == 0 and sa.interactions == sb.interactions
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
