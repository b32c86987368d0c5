"""Cell moments at the edges of their widths: tiles of bodies below 2^21 take 32
and 64-bit sums and a division by an estimate, a heavier body anywhere in the
tile the full width; both against the oracle's exact quadtree."""
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
LIGHT = (1 << 21) - 1  # the heaviest body of a light tile


@pytest.mark.parametrize("K", [2, 700, 2048, 3000])
@pytest.mark.parametrize("kind", ["ones", "light", "mixed", "one-heavy", "heaviest"])
def test_moments_match_oracle(K, kind):
    rng = np.random.default_rng(K)
    mass = {"ones": np.ones(K), "light": np.full(K, LIGHT), "mixed": rng.integers(1, LIGHT + 1, K),
            "one-heavy": np.where(np.arange(K) == K // 2, LIGHT + 1, 3), "heaviest": np.full(K, 2**32 - 1)}[kind]
    mass = mass.astype(np.uint32)
    pos = (rng.random((K, 2)) * 200 - 100).astype(np.float32)
    p = FA2Params(theta=1.2)
    args = (mass, np.zeros(K + 1, np.int32), np.zeros(0, np.int32), np.zeros(0, np.uint32))
    r = G.fa2_forces(pos, *args, p)
    Fr0, inter0 = oracle.bh_repulsion(pos, mass, p)
    assert r["status"] == 0 and r["interactions"] == inter0
    assert G.rel_err(r["Fr"], Fr0) <= 1e-3
    # the run in one cluster (K <= 2,048) or launch by launch: the same bits
    a, b = G.Fa2Device(pos, *args, p), G.Fa2Device(pos, *args, p)
    a.run(3, True)
    B.bgv_fa2_run_timed(b.K, b.nnz, b.off, b.adj, b.w, b.mass, b.params, 3, b.pos, b.F, b.Fprev, b.speed, b.ws)
    for x, y in zip(a.state(), b.state()):
        assert np.array_equal(x, y, equal_nan=True)
