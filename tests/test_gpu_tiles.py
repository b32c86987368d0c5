"""The quadtree from tiles of 1,024 sorted bodies against the oracle's: equal
interaction counts and forces within the tolerance, at sizes around the tiles,
on layouts whose cells end inside a tile, at its edge, and many tiles later."""
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


def _positions(kind, K, rng):
    if kind == "uniform":
        return rng.random((K, 2)) * 200 - 100
    if kind == "line":  # deep chains: every level splits off one side
        t = 2.0 ** -rng.uniform(0, 22, K)
        return np.stack([t, t * 0.5], 1) * 100
    if kind == "clumps":  # clusters of hundreds to thousands of bodies, far apart, at several scales
        c = rng.integers(0, 7, K)
        return np.stack([c * 37.0, (c % 3) * 53.0], 1) + rng.normal(size=(K, 2)) * (10.0 ** -(c % 4))[:, None]
    p = rng.random((max(1, K // 40), 2)) * 100  # "coincident": runs of equal positions, some across a tile's edge
    return p[np.sort(rng.integers(0, p.shape[0], K))]


@pytest.mark.parametrize("K", [2, 3, 1023, 1024, 1025, 2047, 2048, 2049, 5000, 66_561, 140_000])
@pytest.mark.parametrize("kind", ["uniform", "line", "clumps", "coincident"])
@pytest.mark.parametrize("leaf_cap,L", [(1, 24), (5, 24), (1, 6)])
def test_tree_matches_oracle(K, kind, leaf_cap, L):
    rng = np.random.default_rng(K + L)
    pos = _positions(kind, K, rng)[rng.permutation(K)].astype(np.float32)
    mass = rng.integers(1, 1000, K).astype(np.uint32)
    p = FA2Params(theta=1.2, leaf_cap=leaf_cap, max_depth=L)
    if K > 6000 and (leaf_cap > 1 or L < 24 or kind == "coincident"):
        pytest.skip("the oracle takes long here")
    off = np.zeros(K + 1, np.int32)
    r = G.fa2_forces(pos, mass, off, np.zeros(0, np.int32), np.zeros(0, np.uint32), p)
    Fr0, inter0 = oracle.bh_repulsion(pos, mass, p)
    assert r["status"] == 0
    assert r["interactions"] == inter0
    if kind == "uniform":
        assert G.rel_err(r["Fr"], Fr0) <= 1e-3
